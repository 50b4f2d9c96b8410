// noalloc.cu -- tube counts for caller-chosen grain pairs of one small view,
// with every intermediate buffer in one fixed, file-scope device array.
//
// Who needs this: callers that cannot call cudaMalloc.  Examples are a
// scanning microscope's acquisition loop that may not block (cudaMalloc can
// synchronise the whole device), code running inside a host function enqueued
// on a stream (CUDA API calls are not allowed there), and applications whose
// framework has reserved the free device memory for its own pool.  They pass
// device pointers to their grains, their pairs and an output array, and this
// entry point uses only the scratch array below.
//
// The scratch array lives on every GPU that loads the library until the
// process exits.  In host code its name is only a stand-in: the device
// address is obtained once per device with cudaGetSymbolAddress (on the first
// call on that device, which should therefore happen before any stream
// capture) and passed to the kernels.  The address is cached together with
// the device's current CUDA context; after a device reset the context
// differs, and the next call looks the address up again.  Every call shares
// the array and leaves its contents behind; calls whose work overlaps on the
// GPU race with each other, so callers must order them (one stream, or
// events).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>

#include "runtime.h"
#include "walk.cuh"

namespace et {

namespace {

constexpr long long NA_MAX_GRAINS = ET_NOALLOC_MAX_GRAINS;
constexpr long long NA_MAX_CELLS = ET_NOALLOC_MAX_CELLS;

// Two cell lists (rows along x and along y, as the regular path's) of at most
// half the cells each.
constexpr long long NA_LIST_CELLS = NA_MAX_CELLS / 2;

// Layout of the scratch array (byte offsets, 256-aligned).
constexpr size_t NA_ALIGN = 256;
constexpr size_t na_up(size_t v) { return (v + NA_ALIGN - 1) / NA_ALIGN * NA_ALIGN; }
constexpr size_t NA_OFF_GRAINS = 0;                                                       // u64[2 MAX_GRAINS]
constexpr size_t NA_OFF_START = NA_OFF_GRAINS + sizeof(u64) * 2 * NA_MAX_GRAINS;          // u32[2 LIST_CELLS + 1]
constexpr size_t NA_OFF_CURSOR = NA_OFF_START + na_up(sizeof(u32) * (2 * NA_LIST_CELLS + 1));   // u32[2][LIST_CELLS]
constexpr size_t NA_OFF_CTL = NA_OFF_CURSOR + sizeof(u32) * NA_MAX_CELLS;                 // NaCtl
constexpr size_t NA_BYTES = NA_OFF_CTL + NA_ALIGN;

static __device__ __align__(256) unsigned char g_noalloc_scratch[NA_BYTES];

struct NaCtl {
    u64 ticket;   // pairs taken by the counting warps
    u32 bad;      // a coordinate lies outside the extent
};

struct NaScratch {
    u64 *grains;               // packed, x-row list then (at N) y-row list
    u32 *start[2], *cursor[2];
    NaCtl *ctl;
};

// n0: cells of the first list (the second list's starts follow them)
NaScratch carve(unsigned char *base, long long n0) {
    NaScratch s;
    s.grains = (u64 *)(base + NA_OFF_GRAINS);
    for (int l = 0; l < 2; ++l) {
        s.cursor[l] = (u32 *)(base + NA_OFF_CURSOR) + l * NA_LIST_CELLS;
    }
    s.start[0] = (u32 *)(base + NA_OFF_START);
    s.start[1] = s.start[0] + n0;
    s.ctl = (NaCtl *)(base + NA_OFF_CTL);
    return s;
}

__global__ void k_na_clear(NaScratch s, int n0, int n1) {
    griddep_launch();
    griddep_wait();
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < max(n0, n1); c += gridDim.x * blockDim.x) {
        if (c < n0) s.cursor[0][c] = 0;
        if (c < n1) s.cursor[1][c] = 0;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        s.ctl->ticket = 0;
        s.ctl->bad = 0;
    }
}

__device__ __forceinline__ bool na_inside(const Batch &b, int x, int y, int z) {
    return x >= 0 && x < b.ext[0] && y >= 0 && y < b.ext[1] && z >= 0 && z < b.ext[2];
}
__device__ __forceinline__ int na_cell_x(const Batch &b, int x, int y, int z) {
    return x / b.cs[0] + b.nc[0] * (y / b.cs[1] + b.nc[1] * (z / b.cs[2]));
}
__device__ __forceinline__ int na_cell_y(const Batch &b, int x, int y, int z) {
    return y / b.csy[1] + b.ncy[1] * (x / b.csy[0] + b.ncy[0] * (z / b.csy[2]));
}

__global__ void k_na_count(Batch b, const int *xyz, NaScratch s) {
    griddep_launch();
    griddep_wait();
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < b.N; i += gridDim.x * blockDim.x) {
        const int x = xyz[3 * i], y = xyz[3 * i + 1], z = xyz[3 * i + 2];
        if (!na_inside(b, x, y, z)) {
            atomicOr(&s.ctl->bad, 1u);
            continue;
        }
        atomicAdd(&s.cursor[0][na_cell_x(b, x, y, z)], 1u);
        atomicAdd(&s.cursor[1][na_cell_y(b, x, y, z)], 1u);
    }
}

// Block l scans the cell counts of list l into cell starts, which also become
// the fill cursors: tiles of NA_SC x 1024 cells, the next tile's counts loaded
// before the current one is scanned.  2 x 34k cells (29k grains) take 39 us, the
// larger part of what a call needs before it counts.
constexpr int NA_SC = 8;

__global__ void __launch_bounds__(1024) k_na_scan(NaScratch s, int n0, int n1, u32 N) {
    griddep_launch();
    griddep_wait();
    __shared__ u32 part[32];
    const int list = blockIdx.x, n = list ? n1 : n0, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    u32 *cur = s.cursor[list], *start = s.start[list];
    u32 carry = list ? N : 0u, v[NA_SC], next[NA_SC];   // the second list lies behind N
    auto load = [&](int base, u32 (&d)[NA_SC]) {
        const int c = base + (int)threadIdx.x * NA_SC;
#pragma unroll
        for (int k = 0; k < NA_SC; ++k) d[k] = c + k < n ? cur[c + k] : 0u;
    };
    load(0, next);
    for (int base = 0; base < n; base += 1024 * NA_SC) {
        u32 sum = 0;
#pragma unroll
        for (int k = 0; k < NA_SC; ++k) {
            v[k] = next[k];
            sum += v[k];
        }
        load(base + 1024 * NA_SC, next);
        u32 inc = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const u32 t = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += t;
        }
        if (lane == 31) part[w] = inc;
        __syncthreads();
        u32 ps = part[lane];   // every warp scans the warp sums itself
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const u32 t = __shfl_up_sync(0xffffffffu, ps, o);
            if (lane >= o) ps += t;
        }
        const u32 before = w ? __shfl_sync(0xffffffffu, ps, w - 1) : 0u;
        u32 run = carry + before + inc - sum;
        carry += __shfl_sync(0xffffffffu, ps, 31);
        const int c = base + (int)threadIdx.x * NA_SC;
#pragma unroll
        for (int k = 0; k < NA_SC; ++k) {
            if (c + k < n) {
                start[c + k] = run;
                cur[c + k] = run;
            }
            run += v[k];
        }
        __syncthreads();   // part is written again
    }
    // the first list's end is the second one's first start, written by its block
    if (threadIdx.x == 0 && list) start[n] = carry;
}

__global__ void k_na_scatter(Batch b, const int *xyz, NaScratch s) {
    griddep_launch();
    griddep_wait();
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < b.N; i += gridDim.x * blockDim.x) {
        const int x = xyz[3 * i], y = xyz[3 * i + 1], z = xyz[3 * i + 2];
        if (!na_inside(b, x, y, z)) continue;
        const u64 g = pack_xyz(x, y, z);
        s.grains[atomicAdd(&s.cursor[0][na_cell_x(b, x, y, z)], 1u)] = g;
        s.grains[atomicAdd(&s.cursor[1][na_cell_y(b, x, y, z)], 1u)] = g;
    }
}

// The tube walk of the regular path (walk.cuh) over the caller's pairs: a warp
// takes 32 pairs (fewer, at least 4, when there are too few to give every warp
// 32) and deals their cell rows and grains over its lanes.
// A pair with an index outside [0, n) or equal indices, a pair whose two
// grains coincide or lie seed_max or more apart on some axis, and every pair
// when a coordinate was out of range, gets -1.  The separation bound keeps
// every cross-product component an exact int32 (|d_e w_f| + |d_f w_e| <
// (extent_e + extent_f) seed_max < 2^31, the parameter precondition) and the
// squared norms within 64 bits, as for the seeds of the regular path.
// Bound by instruction issue like the regular tube counts.  With one thread
// per pair the lanes of a warp waited for the longest of 32 walks: 400,001
// pairs of a 28k-grain view took 377 us of a 431 us call; the call now takes
// 135 us, 87 of them here.
constexpr int NA_W = 8;   // warps per block

__global__ void __launch_bounds__(NA_W * 32, 4) k_na_tube(Batch b, const int *xyz, const int *pairs,
                                                          long long n_pairs, int *counts, NaScratch s) {
    griddep_launch();
    griddep_wait();
    __shared__ SeedTab sp[NA_W];
    __shared__ int4 tbl[NA_W][32];
    __shared__ u32 scount[NA_W][32];
    __shared__ int nit[NA_W][32];   // items of each line
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const bool bad_view = *(volatile u32 *)&s.ctl->bad != 0;
    const long long nwarps = (long long)gridDim.x * NA_W;
    const int lines = (int)max(4ll, min(32ll, (n_pairs + 2 * nwarps - 1) / (2 * nwarps)));
    // a warp's first pairs follow from its number, the next ones, about half of a list
    // that would do with one share a warp, from the counter, as pairs differ in
    // their grains: 100k pairs of 115 grains 30 us, 34 with every pair taken from
    // the counter; 75k pairs of 10k crowded grains 232 us, 322 with one share a warp
    u64 k0 = ((u64)blockIdx.x * NA_W + wib) * (u64)lines;
    const u64 first = (u64)nwarps * (u64)lines;
    while (k0 < (u64)n_pairs) {
        const u64 k = k0 + lane;
        const bool mine = lane < lines && k < (u64)n_pairs;
        bool good = false;
        int4 a = make_int4(0, 0, 0, 0), c = a;
        if (mine) {
            const int i = pairs[2 * k], j = pairs[2 * k + 1];
            if (!bad_view && i >= 0 && i < b.N && j >= 0 && j < b.N && i != j) {
                a = make_int4(xyz[3 * i], xyz[3 * i + 1], xyz[3 * i + 2], 0);
                c = make_int4(xyz[3 * j], xyz[3 * j + 1], xyz[3 * j + 2], 0);
                const int dx = abs(c.x - a.x), dy = abs(c.y - a.y), dz = abs(c.z - a.z);
                good = (dx | dy | dz) != 0 && dx < b.smax && dy < b.smax && dz < b.smax;
            }
        }
        // the walk's lines are the first lanes', so the pairs to count move up
        // past the others
        const unsigned gm = __ballot_sync(0xffffffffu, good);
        const int slot = __popc(gm & ((1u << lane) - 1u));
        if (gm) {
            scount[wib][lane] = 0;
            if (good) {
                SeedSm q;
                nit[wib][slot] = seed_setup(b, a, c, 0, q);
                sp[wib].put(slot, q);
            }
            __syncwarp();
            u32 tests = 0;
            warp_items<true, true, WALK_SERIAL>(b, sp[wib], tbl[wib], lane < __popc(gm) ? nit[wib][lane] : 0, tests,
                                                scount[wib], [&](int own, int4) { atomicAdd(&scount[wib][own], 1u); });
            __syncwarp();
        }
        if (mine) counts[k] = good ? (int)scount[wib][slot] : -1;
        __syncwarp();
        if (first >= (u64)n_pairs) break;
        if (lane == 0) k0 = first + atomicAdd(&s.ctl->ticket, (u64)lines);
        k0 = __shfl_sync(0xffffffffu, k0, 0);
    }
}

std::mutex g_na_mu;
unsigned char *g_na_base[64] = {};
int g_na_sms[64] = {};
void *g_na_ctx[64] = {};   // the CUDA context the cached address belongs to

// The calling thread's current CUDA context (a driver handle), through the
// runtime's driver entry point so that the library needs no -lcuda.
void *current_context() {
    typedef int (*GetCurrent)(void **);
    static GetCurrent fn = nullptr;
    static bool looked = false;
    if (!looked) {
        void *f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (GetCurrent)f;
        cudaGetLastError();
        looked = true;
    }
    void *c = nullptr;
    if (fn && fn(&c) != 0) c = nullptr;
    return c;
}

}  // namespace

}  // namespace et

using namespace et;

extern "C" et_status et_tube_count_noalloc(const int32_t *d_xyz, int64_t n, const et_params *params,
                                           const int32_t *d_pairs, int64_t n_pairs, int32_t *d_counts,
                                           void *stream) {
    et_status st = check_params(params);
    if (st != ET_OK) return st;
    if (n < 0 || n_pairs < 0) return fail(ET_ERR_INVALID_ARG, "negative size");
    if (n > NA_MAX_GRAINS)
        return fail(ET_ERR_INVALID_ARG, "view of %lld grains exceeds the fixed scratch limit of %lld grains",
                    (long long)n, NA_MAX_GRAINS);
    if (n_pairs == 0) return ET_OK;
    if (!d_xyz || !d_pairs || !d_counts) return fail(ET_ERR_INVALID_ARG, "null device pointer");
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_fail(e, "cudaGetDevice");
    if (dev < 0 || dev >= 64) return fail(ET_ERR_INVALID_ARG, "device %d beyond the supported 64", dev);
    unsigned char *base = nullptr;
    int sms = 1;
    {
        std::lock_guard<std::mutex> g(g_na_mu);
        void *cur = current_context();
        if (!g_na_base[dev] || cur != g_na_ctx[dev]) {
            void *p = nullptr;
            e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
            if (e != cudaSuccess) return cuda_fail(e, "cudaGetSymbolAddress of the scratch array");
            cudaDeviceGetAttribute(&g_na_sms[dev], cudaDevAttrMultiProcessorCount, dev);
            if (g_na_sms[dev] <= 0) g_na_sms[dev] = 1;
            g_na_base[dev] = (unsigned char *)p;
            g_na_ctx[dev] = current_context();
        }
        base = g_na_base[dev];
        sms = g_na_sms[dev];
    }
    // cell grid: the regular path's automatic shape on larger cells (the caller's
    // pairs come in any order, so that a cell's start is seldom in a near cache:
    // 400,001 pairs on 28k grains take 230 us at 0.35 grains per s0 cube, 140 us at
    // 1.4, 144 us at 3), coarsened until both lists fit the scratch limit.  On views
    // of 636 to 65,536 grains with lists of 1 to 1.5 M pairs 0.35 is 1.04 to 2.2 times
    // slower everywhere; 2.8 is faster for few pairs (up to 1.6 times), slower for
    // many near ones (0.88)
    Batch b;
    memset(&b, 0, sizeof b);
    b.V = 1;
    b.N = (int)n;
    for (int k = 0; k < 3; ++k) b.ext[k] = params->extent[k];
    b.r = params->tube_r;
    b.r2 = (long long)params->tube_r * params->tube_r;
    b.smax = params->seed_max;
    const double vol = (double)b.ext[0] * b.ext[1] * b.ext[2];
    double s0 = std::cbrt(1.4 * vol / (double)std::max<int64_t>(n, 1));
    // no more cells than the pairs repay: one block scans a list's cells, some 1.2 us a
    // thousand.  At half a cell a pair and at all that fit, us a call: 65,536 grains with
    // 1, 1,000, 30,000 and 100,000 pairs 37 and 113, 85 and 124, 81 and 130, 122 and 154;
    // 21,783 grains of a thin extent with one pair 35 and 166
    const long long most_cells = std::min<long long>(NA_LIST_CELLS, std::max<long long>(4096, n_pairs / 2));
    long long nx = 0, ny = 0;
    for (int tries = 0; tries < 64; ++tries) {
        nx = ny = 1;
        // the second list's edges along x and y are the first one's along y and x as
        // chosen, not as cut to a thin extent: either list comes down to one cell
        auto edge = [&](int shape, int axis) {
            return (int)std::min<double>(std::max(1.0, std::round(s0 * AUTO_CELL[shape])), b.ext[axis]);
        };
        for (int k = 0; k < 3; ++k) {
            b.cs[k] = edge(k, k);
            b.csy[k] = edge(k == 2 ? 2 : 1 - k, k);
        }
        for (int k = 0; k < 3; ++k) {
            b.nc[k] = (b.ext[k] + b.cs[k] - 1) / b.cs[k];
            b.ncy[k] = (b.ext[k] + b.csy[k] - 1) / b.csy[k];
            b.ics[k] = 1.0f / (float)b.cs[k];
            b.icsy[k] = 1.0f / (float)b.csy[k];
            nx *= b.nc[k];
            ny *= b.ncy[k];
        }
        if (std::max(nx, ny) <= most_cells) break;
        s0 *= 1.26;
    }
    if (std::max(nx, ny) > NA_LIST_CELLS) return fail(ET_ERR_INVALID_ARG, "no cell grid fits the fixed scratch limit");
    b.ncell = (int)nx;
    b.ncelly = (int)ny;
    b.dual = 1;
    const NaScratch s = carve(base, nx);
    b.cell_start = s.start[0];
    b.gp = s.grains;
    cudaStream_t cst = (cudaStream_t)stream;
    const unsigned gc = (unsigned)std::min<long long>((std::max(nx, ny) + 255) / 256, 608);
    const unsigned gn = (unsigned)std::max<long long>(1, (n + 255) / 256);
    launch_dep(k_na_clear, dim3(gc), dim3(256), 0, cst, s, (int)nx, (int)ny);
    launch_dep(k_na_count, dim3(gn), dim3(256), 0, cst, b, d_xyz, s);
    launch_dep(k_na_scan, dim3(2), dim3(1024), 0, cst, s, (int)nx, (int)ny, (u32)n);
    launch_dep(k_na_scatter, dim3(gn), dim3(256), 0, cst, b, d_xyz, s);
    // no more blocks than are resident: the warps of a second wave came late and took
    // the counter once each (100k pairs of 115 grains 46 us, 34 without them)
    const unsigned gp = (unsigned)std::min<long long>((n_pairs + 4 * NA_W - 1) / (4 * NA_W), 4ll * sms);
    launch_dep(k_na_tube, dim3(gp), dim3(NA_W * 32), 0, cst, b, d_xyz, d_pairs, n_pairs, d_counts, s);
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "no-alloc tube count launch");
    return ET_OK;
}
