// frames.cu -- the image front end: filtering and 3D grain recognition of raw
// camera frames (Section 2 of the paper, Fig. 2), from a batch of views to
// their grains, and the C ABI of include/et_frames.h.
//
// One kernel does both steps, k_recognize.  Filtering is monotone in the raw
// value (non-increasing), so f > T holds exactly for raw values below a
// per-pixel cutoff: the count of raw values whose filtered value exceeds T,
// computed once per calibration by k_cutoff from the same formula.  A block
// owns a tile of pixels (256 x 16 on wide frames) and ZC frames: a thread keeps
// the cutoffs of 16 pixels in registers and compares them with its ZC x 16 raw
// bytes, four bytes at a time (SWAR), all loads issued before the first is
// used.  The few voxels that pass (0.2 % of an emulsion view) go to a queue in
// shared memory; once the tile is scanned the block's warps take them 32 at a
// time, one per lane: the lane filters the 3 x 3 x 3 box (its own frame first;
// most candidates end there), applies the maximum test with the raster-order
// tie rule and computes the exact centre-of-mass sums.  The box's bytes were
// loaded by this block or its neighbours a moment ago, so they come from the
// caches.
//
// A grain is counted in its image row (view, frame, row) and linked to the
// row's grains found before it.  The scan of the row counts gives every row's
// place in raster order (and the views' offsets), and k_fr_place ranks each
// grain among its row's few by x.  So the order is independent of the order
// blocks ran in, without a sort.
//
// An earlier form walked each tile's frames through a TMA ring and evaluated
// candidates one at a time with a neighbour per lane: 0.64 ms for 24 full
// views, bound by instruction issue at 0.3 of the copy bandwidth; pruning the
// candidates inside the scanning threads instead took 0.58 ms for the scan
// alone, the lanes of a warp idling while a few of them prune.
#include <algorithm>
#include <cstring>

#include "et_frames.h"
#include "runtime.h"

namespace et {

namespace {

constexpr int FT = 256;       // threads per block
constexpr int ZC = 8;         // frames a scanning thread holds at a time
constexpr int QCAP = 16 * FT; // candidates a block collects on chip: at least one frame of its tile

enum : u32 { FRB_OVF = 1u << 0, FRB_TIMEOUT = 1u << 1, FRB_CROWDED = 1u << 2 };

struct FrCtl {
    u64 n_grains;   // grains appended (may exceed the capacity)
    u64 n_cand;     // voxels with f > T
    u32 error;      // FRB_* bits
    u32 bar[2];     // grid barrier of the scan
    u32 pad;
};

struct FrArgs {
    int W, H, D, P, V;
    int num[3], den[3];
    int chunks;                 // 16-pixel chunks per row
    int zb;                     // frames of a block, a multiple of ZC
    int lc, tiles_x;            // a tile is 2^lc chunks wide and FT / 2^lc rows high; tiles per row
    const unsigned char *raw;
    const unsigned char *cut;       // padded tables: pixel (x, y) at (y + 1) * TP + x + 16
    const unsigned short *cal;      // gain | thr << 8, same layout
    int TP;
    FrCtl *ctl;
    u64 *key;                   // row << 12 | x
    u32 *next;                  // grain of the same row found before (~0: none)
    int4 *rec;
    u64 cap;
    u32 *row_count;             // per image row: grains, then (row_head) the last one found
    u32 *row_head;
};

// Page-locked host memory that the last kernel of a run writes (as Stage of the
// tracking): control block, view offsets and grains where they are few.  A full
// stack of 1,600, 6,400 and 11,900 grains takes 83, 87 and 90 us with copies and 72,
// 78 and 85 us with publication; from some 18,000 grains on the copies are faster
// (34,000 grains: 93 and, in a copy of this code with a larger limit, 109 us).
constexpr u32 FSTAGE_GRAINS = 16384, FSTAGE_VIEWS = 1024;
struct FrStage {
    FrCtl ctl;
    alignas(16) u32 view_off[FSTAGE_VIEWS + 4];
    alignas(16) int xyz[3 * FSTAGE_GRAINS];
    alignas(16) int pulse[FSTAGE_GRAINS];
};

__device__ __forceinline__ int filt(int raw, int g, int t) {
    const int v = min(255, ((255 - raw) * g + 64) >> 7);
    return max(0, v - t);
}

// Per pixel: the number of raw values r in [0, 255] with filt(r) > T; by
// monotonicity exactly the r below it.  filt(255) = 0, so it is at most 255.
__global__ void k_cutoff(const unsigned char *gain, const unsigned char *thr, unsigned char *cut, unsigned short *cal,
                         int n, int T) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int g = gain[i], t = thr[i];
        int c = 0;
        for (int r = 0; r < 256; ++r) c += filt(r, g, t) > T;
        cut[i] = (unsigned char)c;
        cal[i] = (unsigned short)(g | (t << 8));
    }
}

// Tests the candidate (x, y, z) of view v and appends its grain if it is a
// maximum of its 3 x 3 x 3 box.
__device__ __noinline__ void test_candidate(const FrArgs &a, int x, int y, int z, int v) {
    const size_t frame = (size_t)a.H * a.P;
    const unsigned char *at = a.raw + ((size_t)v * a.D + z) * frame + (size_t)y * a.P;   // row start
    const unsigned short *cal = a.cal + (size_t)(y + 1) * a.TP + x + 16;
    u32 c[9];   // calibration of the 3 x 3 pixels
#pragma unroll
    for (int k = 0; k < 9; ++k) c[k] = __ldg(cal + (k / 3 - 1) * a.TP + k % 3 - 1);
    // raw bytes x - 1, x, x + 1 of a row in the low 24 bits
    const int xs = max(x - 1, 0), xw = xs & ~3, sh = 8 * (xs & 3);
    const bool two = (xs & 3) >= 2 && xw + 4 < a.P;
    auto row3 = [&](const unsigned char *row) {
        const u32 w0 = __ldg((const u32 *)(row + xw));
        const u32 w1 = two ? __ldg((const u32 *)(row + xw + 4)) : 0u;
        const u32 w = __funnelshift_r(w0, w1, sh);
        return x > 0 ? w : w << 8;
    };
    const bool left = x > 0, right = x + 1 < a.W;
    auto value = [&](u32 w, int dy, int k) {   // filtered value of byte k (dx = k - 1); outside the frame: -1
        if ((k == 0 && !left) || (k == 2 && !right)) return -1;
        const u32 cc = c[(dy + 1) * 3 + k];
        return filt((int)(w >> (8 * k)) & 255, (int)(cc & 255u), (int)(cc >> 8));
    };
    int S = 0, SX = 0, SY = 0, SZ = 0;
    auto sum = [&](int f, int dx, int dy, int dz) {
        f = max(f, 0);
        S += f;
        SX += dx * f;
        SY += dy * f;
        SZ += dz * f;
    };
    bool alive = true;
    u32 w[3];   // the candidate's frame
#pragma unroll
    for (int dy = -1; dy <= 1; ++dy)
        w[dy + 1] = (unsigned)(y + dy) < (unsigned)a.H ? row3(at + (ptrdiff_t)dy * a.P) : 0u;
    const int fc = value(w[1], 0, 1);
#pragma unroll
    for (int dy = -1; dy <= 1; ++dy) {
        if ((unsigned)(y + dy) >= (unsigned)a.H) continue;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const int f = value(w[dy + 1], dy, k);
            const bool before = dy < 0 || (dy == 0 && k == 0);
            if (dy != 0 || k != 1) alive = alive && (before ? f < fc : f <= fc);
            sum(f, k - 1, dy, 0);
        }
    }
    if (!alive) return;
#pragma unroll
    for (int dz = -1; dz <= 1; dz += 2) {   // the frames before and after
        if ((unsigned)(z + dz) >= (unsigned)a.D) continue;
        const unsigned char *fr = at + (ptrdiff_t)dz * (ptrdiff_t)frame;
#pragma unroll
        for (int dy = -1; dy <= 1; ++dy)
            w[dy + 1] = (unsigned)(y + dy) < (unsigned)a.H ? row3(fr + (ptrdiff_t)dy * a.P) : 0u;
#pragma unroll
        for (int dy = -1; dy <= 1; ++dy) {
            if ((unsigned)(y + dy) >= (unsigned)a.H) continue;
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const int f = value(w[dy + 1], dy, k);
                alive = alive && (dz < 0 ? f < fc : f <= fc);
                sum(f, k - 1, dy, dz);
            }
        }
    }
    if (!alive) return;
    const unsigned won = __activemask();   // the lanes here together share one atomic
    const int lane = threadIdx.x & 31, leader = __ffs(won) - 1;
    u64 slot = 0;
    if (lane == leader) slot = atomicAdd(&a.ctl->n_grains, (u64)__popc(won));
    slot = __shfl_sync(won, slot, leader) + __popc(won & ((1u << lane) - 1u));
    if (slot >= a.cap) {
        atomicOr(&a.ctl->error, FRB_OVF);
        return;
    }
    // coordinate of an axis, rounded half up: floor((2 S g num + 2 So num + S
    // den) / (2 S den)) with the voxel index g and So the offset sum.  With A =
    // 2 g num = a1 (2 den) + a0 it is a1 + floor((S a0 + 2 So num + S den) / (2 S
    // den)), all in int32: A < 2^30, S a0 < 9.1e8, |2 So num| < 3.1e8, S den < 4.6e8
    auto coord = [&](int g, int So, int axis) {
        const int A = 2 * g * a.num[axis], twoden = 2 * a.den[axis];
        const int a1 = A / twoden, a0 = A - a1 * twoden;
        const int m = S * a0 + 2 * So * a.num[axis] + S * a.den[axis], Q = S * twoden;
        int q = m / Q;
        if (m < 0 && q * Q != m) --q;
        return a1 + q;
    };
    const u64 row = ((u64)v * a.D + z) * a.H + y;
    a.key[slot] = (row << 12) | (u64)x;
    a.rec[slot] = make_int4(coord(x, SX, 0), coord(y, SY, 1), coord(z, SZ, 2), S);
    atomicAdd(&a.row_count[row], 1u);
    a.next[slot] = atomicExch(&a.row_head[row], (u32)slot);
}

// Tile blockIdx.x of frames blockIdx.y zb .. of view blockIdx.z.  The floor
// is one read of the raw frames (DRAM), which scan and queue alone reach: 0.48
// ms for 64 full views.  Testing their 6.7 M candidates adds 0.36 ms: the own
// frame 0.10, the frames before and after 0.15, appending the grains 0.10
// (0.835 in all, and 0.822 with those left out that the frame before rules out);
// the blocks' scans and tests overlap on an SM only in part.  With many views a
// block takes the whole depth, whose some 330 candidates keep all its warps
// busy in the test; with few views the depth is split so that the blocks fill
// the device.
__global__ void __launch_bounds__(FT, 4) k_recognize(const __grid_constant__ FrArgs a) {
    griddep_launch();
    griddep_wait();
    __shared__ u32 queue[QCAP];   // thread | pixel << 8 | frame << 12
    __shared__ u32 queued, passed;
    static_assert(FT == 256, "bits of a queue entry");
    const int tid = threadIdx.x;
    if (tid == 0) queued = passed = 0;
    __syncthreads();
    const int tx0 = (blockIdx.x % a.tiles_x) << a.lc, ty0 = (blockIdx.x / a.tiles_x) * (FT >> a.lc);
    const int chunk = tx0 + (tid & ((1 << a.lc) - 1)), y = ty0 + (tid >> a.lc);
    const int v = blockIdx.z, z0 = blockIdx.y * a.zb, nz = min(a.zb, a.D - z0);
    const size_t frame = (size_t)a.H * a.P;
    const bool mine = chunk < a.chunks && y < a.H;
    const unsigned char *src = a.raw + ((size_t)v * a.D + z0) * frame + (size_t)y * a.P + chunk * 16;
    u32 cv[4] = {0u, 0u, 0u, 0u};
    u32 ncand = 0;
    // per byte a < b, four bytes a word (SWAR): with the bytes' high bits a7, b7 and
    // d = (a | 0x80) - (b & 0x7f) (no borrow between bytes), a < b iff
    // (!a7 & b7) | (a7 == b7 & !d7)
    auto below = [](u32 a, u32 b) {
        const u32 d = (a | 0x80808080u) - (b & 0x7f7f7f7fu);
        return ((~a & b) | (~(a ^ b) & ~d)) & 0x80808080u;
    };
    auto bits = [](const u32 (&w)[4]) {   // bit 8 j + k: byte j of word k
        return (w[0] >> 7) | (w[1] >> 6) | (w[2] >> 5) | (w[3] >> 4);
    };
    // queues the pixels r of frame kz below their cutoffs, except those that are no
    // brighter in the frame before (p): calibrated alike and filtered without increasing
    // in the raw value, their pulse there is no smaller, which rules a maximum out.
    // Without that a dark stack queued every voxel.
    auto scan = [&](uint4 r, uint4 p, int kz) {
        const u32 rw[4] = {r.x, r.y, r.z, r.w}, pw[4] = {p.x, p.y, p.z, p.w};
        u32 lt[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) lt[k] = below(rw[k], cv[k]);
        if (lt[0] | lt[1] | lt[2] | lt[3]) {
            ncand += (u32)__popc(bits(lt));
#pragma unroll
            for (int k = 0; k < 4; ++k) lt[k] &= below(rw[k], pw[k]);
            u32 m = bits(lt);
            if (m == 0) return;
            u32 s = atomicAdd(&queued, (u32)__popc(m));
            for (; m && s < QCAP; m &= m - 1, ++s) {
                const int bit = __ffs(m) - 1, px = 4 * (bit & 7) + (bit >> 3);
                queue[s] = (u32)(tid | (px << 8) | (kz << 12));
            }
        }
    };
    auto test_queue = [&](u32 n) {
        for (u32 i = tid; i < n; i += FT) {
            const u32 e = queue[i];
            const int t = (int)(e & 255u);
            test_candidate(a, (tx0 + (t & ((1 << a.lc) - 1))) * 16 + (int)((e >> 8) & 15u), ty0 + (t >> a.lc),
                           z0 + (int)(e >> 12), v);
        }
    };
    if (mine) {
        const uint4 c4 = __ldg((const uint4 *)(a.cut + (size_t)(y + 1) * a.TP + chunk * 16 + 16));
        cv[0] = c4.x;
        cv[1] = c4.y;
        cv[2] = c4.z;
        cv[3] = c4.w;
        uint4 before = make_uint4(~0u, ~0u, ~0u, ~0u);   // the piece's first frame: nothing is ruled out
        for (int z = 0; z < nz; z += ZC) {
            uint4 r[ZC];
#pragma unroll
            for (int k = 0; k < ZC; ++k)
                if (z + k < nz) r[k] = __ldg((const uint4 *)(src + (size_t)(z + k) * frame));
#pragma unroll
            for (int k = 0; k < ZC; ++k)
                if (z + k < nz) scan(r[k], k ? r[k - 1] : before, z + k);
            before = r[ZC - 1];
        }
    }
    ncand = __reduce_add_sync(0xffffffffu, ncand);
    if ((tid & 31) == 0 && ncand) atomicAdd(&passed, ncand);
    __syncthreads();
    const u32 all = queued;
    if (tid == 0 && passed) atomicAdd(&a.ctl->n_cand, (u64)passed);
    if (all <= QCAP) {
        test_queue(all);
        return;
    }
    // a crowded tile: again, a frame at a time (its candidates always fit)
    uint4 before = make_uint4(~0u, ~0u, ~0u, ~0u);
    for (int k = 0; k < nz; ++k) {
        __syncthreads();
        if (tid == 0) queued = 0;
        __syncthreads();
        if (mine) {
            const uint4 r = __ldg((const uint4 *)(src + (size_t)k * frame));
            scan(r, before, k);
            before = r;
        }
        __syncthreads();
        test_queue(queued);
    }
}

// Grains into raster order: a grain's place is its row's start plus its rank by
// x among the row's grains (a few).  Also the views' offsets.  Every grain of a
// row walks its whole chain, so longer rows are left to the two kernels below,
// which the host then launches.  us a call by chains and by those kernels: rows of
// 256 grains 65 and 75 (one row), 150 and 153 (66k grains); of 320, 150 and 153
// (82k grains); of 512, 83 and 85 (one row), 312 and 283 (262k grains); of 1,024,
// 199 and 138 (16k grains); rows of unlike numbers, some above the limit, pay for
// both (46k grains, 320 a row: 172, and 210 with a limit of 384).  Above ROW_FEW
// grains the kernels win from rows of some 100 on: 933k grains of noise, 114 a row,
// 1,344 and 980; 4.2 M grains, 2,048 a row, 9,582 and 6,787.
constexpr u32 ROW_WALK = 768, ROW_WALK_LARGE = 96, ROW_FEW = 1u << 19;

__global__ void k_fr_place(FrArgs a, const u32 *row_start, int *xyz, int *pulse, u32 *view_off) {
    griddep_launch();
    griddep_wait();
    const u64 n = min(a.ctl->n_grains, a.cap);
    const u32 limit = n > ROW_FEW ? ROW_WALK_LARGE : ROW_WALK;
    const u64 tid = (u64)blockIdx.x * blockDim.x + threadIdx.x, stride = (u64)gridDim.x * blockDim.x;
    for (u64 v = tid; v <= (u64)a.V; v += stride) view_off[v] = row_start[v * (u64)a.D * a.H];
    for (u64 i = tid; i < n; i += stride) {
        const u64 k = a.key[i], row = k >> 12;
        const u32 r0 = row_start[row];
        if (row_start[row + 1] - r0 > limit) {
            atomicOr(&a.ctl->error, FRB_CROWDED);
            continue;
        }
        u32 rank = 0;
        for (u32 j = a.row_head[row]; j != ~0u; j = a.next[j]) rank += a.key[j] < k;
        const u64 p = (u64)r0 + rank;
        if (p >= a.cap) continue;   // only after an overflow, when the run is repeated
        const int4 r = a.rec[i];
        xyz[3 * p + 0] = r.x;
        xyz[3 * p + 1] = r.y;
        xyz[3 * p + 2] = r.z;
        pulse[p] = r.w;
    }
}

// Placement where rows are crowded.  First every grain takes a slot of its row's
// part of one array (x << 32 | grain; the row counts count down to 0) ...
__global__ void k_fr_bucket(FrArgs a, const u32 *row_start, u64 *bucket) {
    griddep_launch();
    griddep_wait();
    const u64 n = min(a.ctl->n_grains, a.cap), stride = (u64)gridDim.x * blockDim.x;
    for (u64 i = (u64)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const u64 k = a.key[i], row = k >> 12;
        const u64 p = (u64)row_start[row] + atomicSub(&a.row_count[row], 1u) - 1u;
        bucket[p] = ((k & 4095u) << 32) | i;
    }
}

// ... then it counts the smaller x of its row in that part.  Neighbouring lanes
// are mostly of one row and read the same entries.
__global__ void k_fr_rank(FrArgs a, const u32 *row_start, const u64 *bucket, int *xyz, int *pulse) {
    griddep_launch();
    griddep_wait();
    const u64 n = min(a.ctl->n_grains, a.cap), stride = (u64)gridDim.x * blockDim.x;
    for (u64 q = (u64)blockIdx.x * blockDim.x + threadIdx.x; q < n; q += stride) {
        const u64 e = bucket[q], i = e & 0xffffffffu, row = a.key[i] >> 12;
        const u32 r0 = row_start[row], r1 = row_start[row + 1];
        u64 p = r0;
        for (u32 j = r0; j < r1; ++j) p += bucket[j] < e;   // no two grains of a row share x
        const int4 r = a.rec[i];
        xyz[3 * p + 0] = r.x;
        xyz[3 * p + 1] = r.y;
        xyz[3 * p + 2] = r.z;
        pulse[p] = r.w;
    }
}

// Control block, view offsets and, where they are few, the grains into
// page-locked host memory (16-byte stores in order), for a fetch without device
// copies.
__global__ void k_fr_publish(FrArgs a, const int *xyz, const int *pulse, const u32 *view_off, FrStage *st) {
    griddep_launch();
    griddep_wait();
    const u32 tid = blockIdx.x * blockDim.x + threadIdx.x, stride = gridDim.x * blockDim.x;
    if (tid == 0) st->ctl = *a.ctl;
    for (u32 v = tid; v <= min((u32)a.V, FSTAGE_VIEWS); v += stride) st->view_off[v] = view_off[v];
    const u64 n = min(a.ctl->n_grains, a.cap);
    if (n > FSTAGE_GRAINS) return;
    for (u32 i = tid; i < (3 * (u32)n + 3) / 4; i += stride) ((uint4 *)st->xyz)[i] = ((const uint4 *)xyz)[i];
    for (u32 i = tid; i < ((u32)n + 3) / 4; i += stride) ((uint4 *)st->pulse)[i] = ((const uint4 *)pulse)[i];
}

}  // namespace

// The front end of one camera (geometry and calibration) with its device buffers.
struct FramesRT {
    Ctx *ctx;
    et_frame_params p;
    Group g_tab, g_raw, g_out, g_ctl;
    Group g_bucket;   // for stacks with crowded rows, once there was one
    unsigned char *gain = nullptr, *thr = nullptr, *cut = nullptr;
    unsigned short *cal = nullptr;
    FrCtl *ctl = nullptr;
    // run state
    int V = 0;
    const unsigned char *d_raw = nullptr;
    u64 cap = 0, want = 0;
    u64 *key = nullptr;
    u32 *next = nullptr;
    int4 *rec = nullptr;
    int *xyz = nullptr, *pulse = nullptr;
    u32 *row_count = nullptr, *row_head = nullptr, *row_start = nullptr, *view_off = nullptr;
    void *temp = nullptr;
    int launches = 0;
    cudaStream_t run_stream = nullptr;
    cudaEvent_t ev[4] = {};   // run start, kernel start, kernel end, done
    cudaEvent_t handoff = nullptr;   // a batch's copy of the grains (et_frames_to_batch)
    bool handoff_pending = false;
    bool ran = false, settled = false;
    FrCtl hctl{};
    FrStage *stage = nullptr;   // null: results are copied by the fetch
    et_status run_status = ET_OK;
    float kernel_ms = 0.0f, run_ms = 0.0f;

    FramesRT(Ctx *c, const et_frame_params &pp) : ctx(c), p(pp) {}
    ~FramesRT() {
        if (ran) cudaEventSynchronize(ev[3]);
        if (handoff_pending) cudaEventSynchronize(handoff);
        for (auto &e : ev)
            if (e) cudaEventDestroy(e);
        if (handoff) cudaEventDestroy(handoff);
        ctx->give_stage(1, stage);
        g_tab.release(ctx);
        g_raw.release(ctx);
        g_out.release(ctx);
        g_ctl.release(ctx);
        g_bucket.release(ctx);
    }

    size_t pixels() const { return (size_t)p.width * p.height; }
    // padded calibration tables: 16 columns on either side (16-byte loads), one row
    // above and below
    int table_pitch() const { return (p.width + 15) / 16 * 16 + 32; }
    size_t table_bytes() const { return (size_t)table_pitch() * ((size_t)p.height + 2); }
    size_t rows() const { return (size_t)V * p.depth * p.height; }
    size_t view_bytes() const { return (size_t)p.depth * p.height * p.row_pitch; }

    et_status init() {
        for (auto &e : ev)
            if (cudaEventCreate(&e) != cudaSuccess) return fail(ET_ERR_CUDA, "event creation failed");
        if (cudaEventCreateWithFlags(&handoff, cudaEventDisableTiming) != cudaSuccess)
            return fail(ET_ERR_CUDA, "event creation failed");
        const size_t tb = align_up(table_bytes(), 256);
        if (!g_tab.reserve(ctx, 5 * tb)) return fail(ET_ERR_OOM, "calibration tables");
        gain = (unsigned char *)g_tab.base;
        thr = gain + tb;
        cut = thr + tb;
        cal = (unsigned short *)(cut + tb);
        if (!g_ctl.reserve(ctx, sizeof(FrCtl))) return fail(ET_ERR_OOM, "control block");
        ctl = (FrCtl *)g_ctl.base;
        stage = (FrStage *)ctx->take_stage(1, sizeof(FrStage));
        return ET_OK;
    }

    et_status calibrate(const unsigned char *hg, const unsigned char *ht) {
        if (ran) cudaEventSynchronize(ev[3]);
        cudaStream_t st = ctx->stream;
        const size_t tp = (size_t)table_pitch();
        cudaError_t e = cudaMemsetAsync(gain, 0, 2 * align_up(table_bytes(), 256), st);   // gain and thr
        if (e == cudaSuccess)
            e = cudaMemcpy2DAsync(gain + tp + 16, tp, hg, p.width, p.width, p.height, cudaMemcpyHostToDevice, st);
        if (e == cudaSuccess)
            e = cudaMemcpy2DAsync(thr + tp + 16, tp, ht, p.width, p.width, p.height, cudaMemcpyHostToDevice, st);
        if (e != cudaSuccess) return cuda_fail(e, "calibration upload");
        // zero gain outside the frame gives a zero cutoff there
        const int n = (int)table_bytes();
        k_cutoff<<<std::min((n + 255) / 256, ctx->sms * 8), 256, 0, st>>>(gain, thr, cut, cal, n, p.grain_threshold);
        e = cudaStreamSynchronize(st);   // the caller may free its tables on return
        return e == cudaSuccess ? ET_OK : cuda_fail(e, "cutoff table");
    }

    et_status reserve_out(u64 need) {
        Carver c;
        auto carve = [&](Carver &cv) {
            key = cv.take<u64>(need);
            next = cv.take<u32>(need);
            rec = cv.take<int4>(need);
            xyz = cv.take<int>(3 * need);
            pulse = cv.take<int>(need);
            row_count = cv.take<u32>(rows());
            row_head = cv.take<u32>(rows());
            row_start = cv.take<u32>(rows() + 1);
            view_off = cv.take<u32>((size_t)V + 1);
            temp = cv.take<char>(scan_temp_bytes((long long)rows()));
        };
        cap = last_views = 0;   // until the arrays are there
        carve(c);
        if (!g_out.reserve(ctx, c.off)) return fail(ET_ERR_OOM, "grain buffers (%llu grains)", (unsigned long long)need);
        Carver d;
        d.base = g_out.base;
        carve(d);
        cap = need;
        last_views = (size_t)V;   // the views the row arrays are carved for
        return ET_OK;
    }

    FrArgs args() const {
        FrArgs a;
        memset(&a, 0, sizeof a);
        a.W = p.width;
        a.H = p.height;
        a.D = p.depth;
        a.P = p.row_pitch;
        a.V = V;
        for (int k = 0; k < 3; ++k) {
            a.num[k] = p.pitch_num[k];
            a.den[k] = p.pitch_den[k];
        }
        a.chunks = (p.width + 15) / 16;
        while (a.lc < 4 && (1 << a.lc) < a.chunks) ++a.lc;
        a.tiles_x = (a.chunks + (1 << a.lc) - 1) >> a.lc;
        a.raw = d_raw;
        a.cut = cut;
        a.cal = cal;
        a.TP = table_pitch();
        a.ctl = ctl;
        a.key = key;
        a.next = next;
        a.rec = rec;
        a.cap = cap;
        a.row_count = row_count;
        a.row_head = row_head;
        return a;
    }

    et_status enqueue(cudaStream_t st) {
        cudaMemsetAsync(ctl, 0, sizeof(FrCtl), st);
        cudaMemsetAsync(row_count, 0, sizeof(u32) * rows(), st);
        cudaMemsetAsync(row_head, 0xFF, sizeof(u32) * rows(), st);
        FrArgs a = args();
        const int tile_h = FT >> a.lc, tiles_y = (p.height + tile_h - 1) / tile_h;
        cudaEventRecord(ev[1], st);
        // the depth in as few pieces as give the device 8 blocks per SM
        const long long tiles = (long long)a.tiles_x * tiles_y * V;
        const int steps = (p.depth + ZC - 1) / ZC;
        const int pieces = (int)std::min<long long>(steps, std::max<long long>(1, ((long long)ctx->sms * 8 + tiles - 1) / tiles));
        a.zb = (steps + pieces - 1) / pieces * ZC;
        launch_dep(k_recognize, dim3((unsigned)(a.tiles_x * tiles_y), (unsigned)((p.depth + a.zb - 1) / a.zb), (unsigned)V),
                   dim3(FT), 0, st, a);
        cudaEventRecord(ev[2], st);
        exclusive_scan_u32(row_count, row_start, (long long)rows(), temp, st, &ctl->error, FRB_TIMEOUT, ctl->bar);
        launch_dep(k_fr_place, dim3(ctx->sms * 4), dim3(256), 0, st, a, row_start, xyz, pulse, view_off);
        publish(a, st);
        launches = stage ? 4 : 3;   // recognition, the scan of the row counts, placement, publication
        cudaError_t e = cudaGetLastError();
        return e == cudaSuccess ? ET_OK : cuda_fail(e, "front-end launch");
    }

    void publish(const FrArgs &a, cudaStream_t st) {
        if (stage) launch_dep(k_fr_publish, dim3(16), dim3(512), 0, st, a, (const int *)xyz, (const int *)pulse, (const u32 *)view_off, stage);
    }

    // The placement again, for rows too long to walk.
    et_status place_crowded(cudaStream_t st) {
        if (!g_bucket.reserve(ctx, sizeof(u64) * std::max<u64>(n_grains(), 1)))
            return fail(ET_ERR_OOM, "row order of %llu grains", (unsigned long long)n_grains());
        const FrArgs a = args();
        u64 *bucket = (u64 *)g_bucket.base;
        launch_dep(k_fr_bucket, dim3(ctx->sms * 4), dim3(256), 0, st, a, (const u32 *)row_start, bucket);
        launch_dep(k_fr_rank, dim3(ctx->sms * 8), dim3(256), 0, st, a, (const u32 *)row_start, (const u64 *)bucket, xyz, pulse);
        publish(a, st);
        launches += stage ? 3 : 2;
        cudaError_t e = cudaGetLastError();
        return e == cudaSuccess ? ET_OK : cuda_fail(e, "row order launch");
    }

    et_status run(const unsigned char *raw, int nv, bool on_device, cudaStream_t st) {
        if (ran) cudaEventSynchronize(ev[3]);
        if (handoff_pending) cudaEventSynchronize(handoff);   // buffers may be regrown below
        handoff_pending = false;
        ran = false;   // the shape is the new one: a run that fails leaves nothing to fetch
        V = nv;
        const size_t bytes = (size_t)nv * view_bytes();
        cudaEventRecord(ev[0], st);
        if (on_device) {
            d_raw = raw;
        } else {
            if (!g_raw.reserve(ctx, bytes)) return fail(ET_ERR_OOM, "raw frame buffer (%zu bytes)", bytes);
            cudaError_t e = cudaMemcpyAsync(g_raw.base, raw, bytes, cudaMemcpyHostToDevice, st);
            if (e != cudaSuccess) return cuda_fail(e, "raw frame upload");
            d_raw = (const unsigned char *)g_raw.base;
        }
        const u64 need = std::max(want, std::max<u64>(65536, (u64)nv * p.depth * p.height * p.width / 2000));
        if (cap < need || (size_t)V > last_views) {
            et_status s = reserve_out(std::max(need, cap));
            if (s != ET_OK) {
                if (!on_device) cudaStreamSynchronize(st);   // the upload
                return s;
            }
        }
        want = need;
        et_status s = enqueue(st);
        cudaEventRecord(ev[3], st);
        if (s != ET_OK) {
            cudaEventSynchronize(ev[3]);   // what was launched still writes this handle's memory
            return s;
        }
        run_stream = st;
        ran = true;
        settled = false;
        return ET_OK;
    }
    size_t last_views = 0;

    // Waits for the run; regrows and reruns after an output overflow.
    et_status settle() {
        if (!ran) return fail(ET_ERR_NOT_READY, "nothing has been run");
        if (settled) return run_status;
        bool placed = false;   // this run's crowded rows
        for (int attempt = 0; attempt < 4; ++attempt) {
            cudaError_t e = cudaEventSynchronize(ev[3]);
            if (e != cudaSuccess) return run_status = cuda_fail(e, "front-end run");
            if (stage) hctl = stage->ctl;
            else e = cudaMemcpy(&hctl, ctl, sizeof(FrCtl), cudaMemcpyDeviceToHost);
            if (e != cudaSuccess) return run_status = cuda_fail(e, "control block read");
            if (hctl.error & FRB_TIMEOUT) {
                settled = true;
                return run_status = fail(ET_ERR_TIMEOUT, "the scan of the row counts did not complete in time");
            }
            if ((hctl.error & (FRB_OVF | FRB_CROWDED)) == FRB_CROWDED && !placed) {
                et_status s = place_crowded(ctx->stream);
                cudaEventRecord(ev[3], ctx->stream);
                if (s != ET_OK) {
                    settled = g_bucket.base != nullptr;   // without it nothing was launched: the next call tries again
                    return run_status = s;
                }
                placed = true;
                --attempt;
                continue;
            }
            if (!(hctl.error & FRB_OVF)) {
                cudaEventElapsedTime(&kernel_ms, ev[1], ev[2]);
                cudaEventElapsedTime(&run_ms, ev[0], ev[3]);
                settled = true;
                return run_status = ET_OK;
            }
            const u64 need = hctl.n_grains + hctl.n_grains / 8 + 1024;
            et_status s = reserve_out(need);
            if (s != ET_OK) return run_status = s;
            want = need;
            cudaStream_t st = ctx->stream;
            cudaEventRecord(ev[0], st);
            s = enqueue(st);
            if (s != ET_OK) return run_status = s;
            cudaEventRecord(ev[3], st);
        }
        settled = true;
        return run_status = fail(ET_ERR_CAPACITY, "grain buffer kept overflowing");
    }

    u64 n_grains() const { return std::min(hctl.n_grains, cap); }

    // View offsets of the settled run.
    et_status offsets(std::vector<u32> &off) const {
        off.resize((size_t)V + 1);
        if (stage && V <= (int)FSTAGE_VIEWS) {
            memcpy(off.data(), stage->view_off, sizeof(u32) * off.size());
            return ET_OK;
        }
        const cudaError_t e = cudaMemcpy(off.data(), view_off, sizeof(u32) * off.size(), cudaMemcpyDeviceToHost);
        return e == cudaSuccess ? ET_OK : cuda_fail(e, "view offsets");
    }
};

}  // namespace et

using namespace et;

struct et_frames : public FramesRT {
    using FramesRT::FramesRT;
};

static et_status check_frame_params(const et_frame_params *p) {
    if (!p) return fail(ET_ERR_INVALID_ARG, "params is NULL");
    if (p->width < 1 || p->width > 4096 || p->height < 1 || p->height > 4096 || p->depth < 1 || p->depth > 1024)
        return fail(ET_ERR_INVALID_ARG, "frame size %d x %d x %d outside the limits", p->width, p->height, p->depth);
    if (p->row_pitch < p->width || p->row_pitch % 16 != 0)
        return fail(ET_ERR_INVALID_ARG, "row_pitch %d must be >= width and a multiple of 16", p->row_pitch);
    for (int k = 0; k < 3; ++k)
        if (p->pitch_num[k] < 1 || p->pitch_num[k] > 65535 || p->pitch_den[k] < 1 || p->pitch_den[k] > 65535)
            return fail(ET_ERR_INVALID_ARG, "voxel pitch of axis %d outside [1, 65535]", k);
    if (p->grain_threshold < 0 || p->grain_threshold > 254)
        return fail(ET_ERR_INVALID_ARG, "grain_threshold %d outside [0, 254]", p->grain_threshold);
    if (p->flags != 0) return fail(ET_ERR_INVALID_ARG, "flags must be 0");
    return ET_OK;
}

extern "C" {

et_status et_frames_create(et_ctx *ctx, const et_frame_params *params, const uint8_t *gain, const uint8_t *thr,
                           et_frames **out) {
    GUARD_BEGIN
    if (!ctx || !out || !gain || !thr) return fail(ET_ERR_INVALID_ARG, "NULL argument");
    *out = nullptr;
    et_status s = check_frame_params(params);
    if (s != ET_OK) return s;
    cudaSetDevice(ctx->device);
    et_frames *fr = new et_frames(ctx, *params);
    s = fr->init();
    if (s == ET_OK) s = fr->calibrate(gain, thr);
    if (s != ET_OK) {
        delete fr;
        return s;
    }
    *out = fr;
    return ET_OK;
    GUARD_END
}

et_status et_frames_set_calibration(et_frames *fr, const uint8_t *gain, const uint8_t *thr) {
    GUARD_BEGIN
    if (!fr || !gain || !thr) return fail(ET_ERR_INVALID_ARG, "NULL argument");
    cudaSetDevice(fr->ctx->device);
    return fr->calibrate(gain, thr);
    GUARD_END
}

et_status et_frames_run(et_frames *fr, const uint8_t *raw, int32_t n_views, int32_t on_device, void *stream) {
    GUARD_BEGIN
    if (!fr || !raw) return fail(ET_ERR_INVALID_ARG, "NULL argument");
    if (n_views < 1 || n_views > 65535)
        return fail(ET_ERR_INVALID_ARG, "n_views %d outside the limits", n_views);
    if (on_device && ((uintptr_t)raw & 15u)) return fail(ET_ERR_INVALID_ARG, "device frames must be 16-byte aligned");
    cudaSetDevice(fr->ctx->device);
    cudaStream_t st = stream ? (cudaStream_t)stream : fr->ctx->stream;
    return fr->run(raw, n_views, on_device != 0, st);
    GUARD_END
}

et_status et_frames_sync(et_frames *fr) {
    GUARD_BEGIN
    if (!fr) return fail(ET_ERR_INVALID_ARG, "NULL argument");
    cudaSetDevice(fr->ctx->device);
    return fr->settle();
    GUARD_END
}

et_status et_frames_fetch(et_frames *fr, int64_t *view_offsets, int32_t *xyz, int32_t *pulse, int64_t cap,
                          int64_t *n_grains) {
    GUARD_BEGIN
    if (!fr || !n_grains) return fail(ET_ERR_INVALID_ARG, "NULL argument");
    cudaSetDevice(fr->ctx->device);
    et_status s = fr->settle();
    if (s != ET_OK) return s;
    const int64_t n = (int64_t)fr->n_grains();
    *n_grains = n;
    if (n > 0 && (!xyz || cap < n)) return fail(ET_ERR_CAPACITY, "need room for %lld grains", (long long)n);
    cudaError_t e = cudaSuccess;
    if (fr->stage && n <= (int64_t)FSTAGE_GRAINS) {
        if (n > 0) memcpy(xyz, fr->stage->xyz, sizeof(int32_t) * 3 * (size_t)n);
        if (n > 0 && pulse) memcpy(pulse, fr->stage->pulse, sizeof(int32_t) * (size_t)n);
    } else {
        if (n > 0) e = cudaMemcpy(xyz, fr->xyz, sizeof(int32_t) * 3 * (size_t)n, cudaMemcpyDeviceToHost);
        if (e == cudaSuccess && n > 0 && pulse) e = cudaMemcpy(pulse, fr->pulse, sizeof(int32_t) * (size_t)n, cudaMemcpyDeviceToHost);
    }
    if (e == cudaSuccess && view_offsets) {
        std::vector<u32> off;
        s = fr->offsets(off);
        if (s != ET_OK) return s;
        for (size_t i = 0; i < off.size(); ++i) view_offsets[i] = off[i];
    }
    return e == cudaSuccess ? ET_OK : cuda_fail(e, "grain download");
    GUARD_END
}

et_status et_frames_to_batch(et_frames *fr, et_batch *batch, void *stream) {
    GUARD_BEGIN
    if (!fr || !batch) return fail(ET_ERR_INVALID_ARG, "NULL argument");
    if (batch->ctx != fr->ctx) return fail(ET_ERR_INVALID_ARG, "batch and front end belong to different contexts");
    cudaSetDevice(fr->ctx->device);
    et_status s = fr->settle();
    if (s != ET_OK) return s;
    std::vector<u32> off;
    s = fr->offsets(off);
    if (s != ET_OK) return s;
    std::vector<int64_t> off64(off.begin(), off.end());
    cudaStream_t st = stream ? (cudaStream_t)stream : fr->ctx->stream;
    if (batch->ran) cudaEventSynchronize(batch->done);
    s = batch->load(fr->xyz, off64.data(), fr->V, true, st);
    if (s == ET_OK) {
        cudaEventRecord(fr->handoff, st);   // the next run waits for this copy
        fr->handoff_pending = true;
    }
    return s;
    GUARD_END
}

et_status et_frames_stats_get(et_frames *fr, et_frames_stats *out) {
    if (!fr || !out) return fail(ET_ERR_INVALID_ARG, "NULL argument");
    memset(out, 0, sizeof *out);
    if (!fr->ran || !fr->settled || fr->run_status != ET_OK) return ET_OK;
    out->n_views = fr->V;
    out->n_voxels = (int64_t)fr->V * fr->p.depth * fr->p.height * fr->p.width;
    out->n_candidates = (int64_t)fr->hctl.n_cand;
    out->n_grains = (int64_t)fr->n_grains();
    out->kernel_ms = fr->kernel_ms;
    out->run_ms = fr->run_ms;
    out->kernel_launches = fr->launches;
    return ET_OK;
}

et_status et_frames_destroy(et_frames *fr) {
    if (!fr) return fail(ET_ERR_INVALID_ARG, "NULL argument");
    cudaSetDevice(fr->ctx->device);
    delete fr;
    return ET_OK;
}

}  // extern "C"
