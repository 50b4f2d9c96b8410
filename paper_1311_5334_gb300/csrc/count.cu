// count.cu -- seeds, tube counts, candidates and their member lists.
//
// Seeds (Section 2, Fig. 4a): for each grain a, every grain b of higher
// canonical rank with seed_min^2 <= |g_b - g_a|^2 < seed_max^2.  Higher rank
// means lexicographically larger (x, y, z), so only cells with cx >= cx(a)
// can hold partners.
//
// Tube count (Section 2, Fig. 4b): for each seed, the grains of the whole
// view within tube_r of the infinite line, by the exact test of tube.cuh over
// the cell cover.  Seeds whose count reaches min_hits become candidates.
#include "common.cuh"
#include "walk.cuh"

namespace et {

namespace {

__device__ __forceinline__ u64 warp_sum_u64(u64 v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Work tickets of the warp-balanced walks below.
constexpr int TW = 8;   // warps per block
constexpr int SEED_CHUNK = 32 * 8;   // largest work ticket of a warp (lines)

// Ticket size: SEED_CHUNK lines, smaller when there are too few lines to give
// every warp of the grid a few tickets.
__device__ __forceinline__ u64 ticket_size(u64 n) {
    const u64 unit = 32;
    u64 c = (n / ((u64)gridDim.x * TW * 4) + unit - 1) / unit * unit;
    return c < unit ? unit : (c > (u64)SEED_CHUNK ? (u64)SEED_CHUNK : c);
}

// floor(sqrt(v)) for 0 <= v < 2^62: the float estimate, corrected exactly.
__device__ __forceinline__ int isqrt_ll(long long v) {
    int r = (int)sqrtf((float)v);
    while ((long long)r * r > v) --r;
    while ((long long)(r + 1) * (r + 1) <= v) ++r;
    return r;
}

// Seed generation inside the tube-count kernel.
//
// Seeds (Section 2) are the pairs of grains of one view with
// seed_min^2 <= |g_b - g_a|^2 < seed_max^2, each pair once (a of lower
// canonical rank).  A warp takes SG origins a at a time (1, 2 or 4, a tuning
// choice compiled into one kernel each; consecutive in the
// x-row cell order, one work ticket).  The cell rows that can hold their
// partners -- the (y, z) cells within seed_max - 1 of a, each an x run from
// a's cell to the largest admissible dx -- are dealt to the lanes in rounds
// of 32, and the grains of a round's rows are tested 32 per pass (owner row
// found from one-hot start bits, as in the tube walk).  Accepted pairs queue
// in shared memory; the tube walk takes them 32 at a time.  So seeds are
// walked in the order origin, row, x, and concurrently running warps work on
// nearby origins: no seed list is written to memory.
constexpr int SQ = 64;         // seed queue: < 32 waiting + one pass

template <int SG>
struct GenSm {
    int4 og[SG];      // origin: x, y, z, canonical index
    int4 oc[SG];      // cx0, cx1, cy0, cz0
    int2 on[SG];      // y cells per z slab, cell-table offset of the view
    int ofirst[SG];   // first row item of each origin (the group's total if none)
    int2 tbl[32];     // round's non-empty rows: first position minus pass position, owner origin
    uint2 rr[32];     // per lane: pass position and length of the lane's row in the round
    int ov[SG];       // view of each origin
    int2 q[SQ];       // seeds waiting for the tube walk (lo, hi)
    int qv[SQ];       // their views
};

struct GenState {
    int gtotal = 0;   // row items of the current origin group
    int ibase = 0;    // first row item of the current round
    u32 rtotal = 0;   // grains of the current round
    u32 pbase = 0;    // next pass position in the round
    u32 cnt = 0;      // queued seeds
    u32 pair_tests = 0;   // seed-window tests made by this lane (far below 2^32 in one launch)
};

// Takes the next SG origins; false when none is left.
template <int SG>
__device__ __forceinline__ bool gen_group(const Batch &b, GenSm<SG> &sm, GenState &gs) {
    const int lane = threadIdx.x & 31;
    u64 g0 = 0;
    if (lane == 0) g0 = atomicAdd(&b.ctl->ticket[0], (u64)SG);
    g0 = __shfl_sync(0xffffffffu, g0, 0);
    const u64 N = (u64)b.N;
    if (g0 >= N) return false;
    const int reach = b.smax - 1;   // >= 0: seed_max >= 1
    int nrows = 0;
    if (lane < SG && g0 + lane < N) {
        const int4 g = b.gc[g0 + lane];
        const int v = view_of(b.goff, b.V, g.w);
        const int cx0 = g.x / b.cs[0];
        const int cx1 = min(b.nc[0] - 1, (g.x + reach) / b.cs[0]);
        const int cy0 = max(0, g.y - reach) / b.cs[1];
        const int cy1 = min(b.nc[1] - 1, (g.y + reach) / b.cs[1]);
        const int cz0 = max(0, g.z - reach) / b.cs[2];
        const int cz1 = min(b.nc[2] - 1, (g.z + reach) / b.cs[2]);
        const int ny = cy1 - cy0 + 1;
        nrows = ny * (cz1 - cz0 + 1);
        sm.og[lane] = g;
        sm.oc[lane] = make_int4(cx0, cx1, cy0, cz0);
        sm.on[lane] = make_int2(ny, (int)((u32)v * (u32)b.ncell));
        sm.ov[lane] = v;
    }
    int incl = nrows;
#pragma unroll
    for (int o = 1; o < SG; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane < SG) sm.ofirst[lane] = incl - nrows;
    gs.gtotal = __shfl_sync(0xffffffffu, incl, SG - 1);
    gs.ibase = 0;
    __syncwarp();
    return true;
}

// Resolves the rows of the round at gs.ibase into the pass table.
template <int SG>
__device__ __forceinline__ void gen_round(const Batch &b, GenSm<SG> &sm, GenState &gs) {
    const int lane = threadIdx.x & 31;
    const unsigned lane_lt = (1u << lane) - 1u;
    const int item = gs.ibase + lane;
    u32 beg = 0, n = 0;
    int own = 0;
    if (item < gs.gtotal) {
        // owner: the last origin whose first item is at or before this one
        // (an origin without rows has ofirst = gtotal and is never chosen)
#pragma unroll
        for (int o = 1; o < SG; ++o) own += sm.ofirst[o] <= item ? 1 : 0;
        const int4 g = sm.og[own], oc = sm.oc[own];
        const int2 on = sm.on[own];
        const int j = item - sm.ofirst[own];
        const int jz = j / on.x;
        const int cy = oc.z + (j - jz * on.x), cz = oc.w + jz;
        const long long rz = max(0, max(cz * b.cs[2] - g.z, g.z - (cz * b.cs[2] + b.cs[2] - 1)));
        const long long ry = max(0, max(cy * b.cs[1] - g.y, g.y - (cy * b.cs[1] + b.cs[1] - 1)));
        // the row's nearest point is at least (ry, rz) away in (y, z): it holds
        // partners only up to dx^2 <= seed_max^2 - 1 - ry^2 - rz^2
        const long long left = b.smax2 - 1 - ry * ry - rz * rz;
        if (left >= 0) {
            const int cxr = min(oc.y, (g.x + isqrt_ll(left)) / b.cs[0]);
            const u32 *cs = b.cell_start + (u32)on.y + (size_t)(cz * b.nc[1] + cy) * b.nc[0];
            beg = cs[oc.x];
            n = cs[cxr + 1] - beg;
        }
    }
    u32 rin = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const u32 t = __shfl_up_sync(0xffffffffu, rin, o);
        if (lane >= o) rin += t;
    }
    const u32 rex = rin - n;
    const unsigned nonempty = __ballot_sync(0xffffffffu, n > 0);
    if (n > 0) sm.tbl[__popc(nonempty & lane_lt)] = make_int2((int)(beg - rex), own);
    sm.rr[lane] = make_uint2(rex, n);
    gs.rtotal = __shfl_sync(0xffffffffu, rin, 31);
    gs.pbase = 0;
    __syncwarp();
}

// One pass of 32 grain tests, appending the accepted pairs to the queue;
// false when every origin is done.
template <int SG>
__device__ __forceinline__ bool gen_pass(const Batch &b, GenSm<SG> &sm, GenState &gs) {
    while (gs.pbase >= gs.rtotal) {
        gs.ibase += 32;
        if (gs.ibase >= gs.gtotal && !gen_group(b, sm, gs)) return false;
        gen_round(b, sm, gs);
    }
    const int lane = threadIdx.x & 31;
    const unsigned lane_le = 0xffffffffu >> (31 - lane), lane_lt = lane_le >> 1;
    const uint2 r = sm.rr[lane];
    const u32 base = gs.pbase;
    const bool st = r.y > 0 && r.x >= base && r.x < base + 32;
    const unsigned pm = __reduce_or_sync(0xffffffffu, st ? (1u << (r.x - base)) : 0u);
    const int bef = __popc(__ballot_sync(0xffffffffu, r.y > 0 && r.x < base));
    const u32 i = base + lane;
    bool hit = false;
    int lo = 0, hi = 0, view = 0;
    if (i < gs.rtotal) {
        const int2 t = sm.tbl[bef + __popc(pm & lane_le) - 1];
        const int4 h = b.gc[i + (u32)t.x];
        const int4 g = sm.og[t.y];
        const long long dx = h.x - g.x, dy = h.y - g.y, dz = h.z - g.z;
        const long long d2 = dx * dx + dy * dy + dz * dz;
        hit = h.w > g.w && d2 >= b.smin2 && d2 < b.smax2;
        lo = g.w;
        hi = h.w;
        view = sm.ov[t.y];
        ++gs.pair_tests;
    }
    const unsigned hm = __ballot_sync(0xffffffffu, hit);
    if (hit) {
        const int slot = gs.cnt + __popc(hm & lane_lt);
        sm.q[slot] = make_int2(lo, hi);
        sm.qv[slot] = view;
    }
    gs.cnt += __popc(hm);
    gs.pbase = base + 32;
    __syncwarp();
    return true;
}

// Appends the lanes' accepted seeds (cm: the lanes with is_cand) to the
// candidates, complete: key (2^21 - 1 - count) << 42 | rank_lo << 21 | rank_hi,
// whose ascending order is count descending, then ranks ascending; the place of
// its member list (lists lie in the order the candidates were appended); and
// the input of the candidate-order sort where there is one.
__device__ __forceinline__ void append_candidates(const Batch &b, const Work &w, bool is_cand, unsigned cm, int lo,
                                                  int hi, u32 count, int view) {
    const int lane = threadIdx.x & 31, leader = __ffs(cm) - 1;
    u32 incl = is_cand ? count : 0u;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const u32 t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    const u32 total = __shfl_sync(0xffffffffu, incl, 31);
    u64 idx = 0, m0 = 0;
    if (lane == leader) {
        idx = atomicAdd(&b.ctl->n_cand, (u64)__popc(cm));
        m0 = atomicAdd(&b.ctl->n_members, (u64)total);
    }
    idx = __shfl_sync(0xffffffffu, idx, leader) + __popc(cm & ((1u << lane) - 1u));
    m0 = __shfl_sync(0xffffffffu, m0, leader) + incl - count;
    if (!is_cand) return;
    if (idx >= w.cand_cap) {
        atomicOr(&b.ctl->error, ERRB_OVF_CAND);
        return;
    }
    const u64 g0 = (u64)b.goff[view];
    const u64 key = ((((1ull << 21) - 1ull) - count) << 42) | (((u64)lo - g0) << 21) | ((u64)hi - g0);
    w.c_lo[idx] = lo;
    w.c_hi[idx] = hi;
    w.c_cnt[idx] = count;
    w.c_key[idx] = key;
    w.c_moff[idx] = m0;
    w.c_state[idx] = CS_UNDECIDED;
    if (w.order_k) {
        w.order_k[idx] = cand_sort_key(b, key);
        w.order_v[idx] = (u32)idx;
    }
}

template <int SG>
__global__ void __launch_bounds__(TW * 32, 4) k_tube_count(Batch b, Work w, int record) {
    griddep_launch();
    griddep_wait();
    if (input_failed(b.ctl)) return;
    __shared__ SeedTab sp[TW];
    __shared__ int4 tbl[TW][32];
    __shared__ u32 scount[TW][32];
    __shared__ GenSm<SG> gsm[TW];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    u32 tests = 0, hits = 0;   // per thread: far below 2^32 in one launch
    u64 nseeds = 0;            // per warp (lane 0)
    GenState gs;               // empty: the first pass takes a work ticket
    bool more = true;
    for (;;) {
        while (gs.cnt < 32 && more) more = gen_pass(b, gsm[wib], gs);
        if (gs.cnt == 0) break;
        const u32 m = min(gs.cnt, 32u);
        const bool valid = lane < (int)m;
        int lo = 0, hi = 0, view = 0, n_items = 0;
        if (valid) {
            const int2 sd = gsm[wib].q[lane];
            lo = sd.x;
            hi = sd.y;
            view = gsm[wib].qv[lane];
        }
        __syncwarp();
        if (lane + 32 < (int)gs.cnt) {
            gsm[wib].q[lane] = gsm[wib].q[lane + 32];
            gsm[wib].qv[lane] = gsm[wib].qv[lane + 32];
        }
        gs.cnt -= m;
        nseeds += m;
        if (valid) {
            SeedSm q;
            n_items = seed_setup(b, b.gr[lo], b.gr[hi], view, q);
            sp[wib].put(lane, q);
        }
        scount[wib][lane] = 0;
        __syncwarp();
        warp_items<true, true, WALK_SERIAL>(b, sp[wib], tbl[wib], n_items, tests, scount[wib],
                               [&](int own, int4) { atomicAdd(&scount[wib][own], 1u); });
        __syncwarp();
        const u32 count = valid ? scount[wib][lane] : 0u;
        hits += count;
        if (record) {   // diagnostic per-seed records, appended in blocks of 32
            u64 r0 = 0;
            if (lane == 0) r0 = atomicAdd(&b.ctl->n_record, (u64)m);
            r0 = __shfl_sync(0xffffffffu, r0, 0);
            if (valid) {
                const u64 s = r0 + lane;
                if (s < w.rec_cap) {   // indices into the batch's grains back to back
                    const int vbase = (int)b.goff[view];
                    w.rec_lo[s] = vbase + b.gr[lo].w;
                    w.rec_hi[s] = vbase + b.gr[hi].w;
                    w.rec_cnt[s] = (int)count;
                } else {
                    atomicOr(&b.ctl->error, ERRB_OVF_RECORD);
                }
            }
        }
        const bool is_cand = valid && count >= (u32)b.H;
        const unsigned cm = __ballot_sync(0xffffffffu, is_cand);
        if (cm) append_candidates(b, w, is_cand, cm, lo, hi, count, view);
        __syncwarp();
    }
    const u64 wtests = warp_sum_u64(tests), whits = warp_sum_u64(hits);
    const u64 wpairs = warp_sum_u64(gs.pair_tests);
    if (lane == 0) {
        if (wtests) atomicAdd(&b.ctl->n_tests, wtests);
        if (wpairs) atomicAdd(&b.ctl->n_pair_tests, wpairs);
        if (whits) atomicAdd(&b.ctl->n_hits, whits);
        if (nseeds) atomicAdd(&b.ctl->n_seeds, nseeds);
    }
}

// Member lists of the candidates: the same warp-balanced walk as the counts;
// each in-tube grain takes the next slot of its candidate's member range
// (a shared-memory cursor), so the order inside a list is arbitrary.
__global__ void __launch_bounds__(TW * 32, 4) k_member_fill(Batch b, Work w) {
    griddep_launch();
    griddep_wait();
    if (input_failed(b.ctl)) return;
    if (b.ctl->n_members > w.member_cap) {
        if (blockIdx.x == 0 && threadIdx.x == 0) atomicOr(&b.ctl->error, ERRB_OVF_MEMBERS);
        return;
    }
    const u64 nc = min(b.ctl->n_cand, w.cand_cap);
    __shared__ SeedTab sp[TW];
    __shared__ int4 tbl[TW][32];
    __shared__ u32 cursor[TW][32];            // next slot, relative to the candidate's first
    __shared__ unsigned long long mbase[TW][32];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    int *__restrict__ members = w.members;
    // lines walked together by a warp: 32, or fewer (at least 4) when the
    // candidates cannot give every warp of the grid 32; the rounds a warp
    // walks in sequence, not the work, then set the kernel's duration
    const u64 nwarps = (u64)gridDim.x * TW;
    const u64 per_warp = (nc + nwarps - 1) / nwarps;
    const int lines = per_warp >= 32 ? 32 : (per_warp < 4 ? 4 : (int)per_warp);
    const u64 tsize = lines == 32 ? ticket_size(nc) : (u64)lines;
    for (;;) {
    u64 c0 = 0;
    if (lane == 0) c0 = atomicAdd(&b.ctl->ticket[1], tsize);
    c0 = __shfl_sync(0xffffffffu, c0, 0);
    if (c0 >= nc) break;
    const u64 c1 = min(c0 + tsize, nc);
    for (u64 base = c0; base < c1; base += (u64)lines) {
        const u64 c = base + lane;
        int n_items = 0;
        if (lane < lines && c < c1) {
            const int lo = __ldcs(&w.c_lo[c]), hi = __ldcs(&w.c_hi[c]);
            SeedSm q;
            n_items = seed_setup(b, b.gr[lo], b.gr[hi], view_of(b.goff, b.V, lo), q);
            sp[wib].put(lane, q);
            cursor[wib][lane] = 0;
            mbase[wib][lane] = w.c_moff[c];
        }
        __syncwarp();
        u32 tests = 0;
        warp_items<false, false, WALK_SERIAL>(b, sp[wib], tbl[wib], n_items, tests, cursor[wib], [&](int own, int4 g) {
            members[mbase[wib][own] + atomicAdd(&cursor[wib][own], 1u)] = g.w;
        });
        __syncwarp();
    }
    }
}

unsigned persistent_grid(int blocks_per_sm) {
    static int sms = 0;
    if (!sms) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (sms <= 0) sms = 1;
    }
    return (unsigned)(sms * blocks_per_sm);
}

}  // namespace

void launch_tube_count(const Batch &b, const Work &w, int record, cudaStream_t st) {
    if (b.gen_origins == 1) launch_dep(k_tube_count<1>, dim3(persistent_grid(8)), dim3(TW * 32), 0, st, b, w, record);
    else if (b.gen_origins == 4) launch_dep(k_tube_count<4>, dim3(persistent_grid(8)), dim3(TW * 32), 0, st, b, w, record);
    else launch_dep(k_tube_count<2>, dim3(persistent_grid(8)), dim3(TW * 32), 0, st, b, w, record);
}

void launch_member_fill(const Batch &b, const Work &w, cudaStream_t st) {
    launch_dep(k_member_fill, dim3(persistent_grid(8)), dim3(TW * 32), 0, st, b, w);
}

}  // namespace et
