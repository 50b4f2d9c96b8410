// merge.cu -- exclusive grain association, track order and line fit.
//
// Association (Section 2): "each grain used only once, threshold applied
// again".  The defined result is the sequential greedy pass over candidates
// in key order (count descending, rank lo, rank hi): a candidate keeps its
// unused tube grains and is accepted iff at least min_hits remain.
//
// The device computes exactly that result in rounds.  In a round every
// undecided candidate first counts its unused grains; with fewer than
// min_hits it can never be accepted (its unused set only shrinks), so it is
// rejected.  The others post their key on each unused grain (atomicMin).  A
// candidate holding the minimum key on all its unused grains is "ready": every
// earlier candidate sharing one of those grains is already decided, so its
// unused set is final.  It recounts that set -- a candidate accepted earlier
// in the same phase may have taken some of its grains -- and is accepted iff
// at least min_hits remain, else rejected.  Ready candidates share no unused
// grain, so they mark their grains in parallel.  The lowest undecided key is
// always ready, so every round decides at least one candidate.
//
// Key slots are cleaned by their posters: a candidate decided in phase 2
// resets the slots it holds; one still undecided resets last round's slots of
// all its grains at the start of the next round.
//
// A candidate is only ever blocked by candidates of smaller key, so the
// rounds run over windows of the key-sorted candidate list, one window after
// the other: a window's candidates are decided with every earlier window
// already final and no later one taking part.  The result is the same; a
// candidate joins only the rounds of its own window instead of every round
// until its decision.
//
// Rounds are separated by a grid barrier in one cooperative launch; every
// wait is bounded and a timeout sets ERRB_TIMEOUT instead of hanging.  The
// launch covers the device; a short candidate list keeps only a few of its
// blocks (the result does not depend on how many).
#include "common.cuh"
#include <math.h>

#include <algorithm>

namespace et {

// Device mirror of et_track (include/et.h).
struct TrackOut {
    int seed_i, seed_j, nhits, view;
    long long member_offset;
    float c[3], u[3], tmin, tmax;
    int count, reserved;
};
static_assert(sizeof(TrackOut) == 64, "et_track layout");

namespace {

constexpr int MT = 256;
constexpr unsigned long long BARRIER_SPIN_LIMIT = 1ull << 24;  // x ~128 ns sleep ~ 2 s

__device__ __forceinline__ u32 ld_cg_u32(const u32 *p) { return __ldcg(p); }

// Candidates per block in use: a short candidate list runs on few blocks, whose
// barriers are cheap, a long one on the whole grid.
constexpr u64 MERGE_CANDS_PER_BLOCK = MT / 32;

// Up to four candidates of at most 32 grains (cnt 0: none), or one longer one,
// whose grains are read 128 at a time: bound by the dependent reads, too, 239k
// candidates of 600 grains took 3.42 ms at 32 grains a step and take 1.46 ms.
struct Four {
    int c[4];
    u32 cnt[4];
    u64 m0[4], key[4];
    bool lng;
};

// Calls f for the undecided candidates of this warp's share of the list (of
// the window's candidates in order, without one).  The lanes read the states,
// places and keys of 32 candidates at once, and candidates of at most 32 grains
// are handed out four at a time, so that the dependent reads of one (members,
// owners, keys; all from L2) overlap those of the others: a round over the 34k
// candidates of a 28k-grain view took 29 us one candidate at a time.
template <class F>
__device__ __forceinline__ void for_candidates(const Work &w, const int *list, const u32 *corder, u64 w0, long long nl,
                                               long long gwarp, long long nwarps, F &&f) {
    const int lane = threadIdx.x & 31;
    for (long long i0 = gwarp; i0 < nl; i0 += 32 * nwarps) {
        const long long i = i0 + lane * nwarps;
        int c = 0;
        u32 cnt = 0;
        u64 m0 = 0, key = 0;
        bool open = false;
        if (i < nl) {
            // lists and states are rewritten by other SMs between rounds: read through L2
            c = list ? __ldcg(&list[i]) : (int)(corder ? (long long)corder[w0 + i] : i);
            cnt = w.c_cnt[c];
            m0 = w.c_moff[c];
            key = w.c_key[c];
            open = __ldcg(&w.c_state[c]) == CS_UNDECIDED;
        }
        const unsigned longs = __ballot_sync(0xffffffffu, open && cnt > 32);
        unsigned todo = __ballot_sync(0xffffffffu, open);
        while (todo) {
            Four q;
            q.lng = (longs >> (__ffs(todo) - 1)) & 1u;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int src = todo ? __ffs(todo) - 1 : 0;
                const bool take = todo && (k == 0 || (!q.lng && !((longs >> src) & 1u)));
                q.c[k] = __shfl_sync(0xffffffffu, c, src);
                const u32 n = __shfl_sync(0xffffffffu, cnt, src);
                q.m0[k] = __shfl_sync(0xffffffffu, m0, src);
                q.key[k] = __shfl_sync(0xffffffffu, key, src);
                q.cnt[k] = take ? n : 0u;
                if (take) todo &= todo - 1;
            }
            f(q);
        }
    }
}

// The lane's members (-1: none) of the 128 from base on, of a candidate whose list
// ends at m1.
__device__ __forceinline__ void members_at(const Work &w, u64 base, u64 m1, int (&g)[4]) {
    const u64 m = base + (threadIdx.x & 31);
#pragma unroll
    for (int k = 0; k < 4; ++k) g[k] = m + 32 * k < m1 ? w.members[m + 32 * k] : -1;
}

// Angle cut (ET_FLAG_ANGLE_CUT): keep a track iff
//     nhits >= cut_base + cut_slope * min(tan theta, cut_tmax),
// tan theta = sqrt(wx^2 + wy^2) / |wz| for the seed vector w, in exact
// integers: with A = nhits - cut_base, keep iff A >= 0 and either
// wx^2 + wy^2 >= cut_tmax^2 wz^2 (tan theta capped) and A >= cut_slope cut_tmax,
// or A^2 wz^2 >= cut_slope^2 (wx^2 + wy^2) (128-bit products).
__device__ __forceinline__ bool angle_cut_keeps(const Batch &b, int4 glo, int4 ghi, long long nhits) {
    const long long A = nhits - b.cut_base;
    if (A < 0) return false;
    const long long wx = ghi.x - glo.x, wy = ghi.y - glo.y, wz = ghi.z - glo.z;
    const unsigned long long t2 = (unsigned long long)(wx * wx + wy * wy), z2 = (unsigned long long)(wz * wz);
    const unsigned long long tm = (unsigned long long)b.cut_tmax, sl = (unsigned long long)b.cut_slope;
    if ((unsigned __int128)t2 >= (unsigned __int128)(tm * tm) * z2) return (unsigned long long)A >= sl * tm;
    return (unsigned __int128)((unsigned long long)A * (unsigned long long)A) * z2 >=
           (unsigned __int128)(sl * sl) * t2;
}

// Puts an accepted candidate on the list of tracks (any order), unless the
// angle cut drops it.
__device__ __forceinline__ void take_track(const Batch &b, const Work &w, long long c, u32 nfree) {
    if ((b.flags & ET_FLAG_ANGLE_CUT) && !angle_cut_keeps(b, b.gr[w.c_lo[c]], b.gr[w.c_hi[c]], nfree)) return;
    w.acc[atomicAdd(&b.ctl->n_acc, 1ull)] = (int)c;
}

__global__ void __launch_bounds__(MT, 3) k_merge(Batch b, Work w) {
    griddep_launch();
    griddep_wait();
    Ctl *ctl = b.ctl;
    if (input_failed(ctl)) return;   // decided before launch: uniform over the grid
    const u64 nc = min(ctl->n_cand, w.cand_cap);
    // blocks in use (uniform: every block read the same count)
    const unsigned nb = (unsigned)min((u64)gridDim.x, max((u64)1, (nc + MERGE_CANDS_PER_BLOCK - 1) / MERGE_CANDS_PER_BLOCK));
    if (blockIdx.x >= nb) return;
    const unsigned long long lim = b.spin_limit > 0 ? (unsigned long long)b.spin_limit : BARRIER_SPIN_LIMIT;
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const long long gwarp = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const long long nwarps = ((long long)nb * blockDim.x) >> 5;
    const u32 H = (u32)b.H;
    __shared__ int keep[MT / 32][32];   // per warp: undecided candidates waiting to be appended
    // candidates per window: at least 2^18, at most 128 windows, unless set
    const u64 win = w.window ? w.window : max(ASSOC_WINDOW, (nc + 128 - 1) / 128);
    // one window: its rounds give the same result in any order, and the
    // candidates were not sorted
    const u32 *corder = nc > win ? w.corder : nullptr;
    u32 round = 0;   // counts all rounds: it selects the ping-pong buffers
    for (u64 w0 = 0; w0 < nc; w0 += win) {
    const u64 w1 = min(nc, w0 + win);
    for (u32 wr = 0;; ++wr, ++round) {
        u64 *B = w.best[round & 1];
        u64 *Bp = w.best[(round + 1) & 1];
        // candidates of this round: the window first, then the carried list
        const bool first = wr == 0;
        const int *list = first ? nullptr : w.clist[round & 1];
        const long long nl = first ? (long long)(w1 - w0) : (long long)__ldcg(&ctl->ncl[round & 1]);
        if (blockIdx.x == 0 && threadIdx.x == 0) ctl->ncl[(round + 1) & 1] = 0;
        // ---- phase 1: reject hopeless candidates, post keys on unused grains
        u32 my_active = 0;
        for_candidates(w, list, corder, w0, nl, gwarp, nwarps, [&](const Four &f) {
            int g[4];
            bool fr[4];
            if (f.lng) {   // one candidate of more than 32 grains, 128 at a time
                const u64 m0 = f.m0[0], m1 = m0 + f.cnt[0];
                u32 nfree = 0;
                for (u64 base = m0; base < m1; base += 128) {
                    members_at(w, base, m1, g);
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        if (g[k] >= 0 && !first) Bp[g[k]] = ~0ull;   // entries this candidate posted last round
                        fr[k] = g[k] >= 0 && __ldcg(&w.owner[g[k]]) < 0;
                    }
#pragma unroll
                    for (int k = 0; k < 4; ++k) nfree += __popc(__ballot_sync(0xffffffffu, fr[k]));
                }
                if (nfree < H) {
                    if (lane == 0) w.c_state[f.c[0]] = CS_REJECTED;
                    return;
                }
                for (u64 base = m0; base < m1; base += 128) {
                    if (f.cnt[0] > 128) {   // else they are still at hand
                        members_at(w, base, m1, g);
#pragma unroll
                        for (int k = 0; k < 4; ++k) fr[k] = g[k] >= 0 && __ldcg(&w.owner[g[k]]) < 0;
                    }
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        if (fr[k]) atomicMin(&B[g[k]], f.key[0]);
                }
                ++my_active;
                return;
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) g[k] = lane < (int)f.cnt[k] ? w.members[f.m0[k] + lane] : -1;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                if (g[k] >= 0 && !first) Bp[g[k]] = ~0ull;
                fr[k] = g[k] >= 0 && __ldcg(&w.owner[g[k]]) < 0;
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                if (f.cnt[k] == 0) continue;   // fewer than four
                if (__popc(__ballot_sync(0xffffffffu, fr[k])) < H) {
                    if (lane == 0) w.c_state[f.c[k]] = CS_REJECTED;
                } else {
                    if (fr[k]) atomicMin(&B[g[k]], f.key[k]);
                    ++my_active;
                }
            }
        });
        if (lane == 0 && my_active) atomicAdd(&ctl->active[round & 1], my_active);
        if (!coop_barrier(ctl->bar, nb, &ctl->error, ERRB_TIMEOUT, lim)) return;
        const u32 active = ld_cg_u32(&ctl->active[round & 1]);
        if (blockIdx.x == 0 && threadIdx.x == 0 && round < 64) ctl->round_active[round] = active;
        if (blockIdx.x == 0 && threadIdx.x == 0) ctl->active[(round + 1) & 1] = 0;
        if (active == 0) {   // the window is decided (uniform: every block read the same count)
            ++round;
            // the next window's first round counts into the counter just reset
            if (!coop_barrier(ctl->bar, nb, &ctl->error, ERRB_TIMEOUT, lim)) return;
            break;
        }
        // ---- phase 2: accept ready candidates, carry the others to the next round
        int *next = w.clist[(round + 1) & 1];
        u64 *next_n = &ctl->ncl[(round + 1) & 1];
        int nkeep = 0;   // warp-uniform
        auto carry = [&](int c) {
            if (lane == 0) keep[wib][nkeep] = c;
            if (++nkeep == 32) {
                __syncwarp();
                u64 pos = 0;
                if (lane == 0) pos = atomicAdd(next_n, 32ull);
                pos = __shfl_sync(0xffffffffu, pos, 0);
                next[pos + lane] = keep[wib][lane];
                nkeep = 0;
                __syncwarp();
            }
        };
        auto decide = [&](int c, u32 nfree, bool accept) {   // lane 0
            w.c_nfree[c] = nfree;
            w.c_state[c] = accept ? CS_ACCEPTED : CS_REJECTED;
            if (accept) take_track(b, w, c, nfree);
        };
        for_candidates(w, list, corder, w0, nl, gwarp, nwarps, [&](const Four &f) {
            int g[4];
            bool fr[4], bad[4];
            if (f.lng) {
                const u64 m0 = f.m0[0], m1 = m0 + f.cnt[0], key = f.key[0];
                u32 nfree = 0;
                for (u64 base = m0; base < m1; base += 128) {
                    members_at(w, base, m1, g);
#pragma unroll
                    for (int k = 0; k < 4; ++k) fr[k] = g[k] >= 0 && __ldcg(&w.owner[g[k]]) < 0;
#pragma unroll
                    for (int k = 0; k < 4; ++k) bad[k] = fr[k] && __ldcg(&B[g[k]]) != key;
                    if (__any_sync(0xffffffffu, bad[0] | bad[1] | bad[2] | bad[3])) {
                        carry(f.c[0]);
                        return;
                    }
#pragma unroll
                    for (int k = 0; k < 4; ++k) nfree += __popc(__ballot_sync(0xffffffffu, fr[k]));
                }
                // ready: the unused grains are exactly those where this key is the
                // minimum; nobody else can take them any more
                const bool accept = nfree >= H;
                for (u64 base = m0; base < m1; base += 128) {
                    if (f.cnt[0] > 128) {
                        members_at(w, base, m1, g);
#pragma unroll
                        for (int k = 0; k < 4; ++k) fr[k] = g[k] >= 0 && __ldcg(&w.owner[g[k]]) < 0;
                    }
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        if (fr[k]) {
                            if (accept) w.owner[g[k]] = f.c[0];
                            B[g[k]] = ~0ull;
                        }
                }
                if (lane == 0) decide(f.c[0], nfree, accept);
                return;
            }
            // four candidates' members, owners and keys are read before any of
            // them is decided: one that loses a grain to another of the four still
            // sees that grain's smaller key (or the reset slot) and waits a round
#pragma unroll
            for (int k = 0; k < 4; ++k) g[k] = lane < (int)f.cnt[k] ? w.members[f.m0[k] + lane] : -1;
#pragma unroll
            for (int k = 0; k < 4; ++k) fr[k] = g[k] >= 0 && __ldcg(&w.owner[g[k]]) < 0;
#pragma unroll
            for (int k = 0; k < 4; ++k) bad[k] = fr[k] && __ldcg(&B[g[k]]) != f.key[k];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                if (f.cnt[k] == 0) continue;
                if (__any_sync(0xffffffffu, bad[k])) {
                    carry(f.c[k]);
                    continue;
                }
                const u32 nfree = __popc(__ballot_sync(0xffffffffu, fr[k]));
                const bool accept = nfree >= H;
                if (fr[k]) {
                    if (accept) w.owner[g[k]] = f.c[k];
                    B[g[k]] = ~0ull;
                }
                if (lane == 0) decide(f.c[k], nfree, accept);
            }
        });
        if (nkeep > 0) {
            __syncwarp();
            u64 pos = 0;
            if (lane == 0) pos = atomicAdd(next_n, (u64)nkeep);
            pos = __shfl_sync(0xffffffffu, pos, 0);
            if (lane < nkeep) next[pos + lane] = keep[wib][lane];
            __syncwarp();
        }
        if (!coop_barrier(ctl->bar, nb, &ctl->error, ERRB_TIMEOUT, lim)) return;
    }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) ctl->rounds = round;
}

// Single-pass association (ET_FLAG_SINGLE_PASS), step 1: every grain keeps the
// smallest key of the candidates whose tube holds it (one warp per candidate).
__global__ void k_sp_best(Batch b, Work w) {
    griddep_launch();
    griddep_wait();
    if (input_failed(b.ctl)) return;
    const u64 nc = min(b.ctl->n_cand, w.cand_cap);
    const int lane = threadIdx.x & 31;
    const u64 nw = (u64)gridDim.x * (blockDim.x >> 5);
    for (u64 c = (u64)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); c < nc; c += nw) {
        const u64 key = w.c_key[c], m0 = w.c_moff[c], m1 = m0 + w.c_cnt[c];
        for (u64 m = m0 + lane; m < m1; m += 32) atomicMin(&w.best[0][w.members[m]], key);
    }
}

// Step 2: a candidate owns the grains whose smallest key is its own; it is a
// track iff it owns at least min_hits of them.
__global__ void k_sp_own(Batch b, Work w) {
    griddep_launch();
    griddep_wait();
    if (input_failed(b.ctl)) return;
    const u64 nc = min(b.ctl->n_cand, w.cand_cap);
    const int lane = threadIdx.x & 31;
    const u64 nw = (u64)gridDim.x * (blockDim.x >> 5);
    for (u64 c = (u64)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); c < nc; c += nw) {
        const u64 key = w.c_key[c], m0 = w.c_moff[c], m1 = m0 + w.c_cnt[c];
        u32 own = 0;
        for (u64 m = m0 + lane; m < m1; m += 32) own += w.best[0][w.members[m]] == key;
        own = __reduce_add_sync(0xffffffffu, own);
        const bool accept = own >= (u32)b.H;
        if (accept)
            for (u64 m = m0 + lane; m < m1; m += 32) {
                const int g = w.members[m];
                if (w.best[0][g] == key) w.owner[g] = (int)c;
            }
        if (lane == 0) {
            w.c_nfree[c] = own;
            w.c_state[c] = accept ? CS_ACCEPTED : CS_REJECTED;
            if (accept) take_track(b, w, (long long)c, own);
        }
    }
}

// Accepted candidates -> input of the sort into key order.
__global__ void k_acc_keys(Batch b, Work w, Out o) {
    griddep_launch();
    griddep_wait();
    if (input_failed(b.ctl)) return;
    const u64 na = b.ctl->n_acc;
    const u64 stride = (u64)gridDim.x * blockDim.x;
    for (u64 i = (u64)blockIdx.x * blockDim.x + threadIdx.x; i < na; i += stride) {
        const int c = w.acc[i];
        o.sort_k[0][i] = cand_sort_key(b, w.c_key[c]);
        o.sort_v[0][i] = (u32)c;
    }
}

// The whole order of at most ACC_SMALL accepted tracks in one block: (view,
// key) sorted by a bitonic network in shared memory, then their views, member
// offsets and the views' track offsets.  It replaces five launches (eight with
// more than one view) of the general path below, each a few us on one view.
constexpr int ACC_T = 1024, ACC_SMALL = 4096;

__global__ void __launch_bounds__(ACC_T) k_acc_small(Batch b, Work w, Out o) {
    griddep_launch();
    griddep_wait();
    if (input_failed(b.ctl)) return;
    extern __shared__ __align__(16) u64 acc_smem[];
    u64 *key = acc_smem;
    u32 *val = (u32 *)(acc_smem + ACC_SMALL);
    __shared__ u32 wsum[ACC_T / 32];
    const int t = threadIdx.x, lane = t & 31, wib = t >> 5, kb = 3 * b.rbits;
    const int n = (int)min(b.ctl->n_acc, (u64)ACC_SMALL);
    int n2 = 32;
    while (n2 < n) n2 *= 2;
    for (int i = t; i < n2; i += ACC_T) {
        u64 k = ~0ull;
        u32 c = 0;
        if (i < n) {
            c = (u32)w.acc[i];
            k = cand_sort_key(b, w.c_key[c]);
            if (b.V > 1) k |= (u64)view_of(b.goff, b.V, w.c_lo[c]) << kb;
        }
        key[i] = k;
        val[i] = c;
    }
    __syncthreads();
    for (int size = 2; size <= n2; size *= 2)
        for (int step = size / 2; step > 0; step /= 2) {
            for (int i = t; i < n2 / 2; i += ACC_T) {
                const int x = 2 * i - (i & (step - 1)), y = x + step;
                const bool up = (x & size) == 0;
                const u64 kx = key[x], ky = key[y];
                if ((kx > ky) == up) {
                    const u32 v = val[x];
                    key[x] = ky;
                    key[y] = kx;
                    val[x] = val[y];
                    val[y] = v;
                }
            }
            __syncthreads();
        }
    u32 carry = 0;
    for (int base = 0; base < n; base += ACC_T) {
        const int i = base + t;
        u32 c = 0, nf = 0;
        if (i < n) {
            c = val[i];
            nf = w.c_nfree[c];
            o.acc[i] = (int)c;
            o.trk_view[i] = b.V > 1 ? (int)(key[i] >> kb) : 0;
        }
        u32 incl = nf;
#pragma unroll
        for (int s = 1; s < 32; s <<= 1) {
            const u32 x = __shfl_up_sync(0xffffffffu, incl, s);
            if (lane >= s) incl += x;
        }
        if (lane == 31) wsum[wib] = incl;
        __syncthreads();
        u32 ws = wsum[lane];   // every warp scans the warp sums
#pragma unroll
        for (int s = 1; s < 32; s <<= 1) {
            const u32 x = __shfl_up_sync(0xffffffffu, ws, s);
            if (lane >= s) ws += x;
        }
        const u32 before = wib ? __shfl_sync(0xffffffffu, ws, wib - 1) : 0u;
        if (i < n) o.trk_moff[i] = (u64)(carry + before + incl - nf);
        carry += __shfl_sync(0xffffffffu, ws, 31);
        __syncthreads();
    }
    if (t == 0) {
        o.trk_moff[n] = carry;
        b.ctl->n_out_members = carry;
    }
    for (int v = t; v <= b.V; v += ACC_T) {   // first track of view v
        int lo = 0, hi = n;
        if (b.V == 1) lo = v ? n : 0;
        else
            while (lo < hi) {
                const int mid = (lo + hi) / 2;
                if ((long long)(key[mid] >> kb) < v) lo = mid + 1;
                else hi = mid;
            }
        o.view_trk[v] = lo;
    }
}

// After the key sort: second key = view (stable sort keeps key order).
__global__ void k_view_keys(Batch b, Work w, u64 *k, const u32 *v) {
    griddep_launch();
    griddep_wait();
    if (input_failed(b.ctl)) return;   // a timed-out sort leaves invalid indices
    const u64 na = b.ctl->n_acc;
    const u64 stride = (u64)gridDim.x * blockDim.x;
    for (u64 i = (u64)blockIdx.x * blockDim.x + threadIdx.x; i < na; i += stride)
        k[i] = (u64)view_of(b.goff, b.V, w.c_lo[v[i]]);
}

// Sorted accepted list -> per-track view, nhits (for the member scan) and
// per-view counts (with one view, the view's track offsets).
__global__ void k_track_meta(Batch b, Work w, Out o, const u32 *sorted_c) {
    griddep_launch();
    griddep_wait();
    if (input_failed(b.ctl)) return;
    const u64 na = b.ctl->n_acc;
    const u64 stride = (u64)gridDim.x * blockDim.x;
    for (u64 t = (u64)blockIdx.x * blockDim.x + threadIdx.x; t < na; t += stride) {
        const u32 c = sorted_c[t];
        o.acc[t] = (int)c;
        const int v = view_of(b.goff, b.V, w.c_lo[c]);
        o.trk_view[t] = v;
        o.trk_moff[t] = w.c_nfree[c];
        if (b.V > 1) atomicAdd((unsigned long long *)&o.view_trk[v], 1ull);
    }
    if (b.V == 1 && blockIdx.x == 0 && threadIdx.x == 0) {   // one view: its track offsets directly
        o.view_trk[0] = 0;
        o.view_trk[1] = (long long)na;
    }
}

__device__ __forceinline__ long long warp_sum_ll(long long v) {
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) v += __shfl_xor_sync(0xffffffffu, v, s);
    return v;
}

__device__ __forceinline__ float i128_to_float(__int128 x) {
    const bool neg = x < 0;
    unsigned __int128 m = neg ? (unsigned __int128)(-x) : (unsigned __int128)x;
    const double hi = (double)(unsigned long long)(m >> 64);
    const double lo = (double)(unsigned long long)m;
    const double d = hi * 18446744073709551616.0 + lo;
    return (float)(neg ? -d : d);
}

// Symmetric 3x3 eigen-decomposition by cyclic Jacobi rotations (Golub & Van
// Loan, Matrix Computations, Sec. 8.5), FP32.  Columns of V are eigenvectors.
__device__ void jacobi3f(float A[3][3], float V[3][3]) {
    for (int i = 0; i < 3; ++i)
        for (int j = 0; j < 3; ++j) V[i][j] = (i == j) ? 1.0f : 0.0f;
    for (int sweep = 0; sweep < 12; ++sweep) {
        const float off = A[0][1] * A[0][1] + A[0][2] * A[0][2] + A[1][2] * A[1][2];
        const float dg = A[0][0] * A[0][0] + A[1][1] * A[1][1] + A[2][2] * A[2][2];
        if (off == 0.0f || off <= 1e-16f * dg) break;
#pragma unroll
        for (int m = 0; m < 3; ++m) {
            const int p = m < 2 ? 0 : 1, q = m < 1 ? 1 : 2;
            if (A[p][q] == 0.0f) continue;
            const float tau = (A[q][q] - A[p][p]) / (2.0f * A[p][q]);
            const float t = (tau >= 0.0f ? 1.0f : -1.0f) / (fabsf(tau) + sqrtf(1.0f + tau * tau));
            const float c = 1.0f / sqrtf(1.0f + t * t), s = t * c;
            for (int k = 0; k < 3; ++k) {
                const float akp = A[k][p], akq = A[k][q];
                A[k][p] = c * akp - s * akq;
                A[k][q] = s * akp + c * akq;
            }
            for (int k = 0; k < 3; ++k) {
                const float apk = A[p][k], aqk = A[q][k];
                A[p][k] = c * apk - s * aqk;
                A[q][k] = s * apk + c * aqk;
            }
            for (int k = 0; k < 3; ++k) {
                const float vkp = V[k][p], vkq = V[k][q];
                V[k][p] = c * vkp - s * vkq;
                V[k][q] = s * vkp + c * vkq;
            }
        }
    }
}

// One warp per accepted track: exact integer moments about the lo seed grain,
// FP32 principal axis, member projections, and the members (caller indices) in
// ascending order: a track of up to FIT_RANK of them is sorted by rank (each
// member counts the smaller ones) in the warp's shared memory, one of up to
// FIT_SORT by a bitonic network there (one track of 512: the stage 89 us by rank,
// 40 by the network), longer ones are left to k_long_members.  A global sort of
// all members by (track, index) instead took 39 us on a 28k-grain view with 344
// tracks.
constexpr int FIT_T = 256, FIT_RANK = 64, FIT_SORT = 512;

__global__ void __launch_bounds__(FIT_T) k_fit(Batch b, Work w, Out o) {
    __shared__ int ids[FIT_T / 32][FIT_SORT];
    griddep_launch();
    griddep_wait();
    if (input_failed(b.ctl)) return;
    const u64 na = b.ctl->n_acc;
    const int lane = threadIdx.x & 31;
    const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
    int *id = ids[threadIdx.x >> 5];
    TrackOut *tracks = (TrackOut *)o.tracks;
    for (long long t = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; t < (long long)na; t += nw) {
        const int c = o.acc[t];
        const int lo = w.c_lo[c], hi = w.c_hi[c];
        const int4 ga = b.gr[lo], gb = b.gr[hi];
        const u64 m0 = w.c_moff[c], m1 = m0 + w.c_cnt[c];
        const u64 obase = o.trk_moff[t];
        long long s1[3] = {0, 0, 0}, s2[6] = {0, 0, 0, 0, 0, 0};
        u32 written = 0;
        for (u64 base = m0; base < m1; base += 32) {
            const u64 m = base + lane;
            int g = -1;
            if (m < m1) g = w.members[m];
            const bool own = g >= 0 && w.owner[g] == c;
            const unsigned bal = __ballot_sync(0xffffffffu, own);
            if (own) {
                const int4 p = b.gr[g];
                const long long dx = p.x - ga.x, dy = p.y - ga.y, dz = p.z - ga.z;
                s1[0] += dx; s1[1] += dy; s1[2] += dz;
                s2[0] += dx * dx; s2[1] += dy * dy; s2[2] += dz * dz;
                s2[3] += dx * dy; s2[4] += dx * dz; s2[5] += dy * dz;
                const u32 pos = written + __popc(bal & ((1u << lane) - 1u));
                if (pos < FIT_SORT) id[pos] = p.w;
            }
            written += __popc(bal);
        }
        __syncwarp();
        if (written <= FIT_RANK) {
            for (u32 k = lane; k < written; k += 32) {
                const int mine = id[k];
                u32 rank = 0;
                for (u32 j = 0; j < written; ++j) rank += id[j] < mine;
                o.out_members[obase + rank] = mine;
            }
        } else if (written <= FIT_SORT) {
            u32 n2 = 2 * FIT_RANK;
            while (n2 < written) n2 *= 2;
            for (u32 k = written + lane; k < n2; k += 32) id[k] = 0x7fffffff;
            __syncwarp();
            for (u32 size = 2; size <= n2; size *= 2)
                for (u32 step = size / 2; step > 0; step /= 2) {
#pragma unroll 4
                    for (u32 i = lane; i < n2 / 2; i += 32) {
                        const u32 x = 2 * i - (i & (step - 1)), y = x + step;
                        const int a = id[x], c2 = id[y];
                        const bool swap = (a > c2) == ((x & size) == 0);
                        id[x] = swap ? c2 : a;
                        id[y] = swap ? a : c2;
                    }
                    __syncwarp();
                }
            for (u32 k = lane; k < written; k += 32) o.out_members[obase + k] = id[k];
        } else if (lane == 0) {
            o.long_tracks[atomicAdd(&b.ctl->n_long, 1u)] = (int)t;
        }
        __syncwarp();   // the buffer serves the warp's next track
#pragma unroll
        for (int k = 0; k < 3; ++k) s1[k] = warp_sum_ll(s1[k]);
#pragma unroll
        for (int k = 0; k < 6; ++k) s2[k] = warp_sum_ll(s2[k]);
        const long long n = (long long)written;
        // scatter matrix times n^2 ... exact: M_ab = n S2_ab - S1_a S1_b
        const int ia[6] = {0, 1, 2, 0, 0, 1}, ib[6] = {0, 1, 2, 1, 2, 2};
        float cov[6];
        const float inv_n2 = 1.0f / ((float)n * (float)n);
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            const __int128 M = (__int128)n * s2[k] - (__int128)s1[ia[k]] * s1[ib[k]];
            cov[k] = i128_to_float(M) * inv_n2;
        }
        float A[3][3] = {{cov[0], cov[3], cov[4]}, {cov[3], cov[1], cov[5]}, {cov[4], cov[5], cov[2]}};
        float V[3][3];
        jacobi3f(A, V);
        int best = 0;
        if (A[1][1] > A[best][best]) best = 1;
        if (A[2][2] > A[best][best]) best = 2;
        float u[3] = {V[0][best], V[1][best], V[2][best]};
        const float nrm = sqrtf(u[0] * u[0] + u[1] * u[1] + u[2] * u[2]);
        u[0] /= nrm; u[1] /= nrm; u[2] /= nrm;
        const float dot = u[0] * (float)(gb.x - ga.x) + u[1] * (float)(gb.y - ga.y) + u[2] * (float)(gb.z - ga.z);
        bool flip = dot < 0.0f;
        if (dot == 0.0f) flip = (u[0] != 0.0f) ? u[0] < 0.0f : ((u[1] != 0.0f) ? u[1] < 0.0f : u[2] < 0.0f);
        if (flip) { u[0] = -u[0]; u[1] = -u[1]; u[2] = -u[2]; }
        // centroid relative to the lo grain.  A member's offset from the
        // centroid, times n, is the exact integer n d - S1 (d its offset from
        // the lo grain), so a projection's rounding scales with the
        // projection itself, not with the view or the track length
        const float fn = (float)n;
        const float ca[3] = {(float)s1[0] / fn, (float)s1[1] / fn, (float)s1[2] / fn};
        const float cen[3] = {(float)ga.x + ca[0], (float)ga.y + ca[1], (float)ga.z + ca[2]};
        float tmin = 3.0e38f, tmax = -3.0e38f;
        for (u64 base = m0; base < m1; base += 32) {
            const u64 m = base + lane;
            if (m < m1) {
                const int g = w.members[m];
                if (w.owner[g] == c) {
                    const int4 p = b.gr[g];
                    const long long ex = n * (long long)(p.x - ga.x) - s1[0];
                    const long long ey = n * (long long)(p.y - ga.y) - s1[1];
                    const long long ez = n * (long long)(p.z - ga.z) - s1[2];
                    const float tt = ((float)ex * u[0] + (float)ey * u[1] + (float)ez * u[2]) / fn;
                    tmin = fminf(tmin, tt);
                    tmax = fmaxf(tmax, tt);
                }
            }
        }
#pragma unroll
        for (int s = 16; s > 0; s >>= 1) {
            tmin = fminf(tmin, __shfl_xor_sync(0xffffffffu, tmin, s));
            tmax = fmaxf(tmax, __shfl_xor_sync(0xffffffffu, tmax, s));
        }
        if (lane == 0) {
            TrackOut r;
            r.seed_i = ga.w;
            r.seed_j = gb.w;
            r.nhits = (int)n;
            r.view = o.trk_view[t];
            r.member_offset = (long long)obase;
            r.c[0] = cen[0]; r.c[1] = cen[1]; r.c[2] = cen[2];
            r.u[0] = u[0]; r.u[1] = u[1]; r.u[2] = u[2];
            r.tmin = tmin;
            r.tmax = tmax;
            r.count = (int)w.c_cnt[c];
            r.reserved = 0;
            tracks[t] = r;
        }
    }
}

// Members of the tracks longer than FIT_SORT, one block per track: a bitmap of
// the caller indices (below 2^rbits), LONG_BITS of them at a time, whose set bits
// are written out in order.  A thread scans consecutive words, so word w lies at w
// + w / 32: at w the lanes of a warp met in one bank.  200 tracks of 600 took the
// stage 0.88 ms over all 2^21 indices by 16 blocks, and take 0.09 ms.
constexpr int LONG_T = 1024, LONG_BITS = 1 << 20;

__host__ __device__ constexpr u32 long_word(u32 w) { return w + (w >> 5); }
__host__ __device__ inline u32 long_words(int rbits) { return max(1u, min((u32)LONG_BITS, 1u << rbits) / 32u); }

__global__ void __launch_bounds__(LONG_T) k_long_members(Batch b, Work w, Out o) {
    griddep_launch();
    griddep_wait();
    if (input_failed(b.ctl)) return;
    extern __shared__ __align__(16) u32 bits[];   // long_word(long_words(rbits)) of them
    __shared__ u32 wsum[LONG_T / 32];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const u32 nw = long_words(b.rbits), per = (nw + LONG_T - 1) / LONG_T;   // words, and those a thread scans
    const u32 w0 = min(nw, threadIdx.x * per), w1 = min(nw, w0 + per);
    for (u32 l = blockIdx.x; l < b.ctl->n_long; l += gridDim.x) {
        const int t = o.long_tracks[l], c = o.acc[t];
        const u64 m0 = w.c_moff[c], m1 = m0 + w.c_cnt[c];
        u64 obase = o.trk_moff[t];
        for (int base = 0; base < 1 << b.rbits; base += LONG_BITS) {
            for (u32 i = threadIdx.x; i < nw; i += LONG_T) bits[long_word(i)] = 0;
            __syncthreads();
            for (u64 m = m0 + threadIdx.x; m < m1; m += LONG_T) {
                const int g = w.members[m];
                if (w.owner[g] != c) continue;
                const int i = b.gr[g].w - base;
                if (i >= 0 && i < LONG_BITS) atomicOr(&bits[long_word((u32)i >> 5)], 1u << (i & 31));
            }
            __syncthreads();
            u32 n = 0;
            for (u32 k = w0; k < w1; ++k) n += __popc(bits[long_word(k)]);
            u32 incl = n;
#pragma unroll
            for (int s = 1; s < 32; s <<= 1) {
                const u32 x = __shfl_up_sync(0xffffffffu, incl, s);
                if (lane >= s) incl += x;
            }
            if (lane == 31) wsum[wib] = incl;
            __syncthreads();
            u32 before = 0, total = 0;
            for (int k = 0; k < LONG_T / 32; ++k) {
                if (k < wib) before += wsum[k];
                total += wsum[k];
            }
            u64 pos = obase + before + incl - n;
            for (u32 k = w0; k < w1; ++k)
                for (u32 x = bits[long_word(k)]; x; x &= x - 1) o.out_members[pos++] = base + (int)k * 32 + __ffs(x) - 1;
            obase += total;
            __syncthreads();
        }
    }
}

// The run's control block and small results into page-locked host memory, so
// that the caller's fetch waits once and copies on the host: a device copy
// after the run costs about 10 us each, and a fetch took five of them.
__global__ void k_publish(Batch b, Out o, Stage *st) {
    griddep_launch();
    griddep_wait();
    const u32 t = blockIdx.x * blockDim.x + threadIdx.x, nth = gridDim.x * blockDim.x;
    const Ctl *ctl = b.ctl;
    for (u32 i = t; i < sizeof(Ctl) / sizeof(u32); i += nth) ((u32 *)&st->ctl)[i] = ((const u32 *)ctl)[i];
    const bool whole = !(ctl->error & (ERRB_INPUT_MASK | ERRB_OVF_MASK | ERRB_TIMEOUT)) && ctl->n_acc <= STAGE_TRACKS &&
                       ctl->n_out_members <= STAGE_MEMBERS && b.V <= (int)STAGE_VIEWS;
    if (t == 0) st->whole = whole ? 1u : 0u;
    if (!whole) return;
    const u32 nt = (u32)ctl->n_acc, nm = (u32)ctl->n_out_members;
    for (u32 i = t; i < nt * 4; i += nth) ((uint4 *)st->tracks)[i] = ((const uint4 *)o.tracks)[i];
    for (u32 i = t; i < nm; i += nth) st->members[i] = o.out_members[i];
    for (u32 i = t; i <= (u32)b.V; i += nth) st->view_trk[i] = o.view_trk[i];
}

unsigned sm_count() {
    static int sms = 0;
    if (!sms) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (sms <= 0) sms = 1;
    }
    return (unsigned)sms;
}

int bits_for(unsigned long long maxval) {
    int b = 0;
    while (b < 64 && (maxval >> b) != 0) ++b;
    return b;
}

}  // namespace

int merge_grid_blocks(int device) {
    cudaFuncSetAttribute(k_long_members, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)(long_word(LONG_BITS / 32) * sizeof(u32)));
    cudaFuncSetAttribute(k_acc_small, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)(ACC_SMALL * (sizeof(u64) + sizeof(u32))));
    int sms = 0, per_sm = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_merge, MT, 0);
    if (per_sm > 4) per_sm = 4;
    if (per_sm < 1) per_sm = 1;
    return sms * per_sm;
}

cudaError_t launch_merge_coop(const Batch &b, const Work &w, int grid, cudaStream_t st) {
    Batch bb = b;
    Work ww = w;
    void *args[] = {&bb, &ww};
    return cudaLaunchCooperativeKernel((const void *)k_merge, dim3(grid), dim3(MT), args, 0, st);
}

void launch_publish(const Batch &b, const Out &o, Stage *st_host, cudaStream_t st) {
    launch_dep(k_publish, dim3(8), dim3(512), 0, st, b, o, st_host);
}

const u32 *launch_cand_order(const Batch &b, const Work &w, Out &o, u64 window, void *temp, cudaStream_t st) {
    const int cur = radix_sort_pairs_dev(o.sort_k[0], o.sort_v[0], o.sort_k[1], o.sort_v[1], (long long)o.acc_cap,
                                         &b.ctl->n_cand, 3 * b.rbits, temp, st, &b.ctl->error, ERRB_TIMEOUT,
                                         b.ctl->bar, b.spin_limit, (long long)window);
    return o.sort_v[cur];
}

void launch_single_pass(const Batch &b, const Work &w, cudaStream_t st) {
    const unsigned g = sm_count() * 8;
    launch_dep(k_sp_best, dim3(g), dim3(256), 0, st, b, w);
    launch_dep(k_sp_own, dim3(g), dim3(256), 0, st, b, w);
}

static void launch_fit(const Batch &b, const Work &w, const Out &o, cudaStream_t st) {
    launch_dep(k_fit, dim3(sm_count() * 4), dim3(FIT_T), 0, st, b, w, o);
    // a block for every track that can be this long, one at least
    const unsigned g = (unsigned)std::min<long long>(sm_count(), std::max(1, b.N / (FIT_SORT + 1)));
    launch_dep(k_long_members, dim3(g), dim3(LONG_T), long_word(long_words(b.rbits)) * sizeof(u32), st, b, w, o);
}

// Accepted list sorted by (view, key); per-view track offsets; member offsets;
// fit with the sorted members.  acc_cap sizes the launches; the device counters
// decide the work.
void launch_output(const Batch &b, const Work &w, Out &o, long long acc_cap, void *temp, cudaStream_t st) {
    const unsigned g = sm_count() * 4;
    const int vbits = bits_for((unsigned long long)std::max(b.V - 1, 0));
    if (b.N / b.H <= ACC_SMALL && 3 * b.rbits + vbits < 64) {   // a track owns at least H grains
        launch_dep(k_acc_small, dim3(1), dim3(ACC_T), ACC_SMALL * (sizeof(u64) + sizeof(u32)), st, b, w, o);
        launch_fit(b, w, o, st);
        return;
    }
    launch_dep(k_acc_keys, dim3(g), dim3(256), 0, st, b, w, o);
    u64 *na = &b.ctl->n_acc;
    int cur = radix_sort_pairs_dev(o.sort_k[0], o.sort_v[0], o.sort_k[1], o.sort_v[1], acc_cap, na, 3 * b.rbits,
                                   temp, st, &b.ctl->error, ERRB_TIMEOUT, b.ctl->bar, b.spin_limit);
    if (b.V > 1) {
        launch_dep(k_view_keys, dim3(g), dim3(256), 0, st, b, w, o.sort_k[cur], o.sort_v[cur]);
        int c2 = radix_sort_pairs_dev(o.sort_k[cur], o.sort_v[cur], o.sort_k[cur ^ 1], o.sort_v[cur ^ 1], acc_cap,
                                      na, vbits, temp, st, &b.ctl->error, ERRB_TIMEOUT,
                                      b.ctl->bar, b.spin_limit);
        cur = c2 ? (cur ^ 1) : cur;
    }
    if (b.V > 1) cudaMemsetAsync(o.view_trk, 0, sizeof(long long) * (b.V + 1), st);
    launch_dep(k_track_meta, dim3(g), dim3(256), 0, st, b, w, o, o.sort_v[cur]);
    if (b.V > 1)
        exclusive_scan_u64_dev((const u64 *)o.view_trk, (u64 *)o.view_trk, b.V, nullptr, temp, nullptr, st,
                               &b.ctl->error, ERRB_TIMEOUT, b.ctl->bar, b.spin_limit);
    exclusive_scan_u64_dev(o.trk_moff, o.trk_moff, acc_cap, na, temp, &b.ctl->n_out_members, st, &b.ctl->error,
                           ERRB_TIMEOUT, b.ctl->bar, b.spin_limit);
    launch_fit(b, w, o, st);
}

}  // namespace et
