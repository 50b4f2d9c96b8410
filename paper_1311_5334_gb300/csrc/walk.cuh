// walk.cuh -- the tube walk shared by the tube counts and member lists
// (count.cu) and the allocation-free counts (noalloc.cu).
#pragma once
#include "common.cuh"
#include "tube.cuh"

namespace et {

// Tube walks with warp-level load balancing (tube counts and member lists).
//
// A warp takes 32 lines (one per lane).  Each line's cover is split into work
// items: the slabs of cells along whichever of y or z the line crosses more
// cells of ("outer" axis).  Within one slab the tube meets only 1-3 rows of
// the other ("inner") axis, each row a run of x cells that is one contiguous
// range of the cell-ordered grains, so items cost about the same.  The items
// of the 32 lines are dealt to the lanes in rounds of 32: a lane finds the
// line owning its item from the start positions of the lines that begin in
// the round (an OR-reduction of one-hot masks and a popcount).  Line geometry
// is resolved once into shared memory; per-line results are merged with
// shared-memory atomics.  The geometry is the conservative cover of
// tube.cuh, with the per-slab terms hoisted.
// Cover geometry of one line, resolved once per line into eight 16-byte
// vectors (an item loads the six it needs, a grain test the first two).  Slab t-intervals
// are kept as (lower end at cell 0, step per cell, width) with the direction's
// sign already folded in, so the walk needs no min/max to order their ends.
struct __align__(16) SeedSm {
    int4 e0;      // a x w (three components), wx
    int4 e1;      // wy, wz, R low, R high           (R = r^2 |w|^2)
    float4 e2;    // t0, t1 (span of the line near the view), o0, excl (int bits)
    float4 e3;    // outer slab: lower base, step, width; inner cell count (int bits)
    float4 e4;    // inner slab: lower base, step, width, 1 / inner cell edge
    float4 e5;    // inner axis: a - pad, a + pad, w, flags (int bits: 2 w_inner < 0, 4 w_run < 0)
    float4 e6;    // run axis: a - pad, a + pad, w, 1 / run cell edge
    int4 e7;      // run cell count, row stride of outer cell, of inner cell, view offset in the start table
};

// The records of a warp's 32 lines, vector k of line i at v[k][i]: a lane
// storing its own record writes consecutive 16-byte slots (no bank
// conflicts), and lanes reading different lines' vector k mostly hit
// different banks.
struct SeedTab {
    int4 v[8][32];
    __device__ __forceinline__ void put(int i, const SeedSm &q) {
        v[0][i] = q.e0;
        v[1][i] = q.e1;
        v[2][i] = f4i(q.e2);
        v[3][i] = f4i(q.e3);
        v[4][i] = f4i(q.e4);
        v[5][i] = f4i(q.e5);
        v[6][i] = f4i(q.e6);
        v[7][i] = q.e7;
    }
    __device__ __forceinline__ int4 i4(int k, int i) const { return v[k][i]; }
    __device__ __forceinline__ float4 f4(int k, int i) const {
        const int4 t = v[k][i];
        return make_float4(__int_as_float(t.x), __int_as_float(t.y), __int_as_float(t.z), __int_as_float(t.w));
    }
    static __device__ __forceinline__ int4 f4i(float4 f) {
        return make_int4(__float_as_int(f.x), __float_as_int(f.y), __float_as_int(f.z), __float_as_int(f.w));
    }
};

// Slab k of a cell grid with edge cs spans coordinates [k cs, (k+1) cs - 1];
// padded by pad, the line a + t w meets it for t in
//   [base + k step, base + k step + width]
// (w != 0).  w = 0: every t (the caller restricts k to the cells the line's
// constant coordinate can reach).
__device__ __forceinline__ float3 slab_coeffs(float a, float w, float iw, float cs, float pad) {
    if (w == 0.0f) return make_float3(-3.0e38f, 0.0f, 6.0e38f);
    const float step = cs * iw;
    if (w > 0.0f) return make_float3((-pad - a) * iw, step, (cs - 1.0f + 2.0f * pad) * iw);
    return make_float3((cs - 1.0f + pad - a) * iw, step, -(cs - 1.0f + 2.0f * pad) * iw);
}

// Resolves the cover geometry of the line through ga and gb into q and
// returns its number of items (outer slabs).  There is at least one: a lies in the
// view, so t0 < 0 < t1 (pad > 0 keeps the signs), so [a - pad, a + pad] lies within
// the range of every axis, and its cells from (a - pad) / cell to (a + pad) / cell hold
// a's, as the rounding of either (below 2^21 x 2^-22) is less than pad.  warp_items
// counts on that.
__device__ __forceinline__ int seed_setup(const Batch &b, int4 ga, int4 gb, int view, SeedSm &q) {
    const float pad = (float)b.r + COVER_PAD;
    const int wxi = gb.x - ga.x, wyi = gb.y - ga.y, wzi = gb.z - ga.z;
    const long long R = b.r2 * ((long long)wxi * wxi + (long long)wyi * wyi + (long long)wzi * wzi);
    q.e0 = make_int4(ga.y * wzi - ga.z * wyi, ga.z * wxi - ga.x * wzi, ga.x * wyi - ga.y * wxi, wxi);
    q.e1 = make_int4(wyi, wzi, (int)(unsigned)(R & 0xffffffffll), (int)(R >> 32));
    const float ax = (float)ga.x, ay = (float)ga.y, az = (float)ga.z;
    const float wx = (float)wxi, wy = (float)wyi, wz = (float)wzi;
    const float iwx = wxi ? 1.0f / wx : 0.0f;
    const float iwy = wyi ? 1.0f / wy : 0.0f;
    const float iwz = wzi ? 1.0f / wz : 0.0f;
    float t0 = -3.0e38f, t1 = 3.0e38f;
    if (wxi) {
        float ta = (-pad - ax) * iwx, tb = ((float)(b.ext[0] - 1) + pad - ax) * iwx;
        t0 = fmaxf(t0, fminf(ta, tb)); t1 = fminf(t1, fmaxf(ta, tb));
    }
    if (wyi) {
        float ta = (-pad - ay) * iwy, tb = ((float)(b.ext[1] - 1) + pad - ay) * iwy;
        t0 = fmaxf(t0, fminf(ta, tb)); t1 = fminf(t1, fmaxf(ta, tb));
    }
    if (wzi) {
        float ta = (-pad - az) * iwz, tb = ((float)(b.ext[2] - 1) + pad - az) * iwz;
        t0 = fmaxf(t0, fminf(ta, tb)); t1 = fminf(t1, fmaxf(ta, tb));
    }
    const float xl = ax + fminf(t0 * wx, t1 * wx) - pad, xh = ax + fmaxf(t0 * wx, t1 * wx) + pad;
    const float yl = ay + fminf(t0 * wy, t1 * wy) - pad, yh = ay + fmaxf(t0 * wy, t1 * wy) + pad;
    const float zl = az + fminf(t0 * wz, t1 * wz) - pad, zh = az + fmaxf(t0 * wz, t1 * wz) + pad;
    // rows follow the line's dominant horizontal axis: x rows (first list) or y rows (second)
    const bool ylist = b.dual && abs(wyi) > abs(wxi);
    // per axis: a, w, 1/w, cell edge, 1/cell edge, cells
    float ra, rw, oa, ow, oiw, ocs, ia, iw, iiw, ics_, iinv, rinv;
    int nr, o0, nitems, nci, mo, mi;
    u32 cs_off;
    if (!ylist) {
        const int nx = b.nc[0], ny = b.nc[1], nz = b.nc[2];
        cs_off = (u32)view * (u32)b.ncell;
        ra = ax; rw = wx; rinv = b.ics[0]; nr = nx;
        const int cy0 = max(0, floor_i(yl * b.ics[1])), cy1 = min(ny - 1, floor_i(yh * b.ics[1]));
        const int cz0 = max(0, floor_i(zl * b.ics[2])), cz1 = min(nz - 1, floor_i(zh * b.ics[2]));
        const int nyc = max(0, cy1 - cy0 + 1), nzc = max(0, cz1 - cz0 + 1);
        if (nyc >= nzc) {   // outer y, inner z; row = (cz * ny + cy) * nx
            oa = ay; ow = wy; oiw = iwy; ocs = (float)b.cs[1];
            ia = az; iw = wz; iiw = iwz; ics_ = (float)b.cs[2]; iinv = b.ics[2]; nci = nz;
            mo = nx; mi = ny * nx; o0 = cy0; nitems = nyc;
        } else {            // outer z, inner y
            oa = az; ow = wz; oiw = iwz; ocs = (float)b.cs[2];
            ia = ay; iw = wy; iiw = iwy; ics_ = (float)b.cs[1]; iinv = b.ics[1]; nci = ny;
            mo = ny * nx; mi = nx; o0 = cz0; nitems = nzc;
        }
    } else {                // second list: rows along y, index cy + ny * (cx + nx * cz)
        const int nx = b.ncy[0], ny = b.ncy[1], nz = b.ncy[2];
        cs_off = (u32)b.V * (u32)b.ncell + (u32)view * (u32)b.ncelly;
        ra = ay; rw = wy; rinv = b.icsy[1]; nr = ny;
        const int cx0 = max(0, floor_i(xl * b.icsy[0])), cx1 = min(nx - 1, floor_i(xh * b.icsy[0]));
        const int cz0 = max(0, floor_i(zl * b.icsy[2])), cz1 = min(nz - 1, floor_i(zh * b.icsy[2]));
        const int nxc = max(0, cx1 - cx0 + 1), nzc = max(0, cz1 - cz0 + 1);
        if (nxc >= nzc) {   // outer x, inner z; row = (cz * nx + cx) * ny
            oa = ax; ow = wx; oiw = iwx; ocs = (float)b.csy[0];
            ia = az; iw = wz; iiw = iwz; ics_ = (float)b.csy[2]; iinv = b.icsy[2]; nci = nz;
            mo = ny; mi = nx * ny; o0 = cx0; nitems = nxc;
        } else {            // outer z, inner x
            oa = az; ow = wz; oiw = iwz; ocs = (float)b.csy[2];
            ia = ax; iw = wx; iiw = iwx; ics_ = (float)b.csy[0]; iinv = b.icsy[0]; nci = nx;
            mo = nx * ny; mi = ny; o0 = cz0; nitems = nzc;
        }
    }
    const float3 os = slab_coeffs(oa, ow, oiw, ocs, pad);
    const float3 is = slab_coeffs(ia, iw, iiw, ics_, pad);
    const int flags = (iw < 0.0f ? 2 : 0) | (rw < 0.0f ? 4 : 0);
    q.e2 = make_float4(t0, t1, __int_as_float(o0), __int_as_float(0));
    q.e3 = make_float4(os.x, os.y, os.z, __int_as_float(nci));
    q.e4 = make_float4(is.x, is.y, is.z, iinv);
    q.e5 = make_float4(ia - pad, ia + pad, iw, __int_as_float(flags));
    q.e6 = make_float4(ra - pad, ra + pad, rw, rinv);
    q.e7 = make_int4(nr, mo, mi, (int)cs_off);
    return nitems;
}

// Deals the items of the 32 lines in sp to the lanes of the warp and tests
// the grains of their cell runs; hit(owner_line, g) is called for every grain
// g inside the owner line's tube.  n_items is this lane's own line's item
// count (0 for an idle lane).  The lines are those of the first lanes: no lane
// with a line may follow an idle one.  tests counts the membership tests this lane
// performs.
//
// A round gives one item to each lane.  The lane resolves the item's non-empty
// row ranges (usually one or two; a rare third or later row is tested by the
// lane itself).  The warp then deals all grains of the round's first two row
// ranges to its lanes, 32 at a time: lane j takes grain base + j of the
// concatenated ranges, finds the range owning it from the ranges that start
// in this pass (an OR-reduction of one-hot start bits and a popcount) and reads
// the range from a per-warp table (tbl) indexed by that rank.  So every pass
// tests 32 grains, however unevenly the rows of the round hold them.
// Grain k of the two cell orders back to back (k < N: x-row list, k >= N:
// y-row list): 8-byte packed coordinates (PACKED, w = 0) or the 16-byte
// record with the canonical index.
template <bool PACKED>
__device__ __forceinline__ int4 grain_at(const Batch &b, u32 k) {
    if (PACKED) return unpack_xyz(b.gp[k]);
    return b.gc[k];
}

// Grains of its own rows a lane tests itself before the rest is dealt (1 was
// the fastest of 0, 1, 2, 3, 4 and 6 on the batched, dense, PR1 and stress
// workloads: the lane's own loads touch up to 32 lines per warp load, so more
// than one costs more than dealing them).
constexpr int WALK_SERIAL = 1;

// Adds 1 to a shared-memory counter when p holds, without a branch.
__device__ __forceinline__ void red_add_if(bool p, u32 *addr) {
    const unsigned a = (unsigned)__cvta_generic_to_shared(addr);
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %0, 0;\n\t@q red.shared.add.u32 [%1], 1;\n\t}" ::"r"((unsigned)p),
                 "r"(a)
                 : "memory");
}

// COUNT: in the dealt passes every grain inside the tube of line s adds 1 to
// cnt[s] by a predicated reduction; otherwise hit(s, g) is called for it.
template <bool PACKED, bool COUNT, int SERIAL, class Hit>
__device__ __forceinline__ void warp_items(const Batch &b, SeedTab &sp, int4 *tbl, int n_items, u32 &tests,
                                           u32 *cnt, Hit &&hit) {
    const int lane = threadIdx.x & 31;
    const unsigned lane_le = 0xffffffffu >> (31 - lane);
    const unsigned lane_lt = lane_le >> 1;
    int incl = n_items;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
    }
    const int excl = incl - n_items;
    const int total = __shfl_sync(0xffffffffu, incl, 31);
    if (n_items > 0) sp.v[2][lane].w = excl;
    __syncwarp();
    for (int ibase = 0; ibase < total; ibase += 32) {
        // lines whose first item falls in this round mark its position;
        // a lane's owner is the last line started at or before it
        const bool starts = n_items > 0 && excl >= ibase && excl < ibase + 32;
        const unsigned smask = __reduce_or_sync(0xffffffffu, starts ? (1u << (excl - ibase)) : 0u);
        const int before = __popc(__ballot_sync(0xffffffffu, n_items > 0 && excl < ibase));
        const int own = before + __popc(smask & lane_le) - 1;
        const int item = ibase + lane;
        u32 b0 = 0, n0 = 0, b1 = 0, n1 = 0;
        if (item < total) {
            const float4 e2 = sp.f4(2, own), e3 = sp.f4(3, own);
            const int co = __float_as_int(e2.z) + (item - __float_as_int(e2.w));
            const float olo = fmaf((float)co, e3.y, e3.x);
            const float ta = fmaxf(e2.x, olo), tb = fminf(e2.y, olo + e3.z);
            if (ta <= tb) {
                const float4 e4 = sp.f4(4, own), e5 = sp.f4(5, own), e6 = sp.f4(6, own);
                const int4 e7 = sp.i4(7, own);
                const int flags = __float_as_int(e5.w);
                const bool ineg = (flags & 2) != 0, rneg = (flags & 4) != 0;
                // inner cells reached over [ta, tb]
                const float il = fmaf(ineg ? tb : ta, e5.z, e5.x), ih = fmaf(ineg ? ta : tb, e5.z, e5.y);
                const int nci = __float_as_int(e3.w);
                const int ci0 = max(0, floor_i(il * e4.w)), ci1 = min(nci - 1, floor_i(ih * e4.w));
                const u32 *__restrict__ cs = b.cell_start + (u32)e7.w;
                const int rowo = co * e7.y;
                // cell run of inner cell ci: [s0, s1) into cs, or s0 = s1 = 0
                auto run = [&](int ci, int &s0, int &s1) {
                    s0 = s1 = 0;
                    const float vlo = fmaf((float)ci, e4.y, e4.x);
                    const float za = fmaxf(ta, vlo), zb = fminf(tb, vlo + e4.z);
                    const float r0 = fmaf(rneg ? zb : za, e6.z, e6.x), r1 = fmaf(rneg ? za : zb, e6.z, e6.y);
                    const int cr0 = max(0, floor_i(r0 * e6.w)), cr1 = min(e7.x - 1, floor_i(r1 * e6.w));
                    if (za <= zb && cr0 <= cr1 && ci <= ci1) {
                        const int row = rowo + ci * e7.z;
                        s0 = row + cr0;
                        s1 = row + cr1 + 1;
                    }
                };
                // the first two inner cells (almost every item has at most two):
                // their four start-table loads are issued together
                int sa0, sa1, sb0, sb1;
                run(ci0, sa0, sa1);
                run(ci0 + 1, sb0, sb1);
                const u32 ba = cs[sa0], ea = cs[sa1], bb = cs[sb0], eb = cs[sb1];
                if (ea != ba) {
                    b0 = ba;
                    n0 = ea - ba;
                }
                if (eb != bb) {
                    if (n0 == 0) {
                        b0 = bb;
                        n0 = eb - bb;
                    } else {
                        b1 = bb;
                        n1 = eb - bb;
                    }
                }
                for (int ci = ci0 + 2; ci <= ci1; ++ci) {
                    int s0, s1;
                    run(ci, s0, s1);
                    const u32 beg = cs[s0], end = cs[s1];
                    if (end == beg) continue;
                    if (n0 == 0) {
                        b0 = beg;
                        n0 = end - beg;
                    } else if (n1 == 0) {
                        b1 = beg;
                        n1 = end - beg;
                    } else {   // rare: a third row, tested by this lane alone
                        const int4 e0 = sp.i4(0, own), e1 = sp.i4(1, own);
                        const int3 a = make_int3(e0.x, e0.y, e0.z), d = make_int3(e0.w, e1.x, e1.y);
                        const long long R =
                            (long long)(((unsigned long long)(unsigned)e1.w << 32) | (unsigned)e1.z);
                        tests += end - beg;
                        for (u32 k = beg; k < end; ++k) {
                            const int4 g = grain_at<PACKED>(b, k);
                            if (in_tube(g, a, d, R)) hit(own, g);
                        }
                    }
                }
            }
        }
        tests += n0 + n1;
        if (SERIAL > 0 && __any_sync(0xffffffffu, n0 + n1 > 0)) {
            // the first SERIAL grains of its rows each lane tests itself, with its
            // line's parameters in registers (cheaper per test than dealing);
            // only the grains beyond them are dealt over the warp
            const u32 s0 = min(n0, (u32)SERIAL), s1 = min(n1, (u32)SERIAL - s0);
            if (s0 + s1 > 0) {
                const int4 e0 = sp.i4(0, own), e1 = sp.i4(1, own);
                const long long R = (long long)(((unsigned long long)(unsigned)e1.w << 32) | (unsigned)e1.z);
                const int3 a = make_int3(e0.x, e0.y, e0.z), d = make_int3(e0.w, e1.x, e1.y);
#pragma unroll
                for (int j = 0; j < SERIAL; ++j) {
                    if ((u32)j < s0 + s1) {
                        const u32 k = (u32)j < s0 ? b0 + (u32)j : b1 + ((u32)j - s0);
                        const int4 g = grain_at<PACKED>(b, k);
                        const bool h = in_tube(g, a, d, R);
                        if (COUNT) red_add_if(h, &cnt[own]);
                        else if (h) hit(own, g);
                    }
                }
            }
            b0 += s0;
            n0 -= s0;
            b1 += s1;
            n1 -= s1;
        }
        // deal the remaining grains of all lanes' first two rows over the warp
        const u32 n = n0 + n1;
        u32 rin = n;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const u32 v = __shfl_up_sync(0xffffffffu, rin, o);
            if (lane >= o) rin += v;
        }
        const u32 rtotal = __shfl_sync(0xffffffffu, rin, 31);
        const u32 rex = rin - n;
        const unsigned nonempty = __ballot_sync(0xffffffffu, n > 0);
        if (n > 0)
            tbl[__popc(nonempty & lane_lt)] =
                make_int4((int)(b0 - rex), (int)(rex + n0), (int)(b1 - rex - n0), own);
        __syncwarp();
        // two passes per iteration, so that their table, geometry and grain
        // loads overlap; a last part of at most 32 grains takes one pass
        u32 base = 0;
        for (; base + 32 < rtotal; base += 64) {
            const bool st0 = n > 0 && rex >= base && rex < base + 32;
            const bool st1 = n > 0 && rex >= base + 32 && rex < base + 64;
            const unsigned sm0 = __reduce_or_sync(0xffffffffu, st0 ? (1u << (rex - base)) : 0u);
            const unsigned sm1 = __reduce_or_sync(0xffffffffu, st1 ? (1u << (rex - base - 32)) : 0u);
            const unsigned bm = __ballot_sync(0xffffffffu, n > 0 && rex < base);
            const int bef0 = __popc(bm), bef1 = bef0 + __popc(sm0);
            const u32 i0 = base + lane, i1 = i0 + 32;
            const bool v1 = i1 < rtotal;
            const int4 t0 = tbl[bef0 + __popc(sm0 & lane_le) - 1];
            const int4 t1 = tbl[v1 ? bef1 + __popc(sm1 & lane_le) - 1 : 0];
            const u32 k0 = i0 + (u32)(i0 < (u32)t0.y ? t0.x : t0.z);
            const u32 k1 = i1 + (u32)(i1 < (u32)t1.y ? t1.x : t1.z);
            const int ow0 = t0.w, ow1 = t1.w;
            const int4 p0 = sp.i4(0, ow0), q0 = sp.i4(1, ow0), p1 = sp.i4(0, ow1), q1 = sp.i4(1, ow1);
            const int4 g0 = grain_at<PACKED>(b, k0);
            int4 g1 = make_int4(0, 0, 0, 0);
            if (v1) g1 = grain_at<PACKED>(b, k1);
            const long long R0 = (long long)(((unsigned long long)(unsigned)q0.w << 32) | (unsigned)q0.z);
            const long long R1 = (long long)(((unsigned long long)(unsigned)q1.w << 32) | (unsigned)q1.z);
            const bool h0 = in_tube(g0, make_int3(p0.x, p0.y, p0.z), make_int3(p0.w, q0.x, q0.y), R0);
            const bool h1 = v1 && in_tube(g1, make_int3(p1.x, p1.y, p1.z), make_int3(p1.w, q1.x, q1.y), R1);
            if (COUNT) {
                red_add_if(h0, &cnt[ow0]);
                red_add_if(h1, &cnt[ow1]);
            } else {
                if (h0) hit(ow0, g0);
                if (h1) hit(ow1, g1);
            }
        }
        if (base < rtotal) {
            const bool st = n > 0 && rex >= base && rex < base + 32;
            const unsigned sm = __reduce_or_sync(0xffffffffu, st ? (1u << (rex - base)) : 0u);
            const int bef = __popc(__ballot_sync(0xffffffffu, n > 0 && rex < base));
            const u32 i = base + lane;
            if (i < rtotal) {
                const int4 t = tbl[bef + __popc(sm & lane_le) - 1];
                const u32 k = i + (u32)(i < (u32)t.y ? t.x : t.z);
                const int ow = t.w;
                const int4 e0 = sp.i4(0, ow), e1 = sp.i4(1, ow);
                const int4 g = grain_at<PACKED>(b, k);
                const long long R = (long long)(((unsigned long long)(unsigned)e1.w << 32) | (unsigned)e1.z);
                const bool h = in_tube(g, make_int3(e0.x, e0.y, e0.z), make_int3(e0.w, e1.x, e1.y), R);
                if (COUNT) red_add_if(h, &cnt[ow]);
                else if (h) hit(ow, g);
            }
        }
        __syncwarp();   // the table is rewritten by the next round
    }
}

}  // namespace et
