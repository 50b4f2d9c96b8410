// grid.cu -- canonical order and cell list of every view in a batch.
//
// Canonical rank: the position of a grain in lexicographic (x, y, z) order of
// its view.  It orders seeds (lo = lower rank) and breaks ties between
// candidates, so every result is independent of the caller's grain order and
// of the cell size.  The cell list bins the grains of each view in a uniform
// 3D grid (the paper's 3D hash tables, Section 3 footnote), x fastest, so that
// a run of cells along x is one contiguous range of grains.  The list is a
// counting sort: per-cell counts, their exclusive scan (cell starts), and a
// scatter that takes slots with an atomic cursor per cell.  The second list
// (rows along y) is counted, scanned and filled with the first: its cells follow
// the first list's in one table, so its grains' positions start at N.  The order of the
// grains inside one cell is therefore arbitrary; no result depends on it
// (counts, keys and fits are order-independent, member lists are sorted on
// output).
#include "common.cuh"

namespace et {

namespace {

__global__ void k_canonical_keys(Batch b, u64 *keys, u32 *vals) {
    griddep_launch();
    griddep_wait();
    const long long stride = (long long)gridDim.x * blockDim.x;
    const int sy = b.cbits[2], sx = b.cbits[1] + b.cbits[2];
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < b.N; i += stride) {
        int v = view_of(b.goff, b.V, i);
        int x = b.xyz_in[3 * i + 0], y = b.xyz_in[3 * i + 1], z = b.xyz_in[3 * i + 2];
        bool ok = (x >= 0) & (x < b.ext[0]) & (y >= 0) & (y < b.ext[1]) & (z >= 0) & (z < b.ext[2]);
        if (!ok) {
            atomicOr(&b.ctl->error, ERRB_OUT_OF_RANGE);
            x = min(max(x, 0), b.ext[0] - 1);
            y = min(max(y, 0), b.ext[1] - 1);
            z = min(max(z, 0), b.ext[2] - 1);
        }
        keys[i] = ((u64)v << b.vshift) | ((u64)x << sx) | ((u64)y << sy) | (u64)z;
        vals[i] = (u32)i;
    }
}

// Cells of a grain in the two lists.
__device__ __forceinline__ u32 cell_x(const Batch &b, int v, int x, int y, int z) {
    const int cx = min(x / b.cs[0], b.nc[0] - 1), cy = min(y / b.cs[1], b.nc[1] - 1), cz = min(z / b.cs[2], b.nc[2] - 1);
    return (u32)v * (u32)b.ncell + (u32)(cx + b.nc[0] * (cy + b.nc[1] * cz));
}
__device__ __forceinline__ u32 cell_y(const Batch &b, int v, int x, int y, int z) {
    const int cx = min(x / b.csy[0], b.ncy[0] - 1), cy = min(y / b.csy[1], b.ncy[1] - 1);
    const int cz = min(z / b.csy[2], b.ncy[2] - 1);
    return (u32)v * (u32)b.ncelly + (u32)(cy + b.ncy[1] * (cx + b.ncy[0] * cz));
}

// Grains into canonical order, and the counts of their cells in both lists.
// The keys are sorted from bit bit0 on (view and x); a grain's rank among those
// that agree there, rarely more than one, comes from comparing the full keys.
// Sorting on all bits took 6 instead of 2 passes for one view.  More than
// CROWD grains that agree report ERRB_CROWDED, and the run is repeated with
// the full sort, as are the batch's next ones; those watch whether grains would
// still crowd.
constexpr int CROWD = 64;

__global__ void k_canonical_order(Batch b, const u64 *keys, const u32 *vals, u32 *count, u32 *count_y, int bit0,
                                  int watch) {
    griddep_launch();
    griddep_wait();
    // a coordinate out of range is reported as such; a timed-out sort leaves
    // invalid indices: either way nothing after this point may run
    if (input_failed(b.ctl)) return;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < b.N; q += stride) {
        const int v = view_of(b.goff, b.V, q);   // the views' grains stay in their ranges
        const long long i = vals[q];
        const u64 key = keys[q];
        long long p = q;
        bool twin = false, crowded = false;
        if (bit0 > 0) {
            int steps = 0;
            for (long long j = q - 1; j >= 0 && (keys[j] >> bit0) == (key >> bit0); --j) {
                p -= keys[j] > key;
                twin |= keys[j] == key;
                if ((crowded = ++steps > CROWD)) break;
            }
            for (long long j = q + 1; j < b.N && (keys[j] >> bit0) == (key >> bit0); ++j) {
                p += keys[j] < key;
                if ((crowded |= ++steps > CROWD)) break;
            }
        } else {
            twin = q > b.goff[v] && keys[q - 1] == key;
            if (watch && q + CROWD + 1 < b.N && (keys[q + CROWD + 1] >> watch) == (key >> watch)) b.ctl->crowded = 1;
        }
        if (crowded) {
            atomicOr(&b.ctl->error, ERRB_CROWDED);
            continue;
        }
        const int z = (int)(key & ((1ull << b.cbits[2]) - 1ull));   // the key holds the coordinates
        const int y = (int)((key >> b.cbits[2]) & ((1ull << b.cbits[1]) - 1ull));
        const int x = (int)((key >> (b.cbits[1] + b.cbits[2])) & ((1ull << b.cbits[0]) - 1ull));
        b.gr[p] = make_int4(x, y, z, (int)(i - b.goff[v]));
        if (twin) atomicOr(&b.ctl->error, ERRB_DUPLICATE);
        atomicAdd(&count[cell_x(b, v, x, y, z)], 1u);
        if (b.dual) atomicAdd(&count_y[cell_y(b, v, x, y, z)], 1u);
    }
}

// Scatter of the canonical order into the cell lists: a grain takes the next
// slot of its cells (the cursors begin as the cell starts; the y-row list's
// positions begin at N).
__global__ void k_cell_scatter(Batch b, u32 *cursor, u32 *cursor_y) {
    griddep_launch();
    griddep_wait();
    if (input_failed(b.ctl)) return;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x; p < b.N; p += stride) {
        const int v = view_of(b.goff, b.V, p);
        const int4 g = b.gr[p];
        const u32 q = atomicAdd(&cursor[cell_x(b, v, g.x, g.y, g.z)], 1u);
        b.gc[q] = make_int4(g.x, g.y, g.z, (int)p);
        b.gp[q] = pack_xyz(g.x, g.y, g.z);
        if (b.dual) {
            const u32 qy = atomicAdd(&cursor_y[cell_y(b, v, g.x, g.y, g.z)], 1u);
            b.gc[qy] = make_int4(g.x, g.y, g.z, (int)p);
            b.gp[qy] = pack_xyz(g.x, g.y, g.z);
        }
    }
}

unsigned grid_for(long long n, int threads) {
    long long g = (n + threads - 1) / threads;
    if (g < 1) g = 1;
    if (g > 152 * 32) g = 152 * 32;
    return (unsigned)g;
}

}  // namespace

void launch_canonical_keys(const Batch &b, u64 *keys, u32 *vals, cudaStream_t st) {
    launch_dep(k_canonical_keys, dim3(grid_for(b.N, 256)), dim3(256), 0, st, b, keys, vals);
}

void launch_canonical_order(const Batch &b, const u64 *keys, const u32 *vals, u32 *count, u32 *count_y, int bit0,
                            int watch, cudaStream_t st) {
    launch_dep(k_canonical_order, dim3(grid_for(b.N, 256)), dim3(256), 0, st, b, keys, vals, count, count_y, bit0, watch);
}

void launch_cell_scatter(const Batch &b, u32 *cursor, u32 *cursor_y, cudaStream_t st) {
    launch_dep(k_cell_scatter, dim3(grid_for(b.N, 256)), dim3(256), 0, st, b, cursor, cursor_y);
}

}  // namespace et
