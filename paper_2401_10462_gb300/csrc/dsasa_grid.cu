// Cell-list build for the neighbour search (input preparation and binning).
//
// Atoms are binned per molecule into cells of edge >= 2 R_max + skin + slack along y and z and a
// quarter of that along x, so that every pair of overlapping balls |p_i - p_j| < R_i + R_j lies in
// the same or adjacent rows of cells.  The binning is a counting sort in four kernels that start early behind one another (programmatic
// dependent launch): input pass, bounding boxes and grids (the last block makes the grids, so
// nothing waits); counts; starts; scatter.  The neighbour search reads runs of cells that are
// adjacent along x, so only the cells of one row (fixed y, z) need consecutive starts:
// a row takes its place in the sorted order with one atomic add and needs no scan over all
// cells.  (A batch is built in nine kernels, with its grids and a scan over all cells in
// kernels of their own.)  The order of rows and of the atoms inside a cell is not deterministic, which is
// harmless because each atom later sorts its candidate list by (plane distance, atom index).
// The sorted float4 copy (x, y, z, R) gives coalesced neighbour-tile loads in the atom kernel.
// Bound: the latency of the dependent launches and of their atomics.
#include "dsasa_kernels.cuh"
#include "dsasa_math.cuh"

#include <math.h>

namespace dsasa {

namespace {

__device__ __forceinline__ unsigned fenc(float f) {
    unsigned u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float fdec(unsigned u) {
    return __uint_as_float((u & 0x80000000u) ? (u & 0x7fffffffu) : ~u);
}

// The box of a molecule in 7 words that atomicMax grows from zero: ~min x y z, max x y z, max R
// (fenc of a finite float is above zero, and so is its complement).
__device__ __forceinline__ void box_words(float4 f, unsigned* w) {
    w[0] = ~fenc(f.x); w[1] = ~fenc(f.y); w[2] = ~fenc(f.z);
    w[3] = fenc(f.x); w[4] = fenc(f.y); w[5] = fenc(f.z);
    w[6] = fenc(f.w);
}

// atom i's input pass: inflated radius, float copies; non-finite inputs are replaced and reported
__device__ __forceinline__ float4 prep_atom(const BuildArgs& a, int i, int m) {
    double x = a.xyz[3 * i], y = a.xyz[3 * i + 1], z = a.xyz[3 * i + 2];
    double R = a.radii[i] + a.probe;
    if (!(isfinite(x) && isfinite(y) && isfinite(z) && isfinite(R)) || !(R > 0.0)) {
        atomicOr(a.status, ST_INPUT);
        x = y = z = 0.0;
        R = 1.0;
    }
    a.R[i] = R;
    const float h = (float)R;
    a.Rhl[i] = make_float2(h, (float)(R - (double)h));
    a.ad[i] = AtomD{x, y, z, R};
    a.gh[i] = ghost_hf(R);
    a.molid[i] = m;
    const float4 f = make_float4((float)x, (float)y, (float)z, h);
    a.f4[i] = f;
    return f;
}

// the molecule of atom i: the last m with offsets[m] <= i
__device__ __forceinline__ int molecule_of(const long long* offsets, int n_mol, int i) {
    int lo = 0, hi = n_mol - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (offsets[mid] <= i) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// Grid of one molecule from its box (box_words) and atom count: cell size and dimensions; the
// cell count is returned in base, with one more entry per row of cells for the row's end (-1: no
// edge makes a grid of the box).  No axis may be cut off at its limit of cells: the neighbour search
// relies on an atom lying within its cell.
constexpr float AXIS_CELLS = 1e6f;
__device__ MolGrid make_grid(const unsigned* bb, long long nm, double skin, int cube_limit) {
    MolGrid g;
    if (nm <= 0) {
        for (int k = 0; k < 3; ++k) { g.lo[k] = 0.f; g.dims[k] = 0; }
        g.inv_cell = 1.f;
        g.margin = g.fuzz = 0.f;
        g.rmax = 0.f;
        g.base = g.cubes = 0;
        return g;
    }
    float lo[3], hi[3], amax = 0.f;
    for (int k = 0; k < 3; ++k) {
        lo[k] = fdec(~bb[k]);
        hi[k] = fdec(bb[3 + k]);
        amax = fmaxf(amax, fmaxf(fabsf(lo[k]), fabsf(hi[k])));
    }
    float rmax = fdec(bb[6]);
    // float rounding of coordinates (|x| 2^-24 each), of the difference and of R: slack
    float margin = 1e-5f + 4.0e-7f * (amax + 16.0f);
    float cell = 2.0f * rmax + (float)skin + 2.0f * margin + 1e-3f;
    double cap = 8.0 * (double)nm + 64.0;
    int dims[3];
    double prod = 1.0;
    // the edge grows until the cells fit `cap` and every axis its limit (`axis` times AXIS_CELLS)
    const auto fit = [&](float& edge, float xf, int ends, float axis) {
        for (int it = 0; it < 64; ++it) {
            float longest = 0.f;
            prod = 1.0;
            for (int k = 0; k < 3; ++k) {
                const float d = (hi[k] - lo[k]) / edge * (k == 0 ? xf : 1.f);
                longest = fmaxf(longest, d);
                dims[k] = (int)fminf(d, AXIS_CELLS) + 1;
                prod *= dims[k] + (k == 0 ? ends : 0);
            }
            longest /= axis * AXIS_CELLS;
            if (prod <= cap && longest <= 1.f) return true;
            edge *= (float)fmax(1.01, fmax(cbrt(prod / cap), (double)longest) * 1.01);
        }
        return false;
    };
    g.cubes = 0;
    if (cube_limit > 0) {   // (only where the caller set a limit of his own)
        float edge = cell;
        fit(edge, 1.f, 0, INFINITY);
        g.cubes = (int)prod;
        cap = fmin(cap, (double)cell_store(g.cubes));
    }
    const bool fits = fit(cell, (float)GRID_XF, 1, 1.f);
    for (int k = 0; k < 3; ++k) { g.lo[k] = lo[k]; g.dims[k] = dims[k]; }
    g.inv_cell = 1.0f / cell;
    g.fuzz = margin;
    g.margin = margin + (float)skin;   // candidates within R_i + R_j + skin (Verlet lists)
    g.rmax = rmax;
    g.base = fits ? (dims[0] + 1) * dims[1] * dims[2] : -1;
    return g;
}

__device__ __forceinline__ int cell_of(const MolGrid& g, float4 f) {
    int cx = min(max((int)floorf((f.x - g.lo[0]) * (g.inv_cell * GRID_XF)), 0), g.dims[0] - 1);
    int cy = min(max((int)floorf((f.y - g.lo[1]) * g.inv_cell), 0), g.dims[1] - 1);
    int cz = min(max((int)floorf((f.z - g.lo[2]) * g.inv_cell), 0), g.dims[2] - 1);
    return grid_row(g, cz, cy) + cx;
}

// a user's limit is exceeded by so many cubic cells
__device__ __forceinline__ bool refused(const BuildArgs& a, int cubes) { return a.cube_limit > 0 && cubes > a.cube_limit; }
// the cells of one molecule's grid from make_grid, or more than there may be
__device__ __forceinline__ int cells_or_refused(const BuildArgs& a, const MolGrid& g) {
    return refused(a, g.cubes) || g.base < 0 ? a.max_cells + 1 : g.base;
}

constexpr int PREP_T = 256;
constexpr int SCAN_V = 16, SCAN_TILE = PREP_T * SCAN_V;   // cells that a thread / a block of a scan takes
__host__ __device__ constexpr int tiles_of(int cells) { return cells / SCAN_TILE + (cells % SCAN_TILE != 0); }

// Rows of more than LONG_ROW cells (a fibre along x) are not scanned by one warp each but in tiles
// by whole blocks, whose sums the counting pass gathers.  A warp takes about 0.2 us for 32 cells, so
// 7 us for the longest row that it gets.  Whole calls on 130,000 atoms in one row, with one warp a
// row / with tiles: 280,000 cells 2893 / 646 us, a million cells 9297 / 625 us; 5,000 atoms in a row of
// 11,000 cells 110 / 61 us.
constexpr int LONG_ROW = 1024;

// the words that must be zero later in this call (thread t of nt): the counts of the cells that the
// grids can have (8 per atom and 64 per molecule) ...
__device__ __forceinline__ void clear_counts(const BuildArgs& a, int t, int nt) {
    const int words = min(8 * a.n + 64 * a.n_mol, a.max_cells);
    for (int k = t; k < words / 4; k += nt) ((int4*)a.counts)[k] = make_int4(0, 0, 0, 0);
    if (t < words % 4) a.counts[words - 1 - t] = 0;
    for (int k = t; k < tiles_of(words); k += nt) a.blocksums[k] = 0;
}
// ... and, for the next calls, the skin test's scratch, and the deferred counts of the atom kernels
__device__ __forceinline__ void clear_words(const BuildArgs& a, int t, int nt) {
    if (a.test_words)
        for (int k = t; k < a.test_n; k += nt) a.test_words[k] = 0;
    if (t < 2 && a.zero_word) a.zero_word[t] = 0;
}

// exclusive sum of v over the block's threads (in thread order) and the total
__device__ void block_excl_scan(int v, int& ev, int& tv) {
    __shared__ int sv[PREP_T / 32];
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    int x = v;
    for (int o = 1; o < 32; o <<= 1) {
        const int p = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += p;
    }
    if (lane == 31) sv[wp] = x;
    __syncthreads();
    int pv = 0;
    tv = 0;
    for (int k = 0; k < PREP_T / 32; ++k) {
        if (k == wp) pv = tv;
        tv += sv[k];
    }
    ev = pv + x - v;
    __syncthreads();
}

// Input pass and bounding boxes.  GRIDS: the block that finishes last makes the grid.
template <bool GRIDS>
__global__ void __launch_bounds__(PREP_T) k_prep(BuildArgs a) {
    grid_dep_trigger();
    grid_dep_wait();
    const int tid = threadIdx.x, lane = tid & 31;
    if (GRIDS && blockIdx.x == 0) clear_words(a, tid, PREP_T);
    if (a.skip && *a.skip) return;
    clear_counts(a, blockIdx.x * PREP_T + tid, gridDim.x * PREP_T);
    __shared__ unsigned bb[7];
    __shared__ bool last;
    if (tid < 7) bb[tid] = 0;
    __syncthreads();
    const int i0 = blockIdx.x * PREP_T, i = i0 + tid;
    // one molecule in the whole block: its box is gathered in shared memory first
    int m = 0, mb = 0;
    bool one = true;
    if (a.offsets) {
        const int i1 = min(i0 + PREP_T, a.n) - 1;
        mb = molecule_of(a.offsets, a.n_mol, i0);
        one = a.offsets[mb + 1] > i1;
        m = one ? mb : molecule_of(a.offsets, a.n_mol, min(i, a.n - 1));
    }
    unsigned w[7] = {0, 0, 0, 0, 0, 0, 0};
    if (i < a.n) box_words(prep_atom(a, i, m), w);
    if (one) {
        for (int k = 0; k < 7; ++k) {
            const unsigned v = __reduce_max_sync(0xffffffffu, w[k]);
            if (lane == 0) atomicMax(&bb[k], v);
        }
        __syncthreads();
        if (tid < 7) atomicMax(a.bbox + 8 * mb + tid, bb[tid]);
    } else if (i < a.n) {
        for (int k = 0; k < 7; ++k) atomicMax(a.bbox + 8 * m + k, w[k]);
    }
    if constexpr (!GRIDS) return;
    __threadfence();
    __syncthreads();
    if (tid == 0) last = atomicAdd(a.sync + BUILD_TICKET, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last || tid != 0) return;
    __threadfence();
    unsigned bx[7];
    for (int k = 0; k < 7; ++k) bx[k] = __ldcg(a.bbox + k);
    MolGrid g = make_grid(bx, a.n, a.skin, a.cube_limit);
    const int cells = cells_or_refused(a, g);
    g.base = 0;
    a.sync[BUILD_ROWS] = (unsigned)(g.dims[1] * g.dims[2]);
    a.sync[BUILD_CURSOR] = 0u;
    *a.ncells_out = cells;
    if (cells > a.max_cells) {   // an empty grid keeps every index in range
        for (int k = 0; k < 3; ++k) g.dims[k] = 0;
        atomicOr(a.status, ST_GRID_OVF);
    }
    a.grids[0] = g;
}

// batches: the boxes and the words of clear_words cleared (this call's boxes may lie where another
// batch, with other molecules, or a single molecule left its own)
__global__ void k_bbox_init(BuildArgs a) {
    grid_dep_trigger();
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    clear_words(a, m, gridDim.x * blockDim.x);
    if (m >= a.n_mol) return;
    for (int k = 0; k < 8; ++k) a.bbox[8 * m + k] = 0;
}

// batches: each molecule's grid, its cell count in base
__global__ void k_grid_local(BuildArgs a) {
    grid_dep_trigger();
    grid_dep_wait();
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= a.n_mol) return;
    a.grids[m] = make_grid(a.bbox + 8 * m, a.offsets[m + 1] - a.offsets[m], a.skin, a.cube_limit);
}

// batches: the first cell of each molecule (one block)
__global__ void __launch_bounds__(PREP_T) k_grid_scan(BuildArgs a) {
    grid_dep_trigger();
    grid_dep_wait();
    int cells = 0, cubes = 0;
    bool none = false;   // some molecule has no grid
    for (int m0 = 0; m0 < a.n_mol; m0 += PREP_T) {
        const int m = m0 + threadIdx.x;
        if (a.cube_limit > 0) {
            int e, tot;
            block_excl_scan(m < a.n_mol ? a.grids[m].cubes : 0, e, tot);
            cubes += tot;
        }
        const int own = m < a.n_mol ? a.grids[m].base : 0, v = max(own, 0);
        none |= __syncthreads_or(own < 0) != 0;
        int e, tot;
        block_excl_scan(v, e, tot);
        if (m < a.n_mol) {
            const bool fits = own >= 0 && cells + e + v <= a.max_cells;   // (reported below; an empty grid keeps every index in range)
            a.grids[m].base = fits ? cells + e : 0;
            if (!fits)
                for (int k = 0; k < 3; ++k) a.grids[m].dims[k] = 0;
        }
        cells += tot;
    }
    if (threadIdx.x == 0) {
        if (refused(a, cubes) || none) cells = a.max_cells + 1;
        *a.ncells_out = cells;
        if (cells > a.max_cells) atomicOr(a.status, ST_GRID_OVF);
    }
}

// each atom's cell and its rank there; the single-molecule build's box and ticket are zero again
// afterwards
__global__ void k_count(BuildArgs a) {
    grid_dep_trigger();
    grid_dep_wait();
    if (a.skip && *a.skip) return;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (blockIdx.x == 0) {
        if (threadIdx.x < 8) a.bbox[threadIdx.x] = 0;
        if (threadIdx.x == 8) a.sync[BUILD_TICKET] = 0u;
    }
    if (i >= a.n || *a.ncells_out > a.max_cells) return;
    const MolGrid g = a.grids[a.molid[i]];
    const int c = cell_of(g, a.f4[i]);
    a.cell[i] = c;
    a.rank[i] = atomicAdd(&a.counts[c], 1);
    if (!a.offsets && g.dims[0] > LONG_ROW) {
        // one molecule with long rows: the sums of the tiles (atoms next to one another often share one)
        const int lanes = a.n - (i & ~31);
        const unsigned same = __match_any_sync(lanes >= 32 ? 0xffffffffu : (1u << lanes) - 1u, c / SCAN_TILE);
        if ((threadIdx.x & 31) == __ffs(same) - 1) atomicAdd(&a.blocksums[c / SCAN_TILE], __popc(same));
    }
}

// the starts of a tile's cells, `before` atoms lying in the tiles before it
__device__ __forceinline__ void scan_tile(const BuildArgs& a, int tile, int used, int before) {
    const int base = tile * SCAN_TILE + threadIdx.x * SCAN_V;
    int v[SCAN_V], s = 0, e, tot;
    for (int k = 0; k < SCAN_V; ++k) {
        v[k] = (base + k < used) ? a.counts[base + k] : 0;
        s += v[k];
    }
    block_excl_scan(s, e, tot);
    int pre = before + e;
    for (int k = 0; k < SCAN_V; ++k) {
        if (base + k < used) a.cstart[base + k] = pre;
        pre += v[k];
    }
}

// one molecule: the starts of every row's cells, one warp per row (long rows: one block per tile)
__global__ void __launch_bounds__(PREP_T) k_rows(BuildArgs a) {
    grid_dep_trigger();
    grid_dep_wait();
    if (a.skip && *a.skip) return;
    const int used = *a.ncells_out;
    if (used > a.max_cells) return;
    const int d0 = a.grids[0].dims[0];
    if (d0 > LONG_ROW) {
        // (a cell's end is the next one's start, as for a row's last cell the entry after it, which is empty)
        for (int tile = blockIdx.x; tile < tiles_of(used); tile += gridDim.x) {
            int s = 0, e, before;
            for (int k = threadIdx.x; k < tile; k += PREP_T) s += a.blocksums[k];
            block_excl_scan(s, e, before);
            scan_tile(a, tile, used, before);
        }
        return;
    }
    const int rows = (int)a.sync[BUILD_ROWS];
    const int lane = threadIdx.x & 31;
    for (int r = (blockIdx.x * PREP_T + threadIdx.x) >> 5; r < rows; r += gridDim.x * (PREP_T / 32)) {
        const int c0 = r * (d0 + 1);
        int tot = 0;
        for (int x = lane; x < d0; x += 32) tot += a.counts[c0 + x];
        tot = __reduce_add_sync(0xffffffffu, tot);
        int pos = 0;
        if (lane == 0) pos = (int)atomicAdd(a.sync + BUILD_CURSOR, (unsigned)tot);
        pos = __shfl_sync(0xffffffffu, pos, 0);
        for (int x0 = 0; x0 <= d0; x0 += 32) {   // entry d0: the row's end
            const int x = x0 + lane;
            const int v = x < d0 ? a.counts[c0 + x] : 0;
            int y = v;
            for (int o = 1; o < 32; o <<= 1) {
                const int p = __shfl_up_sync(0xffffffffu, y, o);
                if (lane >= o) y += p;
            }
            if (x <= d0) a.cstart[c0 + x] = pos + y - v;
            pos += __shfl_sync(0xffffffffu, y, 31);
        }
    }
}

// batches: exclusive scan of the counts of the cells in use into cstart (three kernels)
__global__ void __launch_bounds__(PREP_T) k_scan_reduce(BuildArgs a, int* bsum) {
    grid_dep_trigger();
    grid_dep_wait();
    const int used = min(*a.ncells_out, a.max_cells), base = blockIdx.x * SCAN_TILE + threadIdx.x * SCAN_V;
    if (blockIdx.x >= tiles_of(used)) return;
    int s = 0, e, tot;
    for (int k = 0; k < SCAN_V; ++k) s += (base + k < used) ? a.counts[base + k] : 0;
    block_excl_scan(s, e, tot);
    if (threadIdx.x == 0) bsum[blockIdx.x] = tot;
}
__global__ void __launch_bounds__(PREP_T) k_scan_top(BuildArgs a, int* bsum) {
    grid_dep_trigger();
    grid_dep_wait();
    const int nb = tiles_of(min(*a.ncells_out, a.max_cells));
    int carry = 0;
    for (int b0 = 0; b0 < nb; b0 += PREP_T) {
        const int b = b0 + threadIdx.x;
        int e, tot;
        block_excl_scan(b < nb ? bsum[b] : 0, e, tot);
        if (b < nb) bsum[b] = carry + e;
        carry += tot;
    }
}
__global__ void __launch_bounds__(PREP_T) k_scan_down(BuildArgs a, const int* bsum) {
    grid_dep_trigger();
    grid_dep_wait();
    const int used = min(*a.ncells_out, a.max_cells);
    if (blockIdx.x < tiles_of(used)) scan_tile(a, blockIdx.x, used, bsum[blockIdx.x]);
}

__global__ void k_scatter(BuildArgs a) {
    grid_dep_trigger();
    grid_dep_wait();
    if (a.skip && *a.skip) return;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= a.n) return;
    const int pos = *a.ncells_out > a.max_cells ? i : a.cstart[a.cell[i]] + a.rank[i];
    a.sidx[pos] = i;
    a.sf4[pos] = a.f4[i];
}

// The whole build for one molecule of at most kSmallAtoms atoms in one block: below that size
// the launches of the four kernels cost more than their width gains (whole calls, areas + gradient:
// 2,048 atoms in one block 88 us, 2,049 with the four kernels 93).  The line is where a thread
// would take a third atom and the counts more than 66 KB of shared memory.  Same grid, same cells;
// counts in shared memory, starts by one scan over all cells (which also ends every row where
// the next one starts).
constexpr int kSmallT = 1024, kSmallAtoms = 2 * kSmallT, kSmallCells = 8 * kSmallAtoms + 64;
__global__ void __launch_bounds__(kSmallT) k_build_small(BuildArgs a) {
    grid_dep_trigger();
    grid_dep_wait();
    clear_words(a, threadIdx.x, kSmallT);
    if (a.skip && *a.skip) return;
    __shared__ unsigned bb[7];
    __shared__ MolGrid g;
    __shared__ int ws[kSmallT / 32];
    extern __shared__ int cnt[];   // kSmallCells + 1
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    if (tid < 7) bb[tid] = 0;
    __syncthreads();
    float4 f[2];
    unsigned bw[7] = {0, 0, 0, 0, 0, 0, 0};
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int i = tid + h * kSmallT;
        if (i < a.n) {
            f[h] = prep_atom(a, i, 0);
            unsigned v[7];
            box_words(f[h], v);
            for (int k = 0; k < 7; ++k) bw[k] = max(bw[k], v[k]);
        }
    }
    for (int k = 0; k < 7; ++k) {
        const unsigned v = __reduce_max_sync(0xffffffffu, bw[k]);
        if (lane == 0) atomicMax(&bb[k], v);
    }
    __syncthreads();
    if (tid == 0) {
        MolGrid gg = make_grid(bb, a.n, a.skin, a.cube_limit);
        const int ncells = cells_or_refused(a, gg);
        gg.base = 0;
        if (ncells > a.max_cells) {   // an empty grid keeps every index in range
            for (int k = 0; k < 3; ++k) gg.dims[k] = 0;
            atomicOr(a.status, ST_GRID_OVF);
        }
        g = gg;
        a.grids[0] = gg;
        *a.ncells_out = ncells;
    }
    __syncthreads();
    const bool ovf = g.dims[0] == 0;
    const int ncells = (g.dims[0] + 1) * g.dims[1] * g.dims[2];
    for (int c = tid; c <= ncells; c += kSmallT) cnt[c] = 0;
    __syncthreads();
    int cell[2], rank[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        if (tid + h * kSmallT < a.n && !ovf) {
            cell[h] = cell_of(g, f[h]);
            rank[h] = atomicAdd(&cnt[cell[h]], 1);
        }
    }
    __syncthreads();
    // exclusive scan of the counts: each thread scans a contiguous run of cells, one block scan
    // over the run totals
    const int per = (ncells + 1 + kSmallT - 1) / kSmallT;
    const int c0 = min(tid * per, ncells + 1), c1 = min(c0 + per, ncells + 1);
    int run = 0;
    for (int c = c0; c < c1; ++c) run += cnt[c];
    int x = run;
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) ws[w] = x;
    __syncthreads();
    if (w == 0) {
        int t = ws[lane];
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t += y;
        }
        ws[lane] = t;
    }
    __syncthreads();
    int pre = (w > 0 ? ws[w - 1] : 0) + x - run;
    for (int c = c0; c < c1; ++c) {
        const int v = cnt[c];
        if (c < ncells) a.cstart[c] = pre;
        cnt[c] = pre;
        pre += v;
    }
    __syncthreads();
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int i = tid + h * kSmallT;
        if (i < a.n) {
            const int pos = ovf ? i : cnt[cell[h]] + rank[h];
            a.sidx[pos] = i;
            a.sf4[pos] = f[h];
        }
    }
}

cudaError_t launch_build_one(const BuildArgs& a, bool early, cudaStream_t s) {
    const int T = 256, nb = (a.n + T - 1) / T;
    static_assert(PREP_T == 256, "one thread per atom");
    cudaError_t e = launch_dependent(k_prep<true>, nb, PREP_T, s, early, a);
    if (e == cudaSuccess) e = launch_dependent(k_count, nb, T, s, true, a);
    // rows of cells: about one for every 32 atoms of a dense molecule; each warp takes several
    if (e == cudaSuccess) e = launch_dependent(k_rows, min(nb, 1216), T, s, true, a);
    if (e == cudaSuccess) e = launch_dependent(k_scatter, nb, T, s, true, a);
    note_launches(4);
    return e;
}

cudaError_t launch_build_batch(const BuildArgs& a, cudaStream_t s) {
    const int T = 256, nb = (a.n + T - 1) / T, mb = (a.n_mol + T - 1) / T;
    const int nt = (int)scan_scratch_ints(a.max_cells) - 1;   // (blocks past the cells in use return at once)
    cudaError_t e = launch_dependent(k_bbox_init, mb, T, s, false, a);
    if (e == cudaSuccess) e = launch_dependent(k_prep<false>, nb, PREP_T, s, true, a);
    if (e == cudaSuccess) e = launch_dependent(k_grid_local, mb, T, s, true, a);
    if (e == cudaSuccess) e = launch_dependent(k_grid_scan, 1, PREP_T, s, true, a);
    if (e == cudaSuccess) e = launch_dependent(k_count, nb, T, s, true, a);
    if (e == cudaSuccess) e = launch_dependent(k_scan_reduce, nt, PREP_T, s, true, a, a.blocksums);
    if (e == cudaSuccess) e = launch_dependent(k_scan_top, 1, PREP_T, s, true, a, a.blocksums);
    if (e == cudaSuccess) e = launch_dependent(k_scan_down, nt, PREP_T, s, true, a, (const int*)a.blocksums);
    if (e == cudaSuccess) e = launch_dependent(k_scatter, nb, T, s, true, a);
    note_launches(9);
    return e;
}

}  // namespace

size_t scan_scratch_ints(int max_cells) { return (size_t)tiles_of(max_cells) + 1; }

namespace {

constexpr int CHECK_T = 256;

// whether this block is the last of the grid to come here (every thread's writes before it are
// visible to the last block after it)
__device__ bool last_block(unsigned* ticket) {
    __shared__ bool last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    __syncthreads();
    if (last) __threadfence();
    return last;
}

// Verlet skin test (see dsasa_kernels.cuh): the largest displacement, any changed radius and the
// ticket are the words from VSTATE_TEST on; the last block decides.
__global__ void __launch_bounds__(CHECK_T) k_verlet_check(const double* xyz, const double* radii, const double* ref_xyz,
                                                          const double* ref_rad, int n, int valid, float lim2, int* vstate,
                                                          AtomD* ad, float4* f4) {
    grid_dep_trigger();
    const int i = blockIdx.x * CHECK_T + threadIdx.x;
    float d2 = 0.f;
    int changed = 0;
    if (valid && i < n) {
        const double x = xyz[3 * i], y = xyz[3 * i + 1], z = xyz[3 * i + 2];
        ad[i].x = x;
        ad[i].y = y;
        ad[i].z = z;
        f4[i] = make_float4((float)x, (float)y, (float)z, f4[i].w);
        double dx = x - ref_xyz[3 * i], dy = y - ref_xyz[3 * i + 1], dz = z - ref_xyz[3 * i + 2];
        double dd = dx * dx + dy * dy + dz * dz;
        d2 = (float)dd * (1.f + 1e-6f);   // rounded up: the test stays conservative
        if (!(dd == dd)) d2 = INFINITY;
        changed = radii[i] != ref_rad[i];
    }
    const unsigned d2max = __reduce_max_sync(0xffffffffu, __float_as_uint(d2));   // d2 >= 0: bits order as values
    changed = __reduce_or_sync(0xffffffffu, changed);
    int* word = vstate + VSTATE_TEST;
    if ((threadIdx.x & 31) == 0) {
        if (d2max) atomicMax((unsigned*)&word[0], d2max);
        if (changed) atomicOr(&word[1], 1);
    }
    if (!last_block((unsigned*)word + 2) || threadIdx.x != 0) return;
    const float dm = __uint_as_float((unsigned)__ldcg(word));
    const int reuse = valid && __ldcg(word + 1) == 0 && vstate[3] == 0 && dm <= lim2;
    vstate[2] = reuse;
    if (!reuse) vstate[3] = 0;   // the lists are rebuilt by this call
}

// The same test for a batch of resident molecules, per molecule m (atoms [off[m], off[m+1]),
// lists at arena slot base[m] + local index; base[m] < 0: no lists): words[0] is the ticket; of
// words 1 + 3m .. 3 + 3m the first is the largest squared displacement since the lists were built
// (float bits, rounded up), the second says that a radius changed, the third that some atom has no
// valid list (negative length).
__global__ void __launch_bounds__(CHECK_T) k_verlet_check_batch(const double* xyz, const double* radii,
                                                                const double* ref_xyz, const double* ref_rad,
                                                                const int* nbn, const long long* off,
                                                                const long long* base, int n, int n_mol, float lim2,
                                                                int* words, int* reuse) {
    grid_dep_trigger();
    int* vmol = words + 1;
    const int i = blockIdx.x * CHECK_T + threadIdx.x;
    int m = -1;
    unsigned d2b = 0;
    int changed = 0, none = 0;
    if (i < n) {
        m = molecule_of(off, n_mol, i);
        if (base[m] >= 0) {
            const size_t li = (size_t)(base[m] + (i - off[m]));
            const double dx = xyz[3 * i] - ref_xyz[3 * li], dy = xyz[3 * i + 1] - ref_xyz[3 * li + 1],
                         dz = xyz[3 * i + 2] - ref_xyz[3 * li + 2];
            const double dd = dx * dx + dy * dy + dz * dz;
            d2b = __float_as_uint(dd == dd ? (float)dd * (1.f + 1e-6f) : INFINITY);
            changed = radii[i] != ref_rad[li];
            none = nbn[li] < 0;
        }
    }
    // one atomic per warp where its atoms share a molecule
    const int m0 = __shfl_sync(0xffffffffu, m, 0);
    if (__all_sync(0xffffffffu, m == m0)) {
        d2b = __reduce_max_sync(0xffffffffu, d2b);
        changed = __reduce_or_sync(0xffffffffu, changed);
        none = __reduce_or_sync(0xffffffffu, none);
        if (threadIdx.x & 31) m = -1;
    }
    if (m >= 0) {
        if (d2b) atomicMax((unsigned*)&vmol[3 * m], d2b);
        if (changed) atomicOr(&vmol[3 * m + 1], 1);
        if (none) atomicOr(&vmol[3 * m + 2], 1);
    }
    if (!last_block((unsigned*)words)) return;
    for (int k = threadIdx.x; k < n_mol; k += CHECK_T) {
        reuse[k] = base[k] >= 0 && __ldcg(vmol + 3 * k + 1) == 0 && __ldcg(vmol + 3 * k + 2) == 0 &&
                   __uint_as_float((unsigned)__ldcg(vmol + 3 * k)) <= lim2;
    }
}

}  // namespace

cudaError_t launch_verlet_check_batch(const double* xyz, const double* radii, const double* ref_xyz,
                                      const double* ref_rad, const int* nbn, const long long* off,
                                      const long long* base, int n, int n_mol, double skin, int* vmol,
                                      int* reuse, cudaStream_t s) {
    const float lim2 = (float)(0.25 * skin * skin) * (1.f - 1e-6f);
    const int nb = n > 0 ? (n + CHECK_T - 1) / CHECK_T : 1;
    k_verlet_check_batch<<<nb, CHECK_T, 0, s>>>(xyz, radii, ref_xyz, ref_rad, nbn, off, base, n, n_mol, lim2, vmol, reuse);
    note_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_verlet_check(const double* xyz, const double* radii, const double* ref_xyz, const double* ref_rad,
                                int n, int valid, double skin, int* vstate, AtomD* ad, float4* f4,
                                cudaStream_t s) {
    // (skin / 2)^2, rounded down in float
    const float lim2 = (float)(0.25 * skin * skin) * (1.f - 1e-6f);
    const int nb = valid && n > 0 ? (n + CHECK_T - 1) / CHECK_T : 1;
    k_verlet_check<<<nb, CHECK_T, 0, s>>>(xyz, radii, ref_xyz, ref_rad, n, valid, lim2, vstate, ad, f4);
    note_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_build(const BuildArgs& a, cudaStream_t s) {
    if (a.n <= 0) return cudaSuccess;
    // (behind the skin test, the first kernel of the build starts early too)
    const bool early = a.skip != nullptr;
    if (a.n_mol == 1 && a.n <= kSmallAtoms) {
        constexpr size_t smem = sizeof(int) * (kSmallCells + 1);
        // idempotent, and needed once per context: above 48 KB a kernel has to ask
        cudaError_t e = cudaFuncSetAttribute(k_build_small, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        e = launch_dependent_smem(k_build_small, 1, kSmallT, smem, s, early, CARVEOUT_DEFAULT, a);
        note_launches(1);
        return e;
    }
    return a.n_mol == 1 ? launch_build_one(a, early, s) : launch_build_batch(a, s);
}

}  // namespace dsasa
