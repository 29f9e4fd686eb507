// Shared declarations of the dSASA CUDA kernels (host side and device side).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <utility>

namespace dsasa {

// Programmatic dependent launch (the kernels of one call run back to back on one stream): a
// kernel launched by launch_dependent may be scheduled while the previous kernel of the
// stream is still running; it calls grid_dep_wait() before it touches anything, which returns
// once that kernel has completed and its writes are visible.  grid_dep_trigger() lets the
// next kernel be scheduled once every block of this one has started.  Both are no-ops for a
// kernel launched without the attribute.
#ifdef __CUDACC__
__device__ __forceinline__ void grid_dep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_dep_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
#endif
// How much of an SM's memory is shared memory rather than L1 cache, in percent (default: as the runtime
// decides for each kernel's occupancy).  A kernel cannot start beside one that runs with another split,
// so early launches need the same split along the chain.  Molecules small enough for the fused cell
// kernel leave most of an SM idle and gain from the overlap; larger ones need each kernel's own split
// (one split for all, 20k energy + forces: 372 - 400 us against 365, RNA areas 440 - 486 against 424).
constexpr int CARVEOUT_DEFAULT = -1, CARVEOUT_SMALL = 44;
template <class... K, class... A>
cudaError_t launch_dependent_smem(void (*kernel)(K...), int grid, int block, size_t smem, cudaStream_t s, bool early,
                                  int carveout, A&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = early ? 1 : 0;
    cfg.attrs = at;
    at[1].id = cudaLaunchAttributePreferredSharedMemoryCarveout;
    at[1].val.sharedMemCarveout = (unsigned)carveout;
    cfg.numAttrs = carveout < 0 ? 1 : 2;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);
}
template <class... K, class... A>
cudaError_t launch_dependent(void (*kernel)(K...), int grid, int block, cudaStream_t s, bool early, A&&... args) {
    return launch_dependent_smem(kernel, grid, block, 0, s, early, CARVEOUT_DEFAULT, std::forward<A>(args)...);
}

// host: adds k to the library-wide count of kernel launches (dsasa_kernel_launches)
void note_launches(int k);

// words of the single-molecule build's exchange area: the ticket of the input pass (zero before a
// build), the rows of the grid, and the cursor of the sorted order
enum { BUILD_TICKET = 0, BUILD_ROWS = 1, BUILD_CURSOR = 2, BUILD_SYNC_WORDS = 4 };

// device status bits (ORed by kernels, read by dsasa_status_sync)
enum : int {
    ST_CAND_OVF = 1,      // more overlapping neighbours than one warp's candidate table holds
    ST_TRI_OVF = 2,       // cell needed more vertex slots than available
    ST_UNRESOLVED = 4,    // exact expansion capacity exceeded
    ST_DEGENERATE = 8,    // a clip tie that Simulation of Simplicity cannot break (coincident atoms)
    ST_BADCELL = 16,      // inconsistent cell structure detected (atom output set to NaN)
    ST_INPUT = 32,        // non-finite input
    ST_EXPORT_OVF = 64,   // complex export buffer too small
    ST_GRID_OVF = 128,    // cell grid larger than its capacity
    ST_CHECK = 256        // a bounds check of the checked build failed (the access was redirected)
};

// The checked build (-DDSASA_CHECKED): every data-dependent index into a global array of
// atoms (sorted positions, neighbour entries, plane owners, work lists) is verified on the
// device.  A bad index sets ST_CHECK and is replaced by 0, so the access stays inside the
// array; the results of that call are then not to be used.  The normal build checks nothing.
#ifdef DSASA_CHECKED
__device__ __forceinline__ int ds_checked(int idx, int lim, int* status) {
    if ((unsigned)idx < (unsigned)lim) return idx;
    atomicOr(status, ST_CHECK);
    return 0;
}
#define DS_IDX(idx, lim, status) ds_checked((idx), (lim), (status))
#else
#define DS_IDX(idx, lim, status) (idx)
#endif

// An atom as the atom kernels read it in FP64: position and inflated radius in 32 bytes of device
// memory (the caller's coordinates may lie in host memory, and a neighbour's come as two 16-byte
// loads instead of four of 8)
struct alignas(32) AtomD {
    double x, y, z, R;
};
#ifdef __CUDACC__
__device__ __forceinline__ AtomD load_atom(const AtomD* p) {
    const double2 a = ((const double2*)p)[0], b = ((const double2*)p)[1];
    return {a.x, a.y, b.x, b.y};
}
#endif

// cell grid of one molecule, starting at `lo`: along y and z cells reach as far as any overlap (and
// the skin), so an atom's neighbours lie in its own row of cells and the eight around it; along x
// they are GRID_XF times shorter, so that a row's run can be cut close to the atom's reach
constexpr int GRID_XF = 4;
struct MolGrid {
    float lo[3];
    float inv_cell;   // 1 / edge along y and z (GRID_XF times that along x)
    int dims[3];
    int base;         // first global cell of this molecule
    float margin;     // conservative slack of the FP32 neighbour test (A)
    float rmax;       // largest probe-inflated radius of the molecule
    float fuzz;       // margin without the skin: bound of the FP32 error of a distance minus a sum of radii
    int cubes;        // cubic cells of the same edge in its box: what a user's max_cells bounds
};
// the first cell of row (z, y): a row holds dims[0] cells and one more entry for its end
__host__ __device__ inline int grid_row(const MolGrid& g, int z, int y) {
    return g.base + (z * g.dims[1] + y) * (g.dims[0] + 1);
}

#ifdef __CUDACC__
// The atoms that may lie within f.w + rmax + margin of atom f = (x, y, z, R) of the grid, as one index
// space 0 .. total - 1 over the runs of the nine rows of cells around it; called by a whole warp (buf:
// 32 ints of its shared memory).  Nine lanes look the runs up in one memory round trip, each cut to
// what the sphere can reach in its row: about 120 atoms of a globule in 4 full rounds of 32.  (Whole
// cells of the reach along x gave 200, row by row at 23 of 32 lanes, and three times the
// instructions; cells of half the reach in 25 rows gave 80, but their runs of four atoms spread
// every load over eight lines and more: slower than the nine whole rows.)
struct NearRows {
    int off, len, total, rows;
    int* buf;
    unsigned le;
    __device__ __forceinline__ NearRows(const MolGrid& G, const int* cstart, float4 f, int* b) : off(0), len(0), rows(0), buf(b) {
        const int lane = threadIdx.x & 31;
        const unsigned full = 0xffffffffu;
        int beg = 0;
        if (lane < 9) {
            const int z = min(max((int)floorf((f.z - G.lo[2]) * G.inv_cell), 0), G.dims[2] - 1) + lane / 3 - 1;
            const int y = min(max((int)floorf((f.y - G.lo[1]) * G.inv_cell), 0), G.dims[1] - 1) + lane % 3 - 1;
            if (z >= 0 && z < G.dims[2] && y >= 0 && y < G.dims[1]) {
                const float slack = 1e-3f + 2.f * G.fuzz;   // rounding of an atom's place in the grid
                const float cell = __frcp_rn(G.inv_cell), r = f.w + G.rmax + G.margin + slack;
                const float y0 = G.lo[1] + y * cell, z0 = G.lo[2] + z * cell;
                const float dy = fmaxf(fmaxf(y0 - f.y, f.y - (y0 + cell)) - slack, 0.f);
                const float dz = fmaxf(fmaxf(z0 - f.z, f.z - (z0 + cell)) - slack, 0.f);
                const float w2 = r * r - (dy * dy + dz * dz);
                if (w2 > 0.f) {
                    const float w = w2 * rsqrtf(w2) * 1.00001f + slack, ix = G.inv_cell * GRID_XF, x = f.x - G.lo[0];
                    const int x0 = max((int)floorf((x - w) * ix), 0), x1 = min((int)floorf((x + w) * ix), G.dims[0] - 1);
                    if (x0 <= x1) {
                        const int row = grid_row(G, z, y);
                        beg = cstart[row + x0];
                        len = cstart[row + x1 + 1] - beg;
                    }
                }
            }
        }
        const unsigned ne = __ballot_sync(full, len > 0);
        off = len;
#pragma unroll
        for (int o = 1; o < 16; o <<= 1) {
            const int p = __shfl_up_sync(full, off, o);
            if (lane >= o) off += p;
        }
        total = __shfl_sync(full, off, 8);
        off -= len;
        asm("mov.u32 %0, %%lanemask_le;" : "=r"(le));
        if (len > 0) buf[__popc(ne & (le >> 1))] = beg - off;
        __syncwarp();
    }
    // the lane's sorted position of indices f0 .. f0 + 31 (f0 = 0, 32, ... in turn; past total: any)
    __device__ __forceinline__ int at(int f0) {
        const int p = off - f0;
        const unsigned m = __reduce_or_sync(0xffffffffu, len > 0 && (unsigned)p < 32u ? 1u << p : 0u);
        const int r = rows + __popc(m & le) - 1;
        rows += __popc(m);
        return buf[r] + f0 + (int)(threadIdx.x & 31);
    }
};
#endif

struct BuildArgs {
    const double* xyz;
    const double* radii;
    double probe;
    int n;
    int n_mol;
    const long long* offsets;   // device, n_mol + 1 (NULL: one molecule)
    double skin;
    const int* skip;   // non-NULL and *skip != 0: the previous cell list is reused (nothing to do)
    int* zero_word;    // non-NULL: zero_word[0..1] set to 0 by the build's first kernel (the next atom
                       // kernels' deferred count, and a spare word)
    // The words that kernels count up start every call at zero whatever came before: a call that
    // overlapped another on the same scratch (which no caller may do) spoils itself, not the later
    // ones.  The counts of the cells are cleared before they are used; the box and the ticket of the
    // input pass and the skin test's words by a kernel of the same call after it.
    int* test_words;   // the skin test's scratch (test_n words), set to 0 by the build's first kernel
    int test_n;
    int max_cells;     // cells (and row ends) that counts and cstart hold
    int cube_limit;    // > 0: more cubic cells than this are refused (cell_store makes room for what they become)
    // outputs / scratch
    double* R;         // n
    float2* Rhl;       // n: R as a float pair (hi, lo), for the float-float area terms
    AtomD* ad;         // n: position and R
    float* gh;         // n: half-width of the atom's initial cell (ghost_h, exact in float)
    float4* f4;        // n  (x, y, z, R) float
    int* molid;        // n
    int* rank;         // n
    int* cell;         // n
    unsigned* bbox;    // n_mol * 8 (box words, pad); molecule 0's are zero before a build
    MolGrid* grids;    // n_mol
    int* counts;       // max_cells + 1, 16-byte aligned
    int* cstart;       // max_cells + 1
    int* sidx;         // n
    float4* sf4;       // n
    int* blocksums;    // scan_scratch_ints(max_cells): atoms in each run of SCAN_TILE cells (batches; long rows)
    unsigned* sync;    // BUILD_SYNC_WORDS
    int* status;
    int* ncells_out;   // device int: total cells used
};

struct AtomArgs {
    const double* xyz;
    const double* R;
    const float2* Rhl;      // R as (hi, lo) floats
    const AtomD* ad;        // position and R (of this call's coordinates, also when the lists are reused)
    const float* gh;        // half-width of the initial cell
    const float4* f4;       // (x, y, z, R) in float, by atom (current, like ad)
    const float4* sf4;
    const int* sidx;
    const int* molid;
    const int* cstart;
    const MolGrid* grids;
    const double* w;        // NULL = ones
    double* areas;
    double* grad;           // NULL = no gradient
    double* vol;            // per-atom volumes vol(B_i cap L_i); NULL = not computed
    double* vgrad;          // d(sum_i vw_i V_i) / dx (n x 3); NULL = not computed
    const double* vw;       // volume weights vw (n); NULL = ones (the union volume's gradient)
    // per-molecule completion (NULL = off; not with volumes): every atom adds 1 to
    // mol_done[molid] (device memory, zero at the start) once its area and gradient are final,
    // after a system-scope fence; the molecule's last atom then sets mol_ready[molid] = 1
    // (caller memory, which may be mapped host memory)
    int* mol_done;
    int* mol_ready;
    const long long* mol_off;   // batch offsets (n_mol + 1, device): molecule m is [off[m], off[m+1])
    // resident Verlet lists of a batch (NULL = none): molecule m's lists live at arena index
    // mol_base[m] + (i - mol_off[m]) with molecule-local entries (mol_base[m] < 0: no lists);
    // mol_reuse[m] != 0: reuse them; an atom whose list overflows marks its slot invalid
    const long long* mol_base;
    const int* mol_reuse;
    // the cell list holds the skin band too (skin > 0): keep only the balls that overlap B_i
    // now in the plane table
    int skin_band;
    // single-molecule calls with neighbour lists: the carry kernel keeps each atom's cell from
    // the previous call where it can (list-reusing calls) and appends the other atoms (sorted
    // positions) to redo_list, counted in *redo_count (zero when the kernels start); the cell
    // kernel then builds those
    int carry;
    int* redo_list;
    int* redo_count;
    int n;
    int* status;
    // complex export (NULL = off): records {i, v0, v1, v2, v3}
    int* rec;
    long long max_rec;
    unsigned long long* nrec;
    // deferral: the fast pass appends sorted positions it cannot hold to defer_list; the
    // large pass reads work_list[0 .. *work_count)
    int* defer_list;
    int* defer_count;       // zero when the first atom kernel starts (cleared by the cell-list build)
    const int* work_list;
    const int* work_count;
    // per-atom cell records (by sorted position) between the cell kernel and the terms
    // kernel; NULL = one fused kernel
    void* cells;
    // optional timing: events recorded on the stream after the cell, classification, terms
    // and large-capacity kernels (NULL = none)
    cudaEvent_t* ev;
    // Verlet neighbour lists (single molecule, skin > 0; NULL = none): candidates of atom i
    // at nbl[i * NBL_CAP .. + nbn[i]).  *reuse != 0: take the candidates from the lists (the
    // cell list was not rebuilt); else gather them from the cell list and store them with
    // the reference coordinates and radii.  Either way only the balls that overlap B_i at
    // the current positions enter the plane table.  *lists_bad is set when a list cannot
    // hold its atom's candidates (the next call rebuilds).
    int* nbl;
    int* nbn;
    const int* reuse;
    int* lists_bad;
    double* ref_xyz;
    double* ref_rad;
    const double* radii_in;
};
constexpr int NBL_CAP = 122;   // list capacity per atom (atoms within R_i + R_j + skin)

// Shrake-Rupley numerical SASA (cross-check): m unit vectors pts[3m] (device)
struct SRArgs {
    const double* xyz;
    const double* R;
    const float4* sf4;
    const int* sidx;
    const int* molid;
    const int* cstart;
    const MolGrid* grids;
    const float* pts;
    int m;
    int n;
    double* areas;
    int* exposed;                 // NULL = not written
    unsigned long long* tests;    // NULL = not counted: point-neighbour tests performed
    int* status;
};

cudaError_t launch_build(const BuildArgs& a, cudaStream_t s);
// Verlet skin test: vstate[2] = reuse the lists (valid, every atom within skin/2 of its
// reference position, radii unchanged, no list overflow); the positions go to ad and f4, which a
// build that is not needed does not write; vstate[3] overflow; VSTATE_TEST .. + VSTATE_TEST_N - 1
// scratch, which starts at zero (BuildArgs.test_words of the build that follows)
enum { VSTATE_TEST = 4, VSTATE_TEST_N = 3, VSTATE_WORDS = 8 };
cudaError_t launch_verlet_check(const double* xyz, const double* radii, const double* ref_xyz, const double* ref_rad,
                                int n, int valid, double skin, int* vstate, AtomD* ad, float4* f4,
                                cudaStream_t s);
// the Verlet skin test of a batch of resident molecules: reuse[m] for each molecule (see
// k_verlet_check_batch); vmol: 1 + 3 n_mol ints of scratch, which start at zero
cudaError_t launch_verlet_check_batch(const double* xyz, const double* radii, const double* ref_xyz,
                                      const double* ref_rad, const int* nbn, const long long* off,
                                      const long long* base, int n, int n_mol, double skin, int* vmol,
                                      int* reuse, cudaStream_t s);
cudaError_t launch_sr(const SRArgs& a, cudaStream_t s);
// the classified cell records of every atom (a.cells), for the terms of either precision
cudaError_t launch_cells(const AtomArgs& a, cudaStream_t s);
bool cells_fused(int n);   // (dsasa_atoms_f32.cu)
cudaError_t launch_atoms_f32(const AtomArgs& a, bool grad, cudaStream_t s);
cudaError_t launch_atoms_f64(const AtomArgs& a, bool grad, cudaStream_t s);
size_t scan_scratch_ints(int max_cells);
// entries that `cubes` cubic cells can become: a quarter as long along x, and an end for each row
__host__ __device__ inline int64_t cell_store(int64_t cubes) { return (GRID_XF + 1) * cubes; }
size_t cell_record_bytes();

}  // namespace dsasa
