// FP32 instantiations of the per-atom kernels: the cell construction and classification of both
// precisions (FP32 -> FP64 -> exact predicates) and the mixed form's terms (see
// dsasa_atoms.cuh).
#include "dsasa_atoms.cuh"

namespace dsasa {

// Whether the cell construction and the classification run as one kernel: up to 20 atoms a
// multiprocessor (3,040 on a GB300), all resident at once.  There an atom's classification overlaps the
// slowest cells and one launch and the trip of the records through memory are saved; with more atoms the
// split kernels win, whose smaller instruction streams stay in the cache and which hold 32 warps (fused /
// split, us per call with the gradient: 304 atoms 66 / 80, 700 66 / 88, 1,200 110 / 131, 2,003 87 / 101,
// 3,000 96 / 116, 4,200 125 / 124).
bool cells_fused(int n) {
    static int cap = -1;
    if (cap < 0) {
        int dev = 0, sms = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        cap = 20 * sms;
    }
    return n <= cap;
}

// The cell records of every atom, classified (Steps 1 and 2).
cudaError_t launch_cells(const AtomArgs& a, cudaStream_t s) {
    AtomArgs fast = a;
    fast.work_list = nullptr;
    fast.work_count = nullptr;
    fast.ev = nullptr;
    auto mark = [&](int k) {
        if (a.ev) cudaEventRecord(a.ev[k], s);
    };
    auto nb = [&](int w) { return (a.n + w - 1) / w; };
    const bool small = cells_fused(a.n);
    AtomLaunch go{s, small ? CARVEOUT_SMALL : CARVEOUT_DEFAULT};
    if (!a.carry && small) {
        go(k_atoms<float, false, 64, 64, PH_CC>, nb(WARPS_CELL), WARPS_CELL * 32, fast);
        mark(0);
    } else {
        if (a.carry) {
            // the carried cells, then the cell kernel over the redo list (its grid covers every
            // atom; the warps past the list's length return at once)
            go(k_atoms<float, false, 64, 64, PH_CARRY>, nb(WARPS_CELL), WARPS_CELL * 32, fast);
            AtomArgs redo = fast;
            redo.work_list = a.redo_list;
            redo.work_count = a.redo_count;
            go(k_atoms<float, false, 64, 64, PH_CELL>, nb(WARPS_CELL), WARPS_CELL * 32, redo);
        } else {
            go(k_atoms<float, false, 64, 64, PH_CELL>, nb(WARPS_CELL), WARPS_CELL * 32, fast);
        }
        mark(0);
        go(k_class<WARPS_CLASS>, nb(WARPS_CLASS), WARPS_CLASS * 32, fast);
    }
    mark(1);
    return go.err;
}

cudaError_t launch_atoms_f32(const AtomArgs& a, bool grad, cudaStream_t s) { return launch_atoms_t<float>(a, grad, s); }
// bytes of one atom's cell record between the kernels
size_t cell_record_bytes() { return sizeof(CellRecF); }
}  // namespace dsasa
