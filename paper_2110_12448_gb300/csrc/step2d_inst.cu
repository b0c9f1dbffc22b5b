// step2d_inst.cu -- the 2D step kernels of one precision and one scheme:
// compiled once for each (PF_REAL, PF_SCHEME), so that the build runs them in
// parallel.  Launches and occupancy queries go through step2d.cu.
#include "step2d_kernel.cuh"
#include "step2d_launch.cuh"

namespace pf {

namespace {

PF_BOUNDS_READER(bounds_read)

template <typename T, int S> struct Table {
    using K = void (*)(const WorkItem*, int, const InstRec*, int, StepClock);
    template <int MODE> static K pick(int var, int fr) {
        if (var == 0) {
            if constexpr (MODE == 0) {
                if (fr == FR_ONE) return k_step2d<T, S, 0, FR_ONE, 0>;
                if (fr == FR_CELL) return k_step2d<T, S, 0, FR_CELL, 0>;
            }
            return nullptr;  // the two-kernel form runs at the T0 level (variant 1 or 2)
        }
        if (var == 1) {
            if (fr == FR_ONE) return k_step2d<T, S, 1, FR_ONE, MODE>;
            if (fr == FR_CELL) return k_step2d<T, S, 1, FR_CELL, MODE>;
            if (fr == FR_ANY) return k_step2d<T, S, 1, FR_ANY, MODE>;
        }
        if (var == 2) {
            if (fr == FR_ONE) return k_step2d<T, S, 2, FR_ONE, MODE>;
            if (fr == FR_CELL) return k_step2d<T, S, 2, FR_CELL, MODE>;
        }
        return nullptr;
    }
    static K get(int var, int fr, int mode) {
        return mode == 0 ? pick<0>(var, fr) : mode == 1 ? pick<1>(var, fr) : mode == 2 ? pick<2>(var, fr) : nullptr;
    }
};

}  // namespace

template <> bool step2d_launch<PF_REAL, PF_SCHEME>(const Step2DArgs& a, int grid, cudaStream_t st) {
    const auto k = Table<PF_REAL, PF_SCHEME>::get(a.var, a.fr, a.mode);
    if (!k) return false;
    launch_next(k, grid, 32, 0, st, a.work, a.n_work, a.recs, a.launch_parity, a.clk);
    return true;
}
template <> int step2d_occupancy<PF_REAL, PF_SCHEME>(int var, int fr, int mode) {
    const auto k = Table<PF_REAL, PF_SCHEME>::get(var, fr, mode);
    int n = 0;
    if (!k || cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, 32, 0) != cudaSuccess) return 0;
    return n;
}
template <> int step2d_bounds<PF_REAL, PF_SCHEME>(unsigned long long* count, int* line) { return bounds_read(count, line); }

}  // namespace pf
