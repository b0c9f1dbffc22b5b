// step2d.cu -- dispatch of the 2D step: which compiled kernel a (precision,
// scheme, variant, frames, mode) launches.  The kernels are in
// step2d_kernel.cuh (FP32, FP64) and step2d_c.cu (the compensated state).
#include "step2d_launch.cuh"

namespace pf {

namespace {

constexpr int STRIP = 64;  // columns a warp holds: the only compiled block_x

template <typename F> auto by_scheme(int prec, int scheme, F f) -> decltype(f.template operator()<float, S10>()) {
    if (prec == 0) {
        if (scheme == S10) return f.template operator()<float, S10>();
        if (scheme == S21) return f.template operator()<float, S21>();
        if (scheme == SBAR21) return f.template operator()<float, SBAR21>();
    } else {
        if (scheme == S10) return f.template operator()<double, S10>();
        if (scheme == S21) return f.template operator()<double, S21>();
        if (scheme == SBAR21) return f.template operator()<double, SBAR21>();
    }
    return {};
}

struct Launch {
    const Step2DArgs& a;
    int grid;
    cudaStream_t st;
    template <typename T, int S> bool operator()() const { return step2d_launch<T, S>(a, grid, st); }
};
struct Occupancy {
    int var, fr, mode;
    template <typename T, int S> int operator()() const { return step2d_occupancy<T, S>(var, fr, mode); }
};
struct Bounds {
    unsigned long long* count;
    int* line;
    template <typename T, int S> int operator()() const { return step2d_bounds<T, S>(count, line); }
};

}  // namespace

// totals over the units; the first line of the first unit that has one
int bounds_step2d(unsigned long long* count, int* line) {
    *count = 0;
    *line = 0;
    int rc = 0;
    for (int prec = 0; prec < 2; ++prec)
        for (int scheme : {S10, S21, SBAR21}) {
            unsigned long long c = 0;
            int l = 0;
            const int r = by_scheme(prec, scheme, Bounds{&c, &l});
            if (r < 0) return r;
            rc = r;
            *count += c;
            if (*line == 0) *line = l;
        }
    return rc;
}

// The 2D kernel is warp-granular: `bx` must be 64 (columns a warp holds) and
// `grid` counts warps.
bool launch_step2d(int prec, int scheme, int bx, int grid, cudaStream_t st, const WorkItem* work, int n_work,
                   const InstRec* recs, int lp, StepClock clk, int var, int fr, int mode) {
    if (bx != STRIP) return false;
    const Step2DArgs a{work, n_work, recs, lp, clk, var, fr, mode};
    if (prec == 2) return step2c_launch(scheme, a, grid, st);
    return by_scheme(prec, scheme, Launch{a, grid, st});
}

// Warps of the fused kernel (mode 0) or of a pass of the two-kernel form
// resident on one SM (0 if not compiled).
int occupancy_step2d(int prec, int scheme, int bx, int var, int fr, int mode) {
    if (bx != STRIP) return 0;
    if (prec == 2) return mode == 0 ? step2c_occupancy(scheme, var) : 0;
    return by_scheme(prec, scheme, Occupancy{var, fr, mode});
}

}  // namespace pf
