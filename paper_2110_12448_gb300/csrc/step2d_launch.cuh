// step2d_launch.cuh -- the entry points that each (precision, scheme) unit of
// the 2D step kernels defines (step2d_inst.cu) and step2d.cu dispatches to.
#pragma once
#include "pf_internal.cuh"

namespace pf {

struct Step2DArgs {
    const WorkItem* work;
    int n_work;
    const InstRec* recs;
    int launch_parity;
    StepClock clk;
    int var, fr, mode;
};
// false (0) if the combination has no compiled kernel
template <typename T, int S> bool step2d_launch(const Step2DArgs& a, int grid, cudaStream_t st);
template <typename T, int S> int step2d_occupancy(int var, int fr, int mode);
template <typename T, int S> int step2d_bounds(unsigned long long* count, int* line);

#define PF_STEP2D_DECL(T, S)                                                            \
    template <> bool step2d_launch<T, S>(const Step2DArgs& a, int grid, cudaStream_t st); \
    template <> int step2d_occupancy<T, S>(int var, int fr, int mode);                  \
    template <> int step2d_bounds<T, S>(unsigned long long* count, int* line);
PF_STEP2D_DECL(float, S10)
PF_STEP2D_DECL(float, S21)
PF_STEP2D_DECL(float, SBAR21)
PF_STEP2D_DECL(double, S10)
PF_STEP2D_DECL(double, S21)
PF_STEP2D_DECL(double, SBAR21)
#undef PF_STEP2D_DECL

// the compensated state's kernel (step2d_c.cu)
bool step2c_launch(int scheme, const Step2DArgs& a, int grid, cudaStream_t st);
int step2c_occupancy(int scheme, int var);

}  // namespace pf
