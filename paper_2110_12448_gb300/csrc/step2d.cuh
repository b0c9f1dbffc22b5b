// step2d.cuh -- what the 2D step kernels share: scalar helpers, the packed pair
// of the two columns that a lane owns, and the row loads and stores.
#pragma once
#include "pf_internal.cuh"

namespace pf {

// A step kernel starts with after_previous(): its launch may begin before the
// kernel ahead of it on the stream has ended (launch_next), and it reads and
// writes nothing until that kernel has ended and its writes are there.  Its own
// successor may take free slots at once where there is at most a block per SM;
// larger grids leave that to their blocks' exit, because blocks that wait in the
// free slots of a half-full GPU are spread unevenly (1024^2: 14.4 us a step before,
// 12.8 so, 15.5 with a successor that waits beside it).  Fields and grain maps are
// read by plain loads: non-coherent ones (__ldg) are for memory that nothing
// writes while the kernel is there, and this one may be there while the kernel ahead
// still writes (no difference in time: 0-1.4 % on the step workloads).
constexpr int EARLY_GRID = 152;  // the SMs of GB300
__device__ __forceinline__ void after_previous() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (gridDim.x <= EARLY_GRID) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
// Launches a step kernel so (programmatic stream serialisation; a capture keeps
// it as an edge of the graph).  128^2: 6.2 -> 4.6 us a step; 200^2 FP64 72 -> 70;
// full grids gain under 1 %.
template <typename... P, typename... A>
void launch_next(void (*k)(P...), int grid, int threads, size_t smem, cudaStream_t st, A... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute early{};
    early.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    early.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &early;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, k, static_cast<P>(args)...);
}
namespace {

constexpr unsigned FULL = 0xffffffffu;

// ---------------------------------------------------------------------------
// scalar helpers: FP32 uses the single-instruction approximate reciprocal and
// base-2 exponential; FP64 uses IEEE operations
// ---------------------------------------------------------------------------
__device__ __forceinline__ float rcp_approx(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float ex2_approx(float x) {
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
template <typename T> struct M;
#ifndef PF_PRECISE_F32
template <> struct M<float> {
    // tanh(x / sqrt2) = 1 - 2 / (1 + e^{sqrt2 x}) = 1 - 2 / (1 + 2^{sqrt2 log2(e) x});
    // absolute error ~2e-7 over the whole range
    static __device__ __forceinline__ float tanh_isq2(float x) {
        const float e = ex2_approx(x * 2.0402788931935790f);  // sqrt2 * log2(e)
        return fmaf(-2.0f, rcp_approx(1.0f + e), 1.0f);
    }
    static __device__ __forceinline__ float rcp(float x) { return rcp_approx(x); }
    // single-instruction approximate square root (0 at 0): the App. B and
    // <10> anti-trapping magnitudes, guarded where |grad psi| vanishes
    static __device__ __forceinline__ float sqrt_(float x) {
        float r;
        asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
        return r;
    }
};
#else
// correctly rounded division and the library tanh (slower; for accuracy studies)
template <> struct M<float> {
    static __device__ __forceinline__ float tanh_isq2(float x) { return tanhf(x * 0.70710678118654752440f); }
    static __device__ __forceinline__ float rcp(float x) { return 1.0f / x; }
    static __device__ __forceinline__ float sqrt_(float x) { return sqrtf(x); }
};
#endif
template <> struct M<double> {
    static __device__ __forceinline__ double tanh_isq2(double x) { return tanh(x * 0.70710678118654752440); }
    static __device__ __forceinline__ double rcp(double x) { return 1.0 / x; }
    static __device__ __forceinline__ double sqrt_(double x) { return sqrt(x); }
};

// ---------------------------------------------------------------------------
// packed pair of the two columns of a lane
// ---------------------------------------------------------------------------
template <typename T> struct V;
template <> struct V<float> {
    float2 v;
    __device__ __forceinline__ float x() const { return v.x; }
    __device__ __forceinline__ float y() const { return v.y; }
};
template <> struct V<double> {
    double vx, vy;
    __device__ __forceinline__ double x() const { return vx; }
    __device__ __forceinline__ double y() const { return vy; }
};
__device__ __forceinline__ V<float> mk(float a, float b) {
    V<float> r;
    r.v = make_float2(a, b);
    return r;
}
__device__ __forceinline__ V<double> mk(double a, double b) {
    V<double> r;
    r.vx = a;
    r.vy = b;
    return r;
}
template <typename T> __device__ __forceinline__ V<T> bc(T a) { return mk(a, a); }
__device__ __forceinline__ V<float> operator+(V<float> a, V<float> b) {
    V<float> r;
    r.v = __fadd2_rn(a.v, b.v);
    return r;
}
__device__ __forceinline__ V<float> operator-(V<float> a, V<float> b) {
    V<float> r;
    r.v = __ffma2_rn(b.v, make_float2(-1.0f, -1.0f), a.v);  // exactly a - b
    return r;
}
__device__ __forceinline__ V<float> operator*(V<float> a, V<float> b) {
    V<float> r;
    r.v = __fmul2_rn(a.v, b.v);
    return r;
}
__device__ __forceinline__ V<float> fma(V<float> a, V<float> b, V<float> c) {
    V<float> r;
    r.v = __ffma2_rn(a.v, b.v, c.v);
    return r;
}
// (FP64: explicitly rounded as well, so that every kernel that evaluates an
// expression gives the same bits, whatever the compiler would contract)
__device__ __forceinline__ V<double> operator+(V<double> a, V<double> b) {
    return mk(__dadd_rn(a.vx, b.vx), __dadd_rn(a.vy, b.vy));
}
__device__ __forceinline__ V<double> operator-(V<double> a, V<double> b) {
    return mk(__dsub_rn(a.vx, b.vx), __dsub_rn(a.vy, b.vy));
}
__device__ __forceinline__ V<double> operator*(V<double> a, V<double> b) {
    return mk(__dmul_rn(a.vx, b.vx), __dmul_rn(a.vy, b.vy));
}
__device__ __forceinline__ V<double> fma(V<double> a, V<double> b, V<double> c) {
    return mk(__fma_rn(a.vx, b.vx, c.vx), __fma_rn(a.vy, b.vy, c.vy));
}
template <typename T> __device__ __forceinline__ V<T> rcp2(V<T> a) { return mk(M<T>::rcp(a.x()), M<T>::rcp(a.y())); }

// f of each column
template <typename T, typename F> __device__ __forceinline__ V<T> each(V<T> a, F f) { return mk(f(a.x()), f(a.y())); }
template <typename T, typename F> __device__ __forceinline__ V<T> each(V<T> a, V<T> b, F f) {
    return mk(f(a.x(), b.x()), f(a.y(), b.y()));
}

template <typename T> __device__ __forceinline__ T shup(T v) { return __shfl_up_sync(FULL, v, 1); }
template <typename T> __device__ __forceinline__ T shdn(T v) { return __shfl_down_sync(FULL, v, 1); }

// A row as one lane sees it: columns L-2 .. L+3.
template <typename T> struct Row {
    T m2, m1, l, r, p1, p2;
    __device__ __forceinline__ T at(int o) const {
        return o == -2 ? m2 : o == -1 ? m1 : o == 0 ? l : o == 1 ? r : o == 2 ? p1 : p2;
    }
    __device__ __forceinline__ V<T> pat(int o) const { return mk(at(o), at(o + 1)); }
};

// |psi| beyond which the FP64 library tanh of psi / sqrt2 returns exactly
// +-1 (from |psi / sqrt2| ~ 19 on).  FP64 rows beyond it take phi = sign(psi)
// without the tanh, which is expensive at GB300's FP64 rate (+31% for the FP64
// sweep); the FP32 exp2/reciprocal form costs less than the warp vote.
template <typename T> struct Bulk;
template <> struct Bulk<double> { static constexpr double psi = 32.0; };

template <typename T> struct ConstOf;
template <> struct ConstOf<float> {
    static __device__ __forceinline__ const float* get(const InstRec& r) { return r.cf; }
};
template <> struct ConstOf<double> {
    static __device__ __forceinline__ const double* get(const InstRec& r) { return r.cd; }
};

template <typename T> struct Vec2;
template <> struct Vec2<float> { using t = float2; };
template <> struct Vec2<double> { using t = double2; };

// Column index of a ghost column: periodic wrap or cell-centred mirror.
__device__ __forceinline__ int col_idx(int c, int nx, bool per) {
    return per ? ((c % nx) + nx) % nx : mirror_idx(c, nx);
}
// One periodic period applied to a strip column (c in [-2, nx + 62)): the
// wrapped pair stays contiguous, so it keeps the vector load; columns still
// outside [0, nx) (grids narrower than a strip) take the scalar path.
__device__ __forceinline__ int wrap_once(int c, int nx, bool per) {
    return !per ? c : (c < 0 ? c + nx : (c >= nx ? c - nx : c));
}

// Load the pair (c, c+1) of a row; c is even.  Vector load when both columns
// are inside and the row is 2-element aligned, wrapped or mirrored scalar
// loads otherwise.
template <typename T>
__device__ __forceinline__ void load_pair(const T* __restrict__ row, int c, int nx, bool vec, bool per, T& a, T& b) {
    c = wrap_once(c, nx, per);
    if (vec && c >= 0 && c + 1 < nx) {
        const typename Vec2<T>::t v = *reinterpret_cast<const typename Vec2<T>::t*>(row + PF_CHK(c, nx - 1));
        a = v.x;
        b = v.y;
    } else {
        a = row[PF_CHK(col_idx(c, nx, per), nx)];
        b = row[PF_CHK(col_idx(c + 1, nx, per), nx)];
    }
}
__device__ __forceinline__ void load_grain_pair(const int16_t* __restrict__ row, int c, int nx, bool vec, bool per,
                                                int& a, int& b) {
    c = wrap_once(c, nx, per);
    if (vec && c >= 0 && c + 1 < nx) {
        const int v = *reinterpret_cast<const int*>(row + PF_CHK(c, nx - 1));
        a = (int)(int16_t)(v & 0xffff);
        b = (int)(int16_t)((unsigned)v >> 16);
    } else {
        a = row[PF_CHK(col_idx(c, nx, per), nx)];
        b = row[PF_CHK(col_idx(c + 1, nx, per), nx)];
    }
}
template <typename T>
__device__ __forceinline__ void store_pair(T* __restrict__ row, int c, int nx, bool vec, bool okL, bool okR, V<T> v) {
    if (vec && okL && okR) {
        typename Vec2<T>::t o;
        o.x = v.x();
        o.y = v.y();
        *reinterpret_cast<typename Vec2<T>::t*>(row + PF_CHK(c, nx - 1)) = o;
    } else {
        if (okL) row[PF_CHK(c, nx)] = v.x();
        if (okR) row[PF_CHK(c + 1, nx)] = v.y();
    }
}

// App. B: |grad b| at a <10> face (pairs); B(p, q) = b at origin + p normal + q tangent.
template <typename T, typename F> __device__ __forceinline__ V<T> appb_face2(F B, T ih) {
    const V<T> a1 = B(1, 1) - B(0, -1), a2 = B(0, 1) - B(1, -1);
    const V<T> b1 = B(2, 1) - B(-1, -1), b2 = B(-1, 1) - B(2, -1);
    const V<T> c1 = B(1, 2) - B(0, -2), c2 = B(0, 2) - B(1, -2);
    const V<T> dn = (bc<T>(T(35.0 / 48.0)) * (a1 - a2) - bc<T>(T(1.0 / 48.0)) * (b1 - b2) -
                     bc<T>(T(1.0 / 6.0)) * (c1 - c2)) * bc<T>(ih);
    const V<T> dt = (bc<T>(T(35.0 / 96.0)) * (a1 + a2) - bc<T>(T(1.0 / 32.0)) * (b1 + b2) -
                     bc<T>(T(1.0 / 24.0)) * (c1 + c2)) * bc<T>(ih);
    const V<T> m2 = fma(dn, dn, dt * dt);
    return each(m2, [](T m) { return M<T>::sqrt_(m); });
}
// App. B: |grad b| at a corner; B(p, q) = b at origin + p x + q y.
template <typename T, typename F> __device__ __forceinline__ V<T> appb_corner2(F B, T ih) {
    const V<T> a1 = B(1, 1) - B(0, 0), a2 = B(0, 1) - B(1, 0);
    const V<T> b1 = B(2, 1) - B(-1, 0), b2 = B(-1, 1) - B(2, 0);
    const V<T> c1 = B(1, 2) - B(0, -1), c2 = B(0, 2) - B(1, -1);
    const V<T> dx = (bc<T>(T(5.0 / 8.0)) * (a1 - a2) - bc<T>(T(1.0 / 48.0)) * (b1 - b2) -
                     bc<T>(T(1.0 / 16.0)) * (c1 - c2)) * bc<T>(ih);
    const V<T> dy = (bc<T>(T(5.0 / 8.0)) * (a1 + a2) - bc<T>(T(1.0 / 16.0)) * (b1 + b2) -
                     bc<T>(T(1.0 / 48.0)) * (c1 + c2)) * bc<T>(ih);
    const V<T> m2 = fma(dx, dx, dy * dy);
    return each(m2, [](T m) { return M<T>::sqrt_(m); });
}
// App. B magnitude m at a flux point raised to at least half of the two-point
// slope |d| s (s = 1 / |e|): the quotient slope / m, the unit normal's
// component along e, then stays within [-2, 2]; it leaves that range only
// where grad psi has no direction (reading R-A21G)
template <typename T> __device__ __forceinline__ V<T> appb_floor2(V<T> m, V<T> d, T s) {
    return each(m, d, [&](T a, T b) { return fmax(a, T(0.5) * s * fabs(b)); });
}
// f / m per column with the guard on |grad psi| of the standard anti-trapping forms
template <typename T> __device__ __forceinline__ V<T> guarded_div2(V<T> f, V<T> m, T hh) {
    return each(f * rcp2(m), m, [&](T q, T a) { return a * a * hh < Guard<T>::v ? T(0) : q; });
}

}  // namespace
}  // namespace pf
