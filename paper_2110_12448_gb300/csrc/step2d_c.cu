// step2d_c.cu -- the fused 2D step of the compensated FP32 state (PF_F32C):
// psi and U carried as FP32 pairs hi + lo (about 48 significant bits), the lo
// half of a level stored right after its hi half; 2D, isothermal, mirror walls,
// T1.  The strips, the order of a sweep and the discretisations are those of
// step2d_kernel.cuh; here the psi rate is evaluated in double-float pairs and
// the state updates keep their rounding errors.
//
// The kernel is bound by the FMA pipe (1388 FLOP and 23.6 warp instructions per
// cell where everything is evaluated).  Far from the interface phi, 1 - phi^2
// and delta phi are constants to more digits than the state holds, and a third
// of the double-float arithmetic (the exponential, two divisions, the coupling
// term) forms nothing but them: a row whose |psi| exceeds FAR all over the warp
// takes the constants (10 x 1024^2: 366 -> 260 us a step).
#include <cfloat>

#include "step2d.cuh"
#include "step2d_launch.cuh"

namespace pf {
namespace {

// x / y from the reciprocal estimate and one Newton correction of the
// quotient (Markstein): q = x r, then q + (x - q y) r with the residual in
// one FMA.  Within about an ulp of x / y for normal operands, with no
// slow-path test; the compensated state's divisions either feed a residual
// step that corrects the quotient to double-float precision or form small
// increments whose last-bit error is far below the state's lo half.
__device__ __forceinline__ float div_nr(float x, float y) {
    const float r = rcp_approx(y);
    const float q = x * r;
    return fmaf(fmaf(-q, y, x), r, q);
}
// Crystal frames of the two columns (upper 2x2 of crystal -> lab rotations).
struct Rot2 {
    V<float> a, b, c, d;  // (R00, R01, R10, R11) of column L in .x, of column R in .y
};

// Normal component of J - g for face gradients (gx, gy) of both columns, J =
// d(a_s^2 |g|^2 / 2)/dg, without cancellation: crystal components c = R^T g,
// s_p = c_p^2 / |c|^2, q = s_x^2 + s_y^2, a_s = 1 - 3 eps + 4 eps q; with s_x + s_y = 1 in 2D, a - 1 = eps (4q - 3) =
// eps (1 - 8 s_x s_y), a^2 - 1 = (a - 1)(a + 1), and s_x - q = s_y (s_x - s_y),
// s_y - q = -s_x (s_x - s_y), so
//   J'_x - c_x = c_x eps [b (2 + eps b) + 16 a s_y (s_x - s_y)],
//   J'_y - c_y = c_y eps [b (2 + eps b) - 16 a s_x (s_x - s_y)],  b = 1 - 8 s_x s_y,
// every term formed without subtracting nearly equal numbers.
__device__ __forceinline__ V<float> aniso_qn2c(V<float> gx, V<float> gy, const Rot2& R, float eps, float hh, bool xface) {
    const V<float> cx = fma(R.a, gx, R.c * gy);
    const V<float> cy = fma(R.b, gx, R.d * gy);
    const V<float> r2 = fma(cx, cx, cy * cy);
    const V<float> inv = rcp2(r2);
    const V<float> sx = cx * cx * inv, sy = cy * cy * inv;
    const V<float> dxy = (cx - cy) * (cx + cy) * inv;  // s_x - s_y
    const V<float> b = fma(bc<float>(-8.0f) * sx, sy, bc<float>(1.0f));
    const V<float> a = fma(bc<float>(eps), b, bc<float>(1.0f));
    const V<float> B = b * fma(bc<float>(eps), b, bc<float>(2.0f));
    const V<float> t = bc<float>(16.0f) * a * dxy;
    const V<float> jx = cx * bc<float>(eps) * fma(t, sy, B), jy = cy * bc<float>(eps) * fma(t * bc<float>(-1.0f), sx, B);
    const V<float> o = xface ? fma(R.a, jx, R.b * jy) : fma(R.c, jx, R.d * jy);
    return mk(r2.x() * hh < Guard<float>::v ? 0.0f : o.x(), r2.y() * hh < Guard<float>::v ? 0.0f : o.y());
}
// the anisotropic part 4 eps q of a_s = (1 - 3 eps) + 4 eps q (3 eps where
// the normal is undefined, so that a_s = 1): the compensated state forms
// a_s in double-float from it
__device__ __forceinline__ V<float> aniso_w2(V<float> gx, V<float> gy, const Rot2& R, float eps, float hh) {
    const V<float> cx = fma(R.a, gx, R.c * gy);
    const V<float> cy = fma(R.b, gx, R.d * gy);
    const V<float> r2 = fma(cx, cx, cy * cy);
    const V<float> inv = rcp2(r2);
    const V<float> sx = cx * cx * inv, sy = cy * cy * inv;
    const V<float> w = bc<float>(4.0f * eps) * fma(sx, sx, sy * sy);
    return mk(r2.x() * hh < Guard<float>::v ? 3.0f * eps : w.x(), r2.y() * hh < Guard<float>::v ? 3.0f * eps : w.y());
}
// (hi, lo) + d: Knuth's two-sum of hi and d, the rounding error folded into
// lo, renormalised by Dekker's fast two-sum (the _rn intrinsics are never
// contracted into FMAs, which would break the error-free transformations)
__device__ __forceinline__ void cadd(float hi, float lo, float d, float& ho, float& lo_o) {
    const float s = __fadd_rn(hi, d);
    const float bb = __fsub_rn(s, hi);
    const float e = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)), __fsub_rn(d, bb));
    const float l = __fadd_rn(lo, e);
    ho = __fadd_rn(s, l);
    lo_o = __fsub_rn(l, __fsub_rn(ho, s));
}
__device__ __forceinline__ void cadd2(V<float> hi, V<float> lo, V<float> d, V<float>& ho, V<float>& lo_o) {
    float a, b, c, e;
    cadd(hi.x(), lo.x(), d.x(), a, b);
    cadd(hi.y(), lo.y(), d.y(), c, e);
    ho = mk(a, c);
    lo_o = mk(b, e);
}
// phi(psi + d) - phi(psi) = T (1 - phi^2) / (1 + T phi) with T = tanh(d / sqrt2),
// the addition theorem of tanh: the increment keeps its relative accuracy,
// unlike the difference phi' - phi of two rounded values
__device__ __forceinline__ float dphi_acc(float phi, float d) {
    const float T = tanhf(d * 0.70710678118654752440f);
    return div_nr(T * fmaf(-phi, phi, 1.0f), fmaf(T, phi, 1.0f));
}

// ---------------------------------------------------------------------------
// double-float arithmetic on packed FP32 pairs (Dekker's double-length
// arithmetic, 1971: values h + l with |l| <= ulp(h) / 2; error-free two-sum
// and the FMA two-product).  The compensated state evaluates the psi rate this
// way: its terms are O(1) while the rate must be accurate to ~1e-8 absolute
// (a per-step perturbation of psi at the interface is amplified ~1e4-fold
// over 1e4 steps of the free dendrite), beyond FP32's 2^-24.
// ---------------------------------------------------------------------------
struct D2 {
    V<float> h, l;
};
__device__ __forceinline__ D2 d2(V<float> h, V<float> l) { return D2{h, l}; }
__device__ __forceinline__ D2 d2f(V<float> h) { return D2{h, bc<float>(0.0f)}; }
__device__ __forceinline__ D2 d2c(float h, float l) { return D2{bc<float>(h), bc<float>(l)}; }
__device__ __forceinline__ V<float> vneg(V<float> a) { return a * bc<float>(-1.0f); }
// s + e = a + b exactly (Knuth)
__device__ __forceinline__ D2 two_sum(V<float> a, V<float> b) {
    const V<float> s = a + b;
    const V<float> bb = s - a;
    return D2{s, (a - (s - bb)) + (b - bb)};
}
// s + e = a + b exactly when |a| >= |b| (Dekker)
__device__ __forceinline__ D2 fast_two_sum(V<float> a, V<float> b) {
    const V<float> s = a + b;
    return D2{s, b - (s - a)};
}
// p + e = a b exactly
__device__ __forceinline__ D2 two_prod(V<float> a, V<float> b) {
    const V<float> p = a * b;
    return D2{p, fma(a, b, vneg(p))};
}
__device__ __forceinline__ D2 dadd(D2 x, D2 y) {
    const D2 s = two_sum(x.h, y.h);
    return fast_two_sum(s.h, s.l + (x.l + y.l));
}
__device__ __forceinline__ D2 dsub(D2 x, D2 y) { return dadd(x, D2{vneg(y.h), vneg(y.l)}); }
__device__ __forceinline__ D2 dmul(D2 x, D2 y) {
    const D2 p = two_prod(x.h, y.h);
    return fast_two_sum(p.h, fma(x.h, y.l, fma(x.l, y.h, p.l)));
}
__device__ __forceinline__ D2 dscale(D2 x, float c) { return D2{x.h * bc<float>(c), x.l * bc<float>(c)}; }  // c a power of 2
__device__ __forceinline__ D2 ddiv(D2 x, D2 y) {
    const V<float> q1 = mk(div_nr(x.h.x(), y.h.x()), div_nr(x.h.y(), y.h.y()));
    const D2 r = dsub(x, dmul(d2f(q1), y));
    const V<float> q2 = mk(div_nr(r.h.x(), y.h.x()), div_nr(r.h.y(), y.h.y()));
    return fast_two_sum(q1, q2);
}
// (hi_a + lo_a) - (hi_b + lo_b) with the hi difference exact
__device__ __forceinline__ D2 ddiff(V<float> ha, V<float> la, V<float> hb, V<float> lb) {
    const D2 s = two_sum(ha, vneg(hb));
    return D2{s.h, s.l + (la - lb)};
}
// e^x for x <= 0 (|x| < 80) in double-float, relative error ~1e-11: Cody-Waite
// reduction x = k ln2 + r, |r| <= ln2 / 2 (ln2 = L1 + L2 + L3, k L1 exact),
// e^r by its Taylor series (r, r^2/2, r^3/6 in double-float, r^4/24 ..
// r^9/9! in FP32, each below 1e-3 of the sum), then the exact scaling 2^k.
__device__ __forceinline__ D2 dexp_neg(D2 x) {
    const float L1 = 0.693115234375f, L2 = 3.194618329871446e-05f, L3 = 1.6465717678215697e-12f;
    const float kx = rintf(x.h.x() * 1.4426950216293335f), ky = rintf(x.h.y() * 1.4426950216293335f);
    const V<float> k = mk(kx, ky);
    const D2 r0 = two_sum(fma(vneg(k), bc<float>(L1), x.h), vneg(k * bc<float>(L2)));
    const D2 r = fast_two_sum(r0.h, r0.l + (x.l - k * bc<float>(L3)));
    const D2 r2 = dmul(r, r);
    const D2 r3 = dmul(r2, r);
    const V<float> rh = r.h;
    V<float> t = fma(rh, bc<float>(1.0f / 362880.0f), bc<float>(1.0f / 40320.0f));
    t = fma(rh, t, bc<float>(1.0f / 5040.0f));
    t = fma(rh, t, bc<float>(1.0f / 720.0f));
    t = fma(rh, t, bc<float>(1.0f / 120.0f));
    t = fma(rh, t, bc<float>(1.0f / 24.0f));
    t = t * (r2.h * r2.h);
    D2 e = dadd(dmul(r3, d2c(0.1666666716337204f, -4.967053879312289e-09f)), d2f(t));
    e = dadd(e, dscale(r2, 0.5f));
    e = dadd(e, r);
    e = dadd(e, d2c(1.0f, 0.0f));
    const V<float> p2 = mk(__int_as_float(((int)kx + 127) << 23), __int_as_float(((int)ky + 127) << 23));
    return D2{e.h * p2, e.l * p2};
}


// |psi| from which the psi rate takes phi = +-1 and no coupling term.  What that
// leaves out of dt times the rate, 4 e^{-sqrt2 24} = 7.3e-15 times sqrt2 lambda dt |U|
// (and a quarter of it times sqrt2 dt (1 + |grad psi|^2)), is below 2.1e-14 while
// lambda dt |U| <= 2, less than half a unit in the last place of the lo half of such a
// psi (2.8e-14); rows with a larger U, or one that is not finite, are evaluated in full.
constexpr float FAR = 24.0f;

// Resident one-warp blocks per SM asked for: 168 registers a lane and twelve
// resident warps either way, but asking for nine instead of eleven spills 40
// instead of 88 bytes (264 against 274 us a step at sweeps of 50 rows; eight
// blocks at more registers: 284; the dependency chains need the warps).
#ifndef PF_STEP2C_BLOCKS
#define PF_STEP2C_BLOCKS 9
#endif

// a row as one lane sees it: its two columns and their west and east neighbours
struct Tri {
    V<float> W, C, E;
};

// One sweep of a work item.  INSIDE: the whole strip, halo included, lies
// inside the grid and rows are aligned to pairs.
template <int S, bool INSIDE>
__device__ __forceinline__ void sweep2c(const WorkItem& wi, const InstRec& rec, int launch_parity) {
    constexpr bool ISO = (S == S21 || S == SBAR21);
    using V2 = V<float>;
    auto k_ = [](float x) -> V2 { return bc<float>(x); };
    const int lane = threadIdx.x;
    const int nx = rec.nx, ny = rec.ny;
    const int par = rec.parity_offset ^ launch_parity;
    const size_t NN = (size_t)nx * ny;
    const float* __restrict__ psi = static_cast<const float*>(rec.psi[par]);
    const float* __restrict__ Uf = static_cast<const float*>(rec.U[par]);
    const float* __restrict__ psiL = psi + NN;
    const float* __restrict__ UfL = Uf + NN;
    float* __restrict__ psi_o = static_cast<float*>(rec.psi[par ^ 1]);
    float* __restrict__ U_o = static_cast<float*>(rec.U[par ^ 1]);
    const int16_t* __restrict__ grain = rec.grain;
    const float* __restrict__ rot = static_cast<const float*>(rec.rot);
    const float* cst = rec.cf;
    const float ih = cst[C_IH], hh = cst[C_HH], dt = cst[C_DT];
    const float i4h = cst[C_I4H], ih_half = cst[C_IH_HALF];
    const float kk = cst[C_K], omk = cst[C_OMK], eps = cst[C_EPS], lam = cst[C_LAM], Dc = cst[C_D];
    const float ih2 = cst[C_IH2], i6h2 = cst[C_I6H2];
    const float isq2dt = cst[C_ISQ2DT];
    const float u_far = fminf(2.0f / (lam * dt), FLT_MAX);
    const bool one = rec.one_grain != 0;  // every cell in grain 0
    const int x0 = wi.x0, y0 = wi.y0;
    const int y1 = min(y0 + wi.ext, ny);
    const int cL = x0 - 2 + 2 * lane;
    const bool vec = INSIDE || (nx & 1) == 0;
    const bool own = lane >= 1 && lane <= 30;
    const bool realL = cL >= 0 && cL < nx, realR = cL + 1 >= 0 && cL + 1 < nx;
    const unsigned lo8 = lane * 8u;

    auto fetch_row = [&](const float* f, int vr) -> V2 {
        const float* __restrict__ row = f + (size_t)PF_CHK(mirror_idx(vr, ny), ny) * nx;
        if constexpr (INSIDE) {
#ifdef PF_BOUNDS_CHECK
            const float* __restrict__ at = row + PF_CHK(cL, nx - 1);
#else
            const float* __restrict__ at = reinterpret_cast<const float*>(reinterpret_cast<const char*>(row + (x0 - 2)) + lo8);
#endif
            const float2 v = *reinterpret_cast<const float2*>(at);
            return mk(v.x, v.y);
        }
        float a, b;
        load_pair<float>(row, cL, nx, vec, false, a, b);
        return mk(a, b);
    };
    auto store_row = [&](float* f, int row, V2 v) {
        float* __restrict__ o = f + (size_t)PF_CHK(row, ny) * nx;
        if constexpr (INSIDE) {
#ifdef PF_BOUNDS_CHECK
            float* __restrict__ at = o + PF_CHK(cL, nx - 1);
#else
            float* __restrict__ at = reinterpret_cast<float*>(reinterpret_cast<char*>(o + (x0 - 2)) + lo8);
#endif
            if (own) *reinterpret_cast<float2*>(at) = make_float2(v.x(), v.y());
        } else {
            store_pair<float>(o, cL, nx, vec, own && realL, own && realR, v);
        }
    };
    auto tri = [&](V2 c) -> Tri { return Tri{mk(shup(c.y()), c.x()), c, mk(c.y(), shdn(c.x()))}; };
    auto from_west = [&](V2 f) -> V2 { return mk(shup(f.y()), f.x()); };
    auto from_east = [&](V2 f) -> V2 { return mk(f.y(), shdn(f.x())); };
    // delta phi: ghost columns take their mirror cell's value
    auto ghosts = [&](V2 d) -> V2 {
        if constexpr (INSIDE) return d;
        const int qL = mirror_idx(cL, nx) - (x0 - 2), qR = mirror_idx(cL + 1, nx) - (x0 - 2);
        const float aL = __shfl_sync(FULL, d.x(), qL >> 1), bL = __shfl_sync(FULL, d.y(), qL >> 1);
        const float aR = __shfl_sync(FULL, d.x(), qR >> 1), bR = __shfl_sync(FULL, d.y(), qR >> 1);
        return mk(realL ? d.x() : ((qL & 1) ? bL : aL), realR ? d.y() : ((qR & 1) ? bR : aR));
    };
    Rot2 RR;
    auto g_lo = [](int g) -> int { return (int)(int16_t)(g & 0xffff); };
    auto g_hi = [](int g) -> int { return g >> 16; };
    auto set_rot = [&](int g) {
        const float* A = rot + 9 * PF_CHK(g_lo(g), rec.n_grains);
        const float* B = rot + 9 * PF_CHK(g_hi(g), rec.n_grains);
        RR.a = mk(__ldg(A + 0), __ldg(B + 0));
        RR.b = mk(__ldg(A + 1), __ldg(B + 1));
        RR.c = mk(__ldg(A + 3), __ldg(B + 3));
        RR.d = mk(__ldg(A + 4), __ldg(B + 4));
    };
    auto fetch_grain = [&](int row) -> int {
        if (one) return 0;
        int a, b;
        load_grain_pair(grain + (size_t)PF_CHK(row, ny) * nx, cL, nx, vec, false, a, b);
        return (a & 0xffff) | (b << 16);
    };
    // double-float constants of the psi rate
    auto dfc = [&](double x) -> D2 {
        const float h = (float)x;
        return d2c(h, (float)(x - (double)h));
    };
    const double hd = rec.h;
    const D2 kL = dfc(ISO ? 1.0 / (6.0 * hd * hd) : 1.0 / (hd * hd));
    const D2 kG1 = dfc(ISO ? 2.0 / 3.0 / (4.0 * hd * hd) : 0.25 / (hd * hd));
    const D2 kG2 = dfc(ISO ? 1.0 / 3.0 / (8.0 * hd * hd) : 0.0);
    const D2 kS2 = dfc(1.41421356237309504880);
    const D2 kDT = dfc(rec.dt);
    const D2 kA0 = dfc(1.0 - 3.0 * rec.eps4);
    auto dneg = [](D2 x) -> D2 { return D2{vneg(x.h), vneg(x.l)}; };

    // ---------------- state of the sweep (rows as in step2d_kernel.cuh) ----------------
    const int p0 = max(y0 - 1, 0);
    const V2 zero = k_(0.0f);
    Tri Pm = tri(fetch_row(psi, p0 - 1)), P0 = tri(fetch_row(psi, p0));
    Tri Lm = tri(fetch_row(psiL, p0 - 1)), L0 = tri(fetch_row(psiL, p0));
    Tri U0{zero, zero, zero}, UL0 = U0, AD0 = U0, AA0 = U0;
    V2 phin0 = zero, src0 = zero;  // phi' and delta phi of row r
    unsigned live = 0;             // bits: delta phi of rows r + 1, r, r - 1, r - 2 not exactly 0 over the warp
    V2 Yc;                         // anisotropy flux of the face between rows p - 1 and p
    V2 yD = zero, mmD = zero, pmD = zero, kD = zero, yA = zero, mmA = zero, pmA = zero, kA = zero;
    V2 nP = fetch_row(psi, p0 + 1), nPL = fetch_row(psiL, p0 + 1), nU = fetch_row(Uf, p0), nUL = fetch_row(UfL, p0);
    int nG = fetch_grain(p0), gf = nG;
    set_rot(nG);
    Yc = aniso_qn2c(((P0.E + Pm.E) - (P0.W + Pm.W)) * k_(i4h), (P0.C - Pm.C) * k_(ih), RR, eps, hh, false);

    for (int r = p0 - 1; r < y1; ++r) {
        const int p = r + 1;
        const Tri Pp = tri(nP), Lp = tri(nPL), U1 = tri(nU), UL1 = tri(nUL);
        const int g1 = nG;
        nP = fetch_row(psi, r + 3);
        nPL = fetch_row(psiL, r + 3);
        nU = fetch_row(Uf, r + 2);
        nUL = fetch_row(UfL, r + 2);
        nG = fetch_grain(min(r + 2, ny - 1));

        // ---------------- phase 1 at row p (its result is discarded at the ghost row ny) ----------------
        const bool moved = g1 != gf;
        if (moved) set_rot(g1);
        const V2 Xp = aniso_qn2c((P0.E - P0.C) * k_(ih), ((Pp.E + Pp.C) - (Pm.E + Pm.C)) * k_(i4h), RR, eps, hh, true);
        const V2 Yp = aniso_qn2c(((Pp.E + P0.E) - (Pp.W + P0.W)) * k_(i4h), (Pp.C - P0.C) * k_(ih), RR, eps, hh, false);
        V2 Xm = from_west(Xp), Ym = Yc;
        if (!one) {
            // faces whose other side is in another grain, in the cell's own frame
            const int gW = g_hi(shup(g1));
            const bool bL = gW != g_lo(g1), bR = g_lo(g1) != g_hi(g1);
            if (__any_sync(FULL, bL || bR)) {
                const V2 q = aniso_qn2c((P0.C - P0.W) * k_(ih), ((Pp.C + Pp.W) - (Pm.C + Pm.W)) * k_(i4h), RR, eps, hh, true);
                Xm = mk(bL ? q.x() : Xm.x(), bR ? q.y() : Xm.y());
            }
            if (__any_sync(FULL, moved)) {
                const V2 q = aniso_qn2c(((P0.E + Pm.E) - (P0.W + Pm.W)) * k_(i4h), (P0.C - Pm.C) * k_(ih), RR, eps, hh, false);
                Ym = mk(g_lo(gf) != g_lo(g1) ? q.x() : Ym.x(), g_hi(gf) != g_hi(g1) ? q.y() : Ym.y());
            }
            gf = g1;
        }
        Yc = Yp;
        const V2 N = ((Xp - Xm) + (Yp - Ym)) * k_(ih);
        const V2 ex = P0.E - P0.W, ey = Pp.C - Pm.C;
        // The rate in double-float: psi differences to the centre exact (hi
        // differences by two-sum plus the lo differences); L and G from them;
        // phi and 1 - phi^2 from e = exp(-sqrt2 |psi|) as sign (1 - e) / (1 + e)
        // and 4 e / (1 + e)^2; a_s = (1 - 3 eps) + 4 eps q with the FP32
        // anisotropic part; U with its lo half; the O(eps4) face terms N in
        // FP32.  psi' = (hi + lo) + dt rate kept exactly; delta phi from the
        // addition theorem.
        const V2 C0 = P0.C, cl = L0.C;
        D2 Ld, Gd;
        {
            auto dd = [&](V2 hn, V2 ln) { return ddiff(hn, ln, C0, cl); };
            const D2 dW = dd(P0.W, L0.W), dE = dd(P0.E, L0.E), dS = dd(Pm.C, Lm.C), dN = dd(Pp.C, Lp.C);
            const D2 faces = dadd(dadd(dW, dE), dadd(dS, dN));
            const D2 gx = dsub(dE, dW), gy = dsub(dN, dS);
            if constexpr (ISO) {
                const D2 dWm = dd(Pm.W, Lm.W), dEm = dd(Pm.E, Lm.E), dWp = dd(Pp.W, Lp.W), dEp = dd(Pp.E, Lp.E);
                Ld = dmul(dadd(dscale(faces, 4.0f), dadd(dadd(dWm, dEm), dadd(dWp, dEp))), kL);
                const D2 gp = dsub(dEp, dWm), gm = dsub(dEm, dWp);
                Gd = dadd(dmul(dadd(dmul(gx, gx), dmul(gy, gy)), kG1), dmul(dadd(dmul(gp, gp), dmul(gm, gm)), kG2));
            } else {
                Ld = dmul(faces, kL);
                Gd = dmul(dadd(dmul(gx, gx), dmul(gy, gy)), kG1);
            }
        }
        const V2 w = aniso_w2(ex * k_(ih_half), ey * k_(ih_half), RR, eps, hh);
        const D2 ad = dadd(kA0, d2f(w));
        const bool nL = C0.x() < 0.0f, nR = C0.y() < 0.0f;
        const bool far = __all_sync(FULL, fabsf(C0.x()) > FAR && fabsf(C0.y()) > FAR && fabsf(U1.C.x()) <= u_far &&
                                              fabsf(U1.C.y()) <= u_far);
        V2 ph, dph = zero;
        D2 srcd, phG;  // sqrt2 (phi - lambda (1 - phi^2) U) and sqrt2 phi
        if (far) {
            ph = mk(nL ? -1.0f : 1.0f, nR ? -1.0f : 1.0f);
            srcd = phG = D2{kS2.h * ph, kS2.l * ph};
        } else {
            // |psi| (clamped at 40: e < 1e-24 there) and its sign
            const bool cLx = fabsf(C0.x()) > 40.0f, cRx = fabsf(C0.y()) > 40.0f;
            const D2 ap = d2(mk(cLx ? 40.0f : fabsf(C0.x()), cRx ? 40.0f : fabsf(C0.y())),
                             mk(cLx ? 0.0f : (nL ? -cl.x() : cl.x()), cRx ? 0.0f : (nR ? -cl.y() : cl.y())));
            const D2 e = dexp_neg(dmul(ap, dneg(kS2)));
            const D2 unit = d2c(1.0f, 0.0f);
            const D2 ep1 = dadd(unit, e);
            const D2 pa = ddiv(dsub(unit, e), ep1);
            const D2 phd = d2(mk(nL ? -pa.h.x() : pa.h.x(), nR ? -pa.h.y() : pa.h.y()),
                              mk(nL ? -pa.l.x() : pa.l.x(), nR ? -pa.l.y() : pa.l.y()));
            const D2 omp = ddiv(dscale(e, 4.0f), dmul(ep1, ep1));  // 1 - phi^2
            const D2 cpl = dmul(dmul(omp, d2f(k_(lam))), d2(U1.C, UL1.C));
            srcd = dmul(dsub(phd, cpl), kS2);
            phG = dmul(phd, kS2);
            ph = phd.h;  // phi^n, rounded once from double-float
        }
        const D2 E = dadd(dadd(Ld, d2f(N)), srcd);
        const D2 rate = dsub(ddiv(E, dmul(ad, ad)), dmul(phG, Gd));
        const D2 d = dmul(rate, kDT);
        const D2 s1 = two_sum(C0, d.h);
        const D2 s2 = fast_two_sum(s1.h, s1.l + (cl + d.l));
        if (!far) dph = mk(dphi_acc(ph.x(), d.h.x()), dphi_acc(ph.y(), d.h.y()));
        else dph = d.h * k_(0.0f);  // 0, but NaN where the rate is not finite
        V2 phn = ph + dph;
        if (p >= y0 && p < y1) {
            store_row(psi_o, p, s2.h);
            store_row(psi_o + NN, p, s2.l);
        }

        // ---------------- alphas of row p ----------------
        const Tri AD1 = tri(k_(1.0f) - ph);
        // delta phi row exactly 0 over the whole warp: bulk liquid or solid
        const bool still = __all_sync(FULL, dph.x() == 0.0f && dph.y() == 0.0f);
        live = live << 1 | (still ? 0u : 1u);
        Tri AA1{zero, zero, zero};
        V2 src1 = zero;
        if (!still) {
            src1 = ghosts(dph);
            AA1 = tri((k_(1.0f) + k_(omk) * U1.C) * src1 * k_(isq2dt));
        }
        if (p >= ny) {  // the ghost row ny mirrors row ny - 1
            AA1 = AA0;
            live = (live & ~1u) | (live >> 1 & 1u);
        }
        if (r < 0) {  // the ghost row -1 mirrors row 0
            U0 = U1;
            UL0 = UL1;
            AD0 = AD1;
            AA0 = AA1;
            live = (live & 1u) * 3u;
        }

        // ---------------- phase 2 at row r ----------------
        // eight-flux sums of the own columns (x 6 h^2 for the D~_{2,1} forms, x h^2
        // for S_{1,0}); U differences with those of the lo halves
        if (r >= y0 - 1) {
            V2 sD, sA = zero;
            auto dU = [&](V2 hi_diff, V2 lo_diff) -> V2 { return hi_diff + lo_diff; };
            const V2 u0c = U0.C, l0c = UL0.C, p0c = Pm.C;
            const bool act = (live & 7u) != 0;
            if constexpr (S == S10) {
                const V2 half = k_(0.5f);
                const V2 fxD = half * (AD0.C + AD0.E) * dU(U0.E - u0c, UL0.E - l0c);
                const V2 fyD = half * (AD0.C + AD1.C) * dU(U1.C - u0c, UL1.C - l0c);
                sD = (fxD - from_west(fxD)) + (fyD - yD);
                yD = fyD;
                if (act) {
                    const Tri Q = tri(fetch_row(psi, r - 1));
                    const V2 dxp = Pm.E - p0c, dyp = P0.C - p0c;
                    const V2 gx = dxp * k_(ih), gy = ((P0.E + P0.C) - (Q.E + Q.C)) * k_(i4h);
                    const V2 yx = ((P0.E + Pm.E) - (P0.W + Pm.W)) * k_(i4h), yy = dyp * k_(ih);
                    const V2 mx = fma(gx, gx, gy * gy), my = fma(yx, yx, yy * yy);
                    const V2 fxA = guarded_div2<float>(half * (AA0.C + AA0.E) * dxp, mk(M<float>::sqrt_(mx.x()), M<float>::sqrt_(mx.y())), hh);
                    const V2 fyA = guarded_div2<float>(half * (AA0.C + AA1.C) * dyp, mk(M<float>::sqrt_(my.x()), M<float>::sqrt_(my.y())), hh);
                    sA = (fxA - from_west(fxA)) + (fyA - yA);
                    yA = fyA;
                } else {
                    yA = zero;
                }
            } else {
                const V2 q4 = k_(0.25f);
                // corner means: the (+1/2, +1/2) corners of (L, R) and of (L-1, L)
                auto shell = [&](const Tri& a0, const Tri& a1, V2 bx, V2 by, V2 bpp, V2 bmp, V2& kc, V2& KC, V2& KW, V2& fx,
                                 V2& fy, V2& pp, V2& mp) {
                    KC = q4 * ((a0.C + a0.E) + (a1.C + a1.E));
                    KW = q4 * ((a0.W + a0.C) + (a1.W + a1.C));
                    fx = ((a0.C + a0.E) + (KC + kc)) * bx;
                    fy = ((a0.C + a1.C) + (KC + KW)) * by;
                    pp = KC * bpp;
                    mp = KW * bmp;
                    kc = KC;
                };
                // carries for row q+1: its y- face is this y+ face, its (-1/2,-1/2)
                // corner the (+1/2,+1/2) corner of the column to the left, its
                // (+1/2,-1/2) corner the (-1/2,+1/2) corner of the column to the right
                auto gather = [&](V2 fx, V2 fy, V2 pp, V2 mp, V2& yc, V2& mm, V2& pm) -> V2 {
                    const V2 s = ((fx - from_west(fx)) + (fy - yc)) + ((pp + mp) - (mm + pm));
                    yc = fy;
                    mm = from_west(pp);
                    pm = from_east(mp);
                    return s;
                };
                V2 KC, KW, fx, fy, pp, mp;
                shell(AD0, AD1, dU(U0.E - u0c, UL0.E - l0c), dU(U1.C - u0c, UL1.C - l0c), dU(U1.E - u0c, UL1.E - l0c),
                      dU(U1.W - u0c, UL1.W - l0c), kD, KC, KW, fx, fy, pp, mp);
                sD = gather(fx, fy, pp, mp, yD, mmD, pmD);
                if (act) {
                    const V2 dx = Pm.E - p0c, dy = P0.C - p0c, dpp = P0.E - p0c, dmp = P0.W - p0c;
                    shell(AA0, AA1, dx, dy, dpp, dmp, kA, KC, KW, fx, fy, pp, mp);
                    if constexpr (S == S21) {
                        // App. B: each anti-trapping flux divided by |grad psi| at its point, from
                        // the psi rows r-2 .. r+2; ps(dx, dy) = psi at columns (L + dx, R + dx), row r + dy
                        Row<float> Q[5];
#pragma unroll
                        for (int j = 0; j < 5; ++j) {
                            const V2 q = fetch_row(psi, r - 2 + j);
                            Q[j] = Row<float>{shup(q.x()), shup(q.y()), q.x(), q.y(), shdn(q.x()), shdn(q.y())};
                        }
                        auto ps = [&](int i, int j) -> V2 { return Q[2 + j].pat(i); };
                        const float ihd = ih * 0.70710678118654752440f;  // 1 / |e| of the <11> fluxes
                        fx = guarded_div2<float>(fx, appb_floor2<float>(appb_face2<float>([&](int i, int j) { return ps(i, j); }, ih), dx, ih), hh);
                        fy = guarded_div2<float>(fy, appb_floor2<float>(appb_face2<float>([&](int i, int j) { return ps(j, i); }, ih), dy, ih), hh);
                        pp = guarded_div2<float>(pp, appb_floor2<float>(appb_corner2<float>([&](int i, int j) { return ps(i, j); }, ih), dpp, ihd), hh);
                        mp = guarded_div2<float>(mp, appb_floor2<float>(appb_corner2<float>([&](int i, int j) { return ps(i - 1, j); }, ih), dmp, ihd), hh);
                    }
                    sA = gather(fx, fy, pp, mp, yA, mmA, pmA);
                } else {
                    yA = mmA = pmA = kA = zero;
                }
            }
            if (r >= y0) {
                const float cs = (S == S10) ? ih2 : i6h2;
                const V2 num = fma(k_(dt * cs), fma(k_(Dc), sD, sA), fma(k_(omk), u0c, k_(1.0f)) * src0);
                // U' = (hi + lo) + num / (1 + k - (1-k) phi'), kept exactly
                const V2 den = fma(k_(-omk), phin0, k_(1.0f + kk));
                V2 uh, ul;
                cadd2(u0c, l0c, mk(div_nr(num.x(), den.x()), div_nr(num.y(), den.y())), uh, ul);
                store_row(U_o, r, uh);
                store_row(U_o + NN, r, ul);
            }
        }
        phin0 = phn;
        src0 = src1;
        U0 = U1;
        UL0 = UL1;
        AD0 = AD1;
        AA0 = AA1;
        Pm = P0;
        P0 = Pp;
        Lm = L0;
        L0 = Lp;
    }
}

template <int S>
__global__ void __launch_bounds__(32, PF_STEP2C_BLOCKS)
    k_step2c(const WorkItem* __restrict__ work, int n_work, const InstRec* __restrict__ recs, int launch_parity) {
    after_previous();
    for (int w = blockIdx.x; w < n_work; w += gridDim.x) {
        const WorkItem wi = work[w];
        const InstRec& rec = recs[wi.inst];
        if (wi.x0 >= 2 && wi.x0 + 62 <= rec.nx && (rec.nx & 1) == 0)
            sweep2c<S, true>(wi, rec, launch_parity);
        else
            sweep2c<S, false>(wi, rec, launch_parity);
    }
}

using Kernel2C = void (*)(const WorkItem*, int, const InstRec*, int);
Kernel2C kernel2c(int scheme) {
    return scheme == S10 ? k_step2c<S10> : scheme == S21 ? k_step2c<S21> : scheme == SBAR21 ? k_step2c<SBAR21> : nullptr;
}

}  // namespace

PF_BOUNDS_READER(bounds_step2c)

bool step2c_launch(int scheme, const Step2DArgs& a, int grid, cudaStream_t st) {
    const Kernel2C k = kernel2c(scheme);
    if (!k || a.mode != 0 || a.var != 0) return false;
    launch_next(k, grid, 32, 0, st, a.work, a.n_work, a.recs, a.launch_parity);
    return true;
}
int step2c_occupancy(int scheme, int var) {
    const Kernel2C k = kernel2c(scheme);
    int n = 0;
    if (!k || var != 0 || cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, 32, 0) != cudaSuccess) return 0;
    return n;
}

}  // namespace pf
