// step2d_kernel.cuh -- fused explicit time step of the quantitative alloy
// phase-field model in 2D for sm_103a (arXiv:2110.12448, Eqs. PF_a and PF_b).
//
// Warp-per-strip design.  Each warp owns a strip of 60 output columns and
// sweeps it row by row; lane t holds the two columns L = x0-2+2t, R = L+1
// (lanes 0 and 31 carry the halo).  Nothing is shared between warps (the little
// shared memory holds a lane's own state) and there is no block barrier.  The two columns of a lane are
// processed as a packed pair (FP32: the sm_100 float2 FMA/ADD/MUL
// instructions, one issue slot for both columns).  Global traffic per step:
// psi, U and the int16 grain read once, psi' and U' written once (float2 /
// int32 vectors).
//
// The kernel is bound by the FMA pipe and by instruction issue, so the work
// per cell is what the layout is chosen for:
//   - a psi row is kept as differences: C, e = E - C, ex = E - W and sx = E +
//     W - 2C of each column (formed once, with two shuffles), and between rows
//     d = C(p+1) - C(p).  Every operator is a short sum of these, in units of
//     the lattice (all constants fold into the final scale factors):
//       6 h^2 L_{2,1} = 4 (sx(p) + d - d') + sx(p-1) + sx(p+1) + 2 (d - d')
//       6 h^2 G_{2,1} = ex^2 + (d + d')^2 + (s^2 + t^2) / 8, s and t the sum and
//         difference of the two diagonal differences, ex(p+1) + ex(p-1) and
//         sx(p+1) - sx(p-1) + 2 (d + d')
//       4 h times the face gradients: (4 e, e(p+1) - e(p-1) + 2 (d + d')) and
//         (ex(p) + ex(p+1), 4 d)
//     and Eq. PF_a is summed in units of 1 / (6 h^2) (1 / h^2 for S_{1,0});
//   - J - g in an orthonormal crystal frame needs no rotation there and back:
//     with the reflection h = (C2 gx + S2 gy, S2 gx - C2 gy) of g about the
//     crystal axes (C2 = Ra^2 - Rb^2, S2 = Ra Rc - Rb Rd) and the cosine D =
//     g.h / |g|^2 of twice the angle to them, a_s = 1 + eps (2 D^2 - 1) and
//       J - g = K g + T h,  K = eps [(eps - 2) - (4 - 4 eps) D^2 - 12 eps D^4],
//                           T = eps D [8 - 8 eps + 16 eps D^2],
//     no difference of nearly equal numbers;
//   - every face flux is computed once and handed to the other cell that uses
//     it (shuffle across columns, register carry across rows); the four fluxes
//     of a cell (x+, y+ faces, both diagonals of its upper right corner) share
//     that corner's mean, and what the neighbour columns need of them travels
//     in one shuffle.
//
// Iteration r of a sweep (rows are virtual: mirrored at the walls):
//   take psi(r+2), U(r+1), grain(r+1)            (prefetched one row ahead)
//   phase 1 at row p = r+1: d psi/dt of Eq. PF_a, psi' = psi + dt d psi/dt,
//     phi' and delta phi = phi' - phi (also on the ring columns x0-1, x0+60)
//   phase 2 at row r: U' of Eq. PF_b in conservative form
//
// Discretisations (h = lattice spacing):
//   L_{2,1} (Eq. 2D_L21) or L_{1,0} (Eq. 2D_L10);
//   G_{2,1} = 2/3 G_{1,0} + 1/3 G_{0,1} (App. A, Eqs. Grad_10, Grad_11) or G_{1,0};
//   O(eps4) terms: div(J - grad psi) over the four <10> faces, J from the face
//     gradient (two-point normal, four-point tangential difference) in the
//     crystal frame of the cell whose rate is computed; a_s^2 on the left-hand
//     side and in the G term from the centred gradient;
//   D = D~_{2,1}[1 - phi, U] (Eqs. divergence_10/_11, flux_10/_11), or the <10>
//     form with a two-point face mean for S_{1,0};
//   anti-trapping: D~_{2,1}[(1+(1-k)U) dphi/(sqrt2 dt), psi] (Eq. Anti_approx),
//     App. B's A_{2,1} (fluxes divided by the 21-point |grad psi| at the flux
//     point), or the <10> form normalised by the face gradient (S_{1,0});
//   U' = U + [dt (D D + A) + (1+(1-k)U) dphi] / (1+k-(1-k)phi'), D on phi^n,
//     U^n and the anti-trapping on psi^n: the solute integral is conserved
//     exactly with mirror walls.
// Walls: cell-centred mirrors.  Phase-1 results on ghost columns/rows are
// copied from their mirror cells, so the (not mirror-symmetric) anisotropic
// terms of a rotated crystal are never evaluated at a ghost position.
#pragma once
#include "step2d.cuh"

namespace pf {
namespace {

// Which crystal frames an instance has: FR_ONE every cell in grain 0, the
// frame orthonormal (no grain rows are read); FR_CELL per-cell grains,
// orthonormal frames; FR_ANY any matrices (J - g by rotation into the frame
// and back; compiled for the general variant only).
enum : int { FR_ONE = 0, FR_CELL = 1, FR_ANY = 2 };

// Crystal frames of the two columns of a lane: (C2, S2) of the reflection, or
// the upper 2x2 of the crystal -> lab matrices.
template <typename T, int FR> struct Frame {
    V<T> c2, s2, n2;  // n2 = -C2
};
template <typename T> struct Frame<T, FR_ANY> {
    V<T> a, b, c, d;
};
// slots of a rotation-table row that hold C2 and S2 (unused matrix entries in 2D)
constexpr int ROT_C2 = 6, ROT_S2 = 7;

// Constants of K and T, and of a_s.  The fluxes take gradients times 4 h and
// enter the rate in units of 1 / (6 h^2) (iso) or 1 / h^2: `scale` = 6/4 or 1/4.
template <typename T> struct Aniso {
    T k0, k1, k2, t0, t1, a0, a1, eps, scale;
    __device__ __forceinline__ Aniso(T e, T s)
        : k0(s * e * (e - T(2))), k1(s * e * (T(4) * e - T(4))), k2(T(-12) * s * e * e), t0(s * e * (T(8) - T(8) * e)),
          t1(T(16) * s * e * e), a0(T(1) - e), a1(T(2) * e), eps(e), scale(s) {}
};
// guard on 16 |g|^2 h^2 (face gradients times 4 h) and 4 |g|^2 h^2 (centred differences)
template <typename T> struct Low {
    static constexpr T face = T(16) * Guard<T>::v, centre = T(4) * Guard<T>::v;
};

template <typename T>
__device__ __forceinline__ V<T> select_low(V<T> r2, T low, T other, V<T> v) {
    return each(r2, v, [=](T r, T x) { return r < low ? other : x; });
}

// h and g.h of a gradient (orthonormal frames): D = g.h / |g|^2
template <typename T, int FR>
__device__ __forceinline__ V<T> reflect(V<T> gx, V<T> gy, const Frame<T, FR>& F, V<T>& hx, V<T>& hy) {
    hx = fma(F.c2, gx, F.s2 * gy);
    hy = fma(F.s2, gx, F.n2 * gy);
    return fma(gx, hx, gy * hy);
}
// Normal component of J - g at a face (gradients times 4 h; 0 where |g|^2 h^2
// is below the guard), from 1 / |g|^2.
template <typename T, int FR>
__device__ __forceinline__ V<T> face_flux(V<T> gx, V<T> gy, V<T> r2, V<T> inv, const Frame<T, FR>& F, const Aniso<T>& A,
                                          bool xface) {
    if constexpr (FR == FR_ANY) {
        const V<T> cx = fma(F.a, gx, F.c * gy);
        const V<T> cy = fma(F.b, gx, F.d * gy);
        const V<T> c2 = fma(cx, cx, cy * cy);
        const V<T> ic = rcp2(c2);
        const V<T> sx = cx * cx * ic, sy = cy * cy * ic;
        const V<T> q = fma(sx, sx, sy * sy);
        const V<T> a = fma(bc<T>(T(4) * A.eps), q, bc<T>(T(1) - T(3) * A.eps));
        const V<T> c1 = bc<T>(T(16) * A.eps) * a;
        const V<T> c0 = fma(a, a, bc<T>(T(-1))) - c1 * q;
        const V<T> jx = cx * fma(c1, sx, c0), jy = cy * fma(c1, sy, c0);
        return select_low<T>(c2, Low<T>::face, T(0), bc<T>(A.scale) * (xface ? fma(F.a, jx, F.b * jy) : fma(F.c, jx, F.d * jy)));
    } else {
        V<T> hx, hy;
        const V<T> D = reflect<T, FR>(gx, gy, F, hx, hy) * inv;
        const V<T> m = D * D;
        const V<T> K = fma(m, fma(bc<T>(A.k2), m, bc<T>(A.k1)), bc<T>(A.k0));
        const V<T> t = D * fma(bc<T>(A.t1), m, bc<T>(A.t0));
        return select_low<T>(r2, Low<T>::face, T(0), xface ? fma(gx, K, hx * t) : fma(gy, K, hy * t));
    }
}
// a_s of a gradient (1 below the guard, which the caller applies)
template <typename T, int FR>
__device__ __forceinline__ V<T> aniso_as(V<T> gx, V<T> gy, V<T> inv, const Frame<T, FR>& F, const Aniso<T>& A) {
    if constexpr (FR == FR_ANY) {
        const V<T> cx = fma(F.a, gx, F.c * gy);
        const V<T> cy = fma(F.b, gx, F.d * gy);
        const V<T> ic = rcp2(fma(cx, cx, cy * cy));
        const V<T> sx = cx * cx * ic, sy = cy * cy * ic;
        return fma(bc<T>(T(4) * A.eps), fma(sx, sx, sy * sy), bc<T>(T(1) - T(3) * A.eps));
    } else {
        V<T> hx, hy;
        const V<T> D = reflect<T, FR>(gx, gy, F, hx, hy) * inv;
        return fma(bc<T>(A.a1), D * D, bc<T>(A.a0));
    }
}

// Resident one-warp blocks per SM that the launch bounds of the FP32 kernels
// ask for: 17 (120 registers) where one crystal frame and no App. B magnitudes
// are held, else 16 (128).  The row loop advances two rows per pass with one
// crystal frame, so that the row state moves between registers every other row
// only; one with per-cell frames, whose two copies outgrow the registers or the
// instruction cache.  us a step, 10 x 1024^2, sweeps of 32 / 38 rows:
//   S-bar_21  17 blocks 61.0 / 62.4, 16: 67.6 / 66.0, 18: 61.7 / 63.1
//   S_10      17 blocks 54.0 / 56.0, 16: 64.0 / 62.5
//   S_21      (10 x 781^2, 24 rows) 16 blocks 51.2, 17: 70.1
// (17 blocks are five warps of a scheduler: 96 registers a thread, so that 20 are
// resident.)
// (The forms not taken were measured with non-coherent loads, worth up to 1.4 %.)
// 16 polycrystals: 130.8 with 16 blocks and single rows, 161 with 17, 157 with two
// rows.  Earlier forms of the loop: four columns a lane in 8 blocks of 240
// registers 114 (61.0 here), three or four rows per pass 79 and 72 (68); an L2
// prefetch of the rows ahead changes nothing.
template <int S, int FR> constexpr int BLOCKS_F32 = FR == FR_ONE && S != S21 ? 17 : 16;

// How a strip reaches its rows: WALL any strip (mirrored or wrapped columns,
// per lane); PAIRS the whole strip, halo included, lies inside the grid and
// rows are aligned to pairs; SINGLES inside the grid, rows of odd length.  The
// last two leave no wall logic in the row loop.
enum : int { WALL = 0, PAIRS = 1, SINGLES = 2 };

// One sweep of a work item.
template <typename T, int S, int VAR, int FR, int MODE, int ACC>
__device__ __forceinline__ void sweep2d(const WorkItem& wi, const InstRec& rec, int launch_parity, const StepClock& clk,
                                        V<T>* park) {
    constexpr bool ISO = (S == S21 || S == SBAR21);
    constexpr bool DS = VAR == 1;   // frozen temperature / periodic x, T0 from the record
    constexpr bool T0I = VAR == 2;  // isothermal, mirror walls, T0
    using V2 = V<T>;
    auto c_ = [](double x) -> V2 { return bc<T>(T(x)); };
    auto k_ = [](T x) -> V2 { return bc<T>(x); };
    const int lane = threadIdx.x;
    const int nx = rec.nx, ny = rec.ny;
    const int par = rec.parity_offset ^ launch_parity;
    const T* __restrict__ psi = static_cast<const T*>(rec.psi[par]);
    const T* __restrict__ Uf = static_cast<const T*>(rec.U[par]);
    T* __restrict__ psi_o = static_cast<T*>(rec.psi[par ^ 1]);
    T* __restrict__ U_o = static_cast<T*>(rec.U[par ^ 1]);
    T* __restrict__ rate_b = static_cast<T*>(rec.rate);  // d psi/dt of the two-kernel form
    const int16_t* __restrict__ grain = rec.grain;
    const T* __restrict__ rot = static_cast<const T*>(rec.rot);
    const T* cst = ConstOf<T>::get(rec);
    const T omk = cst[C_OMK], opk = cst[C_OPK];
    // Eq. PF_a in units of lap = 1 / (6 h^2) or 1 / h^2
    const T dtl = ISO ? cst[C_DTL21] : cst[C_DTL10];
    const T sq = ISO ? cst[C_SQ21] : cst[C_SQ10], lam2 = ISO ? cst[C_LAM21] : cst[C_LAM10];
    const T cD = ISO ? cst[C_UD21] : cst[C_UD10], cA = ISO ? cst[C_UA21] : cst[C_UA10];
    const Aniso<T> an(cst[C_EPS], ISO ? T(1.5) : T(0.25));
    const bool per = DS && rec.bcx != 0;
    const bool t0 = T0I || (DS && rec.tlevel != 0);  // T0 time level
    // Frozen temperature: zeta at row p = p zA - (zB + n zC) (Eqs. Thermal_F1/_F2) from
    // the row's index alone, so that it does not depend on where a sweep begins; both
    // constants with what their rounding to the field precision leaves (FP32: within an
    // ulp of zeta, however large the two terms are).  The DS variant applies it
    // branch-free (zA = zB = zC = 0 gives zeta = 0, F1 = 1).
    T zA = T(0), zAl = T(0), z0 = T(0), z0l = T(0);
    if (DS) {
        const long long n = clk.clock ? clk.base[wi.inst] + *clk.clock : clk.step;
        const double b = -::fma((double)n, rec.zC, rec.zB);
        zA = (T)rec.zA;
        zAl = (T)(rec.zA - (double)zA);
        z0 = (T)b;
        z0l = (T)(b - (double)z0);
    }

    const int x0 = wi.x0, y0 = wi.y0;
    const int y1 = min(y0 + wi.ext, ny);
    const int cL = x0 - 2 + 2 * lane;
    const bool vec = ACC == PAIRS || (ACC == WALL && (nx & 1) == 0);
    const bool own = lane >= 1 && lane <= 30;  // the first and the last pair are halo
    const bool realL = cL >= 0 && cL < nx, realR = cL + 1 >= 0 && cL + 1 < nx;
    // warp may hold mirror ghost columns (periodic ghosts are real cells, computed in place)
    const bool edge = ACC == WALL && !per;
    // byte offset of the lane within a strip's row: with the row's address
    // uniform, each access is base + 32-bit offset
    const unsigned lo = lane * unsigned(2 * sizeof(T));

    auto load_row = [&](const T* __restrict__ row) -> V2 {
        T a, b;
        if constexpr (ACC != WALL) {
#ifdef PF_BOUNDS_CHECK
            const T* __restrict__ at = row + PF_CHK(cL, nx - 1);
#else
            const T* __restrict__ at = reinterpret_cast<const T*>(reinterpret_cast<const char*>(row + (x0 - 2)) + lo);
#endif
            if constexpr (ACC == PAIRS) {
                const typename Vec2<T>::t v = *reinterpret_cast<const typename Vec2<T>::t*>(at);
                a = v.x;
                b = v.y;
            } else {
                a = at[0];
                b = at[1];
            }
        } else {
            load_pair<T>(row, cL, nx, vec, per, a, b);
        }
        return mk(a, b);
    };
    auto fetch_row = [&](const T* f, int vr) -> V2 { return load_row(f + (size_t)PF_CHK(mirror_idx(vr, ny), ny) * nx); };
    auto store_row = [&](T* f, int row, V2 v) {
        T* __restrict__ o = f + (size_t)PF_CHK(row, ny) * nx;
        if constexpr (ACC != WALL) {
#ifdef PF_BOUNDS_CHECK
            T* __restrict__ at = o + PF_CHK(cL, nx - 1);
#else
            T* __restrict__ at = reinterpret_cast<T*>(reinterpret_cast<char*>(o + (x0 - 2)) + lo);
#endif
            if (own) {
                if constexpr (ACC == PAIRS) {
                    typename Vec2<T>::t q;
                    q.x = v.x();
                    q.y = v.y();
                    *reinterpret_cast<typename Vec2<T>::t*>(at) = q;
                } else {
                    at[0] = v.x();
                    at[1] = v.y();
                }
            }
        } else {
            store_pair<T>(o, cL, nx, vec, own && realL, own && realR, v);
        }
    };
    auto east = [&](V2 c) -> V2 { return mk(c.y(), shdn(c.x())); };       // values of the east neighbours
    auto from_west = [&](V2 f) -> V2 { return mk(shup(f.y()), f.x()); };  // values held by the west neighbours
    // differences of a psi row along x (see the top of this file)
    struct Diff {
        V2 e, ex, sx;
    };
    auto diffs = [&](V2 C) -> Diff {
        Diff q;
        q.e = east(C) - C;
        const V2 wd = from_west(q.e);  // C - W
        q.ex = q.e + wd;
        q.sx = q.e - wd;
        return q;
    };
    // whether f holds for every column that the warp holds
    auto all_of = [&](V2 a, auto f) -> bool { return __all_sync(FULL, f(a.x()) && f(a.y())); };
    // phi of a row; FP64: where |psi| exceeds the saturation bound on the
    // whole row of the warp, phi = sign(psi) exactly (what tanh returns)
    auto phi_of = [&](V2 p) -> V2 {
        if constexpr (sizeof(T) == 8) {
            if (all_of(p, [](T x) { return fabs(x) > Bulk<T>::psi; })) return each(p, [](T x) { return x > T(0) ? T(1) : T(-1); });
        }
        return each(p, [](T x) { return M<T>::tanh_isq2(x); });
    };
    // delta phi: ghost columns take their mirror cell's value (only in
    // warps that hold ghost columns)
    auto ghosts = [&](V2 d) -> V2 {
        if (!edge) return d;
        const int qL = mirror_idx(cL, nx) - (x0 - 2), qR = mirror_idx(cL + 1, nx) - (x0 - 2);
        // a far ghost column (beyond nx + 1) gets an out-of-range source lane,
        // which the shuffle reduces modulo 32; its value reaches no output
        const T aL = __shfl_sync(FULL, d.x(), qL >> 1), bL = __shfl_sync(FULL, d.y(), qL >> 1);
        const T aR = __shfl_sync(FULL, d.x(), qR >> 1), bR = __shfl_sync(FULL, d.y(), qR >> 1);
        return mk(realL ? d.x() : ((qL & 1) ? bL : aL), realR ? d.y() : ((qR & 1) ? bR : aR));
    };
    // T0: delta phi = dt (1 - phi^2) / sqrt2 d psi/dt (rate in units of lap)
    auto t0_dphi = [&](V2 om, V2 ph, V2 rate) -> V2 {
        const V2 q = k_(dtl * T(0.70710678118654752440));
        return (om * fma(q, ph, q)) * rate;
    };

    // crystal frames of the own columns, reloaded when a grain changes;
    // the two int16 grain indices of a lane in one word
    Frame<T, FR> F;
    auto g_lo = [](int g) -> int { return (int)(int16_t)(g & 0xffff); };
    auto g_hi = [](int g) -> int { return g >> 16; };
    auto set_frame = [&](int g) {
        const T* A = rot + 9 * PF_CHK(g_lo(g), rec.n_grains);
        const T* B = rot + 9 * PF_CHK(g_hi(g), rec.n_grains);
        if constexpr (FR == FR_ANY) {
            F.a = mk(__ldg(A + 0), __ldg(B + 0));
            F.b = mk(__ldg(A + 1), __ldg(B + 1));
            F.c = mk(__ldg(A + 3), __ldg(B + 3));
            F.d = mk(__ldg(A + 4), __ldg(B + 4));
        } else {
            F.c2 = mk(__ldg(A + ROT_C2), __ldg(B + ROT_C2));
            F.s2 = mk(__ldg(A + ROT_S2), __ldg(B + ROT_S2));
            F.n2 = F.c2 * c_(-1.0);
        }
    };
    if constexpr (FR == FR_ONE) {  // one frame for all columns
        F.c2 = k_(__ldg(rot + ROT_C2));
        F.s2 = k_(__ldg(rot + ROT_S2));
        F.n2 = k_(-__ldg(rot + ROT_C2));
    }
    auto fetch_grain = [&](int row) -> int {
        if constexpr (FR == FR_ONE) return 0;
        const int16_t* __restrict__ at = grain + (size_t)PF_CHK(row, ny) * nx;
        if constexpr (ACC == PAIRS) return *reinterpret_cast<const int*>(at + PF_CHK(cL, nx - 1));
        int a, b;
        load_grain_pair(at, cL, nx, vec, per, a, b);
        return (a & 0xffff) | (b << 16);
    };

    // ---------------- state of the sweep ----------------
    // rows r (suffix 0 in phase 2), p = r + 1 and p + 1; p0: the first row
    // whose phase 1 is evaluated (the ghost row -1 copies row 0; the psi
    // pass of the two-kernel form needs no row y0 - 1: no U fluxes)
    // With two rows per pass of the loop, a sweep of an odd number of rows starts
    // one row earlier (whose results reach nothing): the loop's remainder, a third
    // copy of the row's code that rounds one product differently, never runs, and
    // a cell's bits do not depend on where a sweep ends.
    constexpr int ROWS = sizeof(T) == 4 && FR == FR_ONE ? 2 : 1;
    static_assert(ROWS == 1 || ROWS == 2, "rows per pass");
    const int r_end = MODE == 1 ? y1 - 1 : y1;
    int p0 = MODE == 1 ? y0 : max(y0 - 1, 0);
    if (ROWS == 2) p0 -= (r_end - p0 + 1) & 1;
    const V2 zero = k_(T(0));
    const V2 Cm = fetch_row(psi, p0 - 1);
    V2 C0 = fetch_row(psi, p0);             // psi row p
    Diff dm_ = diffs(Cm), d0_ = diffs(C0);  // differences along x of rows p - 1, p
    V2 dm = C0 - Cm;                        // row p minus row p - 1
    // U, alphas and carries of row r
    V2 u0 = fetch_row(Uf, p0 - 1);
    V2 ue0 = east(u0) - u0;                // its differences E - C
    V2 aD0 = c_(1.0) - phi_of(Cm);         // 1 - phi
    V2 xD0 = aD0 + east(aD0);              // a + a_E
    V2 kD = zero;                          // corner sum of row r - 1
    V2 yD = zero, ppD = zero, gD = zero;   // y+ flux, +x+y and -x+y corner fluxes of row r - 1
    // The anti-trapping alpha (1 + (1-k) U) delta phi of row r and its sums and
    // carries, likewise, are kept in shared memory: only rows near the interface
    // read and write them, and the registers stay with the other rows.
    struct AT {
        V2 a, x, k, y, pp, g;
    };
    constexpr int ATN = sizeof(AT) / sizeof(V2);
    V2 phin0 = zero;                       // phi' of row r
    V2 rx = zero, ry = zero;               // S_{1,0}: |4 g h|^2 at the x+, y+ faces of row r
    // bit 0, 1: delta phi of rows r, r - 1 not exactly 0 all over the warp (clear before
    // the first row: only its carries toward the next row are read)
    unsigned live = 0;
    V2 Yc = zero;                          // anisotropy flux of the face between rows p - 1 and p
    // prefetch psi row p0 + 1 and U, grain row p0
    V2 nP = fetch_row(psi, p0 + 1), nU = fetch_row(Uf, p0);
    int nG = fetch_grain(max(p0, 0)), gf = nG;     // gf: the grains of the frames, and of the row that Yc was evaluated for
    if constexpr (MODE != 2) {
        // the face below row p0, in that row's frames
        if constexpr (FR != FR_ONE) set_frame(nG);
        const V2 gx = dm_.ex + d0_.ex, gn = c_(4.0) * dm;
        const V2 r2 = fma(gx, gx, gn * gn);
        Yc = face_flux<T, FR>(gx, gn, r2, rcp2(r2), F, an, false);
    }

#pragma unroll ROWS
    for (int r = p0 - 1; r < r_end; ++r) {
        const int p = r + 1;
        const V2 Cp = nP, u1 = nU;
        const int g1 = nG;
        nP = fetch_row(psi, r + 3);
        nU = fetch_row(Uf, r + 2);
        if constexpr (FR != FR_ONE) nG = fetch_grain(min(r + 2, ny - 1));
        const Diff dp_ = diffs(Cp);
        const V2 d0 = Cp - C0;
        const V2 ph = phi_of(C0);
        const V2 aD1 = c_(1.0) - ph;
        V2 den = fma(k_(-omk), phin0, k_(opk));  // 1 + k - (1-k) phi' of row r

        // ---------------- phase 1 at row p (its result is discarded at ghost rows) ----------------
        V2 phn, dph0 = zero, rxn = zero, ryn = zero;  // phi', T0's delta phi
        const V2 ey = d0 + dm, ey2 = ey + ey;
        if constexpr (MODE == 2) {
            // U pass of the two-kernel form: d psi/dt^n from the psi pass,
            // T0 increment, phi^n on the left
            dph0 = t0_dphi(aD1, ph, load_row(rate_b + (size_t)PF_CHK(max(min(p, ny - 1), 0), ny) * nx));
            phn = ph;
            den = rcp2(den);
            if constexpr (S == S10) {
                const V2 gxX = c_(4.0) * d0_.e, gyX = (dp_.e - dm_.e) + ey2;
                const V2 gxY = dp_.ex + d0_.ex, gyY = c_(4.0) * d0;
                rxn = fma(gxX, gxX, gyX * gyX);
                ryn = fma(gxY, gxY, gyY * gyY);
            }
        } else {
            bool moved = false;  // a column's grain is not the previous row's
            if constexpr (FR != FR_ONE) {
                moved = g1 != gf;
                if (moved) set_frame(g1);
            }
            const V2 ly = d0 - dm;
            // x+ and y+ faces, centre
            const V2 gxX = c_(4.0) * d0_.e, gyX = (dp_.e - dm_.e) + ey2;
            const V2 gxY = dp_.ex + d0_.ex, gyY = c_(4.0) * d0;
            const V2 rX = fma(gxX, gxX, gyX * gyX);
            const V2 rY = fma(gxY, gxY, gyY * gyY);
            const V2 rC = fma(d0_.ex, d0_.ex, ey * ey);
            const V2 iX = rcp2(rX), iY = rcp2(rY), iC = rcp2(rC);
            const V2 Xp = face_flux<T, FR>(gxX, gyX, rX, iX, F, an, true);
            const V2 Yp = face_flux<T, FR>(gxY, gyY, rY, iY, F, an, false);
            // x- faces: from the left column; recomputed across grain boundaries.
            // Lane 0 receives its own value: its column x0-2 feeds no output.
            V2 Xm = from_west(Xp), Ym = Yc;
            if constexpr (FR != FR_ONE) {
                const int gW = g_hi(shup(g1));
                const bool bL = gW != g_lo(g1), bR = g_lo(g1) != g_hi(g1);
                if (__any_sync(FULL, bL || bR)) {
                    const V2 gxW = c_(4.0) * (d0_.e - d0_.sx);  // C - W of row p
                    // (W + C)(p+1) - (W + C)(p-1) = 2 ey - (C - W)(p+1) + (C - W)(p-1)
                    const V2 gyW = ey2 - ((dp_.e - dp_.sx) - (dm_.e - dm_.sx));
                    const V2 r2 = fma(gxW, gxW, gyW * gyW);
                    const V2 q = face_flux<T, FR>(gxW, gyW, r2, rcp2(r2), F, an, true);
                    Xm = mk(bL ? q.x() : Xm.x(), bR ? q.y() : Xm.y());
                }
                if (__any_sync(FULL, moved)) {
                    const V2 gx = dm_.ex + d0_.ex, gn = c_(4.0) * dm;
                    const V2 r2 = fma(gx, gx, gn * gn);
                    const V2 q = face_flux<T, FR>(gx, gn, r2, rcp2(r2), F, an, false);
                    Ym = mk(g_lo(gf) != g_lo(g1) ? q.x() : Ym.x(), g_hi(gf) != g_hi(g1) ? q.y() : Ym.y());
                }
                gf = g1;
            }
            Yc = Yp;
            if constexpr (S == S10) {
                rxn = rX;
                ryn = rY;
            }
            const V2 N = (Xp - Xm) + (Yp - Ym);
            // Laplacian and minus sqrt2 times the gradient square
            V2 L, G;
            if constexpr (ISO) {
                L = fma(c_(4.0), d0_.sx + ly, (dm_.sx + dp_.sx) + (ly + ly));
                const V2 s = dp_.ex + dm_.ex, t = (dp_.sx - dm_.sx) + ey2;
                G = fma(c_(-1.41421356237309504880), rC, c_(-1.41421356237309504880 / 8.0) * fma(s, s, t * t));
            } else {
                L = d0_.sx + ly;
                G = c_(-1.41421356237309504880 / 4.0) * rC;
            }
            const V2 as = select_low<T>(rC, Low<T>::centre, T(1), aniso_as<T, FR>(d0_.ex, ey, iC, F, an));
            V2 uc = u1;      // F2 of Eq. PF_a
            T iF1 = T(1);    // 1 / F1
            if (DS) {
                T z = ::fma(T(p), zA, z0);
                if constexpr (sizeof(T) == 4) z += ::fma(T(p), zAl, z0l);
                uc = uc + k_(z);
                iF1 = M<T>::rcp(::fma(-omk, z, T(1)));
            }
            // sqrt2 [phi - lambda (1 - phi) (1 + phi) F2]
            const V2 src = fma(aD1 * fma(k_(-lam2), ph, k_(-lam2)), uc, k_(sq) * ph);
            const V2 E = (L + N) + src;
            den = rcp2(den);
            V2 rate = fma(ph, G, E * rcp2(as * as));
            if (DS) rate = rate * k_(iF1);
            const V2 psin = fma(k_(dtl), rate, C0);
            if constexpr (T0I) {
                // T0: chain-rule increment dt (1 - phi^2)/sqrt2 dpsi/dt and phi^n on the
                // left-hand side; phi' is not needed
                dph0 = t0_dphi(aD1, ph, rate);
                phn = ph;
            } else {
                phn = phi_of(psin);
                if (DS && t0) {
                    dph0 = t0_dphi(aD1, ph, rate);
                    phn = ph;
                }
            }
            if (p >= y0 && p < y1) {
                store_row(psi_o, p, psin);
                if constexpr (MODE == 1) store_row(rate_b, p, rate);  // in units of lap
            }
        }
        if constexpr (MODE != 1) {
            // ---------------- D fluxes at row r ----------------
            // The four owned fluxes of a D~_{2,1} divergence (times 4 x 6 h^2) from the
            // alphas of rows r (a0, x0s) and r+1 and the differences of beta along x, y
            // and both diagonals, and their sum over the cell's eight neighbours: the
            // neighbours' fluxes enter with the opposite sign, those of the column to the
            // left (its x+ face, its two corner fluxes) in one shuffle.
            auto corner = [&](V2 x0s, V2 x1s, V2 a0, V2 a1, V2& k, V2& fx, V2& fy) -> V2 {
                const V2 K = x0s + x1s;
                fx = fma(c_(4.0), x0s, K + k);
                fy = fma(c_(4.0), a0 + a1, K + from_west(K));
                k = K;
                return K;
            };
            auto gather = [&](V2 fx, V2 fy, V2 pp, V2 g, V2& yc, V2& ppc, V2& gc) -> V2 {
                const V2 v = (g - fx) - ppc;
                const V2 s = ((fx + pp) + (fy - yc)) + (from_west(v) - gc);
                yc = fy;
                ppc = pp;
                gc = g;
                return s;
            };
            const V2 ue1 = east(u1) - u1, dy = u1 - u0;
            const V2 xD1 = aD1 + east(aD1);
            V2 sD;
            if constexpr (ISO) {
                V2 fx, fy;
                const V2 K = corner(xD0, xD1, aD0, aD1, kD, fx, fy);
                sD = gather(fx * ue0, fy * dy, K * (ue1 + dy), K * (dy - ue0), yD, ppD, gD);
            } else {
                const V2 fx = c_(0.5) * xD0 * ue0, fy = c_(0.5) * (aD0 + aD1) * dy;
                sD = (fx - from_west(fx)) + (fy - yD);
                yD = fy;
            }

            // ---------------- alphas of row p, anti-trapping fluxes at row r ----------------
            // Where delta phi is exactly 0 over the whole warp (bulk liquid or solid, where
            // phi = +-1 exactly) on the rows r - 1 .. r + 1, every anti-trapping flux that
            // these rows form or carry is exactly 0 and nothing of it is evaluated.
            bool still;
            if constexpr (T0I || MODE == 2) {
                still = all_of(dph0, [](T d) { return d == T(0); });
            } else {
                const bool s2 = DS && t0 ? dph0.x() == T(0) && dph0.y() == T(0) : phn.x() == ph.x() && phn.y() == ph.y();
                still = __all_sync(FULL, s2);
            }
            const bool held = (live & 7u) != 0;  // the previous row left a state
            live = live << 1 | (still ? 0u : 1u);
            if (p >= ny || r < 0) {  // the ghost rows ny, -1 mirror rows ny - 1, 0
                asm volatile("");    // a branch, not selects on every row
                live = p >= ny ? (live & ~1u) | (live >> 1 & 1u) : (live & 1u) * 3u;
            }
            V2 num = zero;
            if (live & 7u) {
                AT at{zero, zero, zero, zero, zero, zero};
                if (held && r >= 0) {
                    V2* q = reinterpret_cast<V2*>(&at);
#pragma unroll
                    for (int i = 0; i < ATN; ++i) q[i] = park[32 * i + lane];
                }
                V2 aA1 = zero, xA1 = zero;
                if (!still) {
                    V2 dph = dph0;
                    if constexpr (!(T0I || MODE == 2))
                        if (!(DS && t0)) dph = phn - ph;
                    // (1 + (1-k) U) delta phi: the source of Eq. PF_b and, times 1 / (sqrt2 dt),
                    // the anti-trapping alpha
                    aA1 = fma(k_(omk), u1, c_(1.0)) * ghosts(dph);
                    xA1 = aA1 + east(aA1);
                }
                if (p >= ny) {
                    aA1 = at.a;
                    xA1 = at.x;
                }
                if (r < 0) {
                    at.a = aA1;
                    at.x = xA1;
                }
                V2 sA;
                if constexpr (ISO) {
                    V2 fx, fy;
                    const V2 Ka = corner(at.x, xA1, at.a, aA1, at.k, fx, fy);
                    V2 px = fx * dm_.e, py = fy * dm, ppp = Ka * (d0_.e + dm), pg = Ka * (dm - dm_.e);
                    if constexpr (S == S21) {
                        // App. B: each anti-trapping flux divided by |grad psi| at its point, from
                        // the psi rows r-2 .. r+2 (read again: only near the interface);
                        // ps(dx, dy) = psi at columns c + dx, row r + dy
                        const T ih = cst[C_IH], hh = cst[C_HH];
                        Row<T> Q[5];
#pragma unroll
                        for (int j = 0; j < 5; ++j) {
                            const V2 q = fetch_row(psi, r - 2 + j);
                            Q[j] = Row<T>{shup(q.x()), shup(q.y()), q.x(), q.y(), shdn(q.x()), shdn(q.y())};
                        }
                        auto ps = [&](int dx, int dyy) -> V2 { return Q[2 + dyy].pat(dx); };
                        const T ihd = ih * T(0.70710678118654752440);  // 1 / |e| of the <11> fluxes
                        const V2 mx = appb_face2<T>([&](int i, int j) { return ps(i, j); }, ih);
                        px = guarded_div2<T>(px, appb_floor2<T>(mx, dm_.e, ih), hh);
                        const V2 my = appb_face2<T>([&](int i, int j) { return ps(j, i); }, ih);
                        py = guarded_div2<T>(py, appb_floor2<T>(my, dm, ih), hh);
                        const V2 mc = appb_corner2<T>([&](int i, int j) { return ps(i, j); }, ih);  // both diagonals
                        ppp = guarded_div2<T>(ppp, appb_floor2<T>(mc, d0_.e + dm, ihd), hh);
                        pg = guarded_div2<T>(pg, appb_floor2<T>(mc, dm - dm_.e, ihd), hh);
                    }
                    sA = gather(px, py, ppp, pg, at.y, at.pp, at.g);
                } else {
                    // divided by |grad psi| of the face (h and the scale of alpha are in cA)
                    auto over = [&](V2 f, V2 r2) -> V2 {
                        return select_low<T>(r2, Low<T>::face, T(0), f * rcp2(each(r2, [](T m) { return M<T>::sqrt_(m); })));
                    };
                    const V2 px = over(c_(0.5) * at.x * dm_.e, rx), py = over(c_(0.5) * (at.a + aA1) * dm, ry);
                    sA = (px - from_west(px)) + (py - at.y);
                    at.y = py;
                }
                num = fma(k_(cA), sA, at.a);
                at.a = aA1;
                at.x = xA1;
                const V2* q = reinterpret_cast<const V2*>(&at);
#pragma unroll
                for (int i = 0; i < ATN; ++i) park[32 * i + lane] = q[i];
            }
            if (r >= y0) store_row(U_o, r, fma(fma(k_(cD), sD, num), den, u0));
            // row p becomes row r
            u0 = u1;
            ue0 = ue1;
            aD0 = aD1;
            xD0 = xD1;
            phin0 = phn;
            rx = rxn;
            ry = ryn;
        }
        dm_ = d0_;
        d0_ = dp_;
        C0 = Cp;
        dm = d0;
    }
}

// VAR 0: isothermal instances with mirror walls at the T1 time level (the
// flags of the others are compile-time false and their code disappears); VAR 1
// (DS): instances with a frozen temperature and/or periodic x, T1 or T0 read
// from the record; VAR 2: isothermal instances with mirror walls at the T0
// time level, T0 fixed at compile time.  FR: the crystal frames (above).  MODE
// (T0 time level only, VAR 1 or 2): 0 the fused step; 1 the psi pass of the
// two-kernel form of Sec. 3.3.1, which stores psi' and d psi/dt
// (InstRec::rate); 2 its U pass, which reads d psi/dt back instead of
// recomputing phase 1 (U' needs only psi^n, U^n and d psi/dt^n at the T0
// level).
template <typename T, int S, int VAR, int FR, int MODE>
__global__ void __launch_bounds__(32, sizeof(T) == 4 ? BLOCKS_F32<S, FR> : 1)
    k_step2d(const WorkItem* __restrict__ work, int n_work, const InstRec* __restrict__ recs, int launch_parity,
             StepClock clk) {
    __shared__ V<T> park[6 * 32];
    after_previous();
    for (int w = blockIdx.x; w < n_work; w += gridDim.x) {
        const WorkItem wi = work[w];
        const InstRec& rec = recs[wi.inst];
        if constexpr (sizeof(T) == 4) {
            // FP64 rows take the general access: its cost disappears behind the FP64 units
            if (wi.x0 >= 2 && wi.x0 + 62 <= rec.nx) {
                if ((rec.nx & 1) == 0)
                    sweep2d<T, S, VAR, FR, MODE, PAIRS>(wi, rec, launch_parity, clk, park);
                else
                    sweep2d<T, S, VAR, FR, MODE, SINGLES>(wi, rec, launch_parity, clk, park);
                continue;
            }
        }
        sweep2d<T, S, VAR, FR, MODE, WALL>(wi, rec, launch_parity, clk, park);
    }
}

}  // namespace
}  // namespace pf
