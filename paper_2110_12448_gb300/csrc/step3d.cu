// step3d.cu -- explicit time step of the quantitative alloy phase-field model
// in 3D for sm_103a (arXiv:2110.12448, Sec. 5-6, Eqs. PF_a and PF_b).
//
// A step is two passes over the grid, the paper's own order: the psi pass
// forms psi' from psi and U; the U pass forms U' from U, psi and psi'.  It
// takes delta phi from psi and psi' cell by cell, so that nothing else travels
// between the passes (the T0 level's increment takes d psi/dt, which the psi
// pass then stores): 28 bytes per cell (FP32) instead of the 16 of one pass.
// HBM has room for that (two passes over 256^3 take 70 us at the copy rate),
// while one pass has to evaluate the psi rate again on a ring around every
// tile (1.42 times the cells with 30 x 6 columns), to exchange planes through
// shared memory under three barriers a plane, and to hold both phases' state:
// it measured 862 us a step on 256^3 where the two passes take 364 (356 before the
// vote on a plane's phase looked for NaN and the fields were read by plain loads).
//
// Both passes share one layout.  A warp owns two rows (y, y + 1) of a strip of
// 32 columns, 16 lanes with a packed pair of columns each, and marches along
// z; nothing is shared between warps, there is no barrier.  A plane is read as
// three rows of the strip (S, own, N; the rows that neighbouring warps of the
// block read too hit L1), one plane ahead; x neighbours come over 16-lane
// shuffles; what later planes need of a plane is kept as differences along x
// and y in registers.  The outer column on each side is halo: 30 of 32 columns
// are outputs (a strip of 64 columns and one row per warp would waste more on
// grids of 64 to 256 cells: 5 strips of 62 for 256 against 9 of 30).
//
// psi pass (see step2d_kernel.cuh for the notation; sy = N + S - 2C, lz the
// same along z, subscript k: planes above and below):
//   6 h^2 L_{1,2,0} = 2 (sx + lz) + 4 (sy + lz) + sx(N) + sx(S) + sx_k + sy_k
//   6 h^2 G_{1,2,0} = (ex^2 + ey^2 + ez^2) / 2 + sum over the three planes of
//     (s^2 + t^2) / 8, s and t the sum and difference of the diagonal differences
//   <100> faces: x- from the west column, z- from the plane below (same grain),
//     y+ and y- both evaluated (they belong to two warps)
// U pass: the eighteen D~_{1,2,0} fluxes of a cell.  A face weighs (times 8)
//   4 (a + a_e) plus the eight alphas beside the pair, an edge (times 32) 6 times
//   the four alphas of its square plus the eight beside it; both diagonals of a
//   square share its weight.  The weights are linear in alpha: each plane adds
//   its part to them when it is read.  Where phi = +-1 exactly on the planes
//   below, at and above the warp's rows, before and after the step, the weights
//   are constants (liquid) or everything is zero (solid) and neither phi nor the
//   anti-trapping term is evaluated: the same bits at a fraction of the work.
// S_{1,0,0}: the <100> shell with a two-point face mean for D and the standard
// anti-trapping normalised by the face gradient.
// Walls: mirrors in y and z, mirror or periodic in x, by the index of the row
// or column that is read.
// What bounds them (256^3, S-bar_{1,2,0}): the psi pass instruction issue and the
// FMA pipe (195 warp instructions per 60 cells, 115 of them packed arithmetic, 54 %
// of the issue slots with 12 warps per SM), the U pass the latency of its rows.
#include <cfloat>

#include "step2d.cuh"

namespace pf {
namespace {

constexpr int SEG = 16;   // lanes of a row

template <typename T> __device__ __forceinline__ T up16(T v) { return __shfl_up_sync(FULL, v, 1, SEG); }
template <typename T> __device__ __forceinline__ T dn16(T v) { return __shfl_down_sync(FULL, v, 1, SEG); }
template <typename T> __device__ __forceinline__ V<T> east3(V<T> c) { return mk(c.y(), dn16(c.x())); }
template <typename T> __device__ __forceinline__ V<T> west3(V<T> f) { return mk(up16(f.y()), f.x()); }
template <typename T, typename F> __device__ __forceinline__ V<T> each3(V<T> a, F f) { return mk(f(a.x()), f(a.y())); }

// the crystal frames of a lane's two columns (crystal -> lab, row-major)
template <typename T> struct Frame3 {
    V<T> R[9];
};

// |psi| beyond which phi is exactly +-1 in the pass's arithmetic (FP32: 2 / (1 +
// e^{sqrt2 |psi|}) below a quarter ulp of 1)
template <typename T> struct Sat;
template <> struct Sat<float> { static constexpr float psi = 14.0f; };
template <> struct Sat<double> { static constexpr double psi = 32.0; };

// max and min that return NaN where an operand is one
__device__ __forceinline__ float max_nan(float a, float b) {
    float r;
    asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float min_nan(float a, float b) {
    float r;
    asm("min.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ double max_nan(double a, double b) { return a > b || isnan(a) ? a : b; }
__device__ __forceinline__ double min_nan(double a, double b) { return a < b || isnan(a) ? a : b; }
template <typename T> struct Largest;
template <> struct Largest<float> { static constexpr float v = FLT_MAX; };
template <> struct Largest<double> { static constexpr double v = DBL_MAX; };

// Component `ax` of (J - g), J = d(a_s^2 |g|^2 / 2)/dg, times `scale`, for
// gradients times 4 h in the lanes' frames: with c = R^T g, t_p = c_p^2, s_p =
// t_p / |c|^2 and q = sum s_p^2, a_s = 1 - 3 eps + 4 eps q and
// J'_p - c_p = c_p (a^2 - 1 - 16 eps a q + 16 eps a s_p).  0 below the guard.
template <typename T> struct Cubic {
    T eps4, base, eps16, scale;  // 4 eps, 1 - 3 eps, 16 eps
    __device__ __forceinline__ Cubic(T e, T s) : eps4(T(4) * e), base(T(1) - T(3) * e), eps16(T(16) * e), scale(s) {}
};
template <typename T>
__device__ __forceinline__ V<T> frame_q(const V<T> g[3], const Frame3<T>& F, V<T> c[3], V<T> t[3], V<T>& r2, V<T>& inv) {
#pragma unroll
    for (int p = 0; p < 3; ++p) {
        c[p] = fma(F.R[p], g[0], fma(F.R[3 + p], g[1], F.R[6 + p] * g[2]));
        t[p] = c[p] * c[p];
    }
    r2 = (t[0] + t[1]) + t[2];
    inv = rcp2(r2);
    return (fma(t[0], t[0], fma(t[1], t[1], t[2] * t[2])) * inv) * inv;
}
template <typename T>
__device__ __forceinline__ V<T> face3(V<T> gx, V<T> gy, V<T> gz, const Frame3<T>& F, const Cubic<T>& A, int ax) {
    const V<T> g[3] = {gx, gy, gz};
    V<T> c[3], t[3], r2, inv;
    const V<T> q = frame_q<T>(g, F, c, t, r2, inv);
    const V<T> a = fma(bc<T>(A.eps4), q, bc<T>(A.base));
    const V<T> c1 = bc<T>(A.eps16) * a;
    const V<T> c0 = fma(a, a, bc<T>(T(-1))) - c1 * q;
    const V<T> ci = c1 * inv;
    V<T> o = F.R[3 * ax] * (c[0] * fma(ci, t[0], c0));
    o = fma(F.R[3 * ax + 1], c[1] * fma(ci, t[1], c0), o);
    o = fma(F.R[3 * ax + 2], c[2] * fma(ci, t[2], c0), o) * bc<T>(A.scale);
    const T low = T(16) * Guard<T>::v;
    return mk(r2.x() < low ? T(0) : o.x(), r2.y() < low ? T(0) : o.y());
}
// a_s of a centred difference (times 2 h); 1 below the guard
template <typename T>
__device__ __forceinline__ V<T> centre3(V<T> gx, V<T> gy, V<T> gz, const Frame3<T>& F, const Cubic<T>& A) {
    const V<T> g[3] = {gx, gy, gz};
    V<T> c[3], t[3], r2, inv;
    const V<T> q = frame_q<T>(g, F, c, t, r2, inv);
    const V<T> a = fma(bc<T>(A.eps4), q, bc<T>(A.base));
    const T low = T(4) * Guard<T>::v;
    return mk(r2.x() < low ? T(1) : a.x(), r2.y() < low ? T(1) : a.y());
}

// Where a lane reads and writes: its pair of columns in the rows S, own, N.
// PAIRS: both columns inside the grid in every lane of the strip and rows
// aligned to pairs (vector accesses); else one access per column, at its
// mirrored or wrapped index.
template <bool PAIRS> struct Where {
    long long oS, o0, oN;  // offsets in a plane of the first column's cell
    int db;                // the second column's offset from the first
    bool okL, okR;         // output columns
    __device__ __forceinline__ Where(const WorkItem& wi, const InstRec& rec, int row) {
        const int nx = rec.nx, ny = rec.ny, l = threadIdx.x & (SEG - 1);
        const int c = wi.x0 - 2 + 2 * l;
        const bool per = rec.bcx != 0;
        const int a = PAIRS ? c : col_idx(c, nx, per), b = PAIRS ? c + 1 : col_idx(c + 1, nx, per);
        const int y = mirror_idx(row, ny);  // rows beyond the last compute a copy that is not stored
        oS = (long long)PF_CHK(mirror_idx(y - 1, ny), ny) * nx + PF_CHK(a, nx);
        o0 = (long long)PF_CHK(y, ny) * nx + PF_CHK(a, nx);
        oN = (long long)PF_CHK(mirror_idx(y + 1, ny), ny) * nx + PF_CHK(a, nx);
        db = PF_CHK(b, nx) - a;
        const bool mine = row < ny;
        okL = mine && l > 0 && c >= 0 && c < nx;
        okR = mine && l < SEG - 1 && c + 1 >= 0 && c + 1 < nx;
    }
    template <typename T> __device__ __forceinline__ V<T> load(const T* __restrict__ plane, long long o) const {
        if constexpr (PAIRS) {
            const typename Vec2<T>::t v = *reinterpret_cast<const typename Vec2<T>::t*>(plane + o);
            return mk(v.x, v.y);
        }
        return mk(plane[o], plane[o + db]);
    }
    template <typename T> __device__ __forceinline__ void store(T* __restrict__ plane, V<T> v) const {
        if (PAIRS && okL && okR) {
            typename Vec2<T>::t q;
            q.x = v.x();
            q.y = v.y();
            *reinterpret_cast<typename Vec2<T>::t*>(plane + o0) = q;
        } else {
            if (okL) plane[o0] = v.x();
            if (okR) plane[o0 + 1] = v.y();
        }
    }
};

// ---------------------------------------------------------------------------
// psi pass
// ---------------------------------------------------------------------------
template <typename T, int S, bool ONE, bool PAIRS>
__device__ __forceinline__ void psi_sweep(const WorkItem& wi, const InstRec& rec, int launch_parity, const StepClock& clk) {
    constexpr bool ISO = S == SBAR120;
    using V2 = V<T>;
    auto c_ = [](double x) -> V2 { return bc<T>(T(x)); };
    auto k_ = [](T x) -> V2 { return bc<T>(x); };
    const int ny = rec.ny, nz = rec.nz;
    const long long sxy = (long long)rec.nx * ny;
    const int par = rec.parity_offset ^ launch_parity;
    const T* __restrict__ psi = static_cast<const T*>(rec.psi[par]);
    const T* __restrict__ Uf = static_cast<const T*>(rec.U[par]);
    T* __restrict__ psi_o = static_cast<T*>(rec.psi[par ^ 1]);
    T* __restrict__ rate_b = static_cast<T*>(rec.rate);  // T0: d psi/dt for the U pass, in units of 1 / (6 h^2) or 1 / h^2
    const int16_t* __restrict__ grain = rec.grain;
    const T* __restrict__ rot = static_cast<const T*>(rec.rot);
    const T* cst = ConstOf<T>::get(rec);
    const T omk = cst[C_OMK];
    const T dtl = ISO ? cst[C_DTL21] : cst[C_DTL10];  // Eq. PF_a in units of 1 / (6 h^2) or 1 / h^2
    const T sq = ISO ? cst[C_SQ21] : cst[C_SQ10], lam2 = ISO ? cst[C_LAM21] : cst[C_LAM10];
    const Cubic<T> an(cst[C_EPS], ISO ? T(1.5) : T(0.25));
    const int row = wi.y0 + 2 * (threadIdx.x >> 5) + ((threadIdx.x & 31) >> 4);
    const Where<PAIRS> at(wi, rec, row);
    // frozen temperature along +y: zeta of the lane's row at this launch's step
    T zc = T(0), iF1 = T(1);
    if (rec.thermal) {
        const long long n = clk.clock ? clk.base[wi.inst] + *clk.clock : clk.step;
        zc = (T)((double)mirror_idx(row, ny) * rec.zA - rec.zB - (double)n * rec.zC);
        iF1 = T(1) / (T(1) - omk * zc);
    }
    auto plane = [&](const T* f, int z) -> const T* { return f + (long long)PF_CHK(mirror_idx(z, nz), nz) * sxy; };

    // what the pass keeps of a plane: the row itself, its differences along x
    // (e = E - C, ex = E - W, sx = E + W - 2C) and y (n = N - C, ey = N - S, sy),
    // and of its neighbour rows what the plane's own operators need
    struct Plane {
        V2 C, e, ex, sx, n, ey, sy;
        V2 exN, exS, sxj, txy, eyX;
    };
    auto make = [&](V2 cS, V2 c0, V2 cN) -> Plane {
        Plane q;
        q.C = c0;
        const V2 eS = east3(cS) - cS, eN = east3(cN) - cN;
        q.e = east3(c0) - c0;
        const V2 wS = west3(eS), w0 = west3(q.e), wN = west3(eN);
        q.ex = q.e + w0;
        q.sx = q.e - w0;
        q.exN = eN + wN;
        q.exS = eS + wS;
        const V2 sN = eN - wN, sS = eS - wS;
        q.n = cN - c0;
        const V2 s = c0 - cS;
        q.ey = q.n + s;
        q.sy = q.n - s;
        const V2 e2 = q.ey + q.ey;
        q.sxj = sN + sS;
        q.txy = (sN - sS) + e2;  // difference of the diagonal differences in the xy plane
        q.eyX = (eN - eS) + e2;  // 4 h times the y component at the x+ face
        return q;
    };
    auto read = [&](int z) -> Plane {
        const T* P = plane(psi, z);
        return make(at.template load<T>(P, at.oS), at.template load<T>(P, at.o0), at.template load<T>(P, at.oN));
    };
    auto grains = [&](int z) -> int {
        if constexpr (ONE) return 0;
        const int16_t* G = grain + (long long)PF_CHK(mirror_idx(z, nz), nz) * sxy + at.o0;
        return (G[0] & 0xffff) | (G[at.db] << 16);
    };
    auto g_lo = [](int g) -> int { return (int)(int16_t)(g & 0xffff); };
    auto g_hi = [](int g) -> int { return g >> 16; };
    Frame3<T> F;
    auto set_frame = [&](int g) {
        const T* A = rot + 9 * PF_CHK(g_lo(g), rec.n_grains);
        const T* B = rot + 9 * PF_CHK(g_hi(g), rec.n_grains);
#pragma unroll
        for (int q = 0; q < 9; ++q) F.R[q] = mk(__ldg(A + q), __ldg(B + q));
    };

    const int z0 = wi.z0, z1 = min(z0 + wi.ext, nz);
    Plane m = read(z0 - 1), o = read(z0);
    V2 dm = o.C - m.C;
    int g0 = grains(z0), gf = g0;  // gf: the grains of the frames, and of the plane that Zc was evaluated for
    set_frame(g0);
    V2 Zc = face3<T>(m.ex + o.ex, m.ey + o.ey, c_(4.0) * dm, F, an, 2);  // the face below plane z0
    V2 nS, n0, nN, nU;
    {
        const T* P = plane(psi, z0 + 1);
        nS = at.template load<T>(P, at.oS);
        n0 = at.template load<T>(P, at.o0);
        nN = at.template load<T>(P, at.oN);
        nU = at.template load<T>(plane(Uf, z0), at.o0);
    }
    for (int z = z0; z < z1; ++z) {
        const Plane p = make(nS, n0, nN);
        const V2 u = nU + k_(zc);
        {
            const T* P = plane(psi, z + 2);
            nS = at.template load<T>(P, at.oS);
            n0 = at.template load<T>(P, at.o0);
            nN = at.template load<T>(P, at.oN);
            nU = at.template load<T>(plane(Uf, z + 1), at.o0);
        }
        const V2 d = p.C - o.C, ez = d + dm, lz = d - dm, ez2 = ez + ez;
        bool moved = false;  // a column's grain is not the plane below's
        if constexpr (!ONE) {
            moved = g0 != gf;
            if (moved) set_frame(g0);
        }
        const V2 Xp = face3<T>(c_(4.0) * o.e, o.eyX, (p.e - m.e) + ez2, F, an, 0);
        const V2 nd = p.n - m.n;
        const V2 Yp = face3<T>(o.ex + o.exN, c_(4.0) * o.n, nd + ez2, F, an, 1);
        // (C + S)(z+1) - (C + S)(z-1) = 2 ez - (C - S)(z+1) + (C - S)(z-1)
        const V2 Ym = face3<T>(o.ex + o.exS, c_(4.0) * (o.ey - o.n), ez2 - ((p.ey - m.ey) - nd), F, an, 1);
        const V2 Zp = face3<T>(o.ex + p.ex, o.ey + p.ey, c_(4.0) * d, F, an, 2);
        V2 Xm = west3(Xp), Zm = Zc;
        if constexpr (!ONE) {
            // faces whose other side is in another grain are evaluated in the cell's own frame
            const int gW = g_hi(up16(g0));
            const bool bL = gW != g_lo(g0), bR = g_lo(g0) != g_hi(g0);
            if (__any_sync(FULL, bL || bR)) {
                const V2 q = face3<T>(c_(4.0) * (o.e - o.sx), ((o.ey + o.ey) + o.txy) - o.eyX,
                                      ez2 - ((p.e - p.sx) - (m.e - m.sx)), F, an, 0);
                Xm = mk(bL ? q.x() : Xm.x(), bR ? q.y() : Xm.y());
            }
            if (__any_sync(FULL, moved)) {
                const V2 q = face3<T>(m.ex + o.ex, m.ey + o.ey, c_(4.0) * dm, F, an, 2);
                Zm = mk(g_lo(gf) != g_lo(g0) ? q.x() : Zm.x(), g_hi(gf) != g_hi(g0) ? q.y() : Zm.y());
            }
            gf = g0;
            g0 = grains(z + 1);
        }
        Zc = Zp;
        const V2 N = ((Xp - Xm) + (Yp - Ym)) + (Zp - Zm);
        const V2 rC = fma(o.ex, o.ex, fma(o.ey, o.ey, ez * ez));
        V2 L, G;  // Laplacian and minus sqrt2 times the gradient square
        if constexpr (ISO) {
            L = fma(c_(2.0), o.sx + lz, fma(c_(4.0), o.sy + lz, (o.sxj + (p.sx + m.sx)) + (p.sy + m.sy)));
            const V2 sxy_ = o.exN + o.exS, sxz = p.ex + m.ex, syz = p.ey + m.ey;
            const V2 txz = (p.sx - m.sx) + ez2, tyz = (p.sy - m.sy) + ez2;
            V2 g = fma(sxy_, sxy_, o.txy * o.txy);
            g = fma(sxz, sxz, fma(txz, txz, g));
            g = fma(syz, syz, fma(tyz, tyz, g));
            G = fma(c_(-1.41421356237309504880 / 2.0), rC, c_(-1.41421356237309504880 / 8.0) * g);
        } else {
            L = (o.sx + o.sy) + lz;
            G = c_(-1.41421356237309504880 / 4.0) * rC;
        }
        const V2 as = centre3<T>(o.ex, o.ey, ez, F, an);
        const V2 ph = each3(o.C, [](T x) {
            if constexpr (sizeof(T) == 8) return fabs(x) > Sat<T>::psi ? (x > T(0) ? T(1) : T(-1)) : M<T>::tanh_isq2(x);
            else return M<T>::tanh_isq2(x);
        });
        const V2 src = fma((c_(1.0) - ph) * fma(k_(-lam2), ph, k_(-lam2)), u, k_(sq) * ph);
        const V2 E = (L + N) + src;
        const V2 rate = fma(ph, G, E * rcp2(as * as)) * k_(iF1);
        at.template store<T>(psi_o + (long long)PF_CHK(z, nz) * sxy, fma(k_(dtl), rate, o.C));
        if (rate_b) at.template store<T>(rate_b + (long long)PF_CHK(z, nz) * sxy, rate);
        m = o;
        o = p;
        dm = d;
    }
}

// ---------------------------------------------------------------------------
// U pass
// ---------------------------------------------------------------------------
// What a divergence keeps between planes: the parts of plane 0's weights (in
// the plane: x, y+, y- faces, xy squares toward N and S; toward the plane
// above: z face, xz square, yz squares toward N and S) and the sums that the
// plane above adds to its own; and the fluxes through plane 0's lower side.
template <typename T> struct Sums3 {
    V<T> px, pyN, pyS, pqN, pqS;       // partial weights of plane 0
    V<T> rx, ryN, ryS, rqN, rqS;       // alpha sums of plane 0 that plane 1's weights take
    V<T> wz, wxz, wyN, wyS;            // plane 0's part of the weights toward plane 1
};
template <typename T> struct Carry3 {
    V<T> fz, pp, g, yz;                // fluxes between planes -1 and 0
};
template <typename T> struct Div3 {
    Sums3<T> s;
    Carry3<T> c;
};
// differences of the divergence's beta in a plane: along x in the rows own, N,
// S, and to the rows N and S
template <typename T> struct Beta3 {
    V<T> C, e, eN, eS, n, s;
};
template <typename T> __device__ __forceinline__ Beta3<T> beta3(V<T> cS, V<T> c0, V<T> cN) {
    Beta3<T> b;
    b.C = c0;
    b.e = east3(c0) - c0;
    b.eN = east3(cN) - cN;
    b.eS = east3(cS) - cS;
    b.n = cN - c0;
    b.s = cS - c0;
    return b;
}
// the weights of plane 0's owned fluxes (faces times 8, edges times 32)
template <typename T> struct Weights3 {
    V<T> x, yN, yS, z, qN, qS, xz, yzN, yzS;
};
// alphas of plane 1 (rows S, own, N): completes plane 0's weights, then makes
// plane 1 the stored plane
template <typename T> __device__ __forceinline__ Weights3<T> weights3(Sums3<T>& D, V<T> aS, V<T> a0, V<T> aN) {
    auto c_ = [](double x) -> V<T> { return bc<T>(T(x)); };
    const V<T> xs = a0 + east3(a0), xN = aN + east3(aN), xS = aS + east3(aS);
    // E + W of each row
    const V<T> t0 = fma(c_(-2.0), a0, xs + west3(xs)), tN = fma(c_(-2.0), aN, xN + west3(xN)),
               tS = fma(c_(-2.0), aS, xS + west3(xS));
    const V<T> yN = a0 + aN, yS = a0 + aS, P = xN + xS, qN = xs + xN, qS = xs + xS;
    const V<T> bN = t0 + tN, bS = t0 + tS;
    Weights3<T> w;
    w.x = D.px + xs;
    w.yN = D.pyN + yN;
    w.yS = D.pyS + yS;
    w.qN = D.pqN + qN;
    w.qS = D.pqS + qS;
    const V<T> wz = fma(c_(4.0), a0, t0 + (aN + aS)), wxz = fma(c_(6.0), xs, P), wyN = fma(c_(6.0), yN, bN),
               wyS = fma(c_(6.0), yS, bS);
    w.z = D.wz + wz;
    w.xz = D.wxz + wxz;
    w.yzN = D.wyN + wyN;
    w.yzS = D.wyS + wyS;
    D.px = fma(c_(4.0), xs, P) + D.rx;
    D.pyN = fma(c_(4.0), yN, bN) + D.ryN;
    D.pyS = fma(c_(4.0), yS, bS) + D.ryS;
    D.pqN = fma(c_(6.0), qN, D.rqN);
    D.pqS = fma(c_(6.0), qS, D.rqS);
    D.rx = xs;
    D.ryN = yN;
    D.ryS = yS;
    D.rqN = qN;
    D.rqS = qS;
    D.wz = wz;
    D.wxz = wxz;
    D.wyN = wyN;
    D.wyS = wyS;
    return w;
}
// a plane (and the one below it) of the same alpha everywhere
template <typename T> __device__ __forceinline__ void uniform3(Sums3<T>& D, T a) {
    D.rx = D.ryN = D.ryS = bc<T>(T(2) * a);
    D.rqN = D.rqS = bc<T>(T(4) * a);
    D.px = D.pyN = D.pyS = bc<T>(T(14) * a);
    D.pqN = D.pqS = bc<T>(T(28) * a);
    D.wz = bc<T>(T(8) * a);
    D.wxz = D.wyN = D.wyS = bc<T>(T(16) * a);
}
template <typename T> __device__ __forceinline__ Weights3<T> const_weights3(T a) {
    Weights3<T> w;
    w.x = w.yN = w.yS = w.z = bc<T>(T(16) * a);
    w.qN = w.qS = w.xz = w.yzN = w.yzS = bc<T>(T(32) * a);
    return w;
}
// Sum over the eighteen neighbours (times 32 x 6 h^2) from plane 0's weights and
// the differences of beta in planes 0 and 1 (d = C1 - C0).  The fluxes of the
// column to the west (its x+ face, its diagonals toward this column) arrive in
// one shuffle, those of the plane below by carry.
template <typename T>
__device__ __forceinline__ V<T> gather3(Carry3<T>& D, const Weights3<T>& w, const Beta3<T>& b0, const Beta3<T>& b1, V<T> d) {
    const V<T> fx = w.x * b0.e;
    const V<T> fz = w.z * d;
    const V<T> pp = w.xz * (b1.e + d), g = w.xz * (d - b0.e);
    // diagonals of the xy squares: to NE, SE, and what the column to the east gets of N, S
    const V<T> ne = fma(w.qN, b0.eN + b0.n, w.qS * (b0.eS + b0.s));
    const V<T> nw = fma(w.qN, b0.n - b0.e, w.qS * (b0.s - b0.e));
    const V<T> v = (nw + g) - (D.pp + fx * bc<T>(T(4)));
    const V<T> faces = (fma(w.yN, b0.n, w.yS * b0.s) + fx) + (fz - D.fz);
    const V<T> yz = fma(w.yzN, b1.n + d, w.yzS * (b1.s + d));
    const V<T> sum = fma(bc<T>(T(4)), faces, ((ne + pp) + (yz + D.yz)) + (west3(v) - D.g));
    D.fz = fz;
    D.pp = pp;
    D.g = g;
    D.yz = fma(w.yzN, b0.n - d, w.yzS * (b0.s - d));
    return sum;
}

template <typename T, int S, bool PAIRS>
__device__ __forceinline__ void u_sweep(const WorkItem& wi, const InstRec& rec, int launch_parity, V<T>* park) {
    constexpr bool ISO = S == SBAR120;
    using V2 = V<T>;
    auto c_ = [](double x) -> V2 { return bc<T>(T(x)); };
    auto k_ = [](T x) -> V2 { return bc<T>(x); };
    const int ny = rec.ny, nz = rec.nz;
    const long long sxy = (long long)rec.nx * ny;
    const int par = rec.parity_offset ^ launch_parity;
    const T* __restrict__ psi = static_cast<const T*>(rec.psi[par]);
    const bool t0 = rec.tlevel != 0;  // T0 time level
    // from the psi pass: psi', or at the T0 level d psi/dt
    const T* __restrict__ psn = static_cast<const T*>(t0 ? rec.rate : rec.psi[par ^ 1]);
    const T* __restrict__ Uf = static_cast<const T*>(rec.U[par]);
    T* __restrict__ U_o = static_cast<T*>(rec.U[par ^ 1]);
    const T* cst = ConstOf<T>::get(rec);
    const T omk = cst[C_OMK], opk = cst[C_OPK];
    const T cD = ISO ? cst[C_UD120] : cst[C_UD100], cA = ISO ? cst[C_UA120] : cst[C_UA100];
    const T dts = (ISO ? cst[C_DTL21] : cst[C_DTL10]) * T(0.70710678118654752440);
    const int row = wi.y0 + 2 * (threadIdx.x >> 5) + ((threadIdx.x & 31) >> 4);
    const Where<PAIRS> at(wi, rec, row);
    auto plane = [&](const T* f, int z) -> const T* { return f + (long long)PF_CHK(mirror_idx(z, nz), nz) * sxy; };
    struct Rows {
        V2 lo, C, hi;  // rows y - 1, y, y + 1
    };
    auto read = [&](const T* f, int z) -> Rows {
        const T* P = plane(f, z);
        return Rows{at.template load<T>(P, at.oS), at.template load<T>(P, at.o0), at.template load<T>(P, at.oN)};
    };
    // phi of every cell the warp reads of a plane: -1 or 1 exactly, before and (T1) after the step; else 0.
    // A NaN is in neither phase, nor is a plane whose d psi/dt (T0) or, where phi = 1, U is not finite:
    // there the products with alphas of 0 are evaluated, so that NaN and infinities reach U' as they would.
    auto phase_of = [&](const Rows& a, const Rows& q, const Rows& u) -> int {
        const Rows b = t0 ? a : q;
        auto hi = [](V2 x, V2 y) -> T { return max_nan(max_nan(x.x(), x.y()), max_nan(y.x(), y.y())); };
        auto lo = [](V2 x, V2 y) -> T { return min_nan(min_nan(x.x(), x.y()), min_nan(y.x(), y.y())); };
        auto finite = [](const Rows& r) -> bool {
            T m = max_nan(fabs(r.C.x()), fabs(r.C.y()));
            m = max_nan(m, max_nan(fabs(r.lo.x()), fabs(r.lo.y())));
            return max_nan(m, max_nan(fabs(r.hi.x()), fabs(r.hi.y()))) <= Largest<T>::v;
        };
        const T B = Sat<T>::psi;
        const T h = max_nan(max_nan(hi(a.lo, b.lo), hi(a.C, b.C)), hi(a.hi, b.hi)),
                l = min_nan(min_nan(lo(a.lo, b.lo), lo(a.C, b.C)), lo(a.hi, b.hi));
        const bool rate = !t0 || finite(q);
        if (__all_sync(FULL, h < -B && rate)) return -1;
        return __all_sync(FULL, l > B && rate && finite(u)) ? 1 : 0;
    };
    auto phi = [](V2 p) -> V2 {
        return each3(p, [](T x) {
            if constexpr (sizeof(T) == 8) return fabs(x) > Sat<T>::psi ? (x > T(0) ? T(1) : T(-1)) : M<T>::tanh_isq2(x);
            else return M<T>::tanh_isq2(x);
        });
    };
    // alphas of a row: 1 - phi, and (1 + (1-k) U) delta phi with its phi'
    auto alphas = [&](V2 p, V2 q, V2 u, V2& aD, V2& aA, V2& phn) {
        const V2 ph = phi(p);
        aD = c_(1.0) - ph;
        V2 dph;
        if (t0) {  // delta phi = dt (1 - phi^2) / sqrt2 d psi/dt, phi^n on the left-hand side
            dph = (aD * fma(k_(dts), ph, k_(dts))) * q;
            phn = ph;
        } else {
            phn = phi(q);
            dph = phn - ph;
        }
        aA = fma(k_(omk), u, c_(1.0)) * dph;
    };

    const int z0 = wi.z0, z1 = min(z0 + wi.ext, nz);
    const V2 zero = k_(T(0));
    // The state that only planes near the interface need lives in shared memory,
    // a slot per thread: the D term's sums, then the anti-trapping divergence.
    Carry3<T> D{zero, zero, zero, zero};
    constexpr int SUMS = sizeof(Sums3<T>) / sizeof(V2), ALL = sizeof(Div3<T>) / sizeof(V2);
    auto put = [&](const void* v, int slot, int n) {
        const V2* q = static_cast<const V2*>(v);
#pragma unroll
        for (int i = 0; i < n; ++i) park[(slot + i) * blockDim.x + threadIdx.x] = q[i];
    };
    auto get = [&](void* v, int slot, int n) {
        V2* q = static_cast<V2*>(v);
#pragma unroll
        for (int i = 0; i < n; ++i) q[i] = park[(slot + i) * blockDim.x + threadIdx.x];
    };
    auto clear = [&](Div3<T>& X) {
        uniform3<T>(X.s, T(0));
        X.c = Carry3<T>{zero, zero, zero, zero};
    };
    // S_{1,0,0}: the two-cell sums of a plane (the face weights times 2)
    auto faces_only = [&](Sums3<T>& X, V2 xS, V2 x, V2 xN) {
        X.rx = x + east3(x);
        X.ryN = x + xN;
        X.ryS = x + xS;
        X.wz = x;
    };
    // plane z0 - 1: its alphas enter the weights; the carries start at zero,
    // and what they leave out reaches only plane z0 - 1
    int c0, cm = 2;  // phases of planes z and z - 1 (2: not the same as any)
    Beta3<T> b0;     // U's differences in plane z
    V2 phn0 = zero, aA0 = zero;  // phi' and the anti-trapping alpha of the own row in plane z
    bool fresh = true;           // the D term's sums in shared memory are plane z's
    unsigned live = 0;           // bit 0: A's state is in use (in shared memory)
    {
        const Rows P0 = read(psi, z0 - 1), Q0 = read(psn, z0 - 1), R0 = read(Uf, z0 - 1);
        c0 = phase_of(P0, Q0, R0);
        b0 = beta3<T>(R0.lo, R0.C, R0.hi);
        V2 aS, a, aN, bS, b, bN, dS, dN;
        alphas(P0.lo, Q0.lo, R0.lo, aS, bS, dS);
        alphas(P0.C, Q0.C, R0.C, a, b, phn0);
        alphas(P0.hi, Q0.hi, R0.hi, aN, bN, dN);
        auto first = [&](Sums3<T>& X, V2 xS, V2 x, V2 xN) {
            uniform3<T>(X, T(0));
            if constexpr (ISO) (void)weights3<T>(X, xS, x, xN);
            else faces_only(X, xS, x, xN);
        };
        Sums3<T> sums;
        first(sums, aS, a, aN);
        put(&sums, 0, SUMS);
        aA0 = b;
        if (c0 == 0) {
            Div3<T> A;
            clear(A);
            first(A.s, bS, b, bN);
            put(&A, SUMS, ALL);
            live = 1;
        }
    }
    Rows Pn = read(psi, z0), Qn = read(psn, z0), Rn = read(Uf, z0);
    for (int z = z0 - 1; z < z1; ++z) {
        const Rows P1 = Pn, Q1 = Qn, R1 = Rn;
        Pn = read(psi, z + 2);
        Qn = read(psn, z + 2);
        Rn = read(Uf, z + 2);
        // an iteration in bulk is shorter than a trip to HBM: the own rows of two planes
        // on go to L2 (256^3: 384 -> 356 us a step; the psi pass gains nothing from it)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(plane(psi, z + 4) + at.o0));
        asm volatile("prefetch.global.L2 [%0];" ::"l"(plane(psn, z + 4) + at.o0));
        asm volatile("prefetch.global.L2 [%0];" ::"l"(plane(Uf, z + 4) + at.o0));
        const int c1 = phase_of(P1, Q1, R1);
        const Beta3<T> b1 = beta3<T>(R1.lo, R1.C, R1.hi);
        const V2 d = b1.C - b0.C;
        V2 inc = zero;  // cD sum D + cA sum A
        V2 phn1 = k_(T(c1)), aA1 = zero;
        const bool same = c0 != 0 && c1 == c0 && cm == c0;
        if (same && c0 > 0) {
            // solid below, at and above: no flux
            D.fz = D.pp = D.g = D.yz = zero;
        } else if (same) {
            if constexpr (ISO) {
                inc = k_(cD) * gather3<T>(D, const_weights3<T>(T(2)), b0, b1, d);
            } else {
                const V2 fx = c_(4.0) * b0.e, fz = c_(4.0) * d;
                inc = k_(cD) * ((fx - west3(fx)) + fma(c_(4.0), b0.n, c_(4.0) * b0.s) + (fz - D.fz));
                D.fz = fz;
            }
        }
        if (same) {
            fresh = false;
        } else {
            Sums3<T> sums;
            if (fresh) {
                get(&sums, 0, SUMS);
            } else {
                // planes z - 1 and z were of one phase
                const T a = c0 < 0 ? T(2) : T(0);
                uniform3<T>(sums, a);
                if constexpr (!ISO) sums.wz = k_(a);
                fresh = true;
            }
            V2 aS, a, aN, bS = zero, bN = zero;
            if (c1 != 0) {
                aS = a = aN = k_(T(1 - c1));
            } else {
                V2 dS, dN;
                alphas(P1.lo, Q1.lo, R1.lo, aS, bS, dS);
                alphas(P1.C, Q1.C, R1.C, a, aA1, phn1);
                alphas(P1.hi, Q1.hi, R1.hi, aN, bN, dN);
            }
            V2 sD;
            if constexpr (ISO) {
                const Weights3<T> w = weights3<T>(sums, aS, a, aN);
                sD = gather3<T>(D, w, b0, b1, d);
            } else {
                const V2 fx = sums.rx * b0.e, fz = (sums.wz + a) * d;
                sD = (fx - west3(fx)) + fma(sums.ryN, b0.n, sums.ryS * b0.s) + (fz - D.fz);
                faces_only(sums, aS, a, aN);
                D.fz = fz;
            }
            put(&sums, 0, SUMS);
            inc = k_(cD) * sD;
            if (c1 == 0 || live) {
                // the anti-trapping divergence: beta = psi
                Div3<T> A;
                if (live) get(&A, SUMS, ALL);
                else clear(A);
                const Rows P0 = read(psi, z);
                const Beta3<T> q0 = beta3<T>(P0.lo, P0.C, P0.hi), q1 = beta3<T>(P1.lo, P1.C, P1.hi);
                const V2 dq = q1.C - q0.C;
                V2 sA;
                if constexpr (ISO) {
                    const Weights3<T> w = weights3<T>(A.s, bS, aA1, bN);
                    sA = gather3<T>(A.c, w, q0, q1, dq);
                } else {
                    // each face flux over |grad psi| of the face (4 h times the gradient's components)
                    const Rows Pm = read(psi, z - 1);
                    const Beta3<T> qm = beta3<T>(Pm.lo, Pm.C, Pm.hi);
                    const V2 ez2 = c_(2.0) * (q1.C - qm.C);
                    const V2 w0 = west3(q0.e), w1 = west3(q1.e), ex0 = q0.e + w0, ey0 = q0.n - q0.s;
                    auto over = [&](V2 f, V2 gx, V2 gy, V2 gz) -> V2 {
                        const V2 r2 = fma(gx, gx, fma(gy, gy, gz * gz));
                        const V2 i = rcp2(each3(r2, [](T v) { return M<T>::sqrt_(v); }));
                        const V2 o = f * i;
                        const T low = T(16) * Guard<T>::v;
                        return mk(r2.x() < low ? T(0) : o.x(), r2.y() < low ? T(0) : o.y());
                    };
                    const V2 f4 = c_(4.0);
                    const V2 fx = over(A.s.rx * q0.e, f4 * q0.e, (q0.eN - q0.eS) + c_(2.0) * ey0, (q1.e - qm.e) + ez2);
                    const V2 fN = over(A.s.ryN * q0.n, ex0 + (q0.eN + west3(q0.eN)), f4 * q0.n, (q1.n - qm.n) + ez2);
                    const V2 fS = over(A.s.ryS * q0.s, ex0 + (q0.eS + west3(q0.eS)), f4 * q0.s, (q1.s - qm.s) + ez2);
                    const V2 fz = over((A.s.wz + aA1) * dq, ex0 + (q1.e + w1), ey0 + (q1.n - q1.s), f4 * dq);
                    sA = (fx - west3(fx)) + (fN + fS) + (fz - A.c.fz);
                    faces_only(A.s, bS, aA1, bN);
                    A.c.fz = fz;
                }
                inc = fma(k_(cA), sA, inc);
                // nothing of planes z and z + 1 is left in the state once both are of one phase
                live = c1 == 0 || c0 == 0 ? 1u : 0u;
                if (live) put(&A, SUMS, ALL);
            }
        }
        if (z >= z0) {
            const V2 den = fma(k_(-omk), phn0, k_(opk));
            at.template store<T>(U_o + (long long)PF_CHK(z, nz) * sxy, fma(inc + aA0, rcp2(den), b0.C));
        }
        b0 = b1;
        phn0 = phn1;
        aA0 = aA1;
        cm = c0;
        c0 = c1;
    }
}

// Rows of a block: two per warp.  Resident blocks asked for (FP32) of 30 x 6
// columns: four of three warps each at 168 registers (S-bar_{1,2,0}; 256^3: 382
// us a step; 405 with five at 128 registers, 474 and up with six, whose spills
// every plane pays; 4 polycrystals 218 against 264), five for S_{1,0,0} (157 x
// 121 x 189: 87 us against 93).
template <int S, int TY> struct Block3 {
    static constexpr int threads = 16 * TY, blocks = TY == 6 ? (S == S100 ? 5 : 4) : 2;
};
// shared memory of the U pass
template <typename T> constexpr size_t park_bytes(int threads) { return (sizeof(Sums3<T>) + sizeof(Div3<T>)) * threads; }

template <typename T, int S, int TY, bool ONE>
__global__ void __launch_bounds__(Block3<S, TY>::threads, sizeof(T) == 4 ? Block3<S, TY>::blocks : 1)
    k_psi3d(const WorkItem* __restrict__ work, int n_work, const InstRec* __restrict__ recs, int launch_parity, StepClock clk) {
    after_previous();
    for (int w = blockIdx.x; w < n_work; w += gridDim.x) {
        const WorkItem wi = work[w];
        const InstRec& rec = recs[wi.inst];
        if ((rec.nx & 1) == 0 && wi.x0 >= 2 && wi.x0 + 30 <= rec.nx)
            psi_sweep<T, S, ONE, true>(wi, rec, launch_parity, clk);
        else
            psi_sweep<T, S, ONE, false>(wi, rec, launch_parity, clk);
    }
}
template <typename T, int S, int TY>
__global__ void __launch_bounds__(Block3<S, TY>::threads, sizeof(T) == 4 ? Block3<S, TY>::blocks : 1)
    k_u3d(const WorkItem* __restrict__ work, int n_work, const InstRec* __restrict__ recs, int launch_parity) {
    extern __shared__ __align__(16) unsigned char smem3[];
    V<T>* park = reinterpret_cast<V<T>*>(smem3);
    after_previous();
    for (int w = blockIdx.x; w < n_work; w += gridDim.x) {
        const WorkItem wi = work[w];
        const InstRec& rec = recs[wi.inst];
        if ((rec.nx & 1) == 0 && wi.x0 >= 2 && wi.x0 + 30 <= rec.nx)
            u_sweep<T, S, true>(wi, rec, launch_parity, park);
        else
            u_sweep<T, S, false>(wi, rec, launch_parity, park);
    }
}

template <typename T, int S, int TY> bool launch_t(const Step3DArgs& a, cudaStream_t st) {
    constexpr int th = Block3<S, TY>::threads;
    if (a.grid_psi > 0) {
        const auto k = a.fr == 0 ? k_psi3d<T, S, TY, true> : k_psi3d<T, S, TY, false>;
        launch_next(k, a.grid_psi, th, 0, st, a.work, a.n_work, a.recs, a.launch_parity, a.clk);
    }
    if (a.grid_u > 0)
        launch_next(k_u3d<T, S, TY>, a.grid_u, th, park_bytes<T>(th), st, a.work, a.n_work, a.recs, a.launch_parity);
    return true;
}
template <typename T, int S, int TY> bool occ_t(int fr, int& psi, int& u) {
    constexpr int th = Block3<S, TY>::threads;
    const cudaError_t e =
        fr == 0 ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&psi, k_psi3d<T, S, TY, true>, th, 0)
                : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&psi, k_psi3d<T, S, TY, false>, th, 0);
    if (e != cudaSuccess ||
        cudaFuncSetAttribute(k_u3d<T, S, TY>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)park_bytes<T>(th)) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&u, k_u3d<T, S, TY>, th, park_bytes<T>(th)) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return psi > 0 && u > 0;
}

// Compiled tiles (block_x, block_y) = (30 + 4, TY + 4): (34, 10), and (34, 18) but for S-bar_{1,2,0} in FP64.
template <typename T, int SCH> constexpr bool WIDE = sizeof(T) == 4 || SCH == S100;
template <typename T, int S> bool launch_s(const Step3DArgs& a, int bx, int by, cudaStream_t st) {
    if constexpr (WIDE<T, S>)
        if (bx == 34 && by == 18) return launch_t<T, S, 14>(a, st);
    if (bx == 34 && by == 10) return launch_t<T, S, 6>(a, st);
    return false;
}
template <typename T, int S> bool occ_s(int bx, int by, int fr, int& psi, int& u) {
    if constexpr (WIDE<T, S>)
        if (bx == 34 && by == 18) return occ_t<T, S, 14>(fr, psi, u);
    if (bx == 34 && by == 10) return occ_t<T, S, 6>(fr, psi, u);
    return false;
}

}  // namespace

PF_BOUNDS_READER(bounds_step3d)

bool launch_step3d(int prec, int scheme, int bx, int by, cudaStream_t st, const Step3DArgs& a) {
    if (prec == 0) {
        if (scheme == S100) return launch_s<float, S100>(a, bx, by, st);
        if (scheme == SBAR120) return launch_s<float, SBAR120>(a, bx, by, st);
    } else {
        if (scheme == S100) return launch_s<double, S100>(a, bx, by, st);
        if (scheme == SBAR120) return launch_s<double, SBAR120>(a, bx, by, st);
    }
    return false;
}

bool occupancy_step3d(int prec, int scheme, int bx, int by, int fr, int& psi, int& u) {
    psi = u = 0;
    if (prec == 0) {
        if (scheme == S100) return occ_s<float, S100>(bx, by, fr, psi, u);
        if (scheme == SBAR120) return occ_s<float, SBAR120>(bx, by, fr, psi, u);
    } else {
        if (scheme == S100) return occ_s<double, S100>(bx, by, fr, psi, u);
        if (scheme == SBAR120) return occ_s<double, SBAR120>(bx, by, fr, psi, u);
    }
    return false;
}

}  // namespace pf
