// observe.cu -- FP64 reductions (solute integral of Eq. Supersaturation,
// solid fraction, non-finite scan, tip tracking of Sec. 3.3.2 / 6.2.2) and
// the seed initialisation, for sm_103a.
//
// Reductions are deterministic: a fixed grid of OBS_BLOCKS blocks walks the
// cells grid-stride, each block reduces in a fixed tree order, and one block
// combines the partials in index order.  The tip candidate is chosen by the
// total order (larger projection, then smaller cell index), so it does not
// depend on the reduction order.  Candidate positions and projections are
// formed with explicitly rounded FP64 operations (no contraction) so that the
// choice is reproducible on any FP64 implementation of the same formula.
#include <cfloat>
#include <math_constants.h>

#include "pf_internal.cuh"

namespace pf {
namespace {

__device__ __forceinline__ bool better(double s1, long long i1, double s2, long long i2) {
    // is (s1, i1) preferred over (s2, i2)?
    if (i2 < 0) return i1 >= 0;
    if (i1 < 0) return false;
    if (s1 > s2) return true;
    if (s1 < s2) return false;
    return i1 < i2;
}

__device__ __forceinline__ void combine(ObsPartial& a, const ObsPartial& b) {
    a.solute += b.solute;
    a.solid += b.solid;
    a.nonfinite += b.nonfinite;
    if (better(b.score, b.tip_index, a.score, a.tip_index)) {
        a.score = b.score;
        a.tip_index = b.tip_index;
        a.tip[0] = b.tip[0];
        a.tip[1] = b.tip[1];
        a.tip[2] = b.tip[2];
    }
}

// 2^y for -1000 < y <= 0: y = n + f with |f| <= 1/2, the Taylor series of e^{f ln 2}
// to the 12th power (remainder below 2e-16), scaled through the exponent bits.
__device__ __forceinline__ double exp2_neg(double y) {
    const double shift = 6755399441055744.0;  // 1.5 x 2^52: the sum's low bits are rint(y)
    const double t = __dadd_rn(y, shift);
    const double f = __dadd_rn(y, -__dadd_rn(t, -shift));
    double e = 2.5678435993488206e-11;  // ln2^12 / 12!
    e = fma(e, f, 4.4455382718708116e-10);
    e = fma(e, f, 7.0549116208011233e-09);
    e = fma(e, f, 1.0178086009239699e-07);
    e = fma(e, f, 1.3215486790144309e-06);
    e = fma(e, f, 1.5252733804059841e-05);
    e = fma(e, f, 1.5403530393381608e-04);
    e = fma(e, f, 1.3333558146428443e-03);
    e = fma(e, f, 9.6181291076284772e-03);
    e = fma(e, f, 5.5504108664821580e-02);
    e = fma(e, f, 2.4022650695910072e-01);
    e = fma(e, f, 6.9314718055994531e-01);
    e = fma(e, f, 1.0);
    return __hiloint2double(__double2hiint(e) + (__double2loint(t) << 20), __double2loint(e));
}
// phi = tanh(psi / sqrt2) = sign (2 / (1 + e) - 1), e = exp(-sqrt2 |psi|), of two
// values with one division; absolute error below 4e-16, which is what the sums
// over phi need.
__device__ __forceinline__ void phi_two(double a, double b, double& fa, double& fb) {
    const double c = -2.0402788931935790;  // -sqrt2 log2(e)
    const double da = 1.0 + exp2_neg(c * fabs(a)), db = 1.0 + exp2_neg(c * fabs(b));
    const double r = 2.0 / (da * db);
    fa = copysign(fma(r, db, -1.0), a);
    fb = copysign(fma(r, da, -1.0), b);
}

__device__ __forceinline__ void clear(ObsPartial& a) {
    a.solute = 0.0;
    a.solid = 0.0;
    a.nonfinite = 0;
    a.score = -DBL_MAX;
    a.tip_index = -1;
    a.tip[0] = a.tip[1] = a.tip[2] = 0.0;
    a.pad = 0.0;
}
// a's lane takes the record of the lane `off` above
__device__ __forceinline__ ObsPartial from_above(const ObsPartial& a, int off) {
    const unsigned all = 0xffffffffu;
    ObsPartial b;
    b.solute = __shfl_down_sync(all, a.solute, off);
    b.solid = __shfl_down_sync(all, a.solid, off);
    b.score = __shfl_down_sync(all, a.score, off);
    b.tip_index = __shfl_down_sync(all, a.tip_index, off);
    b.nonfinite = __shfl_down_sync(all, a.nonfinite, off);
    for (int q = 0; q < 3; ++q) b.tip[q] = __shfl_down_sync(all, a.tip[q], off);
    b.pad = 0.0;
    return b;
}
// The warp's tip in lane 0 (the order of the choice is total, so any tree order gives it).
__device__ __forceinline__ void reduce_tip(ObsPartial& acc) {
    const unsigned all = 0xffffffffu;
    if (!__any_sync(all, acc.tip_index >= 0)) return;
    for (int off = 16; off > 0; off >>= 1) {
        const ObsPartial b = from_above(acc, off);
        if (better(b.score, b.tip_index, acc.score, acc.tip_index)) {
            acc.score = b.score;
            acc.tip_index = b.tip_index;
            for (int q = 0; q < 3; ++q) acc.tip[q] = b.tip[q];
        }
    }
}
// The block's record in thread 0 from one record per warp, in a fixed tree order.
__device__ __forceinline__ void reduce_warps(ObsPartial& acc, ObsPartial* sh) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int W = OBS_THREADS / 32;
    if (lane == 0) sh[warp] = acc;
    __syncthreads();
    if (warp == 0) {
        if (lane < W) acc = sh[lane];
        else clear(acc);
        for (int off = W / 2; off > 0; off >>= 1) {
            const ObsPartial b = from_above(acc, off);
            combine(acc, b);
        }
    }
}

// Cells near the interface that a warp has met and not yet evaluated.
constexpr int OBS_QUEUE = 64 + 4 * 32;
// what a thread, a warp and a block sum before the terms are formed
template <typename T> struct ObsSums {
    long long liq, sol, near, bad;          // cells
    T l_hi, l_lo, s_hi, s_lo;               // U over the liquid, the solid
    double u, phi, phiu;                    // U, phi and phi U near the interface
    float c, cu;                            // sign - phi and (sign - phi) U in the bulk
};
template <typename T> struct ObsShared {
    ObsPartial part[OBS_THREADS / 32];
    ObsSums<T> sums[OBS_THREADS / 32];
    T psi[OBS_THREADS / 32][OBS_QUEUE], U[OBS_THREADS / 32][OBS_QUEUE];
};

// The partial of block `blk` of `nblk` walking the cells of one field pair.
//
// What bounds the observe is FP64 arithmetic (two FP64 lanes per SM and clock),
// so it is kept to the cells that need it.  From |psi| = 18 on, phi = sign (1 - c)
// with c = 2 e^{-sqrt2 |psi|} < 2e-11 (the next term is c^2 / 2): with phi = +-1 those
// cells contribute 1 + (1-k) U (liquid) or k (1 + (1-k) U) (solid) to the solute
// sum and 0 or 1 to the solid sum; they are counted and their U summed, exactly in
// FP32 pairs (Knuth's two-sum: hi + lo carries ~48 bits), and the sums of c and c U, in
// FP32, are 1e-16 of a term per cell accurate (c is below FP64 precision from |psi| =
// 32 on); FP64 fields take plain FP64 sums.  The other cells, and those with |U| >
// 1e18, whose sums could leave the FP32 range, go to a queue of the warp and are evaluated 64 at a
// time, two to a lane, so that no lane idles where the interface crosses a row;
// each adds U, phi and phi U to three FP64 sums.  (Five 1024^2 members with
// mature dendrites: 150 us with the library tanh and both FP64 terms in place, 96
// with the queue and phi_two, 83 with the bulk from 18 instead of 32, 72 with the
// terms formed once a block instead of once a thread, 74 with U near the interface in
// FP64 and the test for large U.  Against 128-bit sums of 60 fields of each precision the
// solute is 1.3e-16 off and the solid fraction 0.8e-16 (rms), as with every term in
// FP64: the last rounding.)  Rows are walked whole (one block per row, threads
// along x), so no cell index is divided.
template <typename T>
__device__ void observe_block(const ObsArgs& a, ObsPartial* __restrict__ partials, long long blk, long long nblk,
                              ObsShared<T>& sh) {
    const T* __restrict__ psi = static_cast<const T*>(a.psi);
    const T* __restrict__ U = static_cast<const T*>(a.U);
    const long long nx = a.nx, ny = a.ny, nz = a.dim == 3 ? a.nz : 1;
    [[maybe_unused]] const long long N = nx * ny * nz;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned all = 0xffffffffu;
    ObsPartial acc;
    clear(acc);
    const double k = a.k, omk = 1.0 - a.k;
    ObsSums<T> z{};
    auto acc2 = [](T& hi, T& lo, T v) {
        if constexpr (sizeof(T) == 4) {
            const T sm = hi + v, bb = sm - hi;
            lo += (hi - (sm - bb)) + (v - bb);
            hi = sm;
        } else {
            hi += v;  // FP64 fields: the plain FP64 sum
        }
    };
    int queued = 0;  // the same in every lane
    // evaluates the first `n` <= 64 queued cells (two to a lane)
    auto evaluate = [&](int n) {
        __syncwarp();
        const bool v0 = lane < n, v1 = lane + 32 < n;
        // (phi = +-1 to FP64 precision well below |psi| = 40)
        auto clamp = [](T x) -> T { return fabs(x) > T(40) ? copysign(T(40), x) : x; };
        const T p0 = v0 ? clamp(sh.psi[warp][lane]) : T(0), p1 = v1 ? clamp(sh.psi[warp][lane + 32]) : T(0);
        const T u0 = v0 ? sh.U[warp][lane] : T(0), u1 = v1 ? sh.U[warp][lane + 32] : T(0);
        double f0, f1;
        phi_two((double)p0, (double)p1, f0, f1);
        if (v0) {
            z.u += (double)u0;
            z.phi += f0;
            z.phiu = fma(f0, (double)u0, z.phiu);
        }
        if (v1) {
            z.u += (double)u1;
            z.phi += f1;
            z.phiu = fma(f1, (double)u1, z.phiu);
        }
        __syncwarp();
    };
    const long long rows = ny * nz;
    // the sums of one cell; true if it is near the interface
    auto sums = [&](T pst, T ut) -> bool {
        if (!isfinite(pst) || !isfinite(ut)) {
            z.bad += 1;
            return false;
        }
        if (fabs(pst) >= T(18) && fabs(ut) <= T(1e18)) {
            float c = 0.0f;
            if (fabs(pst) < T(32)) c = copysignf(2.0f * exp2f(-2.0402788931935790f * fabsf((float)pst)), (float)pst);
            z.c += c;
            z.cu += c * (float)ut;
            if (pst > T(0)) {
                z.sol += 1;
                acc2(z.s_hi, z.s_lo, ut);
            } else {
                z.liq += 1;
                acc2(z.l_hi, z.l_lo, ut);
            }
            return false;
        }
        z.near += 1;
        return true;
    };
    // the tip candidate of one cell
    auto tip = [&](long long i, long long j, long long kk, long long c, T pst, T ut) {
        if (!(pst >= T(0)) || !isfinite(pst) || !isfinite(ut)) return;
        long long ii = i, jj = j, kq = kk;
        if (a.ea == 0) ii += a.es;
        else if (a.ea == 1) jj += a.es;
        else kq += a.es;
        if (ii < 0 || jj < 0 || kq < 0 || ii >= nx || jj >= ny || kq >= nz) return;
        const T pnt = psi[PF_CHK((kq * ny + jj) * nx + ii, N)];
        if (!(pnt < T(0))) return;
        if (a.grain_filter >= 0 && a.grain[c] != a.grain_filter) return;
        const double ps = (double)pst, pn = (double)pnt;
        const double frac = __ddiv_rn(ps, __dsub_rn(ps, pn));
        double p[3] = {__dmul_rn((double)i, a.h), __dmul_rn((double)j, a.h),
                       a.dim == 3 ? __dmul_rn((double)kk, a.h) : 0.0};
        p[a.ea] = __dadd_rn(p[a.ea], __dmul_rn((double)a.es * frac, a.h));
        double sc = 0.0;
        for (int q = 0; q < a.dim; ++q) sc = __dadd_rn(sc, __dmul_rn(__dsub_rn(p[q], a.cg[q]), a.d[q]));
        if (better(sc, c, acc.score, acc.tip_index)) {
            acc.score = sc;
            acc.tip_index = c;
            acc.tip[0] = p[0];
            acc.tip[1] = p[1];
            acc.tip[2] = p[2];
        }
    };
    // whole warps: queues the lanes' near cells, evaluates when 64 are there
    auto push = [&](bool near, T pst, T ut) {
        const unsigned m = __ballot_sync(all, near);
        if (m == 0) return;
        if (near) {
            const int at = queued + __popc(m & ((1u << lane) - 1u));
            sh.psi[warp][at] = pst;
            sh.U[warp][at] = ut;
        }
        queued += __popc(m);
    };
    auto drain = [&]() {
        while (queued >= 64) {
            evaluate(64);
            // the rest moves down (at most 128 cells: the queue holds 64 + 4 x 32)
            queued -= 64;
            T mp[4], mu[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const bool in = lane + 32 * q < queued;
                mp[q] = in ? sh.psi[warp][64 + lane + 32 * q] : T(0);
                mu[q] = in ? sh.U[warp][64 + lane + 32 * q] : T(0);
            }
            __syncwarp();
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (lane + 32 * q < queued) {
                    sh.psi[warp][lane + 32 * q] = mp[q];
                    sh.U[warp][lane + 32 * q] = mu[q];
                }
            __syncwarp();
        }
    };
    // FP32 rows whose length is a multiple of 4 are read four cells at a time
    // (16-byte vector loads: more bytes in flight per thread); other rows cell
    // by cell.  The order of the per-thread sums differs between the two, not
    // the cells each block covers.
    const bool vec4 = sizeof(T) == 4 && (nx & 3) == 0 && ((uintptr_t)psi & 15) == 0 && ((uintptr_t)U & 15) == 0;
    const int per = vec4 ? 4 : 1;
    for (long long row = blk; row < rows; row += nblk) {
        const long long j = row % ny, kk = row / ny;
        const long long base = row * nx;
        // whole warps stay in the loop: lanes beyond the row hold nothing
        for (long long i0 = (long long)per * 32 * warp; i0 < nx; i0 += (long long)per * blockDim.x) {
            const long long i = i0 + per * lane;
            const bool in = i < nx;
            if (vec4) {
                float4 p4 = make_float4(0.f, 0.f, 0.f, 0.f), u4 = p4;
                if (in) {
                    p4 = __ldg(reinterpret_cast<const float4*>(psi + PF_CHK(base + i, N)));
                    u4 = __ldg(reinterpret_cast<const float4*>(U + PF_CHK(base + i, N)));
                }
                const float pv[4] = {p4.x, p4.y, p4.z, p4.w}, uv[4] = {u4.x, u4.y, u4.z, u4.w};
#pragma unroll
                for (int q = 0; q < 4; ++q) push(in && sums((T)pv[q], (T)uv[q]), (T)pv[q], (T)uv[q]);
                // no tip candidate without a cell with psi >= 0
                if (in && fmaxf(fmaxf(p4.x, p4.y), fmaxf(p4.z, p4.w)) >= 0.0f)
                    for (int q = 0; q < 4; ++q) tip(i + q, j, kk, base + i + q, (T)pv[q], (T)uv[q]);
            } else {
                const T pst = in ? psi[PF_CHK(base + i, N)] : T(0), ut = in ? U[PF_CHK(base + i, N)] : T(0);
                push(in && sums(pst, ut), pst, ut);
                if (in) tip(i, j, kk, base + i, pst, ut);
            }
            drain();
        }
    }
    if (queued > 0) evaluate(queued);
    // Sums over the warp, then over the warps, in a fixed tree order: the counts as
    // integers, the FP32 pairs as pairs, the FP64 sums where there are any; thread 0
    // then forms the terms (once a block: FP64 operations and conversions of every
    // thread would cost as much as the interface).
    auto tree = [&](int from) {
        auto pair = [&](T& hi, T& lo) {
            for (int off = from; off > 0; off >>= 1) {
                const T h = __shfl_down_sync(all, hi, off), l = __shfl_down_sync(all, lo, off);
                acc2(hi, lo, h);
                lo += l;
            }
        };
        const bool liq = __any_sync(all, z.liq != 0), sol = __any_sync(all, z.sol != 0), near = __any_sync(all, z.near != 0);
        for (int off = from; off > 0; off >>= 1) {
            z.liq += __shfl_down_sync(all, z.liq, off);
            z.sol += __shfl_down_sync(all, z.sol, off);
            z.near += __shfl_down_sync(all, z.near, off);
            z.bad += __shfl_down_sync(all, z.bad, off);
            z.c += __shfl_down_sync(all, z.c, off);
            z.cu += __shfl_down_sync(all, z.cu, off);
        }
        if (liq) pair(z.l_hi, z.l_lo);
        if (sol) pair(z.s_hi, z.s_lo);
        if (near) {
            for (int off = from; off > 0; off >>= 1) {
                z.u += __shfl_down_sync(all, z.u, off);
                z.phi += __shfl_down_sync(all, z.phi, off);
                z.phiu += __shfl_down_sync(all, z.phiu, off);
            }
        }
    };
    tree(16);
    reduce_tip(acc);
    if (lane == 0) {
        sh.part[warp] = acc;
        sh.sums[warp] = z;
    }
    __syncthreads();
    if (warp != 0) return;
    constexpr int W = OBS_THREADS / 32;
    if (lane < W) {
        acc = sh.part[lane];
        z = sh.sums[lane];
    } else {
        clear(acc);
        z = ObsSums<T>{};
    }
    tree(W / 2);
    reduce_tip(acc);
    if (lane == 0) {
        const double u_liq = (double)z.l_hi + (double)z.l_lo, u_sol = (double)z.s_hi + (double)z.s_lo;
        // near the interface: sum (1 + k - (1-k) phi) (1 + (1-k) U) / 2 and sum (1 + phi) / 2
        acc.nonfinite = z.bad;
        acc.solute = ((double)z.liq + omk * u_liq) + k * ((double)z.sol + omk * u_sol) +
                     0.5 * ((1.0 + k) * ((double)z.near + omk * z.u) - omk * (z.phi + omk * z.phiu)) +
                     0.5 * omk * ((double)z.c + omk * (double)z.cu);
        acc.solid = (double)z.sol + 0.5 * ((double)z.near + z.phi) - 0.5 * (double)z.c;
        partials[blk] = acc;
    }
}

template <typename T>
__global__ void __launch_bounds__(OBS_THREADS, 3) k_observe(ObsArgs a, ObsPartial* __restrict__ partials) {
    __shared__ ObsShared<T> sh;
    observe_block<T>(a, partials, blockIdx.x, gridDim.x, sh);
}

// All members of a group (of one field precision, or not) in one launch: blocks
// (x, m) walk member m's cells exactly as blocks x of k_observe would (same
// partials, same order).
__global__ void __launch_bounds__(OBS_THREADS, 3) k_observe_multi(const ObsJob* __restrict__ jobs) {
    __shared__ union {
        ObsShared<float> f;
        ObsShared<double> d;
    } sh;
    const ObsJob& j = jobs[blockIdx.y];
    if (j.a.prec == 0)
        observe_block<float>(j.a, j.partials, blockIdx.x, gridDim.x, sh.f);
    else
        observe_block<double>(j.a, j.partials, blockIdx.x, gridDim.x, sh.d);
}

// Combine the block partials: thread t folds partials t, t + 256, ... in
// index order, then a fixed tree; deterministic for a fixed partial count.
__device__ void finish_block(const ObsPartial* __restrict__ partials, int n, ObsPartial* __restrict__ out,
                             ObsPartial* sh) {
    ObsPartial acc;
    clear(acc);
    for (int b = threadIdx.x; b < n; b += OBS_THREADS) combine(acc, partials[b]);
    for (int off = 16; off > 0; off >>= 1) {
        const ObsPartial b = from_above(acc, off);
        combine(acc, b);
    }
    reduce_warps(acc, sh);
    if (threadIdx.x == 0) *out = acc;
}

__global__ void __launch_bounds__(OBS_THREADS) k_observe_finish(const ObsPartial* __restrict__ partials, int n,
                                                                ObsPartial* __restrict__ out) {
    __shared__ ObsPartial sh[OBS_THREADS / 32];
    finish_block(partials, n, out, sh);
}

// Block m combines member m's partials into out[m].
__global__ void __launch_bounds__(OBS_THREADS) k_observe_finish_multi(const ObsJob* __restrict__ jobs,
                                                                      ObsPartial* __restrict__ out) {
    __shared__ ObsPartial sh[OBS_THREADS / 32];
    finish_block(jobs[blockIdx.x].partials, OBS_BLOCKS, out + blockIdx.x, sh);
}

// ---------------------------------------------------------------------------
// Tip radius (Sec. 3.3.2, Sec. 6.2.2): the paper fits the parabola
// y = y_tip - (x - x_tip)^2 / (2 rho) to the psi = 0 contour rotated so that
// the measured growth direction is vertical, up to one radius behind the tip
// (3D: rho_x in the plane of the growth axis and its in-plane normal, rho_z in
// the plane of the growth axis and z, 1/rho = (1/rho_x + 1/rho_z) / 2).
// Contour: 64 lines per transverse axis e, r(t) = (tip + s e) - t e_par with
// s = j h (j = -32..-1, 1..32) and t = m h / 4 (m <= 160); psi is interpolated
// multilinearly between cell centres and the first sample with psi >= 0 gives
// the crossing by linear interpolation.  Fit: c = sum t s^2 / sum s^4 over the
// crossings with t <= w, rho = 1 / (2c); w = 40 h, then the previous rho; four
// rounds.  One warp per line (its lanes take 32 samples at a time), then one
// thread per transverse axis fits in line order.  All FP64 operations are
// explicitly rounded (no contraction), so the crossings are reproducible.
constexpr int TIP_J = 32, TIP_M = 160, TIP_ROUNDS = 4;

template <typename T>
__device__ double tip_interp(const TipArgs& a, const T* __restrict__ psi, const double r[3], bool& inside) {
    const int n[3] = {a.nx, a.ny, a.dim == 3 ? a.nz : 1};
    int i0[3] = {0, 0, 0};
    double f[3] = {0.0, 0.0, 0.0};
    inside = true;
    for (int q = 0; q < a.dim; ++q) {
        const double u = __ddiv_rn(r[q], a.h);
        if (!(u >= 0.0) || u > (double)(n[q] - 1)) {
            inside = false;
            return 0.0;
        }
        int i = (int)floor(u);
        if (i > n[q] - 2) i = n[q] - 2;
        i0[q] = i;
        f[q] = __dsub_rn(u, (double)i);
    }
    auto P = [&](int di, int dj, int dk) -> double {
        return (double)psi[PF_CHK(((long long)(i0[2] + dk) * a.ny + (i0[1] + dj)) * a.nx + (i0[0] + di),
                                  (long long)a.nx * a.ny * (a.dim == 3 ? a.nz : 1))];
    };
    auto plane = [&](int dk) -> double {
        const double g0 = __dsub_rn(1.0, f[0]);
        const double lo = __dadd_rn(__dmul_rn(g0, P(0, 0, dk)), __dmul_rn(f[0], P(1, 0, dk)));
        const double hi = __dadd_rn(__dmul_rn(g0, P(0, 1, dk)), __dmul_rn(f[0], P(1, 1, dk)));
        return __dadd_rn(__dmul_rn(__dsub_rn(1.0, f[1]), lo), __dmul_rn(f[1], hi));
    };
    const double v0 = plane(0);
    if (a.dim == 2) return v0;
    return __dadd_rn(__dmul_rn(__dsub_rn(1.0, f[2]), v0), __dmul_rn(f[2], plane(1)));
}

// growth axis e_par and transverse axes e_x, e_z of the fit (explicitly rounded)
__device__ void tip_frame(const TipArgs& a, double frame[3][3]) {
    double ep[3] = {a.axis[0], a.axis[1], a.dim == 3 ? a.axis[2] : 0.0};
    const double na =
        __dsqrt_rn(__dadd_rn(__dadd_rn(__dmul_rn(ep[0], ep[0]), __dmul_rn(ep[1], ep[1])), __dmul_rn(ep[2], ep[2])));
    for (int q = 0; q < 3; ++q) ep[q] = __ddiv_rn(ep[q], na);
    double ex[3], ez[3] = {0.0, 0.0, 0.0};
    if (a.dim == 2) {
        ex[0] = ep[1];
        ex[1] = -ep[0];
        ex[2] = 0.0;
    } else {
        double ref[3] = {0.0, 0.0, 1.0};
        if (fabs(ep[2]) > 1.0 - 1e-6) {
            ref[0] = 1.0;
            ref[2] = 0.0;
        }
        const double pr =
            __dadd_rn(__dadd_rn(__dmul_rn(ref[0], ep[0]), __dmul_rn(ref[1], ep[1])), __dmul_rn(ref[2], ep[2]));
        for (int q = 0; q < 3; ++q) ez[q] = __dsub_rn(ref[q], __dmul_rn(pr, ep[q]));
        const double nz =
            __dsqrt_rn(__dadd_rn(__dadd_rn(__dmul_rn(ez[0], ez[0]), __dmul_rn(ez[1], ez[1])), __dmul_rn(ez[2], ez[2])));
        for (int q = 0; q < 3; ++q) ez[q] = __ddiv_rn(ez[q], nz);
        ex[0] = __dsub_rn(__dmul_rn(ez[1], ep[2]), __dmul_rn(ez[2], ep[1]));
        ex[1] = __dsub_rn(__dmul_rn(ez[2], ep[0]), __dmul_rn(ez[0], ep[2]));
        ex[2] = __dsub_rn(__dmul_rn(ez[0], ep[1]), __dmul_rn(ez[1], ep[0]));
    }
    for (int q = 0; q < 3; ++q) {
        frame[0][q] = ep[q];
        frame[1][q] = ex[q];
        frame[2][q] = ez[q];
    }
}

// One warp per contour line (64 per transverse axis); the lanes evaluate 32
// consecutive samples at once and the first sample that is outside the grid
// or has psi >= 0 ends the line, as in a sequential march.  t[line] = the
// crossing or NaN.
template <typename T> __global__ void __launch_bounds__(TIP_THREADS) k_tip_lines(TipArgs a, double* __restrict__ t) {
    __shared__ double frame[3][3];
    if (threadIdx.x == 0) tip_frame(a, frame);
    __syncthreads();
    const T* __restrict__ psi = static_cast<const T*>(a.psi);
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int gw = blockIdx.x * (TIP_THREADS / 32) + (threadIdx.x >> 5);
    const int half = gw / (2 * TIP_J), l = gw % (2 * TIP_J);  // half 0: e_x lines, 1: e_z lines
    if (half >= (a.dim == 3 ? 2 : 1)) return;                 // whole warps only
    const double* e = frame[1 + half];
    const int j = l < TIP_J ? l - TIP_J : l - TIP_J + 1;
    const double s = __dmul_rn((double)j, a.h);
    const double dt = __dmul_rn(a.h, 0.25);
    double base[3];
    for (int q = 0; q < 3; ++q) base[q] = __dadd_rn(a.tip[q], __dmul_rn(s, e[q]));
    double tc = CUDART_NAN, carry = 0.0;
    for (int m0 = 0; m0 <= TIP_M; m0 += 32) {
        const int m = m0 + lane;
        double v = 0.0;
        bool inside = false;
        if (m <= TIP_M) {
            const double tm = __dmul_rn((double)m, dt);
            double r[3];
            for (int q = 0; q < 3; ++q) r[q] = __dsub_rn(base[q], __dmul_rn(tm, frame[0][q]));
            v = tip_interp<T>(a, psi, r, inside);
        }
        const bool ev = m <= TIP_M && (!inside || v >= 0.0);
        const unsigned b = __ballot_sync(FULL, ev);
        const double vup = __shfl_up_sync(FULL, v, 1);
        const double prev = lane == 0 ? carry : vup;  // psi at sample m - 1
        if (b) {
            const int f = __ffs(b) - 1;
            double tl = CUDART_NAN;
            if (lane == f && inside && v >= 0.0 && m >= 1)
                tl = __dadd_rn(__dmul_rn((double)(m - 1), dt), __dmul_rn(dt, __ddiv_rn(prev, __dsub_rn(prev, v))));
            tc = __shfl_sync(FULL, tl, f);
            break;
        }
        carry = __shfl_sync(FULL, v, 31);
    }
    if (lane == 0) t[half * 2 * TIP_J + l] = tc;
}

// Parabola fits of the crossings in line order (one thread per transverse
// axis), then rho (3D: 2 / (1/rho_x + 1/rho_z)).
__global__ void k_tip_fit(TipArgs a, const double* __restrict__ t, double* __restrict__ out) {
    const int half = threadIdx.x;
    const double dt = __dmul_rn(a.h, 0.25);
    if (half < (a.dim == 3 ? 2 : 1)) {
        double w = __dmul_rn((double)TIP_M, dt), rho = CUDART_NAN;
        int used = 0;
        for (int round = 0; round < TIP_ROUNDS; ++round) {
            double st = 0.0, s4 = 0.0;
            int n = 0;
            for (int k = 0; k < 2 * TIP_J; ++k) {
                const int j = k < TIP_J ? k - TIP_J : k - TIP_J + 1;
                const double s = __dmul_rn((double)j, a.h);
                const double tk = t[half * 2 * TIP_J + k];
                if (!(tk <= w)) continue;
                const double s2 = __dmul_rn(s, s);
                st = __dadd_rn(st, __dmul_rn(tk, s2));
                s4 = __dadd_rn(s4, __dmul_rn(s2, s2));
                ++n;
            }
            used = n;
            if (n == 0 || !(st > 0.0)) {
                rho = CUDART_NAN;
                break;
            }
            rho = __dmul_rn(0.5, __ddiv_rn(s4, st));
            w = rho;
        }
        out[1 + half] = rho;
        out[3 + half] = (double)used;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        if (a.dim == 2) {
            out[2] = CUDART_NAN;
            out[4] = 0.0;
            out[0] = out[1];
        } else {
            out[0] = __ddiv_rn(2.0, __dadd_rn(__ddiv_rn(1.0, out[1]), __ddiv_rn(1.0, out[2])));
        }
    }
}

template <typename T>
__global__ void k_init_seeds(int dim, int nx, int ny, int nz, double h, double U0, const SeedDev* __restrict__ seeds,
                             int n_seeds, T* __restrict__ psi, T* __restrict__ U, int16_t* __restrict__ grain) {
    const long long N = (long long)nx * ny * (dim == 3 ? nz : 1);
    for (long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x; c < N; c += (long long)gridDim.x * blockDim.x) {
        const long long i = c % nx, j = (c / nx) % ny, k = c / ((long long)nx * ny);
        const double x = __dmul_rn((double)i, h), y = __dmul_rn((double)j, h);
        const double z = dim == 3 ? __dmul_rn((double)k, h) : 0.0;
        double best = -DBL_MAX;
        int bs = 0;
        bool any = false;
        for (int s = 0; s < n_seeds; ++s) {
            const double dx = __dsub_rn(x, seeds[s].x), dy = __dsub_rn(y, seeds[s].y);
            const double dz = dim == 3 ? __dsub_rn(z, seeds[s].z) : 0.0;
            const double d2 = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
            const double v = __dsub_rn(seeds[s].r, __dsqrt_rn(d2));
            if (!any || v > best) {
                best = v;
                bs = s;
                any = true;
            }
        }
        psi[c] = (T)best;
        U[c] = (T)U0;
        grain[c] = (int16_t)seeds[bs].grain;
    }
}

// advances the step clock of a group (one thread, after every step launch)
__global__ void k_tick(long long* clock) { *clock += 1; }

template <typename T> __global__ void k_fill(T* __restrict__ p, T v, long long n) {
    for (long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x; c < n; c += (long long)gridDim.x * blockDim.x)
        p[c] = v;
}

// Compensated FP32 state (precision PF_F32C): split an FP64 field into hi =
// fl32(x) and lo = fl32(x - hi) (x - hi is exact in FP64), or join hi + lo
// back into FP64 (exact).
__global__ void k_split(const double* __restrict__ x, float* __restrict__ hi, float* __restrict__ lo, long long n) {
    for (long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x; c < n; c += (long long)gridDim.x * blockDim.x) {
        const double v = x[c];
        const float h = __double2float_rn(v);
        hi[c] = h;
        lo[c] = __double2float_rn(v - (double)h);
    }
}
__global__ void k_join(const float* __restrict__ hi, const float* __restrict__ lo, double* __restrict__ x, long long n) {
    for (long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x; c < n; c += (long long)gridDim.x * blockDim.x)
        x[c] = (double)hi[c] + (double)lo[c];
}

// Frame shift by `rows` cells toward -y: dst(x, y, z) = src(x, y + rows, z)
// for y + rows < ny.  The vacated top rows, k rows beyond the last one, take
// (mode 0) the last row's value, (mode 1) the last row's value plus a k (psi:
// a = -h, a signed distance continued into the melt) or (mode 3) the value
// a + (last - a) exp(-b k) (U: the steady far field a + C exp(-Vp y / D) ahead
// of a front pulled at Vp, b = Vp h / D).  src and dst do not overlap.
template <typename T>
__global__ void k_shift_rows(const T* __restrict__ src, T* __restrict__ dst, int nx, int ny, int nz, int rows, int mode,
                             double a, double b) {
    const long long n = (long long)nx * ny * nz;
    for (long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x; c < n; c += (long long)gridDim.x * blockDim.x) {
        const int x = (int)(c % nx);
        const long long yz = c / nx;
        const int y = (int)(yz % ny), z = (int)(yz / ny);
        const int ys = y + rows;
        const long long plane = (long long)z * ny;
        if (ys < ny) {
            dst[c] = src[(plane + ys) * nx + x];
        } else {
            const T top = src[(plane + ny - 1) * nx + x];
            // product and sum rounded separately (no contraction): top - k h exactly as written
            const double kk = (double)(ys - (ny - 1));
            dst[c] = mode == 0   ? top
                     : mode == 1 ? (T)__dadd_rn((double)top, __dmul_rn(a, kk))
                                 : (T)(a + ((double)top - a) * exp(-b * kk));
        }
    }
}

}  // namespace

// Fixed scratch for pf_observe_fields_noalloc: OBS_BLOCKS block partials and
// one result record (22 KB).  It lives in the module's global memory on every
// device that loads the library, for the life of the process.  Every call of
// that entry point overwrites all of it, so nothing needs clearing; calls whose
// kernels overlap on a device race on it.
static __device__ __align__(256) ObsPartial g_noalloc_scratch[OBS_BLOCKS + 1];

// Device address of the scratch on the current device, looked up on every
// call with cudaGetSymbolAddress (a host-side name of a __device__ array is
// not a device address).  Nothing is cached, so the address stays right after
// the device's context has been torn down and made again (cudaDeviceReset):
// the module is then loaded anew, possibly at another address.
cudaError_t noalloc_scratch(ObsPartial** partials, ObsPartial** result) {
    void* p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess) return e;
    *partials = static_cast<ObsPartial*>(p);
    *result = *partials + OBS_BLOCKS;
    return cudaSuccess;
}

cudaError_t launch_observe_multi(const ObsJob* jobs, int n, ObsPartial* results, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    k_observe_multi<<<dim3(OBS_BLOCKS, n), OBS_THREADS, 0, st>>>(jobs);
    k_observe_finish_multi<<<n, OBS_THREADS, 0, st>>>(jobs, results);
    return cudaGetLastError();
}

cudaError_t launch_observe(const ObsArgs& a, ObsPartial* partials, ObsPartial* result, cudaStream_t st) {
    if (a.prec == 0)
        k_observe<float><<<OBS_BLOCKS, OBS_THREADS, 0, st>>>(a, partials);
    else
        k_observe<double><<<OBS_BLOCKS, OBS_THREADS, 0, st>>>(a, partials);
    k_observe_finish<<<1, OBS_THREADS, 0, st>>>(partials, OBS_BLOCKS, result);
    return cudaGetLastError();
}

PF_BOUNDS_READER(bounds_observe)

cudaError_t launch_tip_radius(const TipArgs& a, double* out, cudaStream_t st) {
    double* t = out + 8;  // 2 x 64 crossings after the five results
    const int blocks = (a.dim == 3 ? 2 : 1) * 2 * TIP_J / (TIP_THREADS / 32);
    if (a.prec == 0)
        k_tip_lines<float><<<blocks, TIP_THREADS, 0, st>>>(a, t);
    else
        k_tip_lines<double><<<blocks, TIP_THREADS, 0, st>>>(a, t);
    k_tip_fit<<<1, 32, 0, st>>>(a, t, out);
    return cudaGetLastError();
}

cudaError_t launch_tick(long long* clock, cudaStream_t st) {
    k_tick<<<1, 1, 0, st>>>(clock);
    return cudaGetLastError();
}

cudaError_t launch_init_seeds(int prec, int dim, int nx, int ny, int nz, double h, double U0, const SeedDev* seeds,
                              int n_seeds, void* psi, void* U, int16_t* grain, cudaStream_t st) {
    const int grid = 4 * 152, block = 256;
    if (prec == 0)
        k_init_seeds<float><<<grid, block, 0, st>>>(dim, nx, ny, nz, h, U0, seeds, n_seeds, static_cast<float*>(psi),
                                                    static_cast<float*>(U), grain);
    else
        k_init_seeds<double><<<grid, block, 0, st>>>(dim, nx, ny, nz, h, U0, seeds, n_seeds,
                                                     static_cast<double*>(psi), static_cast<double*>(U), grain);
    return cudaGetLastError();
}

cudaError_t launch_shift_rows(int kind, const void* src, void* dst, int nx, int ny, int nz, int rows, int mode,
                              double a, double b, cudaStream_t st) {
    const int grid = 4 * 152, block = 256;
    if (kind == 0)
        k_shift_rows<float><<<grid, block, 0, st>>>(static_cast<const float*>(src), static_cast<float*>(dst), nx, ny, nz,
                                                    rows, mode, a, b);
    else if (kind == 1)
        k_shift_rows<double><<<grid, block, 0, st>>>(static_cast<const double*>(src), static_cast<double*>(dst), nx, ny,
                                                     nz, rows, mode, a, b);
    else
        k_shift_rows<int16_t><<<grid, block, 0, st>>>(static_cast<const int16_t*>(src), static_cast<int16_t*>(dst), nx,
                                                      ny, nz, rows, 0, 0.0, 0.0);
    return cudaGetLastError();
}

cudaError_t launch_split(const double* x, float* hi, float* lo, long long n, cudaStream_t st) {
    const int block = 256;
    const int grid = 4 * 152;
    k_split<<<grid, block, 0, st>>>(x, hi, lo, n);
    return cudaGetLastError();
}

cudaError_t launch_join(const float* hi, const float* lo, double* x, long long n, cudaStream_t st) {
    const int block = 256;
    const int grid = 4 * 152;
    k_join<<<grid, block, 0, st>>>(hi, lo, x, n);
    return cudaGetLastError();
}

cudaError_t launch_fill(int prec, void* p, double v, long long n, cudaStream_t st) {
    const int grid = 4 * 152, block = 256;
    if (prec == 0)
        k_fill<float><<<grid, block, 0, st>>>(static_cast<float*>(p), (float)v, n);
    else
        k_fill<double><<<grid, block, 0, st>>>(static_cast<double*>(p), v, n);
    return cudaGetLastError();
}

}  // namespace pf
