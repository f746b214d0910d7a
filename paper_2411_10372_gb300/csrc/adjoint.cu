// adjoint.cu -- reverse mode of the 2D FP64 MacCormack-TVD sweeps (Sec. 3.1)
// for gradients of the time-averaged plate Nusselt number (Eq. mean_Nu).
//
// One sweep Y = L_al(Delta) X is differentiated in stages, each a kernel with
// one thread per node.  First the sweep's intermediates are recomputed from X
// (primitives, F^n, X^P and its primitives).  The quantities that decide the
// limiter's and C(Co)'s branches (primitives, wave speeds, the differences of
// X and their dot products, the ratios and Co) are rounded exactly as in the
// forward kernels (explicit intrinsics); everything else may use multiply-add
// contraction.  Then the adjoint
// runs the stages backwards: TVD term, corrector and average, F^P, X^P,
// predictor, F^n, primitives.  Every stage whose forward reads neighbours is
// written as a gather: a node collects the contributions it made to its
// neighbours' outputs, so no atomics are used and the result is
// deterministic.  Non-smooth points take fixed one-sided derivatives:
// phi'(r) = 2 on 0 < 2r < 1 and 0 elsewhere, d|u|/du = 0 at u = 0, the
// Co(1 - Co) branch for Co <= 1/2, and on a tie of max(A_k, A_k+1) the first
// argument.  dt of each step is a constant (the recorded one).
//
// The limiter's ratio r = <dX_-, dX_+> / <dX_+, dX_+> of the vector TVD term
// is not Lipschitz in X: where dX_+ -> 0 with dX_- not parallel to it, the
// exact derivative of phi(r) dX_+ grows like |dX_-| / |dX_+|.  The tangent map
// of a long run then grows without bound although the run itself stays
// bounded.  AdjWork::frozen_phi = 1 drops the derivative through r (phi' = 0
// everywhere: the limiter's switch values held fixed, C(Co) still
// differentiated), which keeps the reverse pass bounded.
//
// Stretched z-grid (C.zp set): the spans and factors follow the forward
// sweeps' conservative form.  Along z, the flux differences of plane k scale
// with Delta / w_k (the plate half cells with Delta / w_0, Delta / w_K), the
// one-sided derivatives of a flux at plane j divide by h_j (F^n) or h_{j-1}
// (F^P), the TVD flux of interface (s, s+1) enters Y_s with weight rp_s and
// Y_{s+1} with rm_{s+1} and its Courant number divides by h_s; the x sweep's
// central z-differences at plane k divide by sc_k = h_{k-1} + h_k.
//
// Every stage is bound by the FP64 units (two operations per SM and cycle;
// about 8 for a division, 7 for a square root), so nothing is divided that a
// reciprocal serves, what a stage needs of the sweep's Delta comes from the
// host, and the differences of X along the sweep and their dot products are
// formed once per interface (k_prims, k_flux), not by each of the interfaces
// that use them.  With the limiter held fixed only G dX is differentiated, so
// that reading stores and gathers one difference's adjoint instead of three.
// One reverse sweep at 1024 x 256: 378 -> 230 us with the limiter fixed.
#include <cuda_runtime.h>

#include <cstring>

#include "adjoint.h"
#include "kernels.h"

namespace cm {
namespace {

constexpr int kAdjThreads = 256;

__device__ __forceinline__ int wrapx(int a, int n) { return a < 0 ? a + n : (a >= n ? a - n : a); }

// node (i, k) <-> index k * pitch + i; neighbours along the sweep (AL = 2: z,
// AL = 0: x, periodic) and across it
template <int AL>
__device__ __forceinline__ long long nb_al(const Coef<double>& C, int i, int k, int s)
{
    return AL == 2 ? (long long)(k + s) * C.pitch + i : (long long)k * C.pitch + wrapx(i + s, C.nx);
}
template <int AL>
__device__ __forceinline__ long long nb_ac(const Coef<double>& C, int i, int k, int s)
{
    return AL == 2 ? (long long)k * C.pitch + wrapx(i + s, C.nx) : (long long)(k + s) * C.pitch + i;
}

// nodes that carry a flux: F^n (FWD) along z on planes 0..K-1, F^P along z on
// 1..K; along x the interior rows 1..K-1 only
template <int AL, bool FWD>
__device__ __forceinline__ bool has_flux(const Coef<double>& C, int k)
{
    const int K = C.nz - 1;
    if (AL == 2) return FWD ? (k >= 0 && k <= K - 1) : (k >= 1 && k <= K);
    return k >= 1 && k <= K - 1;
}

__device__ __forceinline__ bool interior_row(const Coef<double>& C, int k) { return k >= 1 && k <= C.nz - 2; }

struct Q4 {
    double v[4];
};

__device__ __forceinline__ Q4 ld4(const double* X, long long fs, long long n)
{
    return {{X[n], X[fs + n], X[2 * fs + n], X[3 * fs + n]}};
}

__device__ __forceinline__ void st4(double* X, long long fs, long long n, const Q4& q)
{
    X[n] = q.v[0];
    X[fs + n] = q.v[1];
    X[2 * fs + n] = q.v[2];
    X[3 * fs + n] = q.v[3];
}

// primitives in the forward kernels' operation order (Sec. 2 closures), each
// operation rounded on its own (explicit intrinsics: this unit contracts
// multiply-adds elsewhere), so that T and the wave speed that decide the
// limiter's branches equal the forward run's bit for bit
__device__ __forceinline__ void prims_of(const Q4& q, double z, const Coef<double>& C, double& ux, double& uz,
                                         double& T, double& p)
{
    double v[3] = {q.v[1], q.v[2], q.v[3]};
    quotients(v, q.v[0]);
    ux = v[0];
    uz = v[1];
    const double ke = __dmul_rn(0.5, __dadd_rn(__dmul_rn(ux, ux), __dmul_rn(uz, uz)));
    T = __dmul_rn(C.b, __dsub_rn(__dsub_rn(v[2], ke), __dmul_rn(C.g, z)));
    p = __dmul_rn(__dmul_rn(C.a, q.v[0]), T);
}

// grid-stride loop over the nodes; each iteration defines i, k and the index n = k * pitch + i
#define FOR_NODES(C)                                                                                    \
    for (long long t_ = blockIdx.x * (long long)blockDim.x + threadIdx.x; t_ < (long long)(C).nx * (C).nz; \
         t_ += (long long)gridDim.x * blockDim.x)
#define NODE(C)                                                                                         \
    const int k = (int)(t_ / (C).nx), i = (int)(t_ % (C).nx);                                          \
    const long long n = (long long)k * (C).pitch + i;                                                   \
    (void)i;                                                                                            \
    (void)n

// interfaces (node, next node along the sweep) that exist
template <int AL>
__device__ __forceinline__ bool has_iface(const Coef<double>& C, int k)
{
    return AL == 2 ? k <= C.nz - 2 : interior_row(C, k);
}

// primitives and wave speed of X, and dX to the next node along the sweep (DX)
template <int AL>
__global__ void k_prims(const double* __restrict__ X, const double* __restrict__ zt, Coef<double> C, AdjWork w)
{
    pdl_enter();
    FOR_NODES(C)
    {
        NODE(C);
        double ux, uz, T, p;
        const Q4 x = ld4(X, w.fs, n);
        prims_of(x, zt[k], C, ux, uz, T, p);
        if (has_iface<AL>(C, k)) {
            const Q4 xn = ld4(X, w.fs, nb_al<AL>(C, i, k, 1));
            Q4 dx;
            for (int c = 0; c < 4; ++c) dx.v[c] = xn.v[c] - x.v[c];
            st4(w.DX, w.fs, n, dx);
        }
        w.U0[n] = ux;
        w.U1[n] = uz;
        w.T[n] = T;
        w.P[n] = p;
        w.A[n] = __dadd_rn(fabs(AL == 2 ? uz : ux), __dsqrt_rn(__dmul_rn(C.cs2, T)));
    }
}

// the derivatives a flux at node (i, k) uses: along the sweep one-sided
// (forward for F^n, backward for F^P), across central.  d[0..2] = along
// (u_al, u_across, T), d[3..4] = across (u_al, u_across).
template <int AL, bool FWD>
__device__ __forceinline__ void flux_derivs(const Coef<double>& C, const double* Ux, const double* Uz,
                                            const double* Tt, int i, int k, long long n, double (&d)[5])
{
    const double* Ua = AL == 2 ? Uz : Ux;
    const double* Uc = AL == 2 ? Ux : Uz;
    const long long np = FWD ? nb_al<AL>(C, i, k, 1) : n, nm = FWD ? n : nb_al<AL>(C, i, k, -1);
    // no branch of the reverse pass depends on these, so reciprocal spans suffice
    double ia = AL == 2 ? C.inv_dz : C.inv_dx, ic = AL == 2 ? C.inv_2dx : C.inv_2dz;
    if (C.zp) {
        if (AL == 2) ia = C.zp[FWD ? k : k - 1].ihp;  // spacing spanned by the one-sided difference
        else ic = C.zp[k].isc;                        // distance of planes k-1 and k+1
    }
    d[0] = (Ua[np] - Ua[nm]) * ia;
    d[1] = (Uc[np] - Uc[nm]) * ia;
    d[2] = (Tt[np] - Tt[nm]) * ia;
    const long long cp = nb_ac<AL>(C, i, k, 1), cm_ = nb_ac<AL>(C, i, k, -1);
    d[3] = (Ua[cp] - Ua[cm_]) * ic;
    d[4] = (Uc[cp] - Uc[cm_]) * ic;
}

// F_al of Sec. 3.1 in 2D, by components along (a) and across (c) the sweep:
//   [m_a ; m_a u_a - tau_a + p ; m_c u_a - tau_c ; u_a (E + p) - K dT_a - (u_x tau_x + u_z tau_z)]
//   tau_a = mu (2 d_a u_a + s div), tau_c = mu (d_a u_c + d_c u_a), div = d_a u_a + d_c u_c
template <int AL>
__device__ __forceinline__ Q4 flux_of(const Q4& q, double ux, double uz, double p, const double (&d)[5],
                                      const Coef<double>& C)
{
    constexpr int fa = AL == 2 ? 2 : 1, fc = AL == 2 ? 1 : 2;
    const double ua = AL == 2 ? uz : ux;
    const double div = d[0] + d[4];
    const double ta = C.mu * ((d[0] + d[0]) + C.stokes * div);
    const double tc = C.mu * (d[1] + d[3]);
    const double tx = AL == 2 ? tc : ta, tz = AL == 2 ? ta : tc;
    Q4 F;
    F.v[0] = q.v[fa];
    F.v[fa] = (q.v[fa] * ua - ta) + p;
    F.v[fc] = q.v[fc] * ua - tc;
    F.v[3] = (ua * (q.v[3] + p) - C.kth * d[2]) - (ux * tx + uz * tz);
    return F;
}

// dot product in the forward kernels' order, every operation rounded on its own
__device__ __forceinline__ double dot4q(const Q4& a, const Q4& b)
{
    return __dadd_rn(__dadd_rn(__dadd_rn(__dmul_rn(a.v[0], b.v[0]), __dmul_rn(a.v[1], b.v[1])),
                               __dmul_rn(a.v[2], b.v[2])),
                     __dmul_rn(a.v[3], b.v[3]));
}

// F^n, and of each interface <dX, dX> (DD) and <dX_{-}, dX> (SS)
template <int AL>
__global__ void k_flux(const double* __restrict__ X, Coef<double> C, AdjWork w)
{
    pdl_enter();
    FOR_NODES(C)
    {
        NODE(C);
        if (has_flux<AL, true>(C, k)) {
            double d[5];
            flux_derivs<AL, true>(C, w.U0, w.U1, w.T, i, k, n, d);
            st4(w.F, w.fs, n, flux_of<AL>(ld4(X, w.fs, n), w.U0[n], w.U1[n], w.P[n], d, C));
        }
        if (has_iface<AL>(C, k) && (AL == 0 || k >= 1)) {
            const Q4 d0 = ld4(w.DX, w.fs, n), dm = ld4(w.DX, w.fs, nb_al<AL>(C, i, k, -1));
            w.DD[n] = dot4q(d0, d0);
            w.SS[n] = dot4q(dm, d0);
        }
    }
}

// X^P (predictor, plate half cells for L_z, plate rows unchanged for L_x) and its primitives
template <int AL>
__global__ void k_pred(const double* __restrict__ X, const double* __restrict__ zt, Coef<double> C, AdjWork w,
                       double Delta, double lam)
{
    pdl_enter();
    FOR_NODES(C)
    {
        NODE(C);
        const Q4 x = ld4(X, w.fs, n);
        Q4 xp = x;
        if (interior_row(C, k)) {
            const double lk = (AL == 2 && C.zp) ? Delta * C.zp[k].iw : lam;
            const Q4 f0 = ld4(w.F, w.fs, n), f1 = ld4(w.F, w.fs, nb_al<AL>(C, i, k, -1));
            for (int c = 0; c < 4; ++c) xp.v[c] = x.v[c] - lk * (f0.v[c] - f1.v[c]);
            if (AL == 2) xp.v[2] = xp.v[2] + Delta * (-C.g * x.v[0]);
        } else if (AL == 2) {
            const double lpl = C.zp ? Delta * C.zp[k].iw : 2.0 * lam;  // plate half cell
            xp.v[0] = (k == 0) ? x.v[0] - lpl * w.F[n] : x.v[0] + lpl * w.F[nb_al<AL>(C, i, k, -1)];
            xp.v[1] = xp.v[2] = 0.0;
            xp.v[3] = xp.v[0] * (k == 0 ? C.ebot : C.etop);
        }
        st4(w.XP, w.fs, n, xp);
        double ux, uz, T, p;
        prims_of(xp, zt[k], C, ux, uz, T, p);
        w.UP0[n] = ux;
        w.UP1[n] = uz;
        w.TP[n] = T;
        w.PP[n] = p;
    }
}

// ---- reverse stages -------------------------------------------------------

// stage 1 of the reverse: the TVD terms.  r_tvd_iface: each interface s+1/2
// (stored at node s) takes the reverse of its flux D = G dX once and stores
// the adjoints of its three differences dX_{s-1/2}, dX_{s+1/2}, dX_{s+3/2} (DVm,
// DV0, DVp; with FROZEN the limiter's ratios are constants and only DV0 is not
// zero) and of the wave speeds A_s, A_s+1 (DVA); zero where there is no TVD
// flux.  tvd_gather: node m sums what the four interfaces s = m+1, m, m-1, m-2
// give it (X_m enters dX_{s-1/2} with -1 for s = m+1, +1 for s = m; dX_{s+1/2}
// with -1 for s = m, +1 for s = m-1; dX_{s+3/2} with -1 for s = m-1, +1 for s =
// m-2).  D_{s+1/2} enters Y_s with + and Y_{s+1} with -.
template <int AL, bool FROZEN>
__global__ void __launch_bounds__(kAdjThreads) r_tvd_iface(const double* __restrict__ Ybar, Coef<double> C, AdjWork w,
                                                           double Delta)
{
    pdl_enter();
    const int K = C.nz - 1;
    FOR_NODES(C)
    {
        NODE(C);
        Q4 tm = {{0.0, 0.0, 0.0, 0.0}}, t0 = tm, tp = tm;
        double a0 = 0.0, a1 = 0.0;
        bool on = C.tvd_form != 2 && (AL == 2 ? (k >= 1 && k <= K - 2) : interior_row(C, k));
        double dd = 0.0;
        if (on) {
            dd = w.DD[n];
            on = !is_zero(dd);
        }
        if (on) {
            const long long s1 = nb_al<AL>(C, i, k, 1);
            const Q4 y0 = ld4(Ybar, w.fs, n), y1 = ld4(Ybar, w.fs, s1), d0 = ld4(w.DX, w.fs, n);
            double wp = 1.0, wm = 1.0, h = AL == 2 ? C.hz : C.hx, ih = AL == 2 ? C.inv_dz : C.inv_dx;
            if (AL == 2 && C.zp) {
                wp = C.zp[k].rp;
                wm = C.zp[k + 1].rm;
                h = C.zp[k].hp;
                ih = C.zp[k].ihp;
            }
            Q4 Db;
            for (int c = 0; c < 4; ++c) Db.v[c] = wp * y0.v[c] - wm * y1.v[c];
            // the ratios and the Courant number with the forward kernels' rounding
            double r[2] = {w.SS[n], w.SS[s1]};
            quotients(r, dd);
            const double A0 = w.A[n], A1 = w.A[s1];
            const double Co = courant(Delta, 0.0, A0, A1, h, ih);
            const bool small = Co <= 0.5;
            const double Cc = small ? Co * (1.0 - Co) : 0.25;
            const double Gb = (Db.v[0] * d0.v[0] + Db.v[1] * d0.v[1]) + (Db.v[2] * d0.v[2] + Db.v[3] * d0.v[3]);
            // 1 - phi, phi = max(0, min(2 r, 1)), of each ratio or of their sum,
            // and whether phi' = 2 there; comparisons on the bits
            auto one_minus_phi = [](double v, bool& slope) {
                const double v2 = v + v;
                const long long bits = __double_as_longlong(v2);
                slope = bits > 0 && bits < 0x3ff0000000000000LL;
                if (bits <= 0) return 1.0;
                return slope ? 1.0 - v2 : 0.0;
            };
            bool sl[2] = {false, false};
            double q;  // sum of the 1 - phi
            if (C.tvd_form == 0) {
                q = one_minus_phi(r[0], sl[0]) + one_minus_phi(r[1], sl[1]);
            } else {
                q = one_minus_phi(r[0] + r[1], sl[0]);
                sl[1] = sl[0];
            }
            const double G = 0.5 * Cc * q;
            for (int c = 0; c < 4; ++c) t0.v[c] = G * Db.v[c];
            if (small) {
                const double Ab = Gb * 0.5 * q * (1.0 - 2.0 * Co) * (Delta * ih);
                if (A0 >= A1) a0 = Ab;
                else a1 = Ab;
            }
            if (!FROZEN && (sl[0] || sl[1])) {
                const double rd = __drcp_rn(dd), rb = -Gb * Cc;  // -Gb Cc phi'/2
                const double spb = sl[0] ? rb * rd : 0.0, smb = sl[1] ? rb * rd : 0.0;
                const double ddb2 = -2.0 * (spb * r[0] + smb * r[1]);
                const Q4 dm = ld4(w.DX, w.fs, nb_al<AL>(C, i, k, -1)), dp = ld4(w.DX, w.fs, s1);
                for (int c = 0; c < 4; ++c) {
                    tm.v[c] = spb * d0.v[c];
                    tp.v[c] = smb * d0.v[c];
                    t0.v[c] += spb * dm.v[c] + smb * dp.v[c] + ddb2 * d0.v[c];
                }
            }
        }
        st4(w.DV0, w.fs, n, t0);
        w.DVA[n] = a0;
        w.DVA[w.fs + n] = a1;
        if (!FROZEN) {
            st4(w.DVm, w.fs, n, tm);
            st4(w.DVp, w.fs, n, tp);
        }
    }
}

template <int AL, bool FROZEN>
__device__ __forceinline__ void tvd_gather(const Coef<double>& C, const AdjWork& w, int i, int k, long long n, Q4& acc, double& ab)
{
    const int K = C.nz - 1;
    for (int c = 0; c < 4; ++c) acc.v[c] = 0.0;
    // interface at node m + d along the sweep exists (in the arrays) for these d
    auto ok = [&](int d) { return AL == 0 || (k + d >= 0 && k + d <= K); };
    const Q4 b0 = ld4(w.DV0, w.fs, n);
    for (int c = 0; c < 4; ++c) acc.v[c] -= b0.v[c];
    ab = w.DVA[n];
    if (ok(-1)) {
        const long long nm = nb_al<AL>(C, i, k, -1);
        const Q4 b = ld4(w.DV0, w.fs, nm);
        for (int c = 0; c < 4; ++c) acc.v[c] += b.v[c];
        ab += w.DVA[w.fs + nm];
    }
    if constexpr (!FROZEN) {
        const Q4 a0 = ld4(w.DVm, w.fs, n);
        for (int c = 0; c < 4; ++c) acc.v[c] += a0.v[c];
        if (ok(1)) {
            const Q4 a = ld4(w.DVm, w.fs, nb_al<AL>(C, i, k, 1));
            for (int c = 0; c < 4; ++c) acc.v[c] -= a.v[c];
        }
        if (ok(-1)) {
            const Q4 a = ld4(w.DVp, w.fs, nb_al<AL>(C, i, k, -1));
            for (int c = 0; c < 4; ++c) acc.v[c] -= a.v[c];
        }
        if (ok(-2)) {
            const Q4 a = ld4(w.DVp, w.fs, nb_al<AL>(C, i, k, -2));
            for (int c = 0; c < 4; ++c) acc.v[c] += a.v[c];
        }
    }
}

// adjoint of the average (X^P + X^C)/2 at a node, the plate values folded in
// (L_z plates: Y = (rho, 0, 0, rho e_w)); zero on plate rows of L_x
template <int AL>
__device__ __forceinline__ Q4 y1bar_of(const Coef<double>& C, const double* Ybar, long long fs, int k, long long n)
{
    const Q4 y = ld4(Ybar, fs, n);
    if (interior_row(C, k)) return y;
    Q4 z = {{0.0, 0.0, 0.0, 0.0}};
    if (AL == 2) z.v[0] = y.v[0] + y.v[3] * (k == 0 ? C.ebot : C.etop);
    return z;
}

// stage 2: the nodes' sums of the TVD adjoints, corrector and average.  X^C = X - lam (F^P_{n+1} - F^P_n) + Delta S(X^P)
// on interior nodes; plate densities of L_z: (X^P + X - 2 lam F^P_1)/2 at the
// bottom, (X^P + X)/2 at the top; plate rows of L_x pass X through.
template <int AL, bool FROZEN>
__global__ void r_corr(const double* __restrict__ Ybar, double* __restrict__ Xbar, Coef<double> C, AdjWork w,
                       double Delta, double lam)
{
    pdl_enter();
    FOR_NODES(C)
    {
        NODE(C);
        const Q4 y1 = y1bar_of<AL>(C, Ybar, w.fs, k, n);
        Q4 xb;
        double ab;
        tvd_gather<AL, FROZEN>(C, w, i, k, n, xb, ab);
        w.AB[n] = ab;
        Q4 xpb = {{0.0, 0.0, 0.0, 0.0}};
        if (interior_row(C, k)) {
            for (int c = 0; c < 4; ++c) {
                xb.v[c] += 0.5 * y1.v[c];
                xpb.v[c] = 0.5 * y1.v[c];
            }
            if (AL == 2) xpb.v[0] += Delta * (-C.g) * (0.5 * y1.v[2]);
        } else if (AL == 2) {
            xb.v[0] += 0.5 * y1.v[0];
            xpb.v[0] = 0.5 * y1.v[0];
        } else {
            const Q4 y = ld4(Ybar, w.fs, n);
            for (int c = 0; c < 4; ++c) xb.v[c] += y.v[c];
        }
        st4(Xbar, w.fs, n, xb);
        st4(w.XPB, w.fs, n, xpb);
        if (has_flux<AL, false>(C, k)) {
            const int km = AL == 2 ? k - 1 : k;
            // Delta / w of planes k and k-1, half of the bottom plate's (stretched L_z)
            double lk = lam, lkm = lam, lhb = lam;
            if (AL == 2 && C.zp) {
                lk = Delta * C.zp[k].iw;
                lkm = Delta * C.zp[km].iw;
                lhb = 0.5 * (Delta * C.zp[0].iw);
            }
            Q4 fpb = {{0.0, 0.0, 0.0, 0.0}};
            if (interior_row(C, k))
                for (int c = 0; c < 4; ++c) fpb.v[c] += lk * (0.5 * y1.v[c]);
            const long long nm = nb_al<AL>(C, i, k, -1);
            if (interior_row(C, km)) {
                const Q4 y1m = y1bar_of<AL>(C, Ybar, w.fs, km, nm);
                for (int c = 0; c < 4; ++c) fpb.v[c] -= lkm * (0.5 * y1m.v[c]);
            }
            if (AL == 2 && k == 1) fpb.v[0] += -lhb * y1bar_of<AL>(C, Ybar, w.fs, 0, nm).v[0];
            st4(w.FPB, w.fs, n, fpb);
        }
    }
}

// sum over a warp of a (in lanes 0..15) and of b (in lanes 16..31): the halves
// swap what they do not keep, so both sums take five additions, not ten
__device__ __forceinline__ double warp_sum2(double a, double b)
{
    const bool low = (threadIdx.x & 16) == 0;
    double x = low ? a : b;
    x += __shfl_xor_sync(0xffffffffu, low ? b : a, 16);
    for (int o = 8; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}

// deterministic block sum of two values into part[2 * blockIdx.x + {0, 1}]
__device__ __forceinline__ void block_sum2(double a, double b, double* part)
{
    __shared__ double sh[2][kAdjThreads / 32];
    const double x = warp_sum2(a, b);
    const int lane = threadIdx.x & 31;
    if ((lane & 15) == 0) sh[lane >> 4][threadIdx.x >> 5] = x;
    __syncthreads();
    if (threadIdx.x < 2) {
        double t = 0.0;
        for (int q = 0; q < kAdjThreads / 32; ++q) t += sh[threadIdx.x][q];
        part[2 * blockIdx.x + threadIdx.x] = t;
    }
}

// stages 3 and 6: reverse of the flux at each node that carries one (F^P on
// X^P, or F^n on X), given its adjoint Fbar.  Adds the terms in q to Qbar and
// writes the node's direct adjoints of (u_x, u_z, T) to UB, those of the
// derivatives it used to DA (along) and DC (across), and the block sums of
// <Fbar, dF/dmu> and <Fbar, dF/dK>.
template <int AL, bool FWD>
__global__ void __launch_bounds__(kAdjThreads) r_flux(const double* __restrict__ Q, const double* Ux,
                                                      const double* Uz, const double* Tt, const double* Pp,
                                                      const double* __restrict__ Fbar, double* Qbar, Coef<double> C,
                                                      AdjWork w, double* part)
{
    pdl_enter();
    constexpr int fa = AL == 2 ? 2 : 1, fc = AL == 2 ? 1 : 2;
    const long long fs = w.fs;
    double smu = 0.0, skt = 0.0;
    FOR_NODES(C)
    {
        NODE(C);
        double ub[3] = {0.0, 0.0, 0.0}, da[3] = {0.0, 0.0, 0.0}, dc[2] = {0.0, 0.0};
        if (has_flux<AL, FWD>(C, k)) {
            double d[5];
            flux_derivs<AL, FWD>(C, Ux, Uz, Tt, i, k, n, d);
            const Q4 q = ld4(Q, fs, n), fb = ld4(Fbar, fs, n);
            const double ux = Ux[n], uz = Uz[n], p = Pp[n], T = Tt[n];
            const double ua = AL == 2 ? uz : ux, uc = AL == 2 ? ux : uz;
            const double div = d[0] + d[4];
            const double xa = (d[0] + d[0]) + C.stokes * div, xc = d[1] + d[3];
            const double ta = C.mu * xa, tc = C.mu * xc;
            const double Fr = fb.v[0], Fa = fb.v[fa], Fc = fb.v[fc], FE = fb.v[3];
            Q4 qb = ld4(Qbar, fs, n);
            qb.v[fa] += Fr + Fa * ua;
            qb.v[fc] += Fc * ua;
            qb.v[3] += FE * ua;
            const double pb = Fa + FE * ua;
            const double uab = Fa * q.v[fa] + Fc * q.v[fc] + FE * (q.v[3] + p) - FE * ta;
            const double ucb = -FE * tc;
            const double tab = -Fa - FE * ua, tcb = -Fc - FE * uc;
            da[2] = -FE * C.kth;
            skt += -FE * d[2];
            smu += tab * xa + tcb * xc;
            da[0] = C.mu * tab * (2.0 + C.stokes);
            dc[1] = C.mu * tab * C.stokes;
            da[1] = C.mu * tcb;
            dc[0] = C.mu * tcb;
            qb.v[0] += pb * C.a * T;  // p = a rho T
            ub[0] = AL == 2 ? ucb : uab;
            ub[1] = AL == 2 ? uab : ucb;
            ub[2] = pb * C.a * q.v[0];
            st4(Qbar, fs, n, qb);
        }
        w.UB[n] = ub[0];
        w.UB[fs + n] = ub[1];
        w.UB[2 * fs + n] = ub[2];
        w.DA[n] = da[0];
        w.DA[fs + n] = da[1];
        w.DA[2 * fs + n] = da[2];
        w.DC[n] = dc[0];
        w.DC[fs + n] = dc[1];
    }
    block_sum2(smu, skt, part);
}

// stages 4 and 7: each node gathers the derivative adjoints of the fluxes
// that read its u and T (one-sided along the sweep: forward for F^n, backward
// for F^P; central across), adds the wave-speed adjoint (F^n stage only), and
// takes the reverse of its primitives into Qbar.  With fold (X^P of L_z), the
// plate nodes' X^P = (rho, 0, 0, rho e_w) is folded into rho.
template <int AL, bool FWD>
__global__ void __launch_bounds__(kAdjThreads) r_gather(const double* __restrict__ Q, double* Qbar,
                                                        const double* Ux, const double* Uz, const double* Tt,
                                                        Coef<double> C, AdjWork w, int with_A, int fold)
{
    pdl_enter();
    const long long fs = w.fs;
    const double ia = AL == 2 ? C.inv_dz : C.inv_dx, ic = AL == 2 ? C.inv_2dx : C.inv_2dz;
    const int K = C.nz - 1;
    FOR_NODES(C)
    {
        NODE(C);
        double uab = AL == 2 ? w.UB[fs + n] : w.UB[n];
        double ucb = AL == 2 ? w.UB[n] : w.UB[fs + n];
        double Tb = w.UB[2 * fs + n];
        // along: the flux at j uses (f[j+1] - f[j]) / h (FWD) or (f[j] - f[j-1]) / h (BWD)
        const double sgn = FWD ? -1.0 : 1.0;
        // 1 / span of the along-sweep difference of the flux at plane j (stretched L_z:
        // h_j for F^n, h_{j-1} for F^P); of the across difference (stretched L_x: sc_j)
        auto ia_of = [&](int j) { return (AL == 2 && C.zp) ? C.zp[FWD ? j : j - 1].ihp : ia; };
        auto ic_of = [&](int j) { return (AL == 0 && C.zp) ? C.zp[j].isc : ic; };
        if (has_flux<AL, FWD>(C, k)) {
            const double a = ia_of(k);
            uab += sgn * w.DA[n] * a;
            ucb += sgn * w.DA[fs + n] * a;
            Tb += sgn * w.DA[2 * fs + n] * a;
        }
        const int kj = AL == 2 ? (FWD ? k - 1 : k + 1) : k;
        if (kj >= 0 && kj <= K && has_flux<AL, FWD>(C, kj)) {
            const long long nj = nb_al<AL>(C, i, k, FWD ? -1 : 1);
            const double a = ia_of(kj);
            uab -= sgn * w.DA[nj] * a;
            ucb -= sgn * w.DA[fs + nj] * a;
            Tb -= sgn * w.DA[2 * fs + nj] * a;
        }
        // across: the flux at j uses (f[j+c] - f[j-c]) / 2h (stretched L_x: / sc_j)
        const int kl = AL == 2 ? k : k - 1, ku = AL == 2 ? k : k + 1;
        if (kl >= 0 && has_flux<AL, FWD>(C, kl)) {
            const long long nj = nb_ac<AL>(C, i, k, -1);
            const double a = ic_of(kl);
            uab += w.DC[nj] * a;
            ucb += w.DC[fs + nj] * a;
        }
        if (ku <= K && has_flux<AL, FWD>(C, ku)) {
            const long long nj = nb_ac<AL>(C, i, k, 1);
            const double a = ic_of(ku);
            uab -= w.DC[nj] * a;
            ucb -= w.DC[fs + nj] * a;
        }
        const double ux = Ux[n], uz = Uz[n];
        if (with_A) {
            const double ab = w.AB[n], ua = AL == 2 ? uz : ux;
            uab += ab * (ua > 0.0 ? 1.0 : (ua < 0.0 ? -1.0 : 0.0));
            Tb += ab * (0.5 * C.cs2) * __drcp_rn(w.A[n] - fabs(ua));  // A = |u| + c, c = sqrt(cs2 T)
        }
        // u = m / rho, T = b (E / rho - |u|^2 / 2 - g z)
        const Q4 q = ld4(Q, fs, n);
        Q4 qb = ld4(Qbar, fs, n);
        double uxb = AL == 2 ? ucb : uab, uzb = AL == 2 ? uab : ucb;
        const double ri = __drcp_rn(q.v[0]), tb = Tb * C.b;
        uxb -= tb * ux;
        uzb -= tb * uz;
        qb.v[0] -= (tb * (q.v[3] * ri) + uxb * ux + uzb * uz) * ri;
        qb.v[1] += uxb * ri;
        qb.v[2] += uzb * ri;
        qb.v[3] += tb * ri;
        if (fold && (k == 0 || k == K)) {
            qb.v[0] += qb.v[3] * (k == 0 ? C.ebot : C.etop);
            qb.v[1] = qb.v[2] = qb.v[3] = 0.0;
        }
        st4(Qbar, fs, n, qb);
    }
}

// stage 5: predictor.  X^P = X - lam (F_n - F_{n-1}) + Delta S(X) on interior
// nodes; L_z plate densities X - 2 lam F_0 and X + 2 lam F_{K-1}; L_x plate rows X.
// Adds dX^P/dX to Xbar and writes the adjoint FB of F^n.
template <int AL>
__global__ void r_pred(double* __restrict__ Xbar, Coef<double> C, AdjWork w, double Delta, double lam)
{
    pdl_enter();
    const int K = C.nz - 1;
    const long long fs = w.fs;
    FOR_NODES(C)
    {
        NODE(C);
        const Q4 xpb = ld4(w.XPB, fs, n);
        Q4 xb = ld4(Xbar, fs, n);
        for (int c = 0; c < 4; ++c) xb.v[c] += xpb.v[c];
        if (AL == 2 && interior_row(C, k)) xb.v[0] += Delta * (-C.g) * xpb.v[2];
        st4(Xbar, fs, n, xb);
        if (has_flux<AL, true>(C, k)) {
            const int kp = AL == 2 ? k + 1 : k;
            // Delta / w of planes k and k+1 and of the plate half cells (stretched L_z)
            double lk = lam, lkp = lam, lbot = 2.0 * lam, ltop = 2.0 * lam;
            if (AL == 2 && C.zp) {
                lk = Delta * C.zp[k].iw;
                lkp = Delta * C.zp[kp].iw;
                lbot = Delta * C.zp[0].iw;
                ltop = Delta * C.zp[K].iw;
            }
            Q4 fb = {{0.0, 0.0, 0.0, 0.0}};
            if (interior_row(C, k))
                for (int c = 0; c < 4; ++c) fb.v[c] -= lk * xpb.v[c];
            const long long np = nb_al<AL>(C, i, k, 1);
            if (interior_row(C, kp)) {
                const Q4 xpbp = ld4(w.XPB, fs, np);
                for (int c = 0; c < 4; ++c) fb.v[c] += lkp * xpbp.v[c];
            }
            if (AL == 2 && k == 0) fb.v[0] += -lbot * xpb.v[0];
            if (AL == 2 && k == K - 1) fb.v[0] += ltop * w.XPB[np];
            st4(w.FB, fs, n, fb);
        }
    }
}

// acc[0..1] += the block partial sums of both flux stages, in a fixed order
constexpr int kAccThreads = 1024;
__global__ void __launch_bounds__(kAccThreads) r_acc(const double* __restrict__ part, int nparts, double* acc)
{
    pdl_enter();
    __shared__ double sh[2][kAccThreads / 32];
    double a = 0.0, b = 0.0;
    for (int q = threadIdx.x; q < nparts; q += kAccThreads) {
        a += part[2 * q];
        b += part[2 * q + 1];
    }
    const double x = warp_sum2(a, b);
    const int lane = threadIdx.x & 31;
    if ((lane & 15) == 0) sh[lane >> 4][threadIdx.x >> 5] = x;
    __syncthreads();
    if (threadIdx.x < 32) {
        const double t = warp_sum2(sh[0][lane], sh[1][lane]);
        if ((lane & 15) == 0) acc[lane >> 4] += t;
    }
}

// ---- objective: plane sums of T and their adjoint --------------------------

struct PlaneSet {
    int k[8];
    double w[8];
    int n;
};

__global__ void __launch_bounds__(kAdjThreads) k_plane_T(const double* __restrict__ X, const double* __restrict__ zt,
                                                         Coef<double> C, long long fs, PlaneSet P, double* out)
{
    __shared__ double sh[kAdjThreads];
    const int k = P.k[blockIdx.x];
    double acc = 0.0;
    for (int i = threadIdx.x; i < C.nx; i += blockDim.x) {
        double ux, uz, T, p;
        prims_of(ld4(X, fs, (long long)k * C.pitch + i), zt[k], C, ux, uz, T, p);
        acc += T;
    }
    sh[threadIdx.x] = acc;
    __syncthreads();
    for (int st = blockDim.x / 2; st > 0; st >>= 1) {
        if ((int)threadIdx.x < st) sh[threadIdx.x] += sh[threadIdx.x + st];
        __syncthreads();
    }
    if (threadIdx.x == 0) out[blockIdx.x] = sh[0];
}

__global__ void k_seed_T(double* Xbar, const double* __restrict__ X, const double* __restrict__ zt, Coef<double> C,
                         long long fs, PlaneSet P)
{
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < (long long)P.n * C.nx;
         t += (long long)gridDim.x * blockDim.x) {
        const int q = (int)(t / C.nx), i = (int)(t % C.nx), k = P.k[q];
        const long long n = (long long)k * C.pitch + i;
        const Q4 x = ld4(X, fs, n);
        Q4 xb = ld4(Xbar, fs, n);
        const double Tb = P.w[q], ri = 1.0 / x.v[0];
        const double ux = x.v[1] * ri, uz = x.v[2] * ri;
        xb.v[3] += Tb * C.b * ri;
        xb.v[0] -= Tb * C.b * (x.v[3] * ri) * ri;
        const double uxb = -Tb * C.b * ux, uzb = -Tb * C.b * uz;
        xb.v[1] += uxb * ri;
        xb.v[2] += uzb * ri;
        xb.v[0] -= (uxb * ux + uzb * uz) * ri;
        st4(Xbar, fs, n, xb);
        (void)zt;
    }
}

__global__ void k_record_dt(const DevCtl* ctl, int slot, double cfl, double dt_fixed, double* out)
{
    if (threadIdx.x == 0 && blockIdx.x == 0) out[0] = step_dt(ctl, slot, cfl, dt_fixed);
}

// dJ/dT at fixed p and u: rho = p/(a T), m = rho u, E = rho (|u|^2/2 + T/b + g z)
// give d(rho, m, E)/dT = (-rho, -m, -E + rho T / b) / T
__global__ void k_grad_T(const double* __restrict__ X, const double* __restrict__ Xbar,
                         const double* __restrict__ zt, Coef<double> C, long long fs, double* gT)
{
    FOR_NODES(C)
    {
        NODE(C);
        double g = 0.0;
        if (interior_row(C, k)) {
            const Q4 x = ld4(X, fs, n), xb = ld4(Xbar, fs, n);
            double ux, uz, T, p;
            prims_of(x, zt[k], C, ux, uz, T, p);
            g = (-(xb.v[0] * x.v[0] + xb.v[1] * x.v[1] + xb.v[2] * x.v[2] + xb.v[3] * x.v[3]) +
                 xb.v[3] * x.v[0] * T / C.b) / T;
        }
        gT[(long long)k * C.nx + i] = g;
    }
}

}  // namespace

// ---- host side ---------------------------------------------------------------

// grid-stride launches of the reverse stages: at most 8 blocks per SM
static int adj_blocks(const Coef<double>& C)
{
    static int nsm = 0;
    if (!nsm) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
        if (nsm <= 0) nsm = 1;
    }
    const long long nodes = (long long)C.nx * C.nz;
    long long b = (nodes + kAdjThreads - 1) / kAdjThreads;
    if (b > 8LL * nsm) b = 8LL * nsm;
    return (int)(b < 1 ? 1 : b);
}

cudaError_t adj_work_create(AdjWork* w, const Coef<double>& C)
{
    std::memset(w, 0, sizeof *w);
    w->fs = C.fstride;
    w->nblocks = adj_blocks(C);
    // the arrays, in order, with their field counts
    double** arrays[] = {&w->U0, &w->U1, &w->T, &w->P, &w->A, &w->F, &w->XP, &w->UP0, &w->UP1, &w->TP,
                         &w->PP, &w->XPB, &w->FPB, &w->FB, &w->UB, &w->DA, &w->DC, &w->AB,
                         &w->DVm, &w->DV0, &w->DVp, &w->DVA, &w->DX, &w->DD, &w->SS};
    const int fields[] = {1, 1, 1, 1, 1, 4, 4, 1, 1, 1, 1, 4, 4, 4, 3, 3, 2, 1, 4, 4, 4, 2, 4, 1, 1};
    static_assert(sizeof arrays / sizeof arrays[0] == sizeof fields / sizeof fields[0], "one count per array");
    size_t nfields = 0;
    for (int f : fields) nfields += (size_t)f;
    const size_t bytes = nfields * (size_t)w->fs * sizeof(double) + (size_t)4 * w->nblocks * sizeof(double);
    cudaError_t e = cudaMalloc(&w->base, bytes);
    if (e != cudaSuccess) return e;
    double* p = w->base;
    for (size_t q = 0; q < sizeof fields / sizeof fields[0]; ++q) {
        *arrays[q] = p;
        p += (size_t)fields[q] * w->fs;
    }
    w->part = p;  // 2 flux stages x nblocks x 2 sums
    return cudaMemset(w->base, 0, bytes);
}

void adj_work_free(AdjWork* w)
{
    if (w->base) cudaFree(w->base);
    w->base = nullptr;
}

template <int AL, bool FROZEN>
static cudaError_t vjp_dir(AdjWork* w, double Delta, const double* X, const double* Ybar, double* Xbar,
                           const double* zt, const Coef<double>& C, double* acc, cudaStream_t s)
{
    const dim3 B(w->nblocks), T(kAdjThreads);
    const AdjWork W = *w;
    const double lam = Delta / (AL == 2 ? C.dz : C.dx);
    cudaError_t e = cudaSuccess;
    // each stage waits for the one before it at its entry (pdl_enter)
    auto go = [&](auto kernel, dim3 g, dim3 t, auto... args) {
        if (e == cudaSuccess) e = launch_pdl(true, kernel, g, t, 0, s, args...);
    };
    go(k_prims<AL>, B, T, X, zt, C, W);
    go(k_flux<AL>, B, T, X, C, W);
    go(k_pred<AL>, B, T, X, zt, C, W, Delta, lam);
    go(r_tvd_iface<AL, FROZEN>, B, T, Ybar, C, W, Delta);
    go(r_corr<AL, FROZEN>, B, T, Ybar, Xbar, C, W, Delta, lam);
    go(r_flux<AL, false>, B, T, W.XP, W.UP0, W.UP1, W.TP, W.PP, W.FPB, W.XPB, C, W, W.part);
    go(r_gather<AL, false>, B, T, W.XP, W.XPB, W.UP0, W.UP1, W.TP, C, W, 0, (int)(AL == 2));
    go(r_pred<AL>, B, T, Xbar, C, W, Delta, lam);
    go(r_flux<AL, true>, B, T, X, W.U0, W.U1, W.T, W.P, W.FB, Xbar, C, W, W.part + 2 * w->nblocks);
    go(r_gather<AL, true>, B, T, X, Xbar, W.U0, W.U1, W.T, C, W, 1, 0);
    go(r_acc, dim3(1), dim3(kAccThreads), W.part, 2 * w->nblocks, acc);
    return e;
}

cudaError_t adj_sweep_vjp(AdjWork* w, int dir, double Delta, const double* X, const double* Ybar, double* Xbar,
                          const double* zt, const Coef<double>& C, double* acc, cudaStream_t s)
{
    const bool fr = w->frozen_phi != 0;
    if (dir == 2) return fr ? vjp_dir<2, true>(w, Delta, X, Ybar, Xbar, zt, C, acc, s) : vjp_dir<2, false>(w, Delta, X, Ybar, Xbar, zt, C, acc, s);
    if (dir == 0) return fr ? vjp_dir<0, true>(w, Delta, X, Ybar, Xbar, zt, C, acc, s) : vjp_dir<0, false>(w, Delta, X, Ybar, Xbar, zt, C, acc, s);
    return cudaErrorInvalidValue;
}

static PlaneSet plane_set(const int* kq, const double* wq, int nq)
{
    PlaneSet P;
    std::memset(&P, 0, sizeof P);
    P.n = nq < 8 ? nq : 8;
    for (int q = 0; q < P.n; ++q) {
        P.k[q] = kq[q];
        P.w[q] = wq ? wq[q] : 0.0;
    }
    return P;
}

cudaError_t adj_plane_T(const double* X, const double* zt, const Coef<double>& C, const int* kq, int nq, double* out,
                        cudaStream_t s)
{
    const PlaneSet P = plane_set(kq, nullptr, nq);
    k_plane_T<<<P.n, kAdjThreads, 0, s>>>(X, zt, C, C.fstride, P, out);
    return cudaGetLastError();
}

cudaError_t adj_seed_T(double* Xbar, const double* X, const double* zt, const Coef<double>& C, const int* kq,
                       const double* wq, int nq, cudaStream_t s)
{
    const PlaneSet P = plane_set(kq, wq, nq);
    const long long work = (long long)P.n * C.nx;
    const int blocks = (int)((work + kAdjThreads - 1) / kAdjThreads);
    k_seed_T<<<blocks, kAdjThreads, 0, s>>>(Xbar, X, zt, C, C.fstride, P);
    return cudaGetLastError();
}

cudaError_t adj_record_dt(const DevCtl* ctl, int slot, double cfl, double dt_fixed, double* out, cudaStream_t s)
{
    k_record_dt<<<1, 32, 0, s>>>(ctl, slot, cfl, dt_fixed, out);
    return cudaGetLastError();
}

cudaError_t adj_grad_T(const double* X, const double* Xbar, const double* zt, const Coef<double>& C, double* gT,
                       cudaStream_t s)
{
    k_grad_T<<<adj_blocks(C), kAdjThreads, 0, s>>>(X, Xbar, zt, C, C.fstride, gT);
    return cudaGetLastError();
}

}  // namespace cm
