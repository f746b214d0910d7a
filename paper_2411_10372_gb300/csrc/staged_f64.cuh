// staged_f64.cuh -- the FP64 sweeps L_x, L_y, L_z of Sec. 3.1 as five
// streaming kernels per sweep, 2D and 3D, uniform and stretched z-grids.
//
// What bounds them.  GB300 executes two FP64 operations per SM and cycle; a
// warp's FP64 instruction holds its scheduler's unit for 64 cycles.  A sweep
// is 230 (2D) to 300 (3D) of them per node (counted by the profiler: 38, 54, 39,
// 69 and 31 in the five stages of L_z), so its floor is the number
// of nodes times that, over 608 units, and memory has time to spare (a node's
// sweep takes an SM 110 cycles, its intermediates are 140 bytes).  So nothing
// is computed twice and every unit gets work: each intermediate is computed
// once per node, kept in a scratch array (L2-resident for all but large
// boxes), and one thread takes one node whatever the shape of the grid.  The
// marching kernels of sweep2d.cuh and sweep3d.cuh recompute the halo columns
// of each 28-column strip (14%) and the ramp of each segment, and a small box
// gives them too few warps.
//
//   st_prims   u, T, p of X; |u_al| + c; dX to the next node along the sweep
//   st_flux    F^n (forward differences); the dot products of the limiter
//   st_pred    X^P and its u, T, p
//   st_fluxp   F^P (backward differences); the TVD flux G dX
//   st_out     corrector, average, TVD term, plates; the next dt
//
// 4096 x 1024: 1.90 ms a sweep against 2.2-2.4 of the marching kernels, 256 x 64
// 23 us against 37 (Launch::sweep in kernels_impl.cuh has the other sizes); the
// five launches overlap by programmatic dependent launch, without which 256 x
// 64 takes 33 us.  A stage lets the next one start only after its own wait
// (pdl_enter), so the stages before the previous one are complete when a stage
// starts: what it reads of them -- X, X^P, the TVD coefficient's inputs -- it
// reads before its wait, past L1 (__ldcg): 256 x 64 95 -> 92 us per step, 97 x 81
// x 49 1.35 -> 1.33 ms.  Starting the next stage before the wait took 177 us.
//
// The formulas, their order and their rounding are those of the marching
// kernels.  Boxes larger than the scratch are swept in chunks of planes; a
// chunk recomputes the two planes next to it on each side.
#pragma once
#include "cm_device.cuh"
#include "kernels.h"

namespace cm {

constexpr int kStThreads = 128;
constexpr int kStHead = 2;  // values before the arrays: the sweep's factors

// scratch arrays of a chunk, `n` values each, in this order
template <int ND>
struct StArrays {
    double* base;
    long long n;
    static constexpr int NF = ND + 2;
    static constexpr int kCount = ND + 5 + 3 * NF;
    __device__ double* u(int c) const { return base + c * n; }          // velocity of X, then of X^P
    __device__ double* T() const { return base + ND * n; }              // temperature, likewise
    __device__ double* p() const { return base + (ND + 1) * n; }        // pressure, likewise
    __device__ double* A() const { return base + (ND + 2) * n; }        // |u_al| + c
    __device__ double* ss() const { return base + (ND + 3) * n; }       // dX_{-} . dX
    __device__ double* dd() const { return base + (ND + 4) * n; }       // dX . dX
    __device__ double* F(int f) const { return base + (ND + 5 + f) * n; }           // F^n, then F^P
    __device__ double* XP(int f) const { return base + (ND + 5 + NF + f) * n; }     // X^P
    __device__ double* D(int f) const { return base + (ND + 5 + 2 * NF + f) * n; }  // dX, then the TVD flux
};

template <int ND>
struct StArgs {
    const double* in;
    double* out;
    const double* zt;
    StArrays<ND> s;
    double* head;   // Delta, Delta / h of the sweep
    int kbase;      // plane of scratch row 0
    int ka, kb;     // planes [ka, kb) of this launch
    int k0, k1;     // planes [k0, k1) of the chunk
};

// a thread's node: indices, global offset g, scratch index q
struct StNode {
    int i, j, k;
    long long g, q;
};

template <int ND>
__device__ __forceinline__ bool st_node(const StArgs<ND>& a, const Coef<double>& C, StNode& v)
{
    const unsigned t = blockIdx.x * (unsigned)kStThreads + threadIdx.x;
    const unsigned nx = C.nx, ny = ND == 3 ? C.ny : 1;
    const unsigned row = t / nx;
    v.i = (int)(t - row * nx);
    v.j = ND == 3 ? (int)(row % ny) : 0;
    v.k = a.ka + (int)(ND == 3 ? row / ny : row);
    v.g = ((long long)v.k * ny + v.j) * C.pitch + v.i;
    v.q = ((long long)(v.k - a.kbase) * ny + v.j) * nx + v.i;
    return v.k < a.kb;
}

// offset (in nodes of the scratch, G = false, or of the state) of the
// neighbour one step up or down direction d (0 x, 1 y, 2 z); x, y periodic
template <int ND, bool G = false>
__device__ __forceinline__ long long st_nb(const Coef<double>& C, const StNode& v, int d, int step)
{
    const long long row = G ? C.pitch : C.nx, plane = ND == 3 ? row * C.ny : row;
    if (d == 0) return step > 0 ? (v.i + 1 == C.nx ? 1 - C.nx : 1) : (v.i == 0 ? C.nx - 1 : -1);
    if (d == 1) return (step > 0 ? (v.j + 1 == C.ny ? 1 - C.ny : 1) : (v.j == 0 ? C.ny - 1 : -1)) * row;
    return step > 0 ? plane : -plane;
}

// direction of velocity component c, and component of direction d
template <int ND> __device__ __forceinline__ constexpr int st_dir(int c) { return ND == 3 ? c : 2 * c; }
template <int ND> __device__ __forceinline__ constexpr int st_comp(int d) { return ND == 3 ? d : d / 2; }

template <int ND>
__device__ __forceinline__ void st_prims_of(const double (&X)[ND + 2], double gz, const Coef<double>& C, double (&u)[ND],
                                            double& T, double& p)
{
    double v[ND + 1];
#pragma unroll
    for (int c = 0; c <= ND; ++c) v[c] = X[1 + c];
    quotients(v, X[0]);
#pragma unroll
    for (int c = 0; c < ND; ++c) u[c] = v[c];
    double ke = u[0] * u[0] + u[1] * u[1];
    if constexpr (ND == 3) ke = ke + u[2] * u[2];
    T = C.b * (v[ND] - 0.5 * (ke) - gz);
    p = C.a * X[0] * T;
}

template <int NF>
__device__ __forceinline__ double st_dot(const double (&a)[NF], const double (&b)[NF])
{
    double s = a[0] * b[0];
#pragma unroll
    for (int f = 1; f < NF; ++f) s = s + a[f] * b[f];
    return s;
}

// planes that carry an F^n (FWD) or an F^P: along z all but the last (first)
// plane, along x and y the interior ones
template <int AL, bool FWD>
__device__ __forceinline__ bool st_has_flux(int k, int nz)
{
    if (AL == 2) return FWD ? k <= nz - 2 : k >= 1;
    return k >= 1 && k <= nz - 2;
}

// ---- 1: primitives, wave speed, differences of X along the sweep ----
template <int ND, int AL>
__global__ void __launch_bounds__(kStThreads) st_prims(StArgs<ND> a, const __grid_constant__ Coef<double> C, SweepCtl sc)
{
    constexpr int NF = ND + 2, CA = st_comp<ND>(AL);
    StNode v;
    const bool on = st_node(a, C, v);
    pdl_enter();
    // by the block after the last node's, so that no node waits for it
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) {
        const double dt = step_dt(sc.ctl, sc.slot_in, C.cfl, C.dt_fixed);
        const double Delta = sc.Delta > 0.0 ? sc.Delta : 0.5 * dt;
        a.head[0] = Delta;
        a.head[1] = Delta / (AL == 2 ? C.dz : (AL == 1 ? C.dy : C.dx));
        if (sc.first && a.k0 == 0) {
            sc.ctl->dt_slot[sc.slot_in ^ 1] = 0x7FF0000000000000ULL;
            sc.ctl->t += dt;
            sc.ctl->steps += 1.0;
        }
    }
    if (!on) return;
    double X[NF];
#pragma unroll
    for (int f = 0; f < NF; ++f) X[f] = a.in[f * C.fstride + v.g];
    double u[ND], T, p;
    st_prims_of<ND>(X, C.g * a.zt[v.k], C, u, T, p);
#pragma unroll
    for (int c = 0; c < ND; ++c) a.s.u(c)[v.q] = u[c];
    a.s.T()[v.q] = T;
    a.s.p()[v.q] = p;
    if (AL == 2 ? (v.k <= a.k1 && v.k >= a.k0 - 1) : (v.k >= a.k0 && v.k < a.k1))
        a.s.A()[v.q] = fabs(u[CA]) + sqrt(C.cs2 * T);
    if (AL == 2 ? (v.k <= a.k1 && v.k <= C.nz - 2) : (v.k >= a.k0 && v.k < a.k1)) {
        const long long nb = st_nb<ND, true>(C, v, AL, 1);
#pragma unroll
        for (int f = 0; f < NF; ++f) a.s.D(f)[v.q] = a.in[f * C.fstride + v.g + nb] - X[f];
    }
}

// F_al of Sec. 3.1 at a node from the fields u, T, p of the scratch arrays
// and the conserved values X of the node: one-sided differences along the
// sweep (forward for F^n, backward for F^P), central ones across
template <int ND, int AL, bool ST, bool FWD>
__device__ __forceinline__ void st_flux_of(const StArgs<ND>& a, const Coef<double>& C, const StNode& v,
                                           const double (&X)[ND + 2], double (&F)[ND + 2])
{
    constexpr int CA = st_comp<ND>(AL);
    double u[ND], T = a.s.T()[v.q], p = a.s.p()[v.q];
#pragma unroll
    for (int c = 0; c < ND; ++c) u[c] = a.s.u(c)[v.q];

    // along the sweep: every velocity component and T
    const long long n1 = v.q + st_nb<ND>(C, v, AL, FWD ? 1 : -1);
    double da[ND + 1];
#pragma unroll
    for (int c = 0; c < ND; ++c) da[c] = FWD ? a.s.u(c)[n1] - u[c] : u[c] - a.s.u(c)[n1];
    da[ND] = FWD ? a.s.T()[n1] - T : T - a.s.T()[n1];
    double h = AL == 2 ? C.hz : (AL == 1 ? C.hy : C.hx), ih = AL == 2 ? C.inv_dz : (AL == 1 ? C.inv_dy : C.inv_dx);
    if constexpr (ST && AL == 2) {
        const Plane<double>& P = C.zp[FWD ? v.k : v.k - 1];
        h = P.hp;
        ih = P.ihp;
    }
    quotients(da, h, ih);

    // across: d u_al / d x_d and d u_d / d x_d of each other direction d
    double own[ND], cross[ND];  // by component of d; own[CA] is the one along the sweep
#pragma unroll
    for (int c = 0; c < ND; ++c) {
        const int d = st_dir<ND>(c);
        if (d == AL) {
            own[c] = da[c];
            cross[c] = da[c];
            continue;
        }
        const long long up = v.q + st_nb<ND>(C, v, d, 1), dn = v.q + st_nb<ND>(C, v, d, -1);
        double t[2] = {a.s.u(CA)[up] - a.s.u(CA)[dn], a.s.u(c)[up] - a.s.u(c)[dn]};
        double span = d == 2 ? C.h2z : (d == 1 ? C.h2y : C.h2x), is = d == 2 ? C.inv_2dz : (d == 1 ? C.inv_2dy : C.inv_2dx);
        if constexpr (ST) {
            if (d == 2) {
                span = C.zp[v.k].sc;
                is = C.zp[v.k].isc;
            }
        }
        quotients(t, span, is);
        cross[c] = t[0];
        own[c] = t[1];
    }
    double div = own[0] + own[1];
    if constexpr (ND == 3) div = div + own[2];
    double work = 0.0;
#pragma unroll
    for (int c = 0; c < ND; ++c) {
        const double tau = c == CA ? C.mu * ((da[c] + da[c]) + C.stokes * div) : C.mu * (da[c] + cross[c]);
        F[1 + c] = c == CA ? (X[1 + c] * u[CA] - tau) + p : X[1 + c] * u[CA] - tau;
        work = c == 0 ? u[c] * tau : work + u[c] * tau;
    }
    F[0] = X[1 + CA];
    F[ND + 1] = (u[CA] * (X[ND + 1] + p) - C.kth * da[ND]) - work;
}

// ---- 2: F^n, and the dot products of the differences of X ----
template <int ND, int AL, bool ST>
__global__ void __launch_bounds__(kStThreads) st_flux(StArgs<ND> a, const __grid_constant__ Coef<double> C)
{
    constexpr int NF = ND + 2;
    StNode v;
    const bool on = st_node(a, C, v);
    double X[NF];
    if (on) {
#pragma unroll
        for (int f = 1; f < NF; ++f) X[f] = __ldcg(&a.in[f * C.fstride + v.g]);
    }
    pdl_enter();
    if (!on) return;
    if (st_has_flux<AL, true>(v.k, C.nz)) {
        double F[NF];
        st_flux_of<ND, AL, ST, true>(a, C, v, X, F);
#pragma unroll
        for (int f = 0; f < NF; ++f) a.s.F(f)[v.q] = F[f];
    }
    // dX . dX and dX_{-} . dX of the interface above the node
    if (AL == 2 ? (v.k >= 1 && v.k >= a.k0 - 1 && v.k <= C.nz - 2) : (v.k >= a.k0 && v.k < a.k1)) {
        const long long nb = st_nb<ND>(C, v, AL, -1);
        double d[NF], dm[NF];
#pragma unroll
        for (int f = 0; f < NF; ++f) {
            d[f] = a.s.D(f)[v.q];
            dm[f] = a.s.D(f)[v.q + nb];
        }
        a.s.ss()[v.q] = st_dot(dm, d);
        a.s.dd()[v.q] = st_dot(d, d);
    }
}

// ---- 3: predictor X^P (half cells on the plates of L_z) and its primitives ----
template <int ND, int AL, bool ST>
__global__ void __launch_bounds__(kStThreads) st_pred(StArgs<ND> a, const __grid_constant__ Coef<double> C)
{
    constexpr int NF = ND + 2;
    StNode v;
    const bool on = st_node(a, C, v);
    const bool inner = v.k >= 1 && v.k <= C.nz - 2;
    double X[NF], P[NF];
    const double Delta = __ldcg(&a.head[0]), lam0 = __ldcg(&a.head[1]);
    if (on) {
#pragma unroll
        for (int f = 0; f < NF; ++f) X[f] = __ldcg(&a.in[f * C.fstride + v.g]);
    }
    pdl_enter();
    if (!on) return;
    double lam[1] = {lam0};
    if constexpr (ST && AL == 2) {
        lam[0] = Delta;
        quotients(lam, C.zp[v.k].w, C.zp[v.k].iw);
    }
    const long long nb = v.q + st_nb<ND>(C, v, AL, -1);
    if (inner) {
#pragma unroll
        for (int f = 0; f < NF; ++f) P[f] = X[f] - lam[0] * (a.s.F(f)[v.q] - a.s.F(f)[nb]);
        if (AL == 2) P[ND] = P[ND] + Delta * (-C.g * X[0]);
    } else if (AL == 2) {
        const double half_cell = ST ? lam[0] : 2.0 * lam0;
        P[0] = v.k == 0 ? X[0] - half_cell * a.s.F(0)[v.q] : X[0] + half_cell * a.s.F(0)[nb];
#pragma unroll
        for (int c = 0; c < ND; ++c) P[1 + c] = 0.0;
        P[NF - 1] = P[0] * (v.k == 0 ? C.ebot : C.etop);
    } else {  // plate planes pass through L_x and L_y: X^P = X, primitives as they are
#pragma unroll
        for (int f = 0; f < NF; ++f) a.s.XP(f)[v.q] = X[f];
        return;
    }
#pragma unroll
    for (int f = 0; f < NF; ++f) a.s.XP(f)[v.q] = P[f];
    double u[ND], T, p;
    st_prims_of<ND>(P, C.g * a.zt[v.k], C, u, T, p);
#pragma unroll
    for (int c = 0; c < ND; ++c) a.s.u(c)[v.q] = u[c];
    a.s.T()[v.q] = T;
    a.s.p()[v.q] = p;
}

// ---- 4: F^P, and the TVD flux G dX of the interface above the node ----
template <int ND, int AL, bool ST>
__global__ void __launch_bounds__(kStThreads) st_fluxp(StArgs<ND> a, const __grid_constant__ Coef<double> C)
{
    constexpr int NF = ND + 2;
    StNode v;
    const bool on = st_node(a, C, v);
    // the TVD flux needs nothing of the stage before this one
    const bool tvd = on && (AL == 2 ? (v.k >= 1 && v.k <= C.nz - 3 && v.k < a.k1) : (v.k >= 1 && v.k <= C.nz - 2));
    double G = 0.0;
    if (tvd) {
        const long long nb = v.q + st_nb<ND>(C, v, AL, 1);
        double h = AL == 2 ? C.hz : (AL == 1 ? C.hy : C.hx), ih = AL == 2 ? C.inv_dz : (AL == 1 ? C.inv_dy : C.inv_dx);
        if constexpr (ST && AL == 2) {
            h = C.zp[v.k].hp;
            ih = C.zp[v.k].ihp;
        }
        const double Co = courant(__ldcg(&a.head[0]), 0.0, __ldcg(&a.s.A()[v.q]), __ldcg(&a.s.A()[nb]), h, ih);
        G = tvd_G(__ldcg(&a.s.ss()[v.q]), __ldcg(&a.s.ss()[nb]), __ldcg(&a.s.dd()[v.q]), Co, C.tvd_form);
    }
    pdl_enter();
    if (!on) return;
    if (v.k >= a.k0 && st_has_flux<AL, false>(v.k, C.nz)) {
        double X[NF], F[NF];
#pragma unroll
        for (int f = 1; f < NF; ++f) X[f] = a.s.XP(f)[v.q];
        st_flux_of<ND, AL, ST, false>(a, C, v, X, F);
#pragma unroll
        for (int f = 0; f < NF; ++f) a.s.F(f)[v.q] = F[f];
    }
    if (tvd) {
#pragma unroll
        for (int f = 0; f < NF; ++f) a.s.D(f)[v.q] = G * a.s.D(f)[v.q];
    }
}

// ---- 5: corrector, average, TVD term, plates; LAST: the next dt ----
template <int ND, int AL, bool ST, bool LAST>
__global__ void __launch_bounds__(kStThreads) st_out(StArgs<ND> a, const __grid_constant__ Coef<double> C, SweepCtl sc)
{
    constexpr int NF = ND + 2;
    StNode v;
    const bool on = st_node(a, C, v);
    const double Delta = __ldcg(&a.head[0]), lam0 = __ldcg(&a.head[1]);
    double X[NF], XP[NF];
    if (on) {
#pragma unroll
        for (int f = 0; f < NF; ++f) {
            X[f] = __ldcg(&a.in[f * C.fstride + v.g]);
            XP[f] = __ldcg(&a.s.XP(f)[v.q]);
        }
    }
    pdl_enter();
    // LAST: the next dt is the minimum of h/(|u| + c); a quotient rounds
    // monotonically, so on uniform planes the block's largest |u| + c of each
    // direction decides, one division each, and only they are reduced (as bits)
    unsigned long long speed[ND] = {};
    double vmin = 1e308;
    int bad = 0;
    if (on) {
        const bool inner = v.k >= 1 && v.k <= C.nz - 2;
        double Y[NF];
        double lam[1] = {lam0};
        if constexpr (ST && AL == 2) {
            lam[0] = Delta;
            quotients(lam, C.zp[v.k].w, C.zp[v.k].iw);
        }
        const long long up = v.q + st_nb<ND>(C, v, AL, 1), dn = v.q + st_nb<ND>(C, v, AL, -1);
        if (inner) {
            // TVD fluxes above and below; none next to the plates
            const bool has_up = AL != 2 || v.k <= C.nz - 3, has_dn = AL != 2 || v.k >= 2;
            const double rp = (ST && AL == 2) ? C.zp[v.k].rp : 1.0, rm = (ST && AL == 2) ? C.zp[v.k].rm : 1.0;
#pragma unroll
            for (int f = 0; f < NF; ++f) {
                double xc = X[f] - lam[0] * (a.s.F(f)[up] - a.s.F(f)[v.q]);
                if (AL == 2 && f == ND) xc = xc + Delta * (-C.g * XP[0]);
                const double mean = 0.5 * (XP[f] + xc);
                const double Dn = has_up ? a.s.D(f)[v.q] : 0.0, Dm = has_dn ? a.s.D(f)[dn] : 0.0;
                if constexpr (ST && AL == 2) Y[f] = mean + (rp * Dn - rm * Dm);
                else Y[f] = mean + (Dn - Dm);
            }
        } else if (AL == 2) {
            const double half_cell = ST ? lam[0] : 2.0 * lam0;
            const double xc = v.k == 0 ? X[0] - half_cell * a.s.F(0)[up] : X[0];  // F^P on the top plate is m_z = 0
            Y[0] = (XP[0] + xc) * 0.5;
#pragma unroll
            for (int c = 0; c < ND; ++c) Y[1 + c] = 0.0;
            Y[NF - 1] = Y[0] * (v.k == 0 ? C.ebot : C.etop);
        } else {
#pragma unroll
            for (int f = 0; f < NF; ++f) Y[f] = X[f];
        }
#pragma unroll
        for (int f = 0; f < NF; ++f) a.out[f * C.fstride + v.g] = Y[f];
        if constexpr (LAST) {
            double u[ND], T, p;
            st_prims_of<ND>(Y, C.g * a.zt[v.k], C, u, T, p);
            const double cs = sqrt(C.cs2 * T);
            if constexpr (ST) {
                vmin = C.dx / (fabs(u[0]) + cs);
                if constexpr (ND == 3) vmin = fmin(vmin, C.dy / (fabs(u[1]) + cs));
                vmin = fmin(vmin, C.zp[v.k].hmin / (fabs(u[ND - 1]) + cs));
                if (!(vmin > 0.0) || !(vmin < 1e300)) bad = 1;
            } else {
                unsigned long long any = 0;
#pragma unroll
                for (int c = 0; c < ND; ++c) {
                    speed[c] = (unsigned long long)__double_as_longlong(fabs(u[c]) + cs);
                    if (speed[c] >= 0x7ff0000000000000ULL) bad = 1;  // infinite (dt = 0) or NaN (left out)
                    if (speed[c] > 0x7ff0000000000000ULL) speed[c] = 0;
                    any |= speed[c];
                }
                if (any == 0) bad = 1;
            }
        }
    }
    if constexpr (LAST && ST) block_dt_reduce(vmin, bad, sc.ctl, sc.slot_in ^ 1);
    if constexpr (LAST && !ST) {
        __shared__ unsigned long long top[ND][kStThreads / 32];
        __shared__ int flag[kStThreads / 32];
        const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
        bad = __any_sync(0xffffffffu, bad);
#pragma unroll
        for (int c = 0; c < ND; ++c) {
            for (int o = 16; o > 0; o >>= 1) {
                const unsigned long long t = __shfl_xor_sync(0xffffffffu, speed[c], o);
                speed[c] = t > speed[c] ? t : speed[c];
            }
            if (lane == 0) top[c][w] = speed[c];
        }
        if (lane == 0) flag[w] = bad;
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int q = 1; q < kStThreads / 32; ++q) {
                bad |= flag[q];
                for (int c = 0; c < ND; ++c) speed[c] = top[c][q] > speed[c] ? top[c][q] : speed[c];
            }
            if (bad) atomicOr(&sc.ctl->status, 1);
            double m = C.dx / __longlong_as_double((long long)speed[0]);
            if constexpr (ND == 3) m = fmin(m, C.dy / __longlong_as_double((long long)speed[1]));
            m = fmin(m, C.dz / __longlong_as_double((long long)speed[ND - 1]));
            if (m < __longlong_as_double(0x7FF0000000000000LL))
                atomicMin(&sc.ctl->dt_slot[sc.slot_in ^ 1], (unsigned long long)__double_as_longlong(m));
        }
    }
}

// planes per chunk that `work` values hold (0: too few for a chunk of 8)
template <int ND>
static int st_chunk(const Coef<double>& C)
{
    const long long plane = (long long)C.nx * (ND == 3 ? C.ny : 1);
    const long long rows = (C.work_values - kStHead) / (StArrays<ND>::kCount * plane);
    if (rows >= C.nz) return C.nz;
    return rows >= 12 ? (int)(rows - 4) : 0;
}

template <int ND, int AL, bool ST>
static cudaError_t st_sweep(const double* in, double* out, const double* zt, const Coef<double>& C, const SweepCtl& sc,
                            cudaStream_t s)
{
    const int chunk = st_chunk<ND>(C);
    const long long plane = (long long)C.nx * (ND == 3 ? C.ny : 1);
    for (int k0 = 0; k0 < C.nz; k0 += chunk) {
        const int k1 = std::min(k0 + chunk, C.nz);
        StArgs<ND> a;
        a.in = in;
        a.out = out;
        a.zt = zt;
        a.head = C.work;
        a.s.base = C.work + kStHead;
        a.kbase = std::max(k0 - 2, 0);
        a.s.n = plane * (std::min(k1 + 2, C.nz) - a.kbase);
        a.k0 = k0;
        a.k1 = k1;
        // planes k0 - back .. k1 + ahead, clamped
        auto rows = [&](int back, int ahead) {
            a.ka = std::max(k0 - back, 0);
            a.kb = std::min(k1 + ahead, C.nz);
            return dim3((unsigned)(((long long)(a.kb - a.ka) * plane + kStThreads - 1) / kStThreads));
        };
        const dim3 b(kStThreads);
        cudaError_t e = cudaSuccess;
        dim3 g = rows(2, 2);
        g.x += 1;  // the block that writes the head
        e = launch_pdl(true, st_prims<ND, AL>, g, b, 0, s, a, C, sc);
        if (e != cudaSuccess) return e;
        g = rows(AL == 2 ? 2 : 1, 1);
        if ((e = launch_pdl(true, st_flux<ND, AL, ST>, g, b, 0, s, a, C)) != cudaSuccess) return e;
        g = rows(1, 1);
        if ((e = launch_pdl(true, st_pred<ND, AL, ST>, g, b, 0, s, a, C)) != cudaSuccess) return e;
        g = AL == 2 ? rows(1, 1) : rows(0, 0);
        if ((e = launch_pdl(true, st_fluxp<ND, AL, ST>, g, b, 0, s, a, C)) != cudaSuccess) return e;
        g = rows(0, 0);
        if constexpr (AL == 0) {
            if (sc.last) {
                if ((e = launch_pdl(true, st_out<ND, AL, ST, true>, g, b, 0, s, a, C, sc)) != cudaSuccess) return e;
                continue;
            }
        }
        if ((e = launch_pdl(true, st_out<ND, AL, ST, false>, g, b, 0, s, a, C, sc)) != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace cm
