// sweep3d_x2.cuh -- FP32 3D sweeps with two columns per lane (uniform or, with
// ST, stretched z-grid): L_z and L_y (march kernel) and L_x of Sec. 3.1.
//
// The 2.5D geometry of sweep3d.cuh -- lanes across x, the warps of a block
// across the third direction W (y for L_z and L_x, z for L_y), all marching
// together along M (z for L_z and L_x, y for L_y) -- with the packed
// arithmetic of sweep2d_x2.cuh: every lane carries two adjacent columns as
// float2 and updates both with one FFMA2/FMUL2/FADD2, so a warp covers 64
// columns, of which lanes 1..30 store 60.  Neighbour columns come from one
// shuffle per exchanged quantity; cross derivatives along W from one
// shared-memory exchange per row (double-buffered by row parity) of the
// velocity components the fluxes need, of X at the newest row and of X^P one
// row behind.  The first and the last warp of a block are halo (F^n, X^P and its
// primitives, no F^P); they also stage rho and two momenta of the row beyond
// theirs and put its two velocities into the exchange, so that no warp is
// spent on that row: 10 of 12 warps store (8 of 12 before, 512 x 512 x 128
// 3.11 -> 2.91 ms per step, 256 x 256 x 128 tanh 1.02 -> 0.89).  Rows are staged by a per-thread cp.async ring in shared memory,
// kRing3 rows deep.
//
// What bounds it: at 168 registers 12 warps run on an SM, three a scheduler,
// so latency and the exchange's barrier count (60% of the issue slots used, a
// third of the instructions register moves and address arithmetic before the
// loops ran two rows a trip).  The registers that two rows a trip need come
// from carrying less: pressures are formed where they are used, L_x keeps of
// F^P only its part across until the row above is known, L_z and L_y carry the
// average with F^P added (V).  512 x 512 x 128, us a sweep, one row a trip with
// the old state -> two with the new: L_z 489 -> 447, L_y 477 -> 426, L_x
// 473 -> 458, with the dt 511 -> 490; with the old state two rows spilled.  The
// stretched L_z would spill (192 against 148 us at 256 x 256 x 128): one row.
// The arithmetic is multiplied out as in the 2D sweeps (K3, flux5).  The x kernel reads an exchange one row
// later, so its barrier is split (an mbarrier: arrive after writing, wait at
// the end of the step) and the TVD term and the F^P stage lie in between:
// 0.580 -> 0.513 ms a sweep at 512 x 512 x 128.  The march kernel needs the
// exchange for F^P of the same row; split around its TVD flux it lost more to
// the smaller basic blocks (0.576 against 0.516 ms), so it keeps the plain
// barrier and one block of code behind it.  512 x 512 x 128: 3.40 -> 3.11 ms per
// step from the arithmetic and the split barrier, 256 x 256 x 128 on the tanh
// grid 1.13 -> 1.02 ms.
//
// The march kernel carries the average across rows:
//   H_c = (X^P + X + Delta S^P)_c / 2 - D_{c-1/2},
//   X_new_c = H_c - (lambda/2) (F^P_{c+1} - F^P_c) + D_{c+1/2},
// which is the average (X^P + X^C)/2 plus the TVD term of Sec. 3.1.  H carries
// (lambda/2) F^P_c as well, except in the momentum along the march: its flux
// difference is formed first, as the scheme writes it, so that equal fluxes
// cancel exactly (y-independent data keep m_y = 0 through L_y, whose
// y-momentum flux holds the pressure).
//
// Stretched z-grid (ST): the conservative metric form of the one-column
// kernels.  L_z: flux differences of plane k over its cell width w_k, the
// one-sided derivatives over the spacing they span, the TVD flux through
// (k, k+1) weighted by its spacing over w_k and its Courant number over that
// spacing; L_y: the central z span of the warp's plane; L_x: the central z
// span of each row's plane and its CFL step 1/h_min.  The block copies the
// metric of its segment's planes after the row ring once (fill_planes).
#pragma once
#include "sweep2d_x2.cuh"
#include "sweep3d.cuh"

namespace cm {

constexpr int kRing3 = 4;  // rows in flight per thread
// warps per block (one halo each side): 12 warps of 168 registers run spill-free;
// 16 would cap a thread at 128 registers (spills: 5.95 against 3.48 ms per
// 512 x 512 x 128 step, before the changes above)
constexpr int kNW3p = 12;
// ring bytes of a block: five fields per warp, three of the row beyond each halo warp
constexpr size_t kRing3Bytes = (size_t)kRing3 * (5 * kNW3p + 3 * 2) * 32 * sizeof(float2);

// 3D state of two columns: (rho, m_x, m_y, m_z, E)
struct P5 {
    f2 r, m[3], E;
};

__device__ __forceinline__ P5 p5_right(const P5& q)
{
    return {right_of(q.r), {right_of(q.m[0]), right_of(q.m[1]), right_of(q.m[2])}, right_of(q.E)};
}
__device__ __forceinline__ P5 p5_left(const P5& q)
{
    return {left_of(q.r), {left_of(q.m[0]), left_of(q.m[1]), left_of(q.m[2])}, left_of(q.E)};
}
__device__ __forceinline__ P5 p5_sub(const P5& a, const P5& b)
{
    return {sub2f(a.r, b.r), {sub2f(a.m[0], b.m[0]), sub2f(a.m[1], b.m[1]), sub2f(a.m[2], b.m[2])}, sub2f(a.E, b.E)};
}
__device__ __forceinline__ f2 p5_dot(const P5& a, const P5& b)
{
    return fma2f(a.E, b.E, fma2f(a.m[2], b.m[2], fma2f(a.m[1], b.m[1], fma2f(a.m[0], b.m[0], mul2f(a.r, b.r)))));
}
__device__ __forceinline__ P5 p5_scale(f2 g, const P5& d)
{
    return {mul2f(g, d.r), {mul2f(g, d.m[0]), mul2f(g, d.m[1]), mul2f(g, d.m[2])}, mul2f(g, d.E)};
}
__device__ __forceinline__ P5 p5_zero()
{
    const f2 z = bc(0.f);
    return {z, {z, z, z}, z};
}

// The five fields of a state buffer, addressed by the byte offset of the
// lane's columns within a field (below 2^32: the launcher sees to it).
// ODD (nx odd): a lane whose columns wrap around x holds two that are not
// adjacent in memory, `gap` bytes apart; the warps that have such lanes
// (split) move every column by itself.
template <bool ODD>
struct Fields5 {
    const char* f[5];
    unsigned gap;
    bool split;
    __device__ __forceinline__ Fields5(const float* base, long long fs, unsigned gap_, bool split_) : gap(gap_), split(split_)
    {
#pragma unroll
        for (int q = 0; q < 5; ++q) f[q] = (const char*)(base + q * fs);
    }
    __device__ __forceinline__ f2 load1(int q, unsigned off) const
    {
        if (ODD && split)
            return make_float2(__ldg(reinterpret_cast<const float*>(f[q] + off)), __ldg(reinterpret_cast<const float*>(f[q] + (off + gap))));
        return __ldg(reinterpret_cast<const f2*>(f[q] + off));
    }
    __device__ __forceinline__ P5 load(unsigned off) const
    {
        return {load1(0, off), {load1(1, off), load1(2, off), load1(3, off)}, load1(4, off)};
    }
    // both: the second column is one of the box (always with an even nx)
    __device__ __forceinline__ void store(unsigned off, const P5& q, bool both) const
    {
        const f2 v[5] = {q.r, q.m[0], q.m[1], q.m[2], q.E};
#pragma unroll
        for (int c = 0; c < 5; ++c) {
            char* d = const_cast<char*>(f[c]) + off;
            if (ODD && !both) *reinterpret_cast<float*>(d) = v[c].x;
            else *reinterpret_cast<f2*>(d) = v[c];
        }
    }
};

__device__ __forceinline__ void cp_async_wait_ring3()
{
    asm volatile("cp.async.wait_group %0;\n" ::"n"(kRing3 - 1) : "memory");
}

// per-thread ring [kRing3 slots][5 fields][threads] of float2; a thread reads
// back only what it copied itself; a row goes into the slot of the row
// consumed last.  The two halo warps (outer) also stage rho, m_A and m_B of
// the row beyond theirs, d_out bytes from their own.
template <bool ODD, int A, int B>
struct Ring5 {
    static constexpr int kT = kNW3p * 32;
    f2 *mine, *beyond;
    unsigned d_out;
    bool outer;
    int take_at = 0, free_at = kRing3 - 1;
    __device__ __forceinline__ Ring5(f2* ring, bool outer_, unsigned d)
        : mine(ring + threadIdx.x), beyond(ring + kRing3 * 5 * kT + (threadIdx.x >= 32 ? 32 : 0) + (threadIdx.x & 31)),
          d_out(d), outer(outer_)
    {
    }
    __device__ __forceinline__ void copy(f2* d, const Fields5<ODD>& in, int q, unsigned off) const
    {
        if (ODD && in.split) {
            cp_async4(&d->x, in.f[q] + off);
            cp_async4(&d->y, in.f[q] + (off + in.gap));
        } else {
            cp_async8(d, in.f[q] + off);
        }
    }
    __device__ __forceinline__ void request_into(int slot, const Fields5<ODD>& in, unsigned off) const
    {
        f2* d = mine + slot * 5 * kT;
#pragma unroll
        for (int q = 0; q < 5; ++q) copy(d + q * kT, in, q, off);
        if (outer) {
            f2* o = beyond + slot * 3 * 64;
#pragma unroll
            for (int q = 0; q < 3; ++q) copy(o + q * 64, in, q == 0 ? 0 : q == 1 ? 1 + A : 1 + B, off + d_out);
        }
    }
    // u_A, u_B of the row beyond, after step(): that step's row
    __device__ __forceinline__ void beyond_u(f2& ua, f2& ub) const
    {
        const f2* o = beyond + free_at * 3 * 64;
        const f2 ri = rcp2(o[0]);
        ua = mul2f(o[64], ri);
        ub = mul2f(o[128], ri);
    }
    __device__ __forceinline__ P5 step(const Fields5<ODD>& in, unsigned off, bool wanted)
    {
        if (wanted) request_into(free_at, in, off);
        cp_async_commit();
        cp_async_wait_ring3();
        const f2* d = mine + take_at * 5 * kT;
        const P5 q = {d[0], {d[kT], d[2 * kT], d[3 * kT]}, d[4 * kT]};
        free_at = take_at;
        take_at = take_at == kRing3 - 1 ? 0 : take_at + 1;
        return q;
    }
};

// A block barrier in two halves.  arrive: this warp has written its part of
// the exchange; wait: every warp has arrived as often as this one.  Each warp
// arrives once per row, so the wait of one row cannot be overtaken by the
// next; it ends as soon as the slowest warp has arrived.  The wait is bounded
// all the same: past the limit it sets the sticky status and goes on.
struct RowBarrier {
    unsigned bar;
    unsigned phase = 0;
    __device__ __forceinline__ explicit RowBarrier(unsigned long long* b) : bar((unsigned)__cvta_generic_to_shared(b))
    {
        if (threadIdx.x == 0) asm volatile("mbarrier.init.shared.b64 [%0], %1;\n" ::"r"(bar), "r"(kNW3p) : "memory");
        __syncthreads();
    }
    __device__ __forceinline__ void arrive() const
    {
        __syncwarp();
        if ((threadIdx.x & 31) == 0) asm volatile("{ .reg .b64 t; mbarrier.arrive.shared.b64 t, [%0]; }\n" ::"r"(bar) : "memory");
    }
    __device__ __forceinline__ void wait(DevCtl* ctl)
    {
        unsigned done = 0;
        for (int n = 0; n < (1 << 22) && !done; ++n)
            asm volatile("{ .reg .pred p; mbarrier.try_wait.parity.shared.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }\n"
                         : "=r"(done)
                         : "r"(bar), "r"(phase)
                         : "memory");
        if (!done) atomicOr(&ctl->status, 1);
        phase ^= 1;
    }
};

// coefficients of one sweep along AL with the directions B1, B2 across, both
// columns alike (see K2 of the 2D sweeps)
struct K3 {
    f2 ab, cs2b;        // p = (a b) rho e, c^2 = (cs2 b) e
    f2 nal, nal2;       // along, per unit difference: -mu/h, -(2 + s) mu/h
    f2 nc1, ns1;        // across B1, per central difference: -mu/(2 h1), -s mu/(2 h1)
    f2 nc2, ns2;        // across B2
    f2 nk;              // -K b/h
    __device__ __forceinline__ K3(const Coef<float>& C, float inv_al, float inv_b1, float inv_b2)
        : ab(bc(C.a * C.b)), cs2b(bc(C.cs2 * C.b)), nal(bc(-C.mu * inv_al)), nal2(bc(-(2.f + C.stokes) * C.mu * inv_al)),
          nc1(bc(-C.mu * inv_b1)), ns1(bc(-C.stokes * C.mu * inv_b1)), nc2(bc(-C.mu * inv_b2)),
          ns2(bc(-C.stokes * C.mu * inv_b2)), nk(bc(-C.kth * C.b * inv_al))
    {
    }
};

// primitives (Sec. 2 closures): u = m/rho, e = E/rho - u^2/2 - g z (T = b e), p = a b rho e; gz = -g z
__device__ __forceinline__ void prims5(const P5& q, f2 gz, const K3& K, f2 (&u)[3], f2& e, f2& p)
{
    const f2 ri = rcp2(q.r);
    u[0] = mul2f(q.m[0], ri);
    u[1] = mul2f(q.m[1], ri);
    u[2] = mul2f(q.m[2], ri);
    const f2 ke = fma2f(u[2], u[2], fma2f(u[1], u[1], mul2f(u[0], u[0])));
    e = fma2f(q.E, ri, fma2f(ke, bc(-0.5f), gz));
    p = mul2f(mul2f(K.ab, q.r), e);
}

__device__ __forceinline__ f2 pressure5(f2 r, f2 e, const K3& K) { return mul2f(mul2f(K.ab, r), e); }

// |u| + c of both columns
__device__ __forceinline__ f2 speed5(f2 u, f2 e, const K3& K)
{
    const f2 c = sqrt2(mul2f(K.cs2b, e));
    return make_float2(__fadd_rn(fabsf(u.x), c.x), __fadd_rn(fabsf(u.y), c.y));
}

// F_AL of Sec. 3.1 for two columns from the differences along the sweep (da of
// u, de of e) and the central differences across: ca1, ca2 of u_AL along B1,
// B2; cb1 of u_B1 along B1, cb2 of u_B2 along B2.  With the negated stresses
// nt[i] = -tau_{i AL}:
//   [m_AL ; m_i u_AL + nt_i + p delta ; u_AL (E + p + nt_AL) + u_B1 nt_B1 + u_B2 nt_B2 - K dT]
template <int AL>
__device__ __forceinline__ P5 flux5(const P5& q, const f2 (&u)[3], f2 p, const f2 (&da)[3], f2 de, f2 ca1, f2 cb1, f2 ca2,
                                    f2 cb2, const K3& K)
{
    constexpr int B1 = AL == 0 ? 1 : 0, B2 = AL == 2 ? 1 : 2;  // the two directions across
    const f2 nta = fma2f(K.nal2, da[AL], fma2f(K.ns1, cb1, mul2f(K.ns2, cb2)));
    const f2 nt1 = fma2f(K.nal, da[B1], mul2f(K.nc1, ca1));
    const f2 nt2 = fma2f(K.nal, da[B2], mul2f(K.nc2, ca2));
    const f2 pt = add2f(p, nta);
    P5 F;
    F.r = q.m[AL];
    F.m[AL] = fma2f(q.m[AL], u[AL], pt);
    F.m[B1] = fma2f(q.m[B1], u[AL], nt1);
    F.m[B2] = fma2f(q.m[B2], u[AL], nt2);
    F.E = fma2f(u[AL], add2f(q.E, pt), fma2f(u[B1], nt1, fma2f(u[B2], nt2, mul2f(K.nk, de))));
    return F;
}

// L_z (AL = 2: march z, W = y) or L_y (AL = 1: march y, W = z).  Row
// pipeline at step j (row j of the march just taken from the ring):
// F^n_{j-1} (forward along the march, central across x from shuffles and
// across W from the exchange of row j-1 one step earlier), X^P_{j-1} and its
// primitives; exchange; F^P_{j-1} (backward along the march); the TVD flux
// across (j-2, j-1) from the input state; output row j-2; H_{j-1}.  Plates:
// for L_z at the ends of the march (half-cell density, m = 0, T = T_w); for
// L_y the plate planes are W rows that pass through unchanged.
template <int AL, bool ST, bool ODD>
__global__ void __launch_bounds__(kNW3p * 32, 1)
sweep3d_march_x2(Sweep3IO<float> io, const __grid_constant__ Coef<float> C, SweepCtl sc)
{
    extern __shared__ f2 ring3_mem[];
    // [row parity][u_AL, u_W of X at row j; u_AL, u_W of X^P at row j-1][row beyond, warps, row beyond][lane]
    __shared__ f2 xs[2][4][kNW3p + 2][32];
    constexpr int WD = (AL == 2) ? 1 : 2;  // direction across the warps

    const int lane = threadIdx.x & 31;
    const int w = threadIdx.x >> 5;
    const bool halo = w == 0 || w == kNW3p - 1;
    const int cw = blockIdx.y * (kNW3p - 2) - 1 + w;  // W coordinate of this warp
    const int ks = blockIdx.z * io.seg;               // first output row of the segment
    const int nz = C.nz, ny = C.ny, nx = C.nx;
    const unsigned pitch4 = C.pitch * (unsigned)sizeof(float);
    const int ke = min(ks + io.seg, io.nmarch);
    const Cols<ODD> col(blockIdx.x, lane, nx);
    // W row this warp reads: periodic in y, clamped in z (out-of-range warps compute unused values)
    auto w_row = [&](int a) -> int { return (WD == 1) ? wrap(a, ny) : min(max(a, 0), nz - 1); };
    const int cwr = w_row(cw);
    const bool own = lane >= 1 && lane <= 30 && col.i < nx && !halo && cw < io.nw;
    const bool passthru = (AL == 1) && (cwr == 0 || cwr == nz - 1);  // L_y leaves the plate planes unchanged

    pdl_enter();
    const float Df = sweep_delta_f32(sc, C);  // Delta = dt/2
    const float lamf = Df * ((AL == 2) ? C.inv_dz : C.inv_dy);
    const f2 lam = bc(lamf), hlam = bc(0.5f * lamf), lam2 = bc(2.f * lamf);
    const f2 mDg = bc(-Df * C.g);  // Delta times the source per unit density (L_z)
    const f2 half = bc(0.5f), z0 = bc(0.f);
    // across W: uniform y (L_z); for L_y on a stretched grid the central span
    // of the warp's own plane.  Stretched L_z: differences along come divided
    const K3 K(C, AL == 2 ? (ST ? 1.f : C.inv_dz) : C.inv_dy, C.inv_2dx,
               (WD == 1) ? C.inv_2dy : (ST ? C.zp[min(max(cw, 0), nz - 1)].isc : C.inv_2dz));
    // stretched L_z: plate half cells Delta / w (predictor) and Delta / (2 w) (average)
    f2 lam_bot = lam2, lam_top = lam2, hlam_bot = lam;
    if constexpr (ST && AL == 2) {
        lam_bot = bc(Df * C.zp[0].iw);
        lam_top = bc(Df * C.zp[nz - 1].iw);
        hlam_bot = bc(0.5f * Df * C.zp[0].iw);
    }

    if (sc.first && blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0 && threadIdx.x == 0) step_bookkeeping(sc, C);

    // byte offset of march row j of this warp's W row
    const unsigned rs = (AL == 2) ? ny * pitch4 : pitch4;
    auto row_off = [&](int j) -> unsigned {
        if (AL == 2) return ((unsigned)min(max(j, 0), nz - 1) * ny + cwr) * pitch4 + col.at;
        return ((unsigned)cwr * ny + wrap(j, ny)) * pitch4 + col.at;
    };
    const Fields5<ODD> fin(io.in, C.fstride, col.gap, col.split), fout(io.out, C.fstride, 0, false);
    const unsigned ws = (AL == 2) ? pitch4 : ny * pitch4;  // from one W row to the next
    Ring5<ODD, AL, WD> ring(ring3_mem, halo, (unsigned)(w_row(w == 0 ? cw - 1 : cw + 1) - cwr) * ws);
    // stretched L_z: the block's plane cache after the ring, {1/hp, 1/w, rp, rm}
    // of planes ks - 4 .. ke (clamped); every warp marches the same rows
    float* pz = reinterpret_cast<float*>(ring3_mem + kRing3Bytes / sizeof(f2));
    if constexpr (ST && AL == 2) fill_planes<float, 4>(pz, C, ks, ke, true);
    auto pl = [&](int k, int q) -> float { return pz[(k - (ks - kPlaneBack)) * 4 + q]; };
    // -g z of march row j (L_z; read one row ahead) or of the warp's plane (L_y)
    auto z_of = [&](int j) -> float { return __ldg(&io.zt[(AL == 2) ? min(max(j, 0), nz - 1) : cwr]); };

    const int j0 = ks - 2;  // first step; the first stored row is ks, at step ks + 2
    for (int q = 0; q < kRing3 - 1; ++q) {
        if (j0 + q <= ke + 1) ring.request_into(q, fin, row_off(j0 + q));
        cp_async_commit();
    }
    // next row to request and its offset; next row to store
    int jr = j0 + kRing3 - 1, jrw = (AL == 1) ? wrap(jr, ny) : 0;
    unsigned gin = row_off(jr), gout = row_off(ks);

    P5 Xm1 = fin.load(row_off(j0 - 1));  // X_{j-1}
    f2 gz1 = bc(-C.g * z_of(j0 - 1));
    float znext = z_of(j0);
    f2 u1[3], e1, unused;
    prims5(Xm1, gz1, K, u1, e1, unused);
    f2 A1 = z0, A2 = z0;        // |u_AL| + c of rows j-1, j-2
    // carried from row to row; each is replaced as soon as its new value
    // exists (which shortens what is live across the exchange)
    P5 F2 = p5_zero();   // F^n_{j-2}
    f2 FPa2 = z0;        // its momentum along the march of F^P_{j-2}
    P5 H = p5_zero();    // H_{j-2}
    P5 d1 = p5_zero();   // X_{j-1} - X_{j-2}
    f2 pp2[3] = {u1[0], u1[1], u1[2]}, ppe2 = e1;  // primitives of X^P_{j-2}
    f2 dd1 = z0, ss2 = z0;      // <d1, d1>, <X_{j-2} - X_{j-3}, d1>

// two rows a trip: the carried rows swap roles instead of being copied
#pragma unroll (AL == 2 && ST ? 1 : 2)
    for (int j = j0; j <= ke + 1; ++j) {
        const P5 X0 = ring.step(fin, gin, jr <= ke + 1);
        if (AL == 2) {
            if (jr >= 0 && jr < nz - 1) gin += rs;
        } else {
            gin += rs;
            if (++jrw == ny) {
                jrw = 0;
                gin -= ny * rs;
            }
        }
        ++jr;
        const f2 gz0 = bc(-C.g * znext);
        znext = z_of(j + 1);
        f2 u0[3], e0;
        prims5(X0, gz0, K, u0, e0, unused);

        // row m = j-1: F^n, X^P and its primitives 
        const int m = j - 1;
        P5 XP1 = Xm1, F1 = p5_zero();
        f2 pp1[3] = {u1[0], u1[1], u1[2]}, ppe1 = e1, ppp1 = z0;
        // stretched L_z: 1/(spacing above m), 1/(spacing below m), Delta / w_m
        f2 ia_f = half, ia_b = half, lam_m = lam;
        if constexpr (ST && AL == 2) {
            ia_f = bc(pl(m, 0));
            ia_b = bc(pl(m - 1, 0));
            lam_m = bc(Df * pl(m, 1));
        }
        if (m >= ks - 2) {
            f2 da[3], de = sub2f(e0, e1);
#pragma unroll
            for (int c = 0; c < 3; ++c) da[c] = sub2f(u0[c], u1[c]);
            if constexpr (ST && AL == 2) {
#pragma unroll
                for (int c = 0; c < 3; ++c) da[c] = mul2f(da[c], ia_f);
                de = mul2f(de, ia_f);
            }
            // across W: the exchange of one step earlier (its buffer is written
            // again only after this step's barrier)
            f2(*b1)[kNW3p + 2][32] = xs[m & 1];
            F1 = flux5<AL>(Xm1, u1, pressure5(Xm1.r, e1, K), da, de, sub2f(right_of(u1[AL]), left_of(u1[AL])),
                           sub2f(right_of(u1[0]), left_of(u1[0])), sub2f(b1[0][w + 2][lane], b1[0][w][lane]),
                           sub2f(b1[1][w + 2][lane], b1[1][w][lane]), K);
            if (AL == 2) {
                if (m >= 1 && m <= nz - 2) {
                    XP1.r = fnma2f(lam_m, sub2f(F1.r, F2.r), Xm1.r);
#pragma unroll
                    for (int c = 0; c < 3; ++c) XP1.m[c] = fnma2f(lam_m, sub2f(F1.m[c], F2.m[c]), Xm1.m[c]);
                    XP1.m[2] = fma2f(mDg, Xm1.r, XP1.m[2]);
                    XP1.E = fnma2f(lam_m, sub2f(F1.E, F2.E), Xm1.E);
                } else if (m <= 0) {
                    XP1.r = fnma2f(lam_bot, F1.r, Xm1.r);
                    XP1.m[0] = XP1.m[1] = XP1.m[2] = z0;
                    XP1.E = mul2f(XP1.r, bc(C.ebot));
                } else {
                    XP1.r = fma2f(lam_top, F2.r, Xm1.r);
                    XP1.m[0] = XP1.m[1] = XP1.m[2] = z0;
                    XP1.E = mul2f(XP1.r, bc(C.etop));
                }
            } else if (!passthru) {
                XP1.r = fnma2f(lam, sub2f(F1.r, F2.r), Xm1.r);
#pragma unroll
                for (int c = 0; c < 3; ++c) XP1.m[c] = fnma2f(lam, sub2f(F1.m[c], F2.m[c]), Xm1.m[c]);
                XP1.E = fnma2f(lam, sub2f(F1.E, F2.E), Xm1.E);
            }
            prims5(XP1, gz1, K, pp1, ppe1, ppp1);
            F2 = F1;
        }

        // exchange across W: u of X at row j and of X^P at row m
        f2(*buf)[kNW3p + 2][32] = xs[j & 1];
        buf[0][w + 1][lane] = u0[AL];
        buf[1][w + 1][lane] = u0[WD];
        buf[2][w + 1][lane] = pp1[AL];
        buf[3][w + 1][lane] = pp1[WD];
        if (halo) ring.beyond_u(buf[0][w == 0 ? 0 : w + 2][lane], buf[1][w == 0 ? 0 : w + 2][lane]);
        __syncthreads();

        const int c = j - 2;
        f2 dd0 = z0, ss1 = z0, A0 = z0;
        P5 nD = p5_zero();

        if (!halo) {
            // minus the TVD flux across (c, m) from the input state
            A0 = speed5(u0[AL], e0, K);
            const P5 d0 = p5_sub(X0, Xm1);
            dd0 = p5_dot(d0, d0);
            ss1 = p5_dot(d1, d0);
            const bool tvd_on = (AL == 2) ? (c >= 1 && c <= nz - 3) : !passthru;
            // Courant number of interface (c, c+1): Delta over its spacing
            const f2 lamh_c = (ST && AL == 2) ? bc(Df * pl(c, 0)) : lam;
            if (tvd_on) nD = p5_scale(tvd_nG2f(ss2, ss1, dd1, mul2f(lamh_c, max2(A2, A1)), C.tvd_form), d1);
            d1 = d0;

            // F^P at row m (backward along the march)
            f2 da[3], de = sub2f(ppe1, ppe2);
#pragma unroll
            for (int q = 0; q < 3; ++q) da[q] = sub2f(pp1[q], pp2[q]);
            if constexpr (ST && AL == 2) {
#pragma unroll
                for (int q = 0; q < 3; ++q) da[q] = mul2f(da[q], ia_b);
                de = mul2f(de, ia_b);
            }
            const P5 FP1 = flux5<AL>(XP1, pp1, ppp1, da, de, sub2f(right_of(pp1[AL]), left_of(pp1[AL])),
                                     sub2f(right_of(pp1[0]), left_of(pp1[0])), sub2f(buf[2][w + 2][lane], buf[2][w][lane]),
                                     sub2f(buf[3][w + 2][lane], buf[3][w][lane]), K);

            // V = (lambda/2) F^P - D enters row c with - and H of row m with +;
            // without F^P in the momentum along the march
            P5 V = nD;
            if constexpr (!(ST && AL == 2)) {
                V.r = fma2f(hlam, FP1.r, nD.r);
#pragma unroll
                for (int q = 0; q < 3; ++q)
                    if (q != AL) V.m[q] = fma2f(hlam, FP1.m[q], nD.m[q]);
                V.E = fma2f(hlam, FP1.E, nD.E);
            }

            // output row c
            if (own && c >= ks) {
                P5 Xn;
                const bool interior = (AL == 2) ? (c >= 1 && c <= nz - 2) : !passthru;
                if (interior) {
                    if constexpr (ST && AL == 2) {
                        // Delta / (2 w_c) on the corrector's flux; the TVD flux
                        // through (c, c+1) weighted by its spacing over w_c
                        const f2 hl = bc(0.5f * Df * pl(c, 1)), rp = bc(pl(c, 2));
                        Xn.r = fnma2f(rp, nD.r, fnma2f(hl, FP1.r, H.r));
#pragma unroll
                        for (int q = 0; q < 3; ++q)
                            Xn.m[q] = fnma2f(rp, nD.m[q], fnma2f(hl, q == AL ? sub2f(FP1.m[q], FPa2) : FP1.m[q], H.m[q]));
                        Xn.E = fnma2f(rp, nD.E, fnma2f(hl, FP1.E, H.E));
                    } else {
                        Xn.r = sub2f(H.r, V.r);
#pragma unroll
                        for (int q = 0; q < 3; ++q)
                            Xn.m[q] = sub2f(q == AL ? fnma2f(hlam, sub2f(FP1.m[q], FPa2), H.m[q]) : H.m[q], V.m[q]);
                        Xn.E = sub2f(H.E, V.E);
                    }
                } else if (AL == 2) {
                    // plates: rho = (rho^P + rho^C)/2 with the half-cell corrector
                    Xn.r = (c == 0) ? fnma2f(hlam_bot, FP1.r, H.r) : H.r;
                    Xn.m[0] = Xn.m[1] = Xn.m[2] = z0;
                    Xn.E = mul2f(Xn.r, bc(c == 0 ? C.ebot : C.etop));
                } else {
                    Xn = H;  // plate planes of L_y: the input row
                }
                fout.store(gout, Xn, col.both);
            }

            // H of row m for the next step
            const bool interior_m = (AL == 2) ? (m >= 1 && m <= nz - 2) : !passthru;
            if (interior_m) {
                if constexpr (ST && AL == 2) {
                    V = p5_scale(bc(pl(m, 3)), nD);  // the flux through (m-1, m): its spacing over w_m
                    const f2 hl = mul2f(half, lam_m);
                    V.r = fma2f(hl, FP1.r, V.r);
                    V.m[0] = fma2f(hl, FP1.m[0], V.m[0]);
                    V.m[1] = fma2f(hl, FP1.m[1], V.m[1]);
                    V.E = fma2f(hl, FP1.E, V.E);
                }
                H.r = fma2f(half, add2f(XP1.r, Xm1.r), V.r);
                H.m[0] = fma2f(half, add2f(XP1.m[0], Xm1.m[0]), V.m[0]);
                H.m[1] = fma2f(half, add2f(XP1.m[1], Xm1.m[1]), V.m[1]);
                if (AL == 2) H.m[2] = fma2f(half, fma2f(mDg, XP1.r, add2f(XP1.m[2], Xm1.m[2])), V.m[2]);
                else H.m[2] = fma2f(half, add2f(XP1.m[2], Xm1.m[2]), V.m[2]);
                H.E = fma2f(half, add2f(XP1.E, Xm1.E), V.E);
            } else if (AL == 2) {
                H = p5_zero();
                H.r = mul2f(half, add2f(XP1.r, Xm1.r));
            } else {
                H = Xm1;
            }
            FPa2 = FP1.m[AL];
        }
        if (c >= ks) gout += rs;

        Xm1 = X0;
        gz1 = gz0;
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            u1[q] = u0[q];
            pp2[q] = pp1[q];
        }
        e1 = e0;
        A2 = A1;
        A1 = A0;
        ppe2 = ppe1;
        dd1 = dd0;
        ss2 = ss1;
    }
    cp_async_drain();
}

// L_x in 3D, march z, warps across y; the x stencil across lanes as in the
// 2D packed x sweep, plate planes pass through.  Row pipeline at step j: for
// row m = j-1, F^n (forward x; d/dz from rows j, j-2; d/dy from the exchange of
// one step earlier), X^P, minus the TVD flux nD across (i-1, i), F^P without
// its differences across x (backward x), V = (lambda/2) F^P + nD and
//   K_m = (X^P + X)_m/2 + V_i - V_{i+1};
// exchange; then for row c = j-2 the rest Q of F^P, which is linear in d/dz of
// X^P (rows j-1, j-3) and d/dy (exchange of row j-2), and
//   X_new_c = K_c - (lambda/2) (Q_{i+1} - Q_i).
// The last sweep of a step (DT) also reduces the next dt from the stored nodes.
template <bool ST, bool ODD, bool DT>
__global__ void __launch_bounds__(kNW3p * 32, 1)
sweep3d_x_x2(Sweep3IO<float> io, const __grid_constant__ Coef<float> C, SweepCtl sc)
{
    extern __shared__ f2 ring3_mem[];
    // [row parity][u_x, u_y of X at row j; u_x, u_y of X^P at row j-1][row beyond, warps, row beyond][lane]
    __shared__ f2 xs[2][4][kNW3p + 2][32];
    __shared__ unsigned long long bar_mem;
    RowBarrier bar(&bar_mem);
    const int lane = threadIdx.x & 31;
    const int w = threadIdx.x >> 5;
    const bool halo = w == 0 || w == kNW3p - 1;
    const int cw = blockIdx.y * (kNW3p - 2) - 1 + w;  // y row of this warp
    const int ks = blockIdx.z * io.seg;
    const int nz = C.nz, ny = C.ny, nx = C.nx;
    const unsigned pitch4 = C.pitch * (unsigned)sizeof(float);
    const int ke = min(ks + io.seg, nz);
    const Cols<ODD> col(blockIdx.x, lane, nx);
    const int cwr = wrap(cw, ny);
    const bool own = lane >= 1 && lane <= 30 && col.i < nx && !halo && cw < ny;

    pdl_enter();
    const float lamf = sweep_delta_f32(sc, C) * C.inv_dx;  // Delta / dx, Delta = dt/2
    const f2 lam = bc(lamf), hlam = bc(0.5f * lamf), half = bc(0.5f), z0 = bc(0.f);
    const K3 K(C, C.inv_dx, C.inv_2dy, ST ? 1.f : C.inv_2dz);  // stretched: z differences come divided
    if (sc.first && blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0 && threadIdx.x == 0) step_bookkeeping(sc, C);
    const unsigned rs = ny * pitch4;
    auto row_off = [&](int k) -> unsigned { return ((unsigned)min(max(k, 0), nz - 1) * ny + cwr) * pitch4 + col.at; };
    auto z_of = [&](int k) -> float { return __ldg(&io.zt[min(max(k, 0), nz - 1)]); };

    // next dt: running maxima of |u_x| + c, |u_y| + c, |u_z| + c over the
    // stored nodes (NaN-propagating), times 1/dx, 1/dy, 1/dz once at the end
    // (equal to the maximum of the per-node products: rounding is monotone)
    float ax = 0.f, ay = 0.f, az = 0.f;
    const Fields5<ODD> fin(io.in, C.fstride, col.gap, col.split), fout(io.out, C.fstride, 0, false);
    Ring5<ODD, 0, 1> ring(ring3_mem, halo, (unsigned)(wrap(w == 0 ? cw - 1 : cw + 1, ny) - cwr) * pitch4);
    // stretched grid: the block's plane cache after the ring, {1/(central z
    // span), 1/(smaller spacing)} of planes ks - 4 .. ke (clamped)
    float* pz = reinterpret_cast<float*>(ring3_mem + kRing3Bytes / sizeof(f2));
    if constexpr (ST) fill_planes<float, 2>(pz, C, ks, ke, false);
    auto pl = [&](int k, int q) -> float { return pz[(k - (ks - kPlaneBack)) * 2 + q]; };
    const int j0 = ks - 1;  // first step: X^P starts with row ks - 1, at step ks
    for (int q = 0; q < kRing3 - 1; ++q) {
        if (j0 + q <= ke + 1) ring.request_into(q, fin, row_off(j0 + q));
        cp_async_commit();
    }
    int jr = j0 + kRing3 - 1;
    unsigned gin = row_off(jr), gout = row_off(ks);

    P5 Xm1 = fin.load(row_off(j0 - 1));
    f2 gz1 = bc(-C.g * z_of(j0 - 1)), gz2 = gz1;
    float znext = z_of(j0);
    f2 u1[3], e1, unused;
    prims5(Xm1, gz1, K, u1, e1, unused);
    f2 u2x = u1[0], u2z = u1[2];            // u_x, u_z of X at row j-2
    f2 dwx1 = z0, dwy1 = z0;                // differences along y of u_x, u_y of X at row j-1
    P5 K2 = Xm1;                            // K of row j-2
    f2 pp2[3] = {u1[0], u1[1], u1[2]};      // velocities of X^P_{j-2}
    f2 pp3x = u1[0], pp3z = u1[2];          // u_x, u_z of X^P at row j-3
    f2 dwpx2 = z0, dwpy2 = z0;              // differences along y of u_x, u_y of X^P at row j-2

#pragma unroll 2
    for (int j = j0; j <= ke + 1; ++j) {
        const P5 X0 = ring.step(fin, gin, jr <= ke + 1);
        if (jr >= 0 && jr < nz - 1) gin += rs;
        ++jr;
        const f2 gz0 = bc(-C.g * znext);
        znext = z_of(j + 1);
        f2 u0[3], e0;
        prims5(X0, gz0, K, u0, e0, unused);

        // row m = j-1: F^n (forward x), X^P, the TVD term along x and K
        const int m = j - 1;
        P5 XP1 = Xm1, K1 = Xm1;  // plate planes pass through
        f2 pp1[3] = {u1[0], u1[1], u1[2]}, ppe1 = e1, ppp1 = z0;
        if (m >= ks - 1 && m >= 1 && m <= nz - 2) {
            f2 da[3], de = sub2f(right_of(e1), e1);
#pragma unroll
            for (int c = 0; c < 3; ++c) da[c] = sub2f(right_of(u1[c]), u1[c]);
            f2 czx = sub2f(u0[0], u2x), czz = sub2f(u0[2], u2z);
            if constexpr (ST) {
                const f2 i2dz_m = bc(pl(m, 0));  // 1/(central z span) of plane m
                czx = mul2f(czx, i2dz_m);
                czz = mul2f(czz, i2dz_m);
            }
            const P5 F1 = flux5<0>(Xm1, u1, pressure5(Xm1.r, e1, K), da, de, dwx1, dwy1, czx, czz, K);
            const P5 Fl = p5_left(F1);
            XP1.r = fnma2f(lam, sub2f(F1.r, Fl.r), Xm1.r);
#pragma unroll
            for (int c = 0; c < 3; ++c) XP1.m[c] = fnma2f(lam, sub2f(F1.m[c], Fl.m[c]), Xm1.m[c]);
            XP1.E = fnma2f(lam, sub2f(F1.E, Fl.E), Xm1.E);
            prims5(XP1, gz1, K, pp1, ppe1, ppp1);
        }

        // exchange across y: u_x, u_y of X at row j and of X^P at row m, read
        // at the end of the step
        f2(*buf)[kNW3p + 2][32] = xs[j & 1];
        buf[0][w + 1][lane] = u0[0];
        buf[1][w + 1][lane] = u0[1];
        buf[2][w + 1][lane] = pp1[0];
        buf[3][w + 1][lane] = pp1[1];
        if (halo) ring.beyond_u(buf[0][w == 0 ? 0 : w + 2][lane], buf[1][w == 0 ? 0 : w + 2][lane]);
        bar.arrive();

        const int c = j - 2;
        if (!halo && m >= ks && m >= 1 && m <= nz - 2) {
            // TVD across (i - 1, i) of row m from the input state
            const P5 dl = p5_sub(Xm1, p5_left(Xm1));
            const f2 dd = p5_dot(dl, dl);
            const f2 sp = p5_dot(dl, p5_right(dl));
            const f2 A = speed5(u1[0], e1, K);
            const f2 nG = tvd_nG2f(left_of(sp), sp, dd, mul2f(lam, max2(left_of(A), A)), C.tvd_form);
            // F^P without its differences across (backward x)
            const f2 nta = mul2f(K.nal2, sub2f(pp1[0], left_of(pp1[0])));
            const f2 nt1 = mul2f(K.nal, sub2f(pp1[1], left_of(pp1[1])));
            const f2 nt2 = mul2f(K.nal, sub2f(pp1[2], left_of(pp1[2])));
            const f2 pt = add2f(ppp1, nta);
            P5 V = p5_scale(nG, dl);  // minus the TVD flux
            V.r = fma2f(hlam, XP1.m[0], V.r);
            V.m[0] = fma2f(hlam, fma2f(XP1.m[0], pp1[0], pt), V.m[0]);
            V.m[1] = fma2f(hlam, fma2f(XP1.m[1], pp1[0], nt1), V.m[1]);
            V.m[2] = fma2f(hlam, fma2f(XP1.m[2], pp1[0], nt2), V.m[2]);
            V.E = fma2f(hlam, fma2f(pp1[0], add2f(XP1.E, pt), fma2f(pp1[1], nt1, fma2f(pp1[2], nt2, mul2f(K.nk, sub2f(ppe1, left_of(ppe1)))))), V.E);
            const P5 dV = p5_sub(V, p5_right(V));
            K1.r = fma2f(half, add2f(XP1.r, Xm1.r), dV.r);
#pragma unroll
            for (int q = 0; q < 3; ++q) K1.m[q] = fma2f(half, add2f(XP1.m[q], Xm1.m[q]), dV.m[q]);
            K1.E = fma2f(half, add2f(XP1.E, Xm1.E), dV.E);
        }
        if (!halo && c >= ks) {
            // row c = j-2: the rest of F^P and the output
            P5 Xn = K2;
            if (c >= 1 && c <= nz - 2) {
                f2 czx = sub2f(pp1[0], pp3x), czz = sub2f(pp1[2], pp3z);
                if constexpr (ST) {
                    const f2 i2dz_c = bc(pl(c, 0));  // 1/(central z span) of plane c
                    czx = mul2f(czx, i2dz_c);
                    czz = mul2f(czz, i2dz_c);
                }
                const f2 Q[3] = {fma2f(K.ns1, dwpy2, mul2f(K.ns2, czz)), mul2f(K.nc1, dwpx2), mul2f(K.nc2, czx)};
                const f2 QE = fma2f(pp2[0], Q[0], fma2f(pp2[1], Q[1], mul2f(pp2[2], Q[2])));
#pragma unroll
                for (int q = 0; q < 3; ++q) Xn.m[q] = fnma2f(hlam, sub2f(right_of(Q[q]), Q[q]), K2.m[q]);
                Xn.E = fnma2f(hlam, sub2f(right_of(QE), QE), K2.E);
            }
            if (own) fout.store(gout, Xn, col.both);
            gout += rs;
            if constexpr (DT) {
                // every lane of a storing warp evaluates; only kept nodes count
                f2 un[3], en;
                prims5(Xn, gz2, K, un, en, unused);
                f2 cs = sqrt2(mul2f(K.cs2b, en));
                if (ODD && !col.both) {  // the second column is another strip's
                    un[0].y = un[0].x; un[1].y = un[1].x; un[2].y = un[2].x;
                    cs.y = cs.x;
                }
                const float vx = fmax_nan(fabsf(un[0].x) + cs.x, fabsf(un[0].y) + cs.y);
                const float vy = fmax_nan(fabsf(un[1].x) + cs.x, fabsf(un[1].y) + cs.y);
                float vz = fmax_nan(fabsf(un[2].x) + cs.x, fabsf(un[2].y) + cs.y);
                if constexpr (ST) vz *= pl(c, 1);  // the plane's CFL z step, 1/h_min
                if (own) {
                    ax = fmax_nan(ax, vx);
                    ay = fmax_nan(ay, vy);
                    az = fmax_nan(az, vz);
                }
            }
        }

        bar.wait(sc.ctl);
        dwx1 = sub2f(buf[0][w + 2][lane], buf[0][w][lane]);
        dwy1 = sub2f(buf[1][w + 2][lane], buf[1][w][lane]);
        dwpx2 = sub2f(buf[2][w + 2][lane], buf[2][w][lane]);
        dwpy2 = sub2f(buf[3][w + 2][lane], buf[3][w][lane]);

        Xm1 = X0;
        gz2 = gz1;
        gz1 = gz0;
        u2x = u1[0];
        u2z = u1[2];
#pragma unroll
        for (int q = 0; q < 3; ++q) u1[q] = u0[q];
        e1 = e0;
        K2 = K1;
        pp3x = pp2[0];
        pp3z = pp2[2];
#pragma unroll
        for (int q = 0; q < 3; ++q) pp2[q] = pp1[q];
    }
    cp_async_drain();
    if constexpr (DT) {
        const float r = fmax_nan(fmax_nan(ax * C.inv_dx, ay * C.inv_dy), ST ? az : az * C.inv_dz);
        block_rmax_dt<kNW3p>(r, sc.ctl, sc.slot_in ^ 1);
    }
}

}  // namespace cm
