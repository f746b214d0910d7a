// sweep2d_x2.cuh -- FP32 sweeps with two columns per lane.
//
// Same scheme and row pipeline as sweep2d.cuh, but every lane carries the
// state of two adjacent columns as float2 and does the arithmetic with the
// packed FP32x2 instructions of sm_100+ (__fadd2_rn, __fmul2_rn,
// __ffma2_rn): one instruction updates both columns.  A warp covers 64
// columns; the stencil and the cross derivatives reach two columns, one
// lane, to each side, so lanes 1..30 produce 60 output columns per strip.
// Neighbour columns come from one shuffle per exchanged quantity:
//   value at c+1 = (own.y, lane+1 .x),  value at c-1 = (lane-1 .y, own.x).
// Loads and stores are 8-byte vectors (the strip origin is even); with an odd
// nx, the warps whose columns reach around x move single columns (Cols).  An
// odd nx took the one-column kernels before: 1001 x 301 0.064 -> 0.027 ms per
// step, 3001 x 1501 tanh 0.44 -> 0.13, 129 x 129 x 65 0.27 -> 0.24.
//
// The sweep bodies (sweep2d_x2_body.inc) are compiled twice.  Namespace pkf
// uses the compiler intrinsics and specialised first steps: the fastest
// form, reproducible bit for bit for a given segment length, but a node's
// FP32 rounding may differ by an ulp with the segment length, because the
// compiler may round separately inlined copies of a step differently.
// Namespace pkx (cm_params.layout_exact) issues every packed operation as an
// opaque PTX instruction and runs interior segments through the same two
// copies of the step from their first step on, so results are bit for bit
// independent of the segment lengths the tuner picks (~6% slower at 4096 x
// 1024).
#pragma once
#include "cm_device.cuh"
#include "sweep2d_x2_types.h"

namespace cm {


typedef float2 f2;

__host__ __device__ __forceinline__ f2 bc(float s) { return make_float2(s, s); }
// Packed FP32x2 arithmetic as compiler intrinsics, rounded once per
// operation: the 3D kernels use these directly; the 2D sweeps below take one
// of two sets of their own (namespaces pkf and pkx).
__device__ __forceinline__ f2 add2f(f2 a, f2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ f2 mul2f(f2 a, f2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ f2 fma2f(f2 a, f2 b, f2 c) { return __ffma2_rn(a, b, c); }
// a - b, rounded once
__device__ __forceinline__ f2 sub2f(f2 a, f2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }
// a - s*b
__device__ __forceinline__ f2 fnma2f(f2 s, f2 b, f2 a) { return __ffma2_rn(make_float2(-s.x, -s.y), b, a); }

__device__ __forceinline__ f2 right_of(f2 v) { return make_float2(v.y, __shfl_down_sync(0xffffffffu, v.x, 1)); }
__device__ __forceinline__ f2 left_of(f2 v) { return make_float2(__shfl_up_sync(0xffffffffu, v.y, 1), v.x); }

struct S2 { f2 r, mx, mz, E; };

__device__ __forceinline__ S2 right_of(const S2& q) { return {right_of(q.r), right_of(q.mx), right_of(q.mz), right_of(q.E)}; }
__device__ __forceinline__ S2 left_of(const S2& q) { return {left_of(q.r), left_of(q.mx), left_of(q.mz), left_of(q.E)}; }

// The two columns of a lane.  at: byte offset of the first within a row; gap:
// distance to the second.  ODD (nx odd): a lane whose columns reach around x
// holds two that are not adjacent in memory or not aligned as a pair; the
// warps that have such lanes (split) move every column by itself, the others
// are those of an even nx.  both: the second column belongs to the box.
template <bool ODD>
struct Cols {
    int i;                 // first column, before wrapping
    unsigned at, gap;
    bool split, both;
    __device__ __forceinline__ Cols(int strip, int lane, int nx)
    {
        i = strip * kOutW2 - 2 + 2 * lane;
        int c0 = i % nx;
        if (c0 < 0) c0 += nx;
        at = c0 * (unsigned)sizeof(float);
        gap = sizeof(float);
        split = false;
        both = true;
        if constexpr (ODD) {
            const int c1 = c0 + 1 == nx ? 0 : c0 + 1;
            gap = (unsigned)(c1 - c0) * (unsigned)sizeof(float);
            split = strip == 0 || strip * kOutW2 + 62 > nx;
            both = i + 1 < nx;
        }
    }
};

// The four fields of a state buffer.  A row is addressed by the byte offset
// of the lane's columns within a field (below 2^32: the launcher sees to it),
// one 32-bit add per row for all four fields.
template <bool ODD>
struct Fields2 {
    const char* f[4];
    unsigned gap;
    bool split;
    __device__ __forceinline__ Fields2(const float* base, long long fs, unsigned gap_, bool split_)
        : f{(const char*)base, (const char*)(base + fs), (const char*)(base + 2 * fs), (const char*)(base + 3 * fs)}, gap(gap_),
          split(split_)
    {
    }
    __device__ __forceinline__ f2 load1(int q, unsigned off) const
    {
        if (ODD && split)
            return make_float2(__ldg(reinterpret_cast<const float*>(f[q] + off)),
                               __ldg(reinterpret_cast<const float*>(f[q] + (off + gap))));
        return __ldg(reinterpret_cast<const f2*>(f[q] + off));
    }
    __device__ __forceinline__ S2 load(unsigned off) const { return {load1(0, off), load1(1, off), load1(2, off), load1(3, off)}; }
    __device__ __forceinline__ void store1(int q, unsigned off, f2 v, bool both) const
    {
        char* d = const_cast<char*>(f[q]) + off;
        if (ODD && !both) *reinterpret_cast<float*>(d) = v.x;
        else *reinterpret_cast<f2*>(d) = v;
    }
    __device__ __forceinline__ void store(unsigned off, const S2& q, bool both) const
    {
        store1(0, off, q.r, both);
        store1(1, off, q.mx, both);
        store1(2, off, q.mz, both);
        store1(3, off, q.E, both);
    }
};

// reciprocal and square root on the special-function unit alone (one MUFU
// instruction each, ~1 ulp, denormals flushed): the FP32 path's tolerance
// is far above that
__device__ __forceinline__ float rcp_fast(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float sqrt_fast(float x)
{
    float r;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ f2 rcp2(f2 a) { return make_float2(rcp_fast(a.x), rcp_fast(a.y)); }
// max(a, b) that returns NaN if either is NaN (fmaxf would drop it)
__device__ __forceinline__ float fmax_nan(float a, float b)
{
    float r;
    asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
    return r;
}

// Delta of a sweep (dt/2 from the step's dt slot, or the single-sweep
// Delta) in FP32, with two FP64 multiplies and one conversion: equal to
// (float)Delta of the FP64 rule.  FP64 issues at a small fraction of the
// FP32 rate on this GPU and every thread of a sweep needs this value at its
// start, where an FP64 division per thread held the warps back at each
// launch.
__device__ __forceinline__ float sweep_delta_f32(const SweepCtl& sc, const Coef<float>& C)
{
    if (sc.Delta > 0.0) return (float)sc.Delta;
    if (C.dt_fixed > 0.0) return (float)(0.5 * C.dt_fixed);
    return (float)(0.5 * (C.cfl * __longlong_as_double((long long)sc.ctl->dt_slot[sc.slot_in])));
}

// the step's advance of t and the step counter, and the reset of the other
// dt slot, by one thread in the first sweep of a step (FP64)
__device__ __forceinline__ void step_bookkeeping(const SweepCtl& sc, const Coef<float>& C)
{
    sc.ctl->dt_slot[sc.slot_in ^ 1] = 0x7FF0000000000000ULL;
    sc.ctl->t += step_dt(sc.ctl, sc.slot_in, C.cfl, C.dt_fixed);
    sc.ctl->steps += 1.0;
}

__device__ __forceinline__ f2 max2(f2 a, f2 b) { return make_float2(fmaxf(a.x, b.x), fmaxf(a.y, b.y)); }
__device__ __forceinline__ f2 sqrt2(f2 a) { return make_float2(sqrt_fast(a.x), sqrt_fast(a.y)); }
// next dt from the FP32 sweeps: the block's maximum of r = max (|u|+c)/h
// over its nodes (NaN-propagating), then one thread stores 1/r in FP64 into
// the dt slot; 1/r is monotone, so this is the minimum of h/(|u|+c) over the
// nodes.  A non-finite maximum sets the sticky status instead.  Every thread
// of the block calls it.
template <int NWARPS>
__device__ __forceinline__ void block_rmax_dt(float r, DevCtl* ctl, int slot)
{
    for (int o = 16; o > 0; o >>= 1) r = fmax_nan(r, __shfl_xor_sync(0xffffffffu, r, o));
    float m = r;
    if constexpr (NWARPS > 1) {
        __shared__ float sm[32];
        if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = r;
        __syncthreads();
        m = sm[0];
        for (int i = 1; i < NWARPS; ++i) m = fmax_nan(m, sm[i]);
    }
    if (threadIdx.x == 0) {
        if (!(m < 1e30f)) {
            atomicOr(&ctl->status, 1);
        } else if (m > 0.f) {
            // the slot only falls while a sweep runs: a block that is already
            // above it has nothing to add (one block is one warp in 2D)
            const unsigned long long v = (unsigned long long)__double_as_longlong(1.0 / (double)m);
            if (v < *(volatile unsigned long long*)&ctl->dt_slot[slot]) atomicMin(&ctl->dt_slot[slot], v);
        }
    }
}

// coefficients of one sweep, both columns alike.  The kernels carry the
// internal energy e = T/b instead of T, and the viscous and heat terms with
// their factors multiplied out (below): 96 packed operations a node and z
// sweep instead of 128, most of them multiply-adds.
struct K2 {
    f2 ab, cs2b;       // p = (a b) rho e, c^2 = (cs2 b) e
    f2 nal, nal2;      // along the sweep, per unit difference: -mu/h, -(2 + s) mu/h
    f2 nac, nacs;      // across, per central difference: -mu/(2 h'), -s mu/(2 h')
    f2 nk;             // -K b/h
    // inv_al: 1/h along the sweep (1 on a stretched grid, where the differences
    // come divided), inv_ac: 1/(2 h') across (likewise)
    __host__ __device__ __forceinline__ K2(const Coef<float>& C, float inv_al, float inv_ac)
        : ab(bc(C.a * C.b)), cs2b(bc(C.cs2 * C.b)), nal(bc(-C.mu * inv_al)), nal2(bc(-(2.f + C.stokes) * C.mu * inv_al)),
          nac(bc(-C.mu * inv_ac)), nacs(bc(-C.stokes * C.mu * inv_ac)), nk(bc(-C.kth * C.b * inv_al))
    {
    }
};


// minus the TVD coefficient G of the flux G dX, both columns at once:
//   C = c(1 - c), c = min(Co, 1/2);  phi(s) = clamp(2 s / dd, 0, 1)
//   Davis form: G = C (1 - (phi(sp) + phi(sm)) / 2);  printed form: C (1 - phi(sp + sm)) / 2
// One reciprocal of dd serves both ratios; the clamps are the saturation of
// the multiplies.  dd = 0 (dX = 0) gives 0 * inf = NaN, which saturates to 0;
// the flux G dX is 0 there anyway.
__device__ __forceinline__ f2 tvd_nG2f(f2 sp, f2 sm, f2 dd, f2 Co, int form)
{
    const f2 c = make_float2(fminf(Co.x, 0.5f), fminf(Co.y, 0.5f));
    const f2 C = fma2f(make_float2(-c.x, -c.y), c, c);
    const f2 r2 = mul2f(bc(2.f), rcp2(dd));
    if (form == 0) {
        const f2 phis = add2f(make_float2(__saturatef(__fmul_rn(sp.x, r2.x)), __saturatef(__fmul_rn(sp.y, r2.y))),
                              make_float2(__saturatef(__fmul_rn(sm.x, r2.x)), __saturatef(__fmul_rn(sm.y, r2.y))));
        return mul2f(C, fma2f(bc(0.5f), phis, bc(-1.f)));
    }
    if (form == 1) {
        const f2 s = add2f(sp, sm);
        const f2 phi = make_float2(__saturatef(__fmul_rn(s.x, r2.x)), __saturatef(__fmul_rn(s.y, r2.y)));
        return mul2f(C, fma2f(bc(0.5f), phi, bc(-0.5f)));
    }
    return make_float2(0.f, 0.f);
}

struct SweepIO2 {
    const float* in;
    float* out;
    const float* zt;
    int seg_rows;
    int nstrips;  // ceil(nx / kOutW2)
};

// ---- asynchronous row loads: each lane copies its own two columns of the
// four fields into a per-thread ring in shared memory (cp.async), kRing rows
// deep, so a row is requested kRing-1 rows before it is consumed without
// holding registers.  A lane only ever reads back what it copied itself, so
// cp.async.wait_group is the only ordering needed.  (Eight rows: 0.109 ms per
// 4096 x 1024 step instead of 0.104.)
constexpr int kRing = 4;

__device__ __forceinline__ void cp_async8(f2* smem, const void* gmem)
{
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async4(float* smem, const void* gmem)
{
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_ring() { asm volatile("cp.async.wait_group %0;\n" ::"n"(kRing - 1) : "memory"); }
__device__ __forceinline__ void cp_async_drain() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

constexpr int kThreads2 = kWarpsX2 * 32;  // block size of the packed kernels

// per-thread ring [kRing slots][4 fields][kThreads2] of float2 in shared
// memory; a row goes into the slot of the row consumed last, so one running
// byte offset serves both ends
template <bool ODD>
struct RowRing {
    static constexpr unsigned kRow = 4 * kThreads2 * sizeof(f2), kMask = kRing * kRow - 1;
    f2* mine;       // this thread's element of slot 0, field 0
    unsigned take_at = 0, free_at = (kRing - 1) * kRow;
    __device__ __forceinline__ explicit RowRing(f2* m) : mine(m) {}
    __device__ __forceinline__ f2* at(unsigned off) const { return reinterpret_cast<f2*>(reinterpret_cast<char*>(mine) + off); }
    __device__ __forceinline__ void request_into(unsigned slot_off, const Fields2<ODD>& in, unsigned off) const
    {
        f2* d = at(slot_off);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if (ODD && in.split) {
                cp_async4(&d[q * kThreads2].x, in.f[q] + off);
                cp_async4(&d[q * kThreads2].y, in.f[q] + (off + in.gap));
            } else {
                cp_async8(d + q * kThreads2, in.f[q] + off);
            }
        }
    }
    // the row kRing-1 ahead, if wanted, then this row
    __device__ __forceinline__ S2 step(const Fields2<ODD>& in, unsigned off, bool wanted)
    {
        if (wanted) request_into(free_at, in, off);
        cp_async_commit();
        cp_async_wait_ring();
        const f2* d = at(take_at);
        const S2 q = {d[0], d[kThreads2], d[2 * kThreads2], d[3 * kThreads2]};
        free_at = take_at;
        take_at = (take_at + kRow) & kMask;
        return q;
    }
};
static_assert((kRing & (kRing - 1)) == 0, "the ring offset wraps by a mask");

// Stretched z-grid: each warp copies the metric of the planes its segment
// touches (ks - 3 .. ke + 1, clamped; ke + 2 for the extra step of an odd
// interior segment in pkx) into its own slice of shared memory,
// after the row ring, so that every row reads it by broadcast.  NV values
// per plane; entry e holds plane clamp(ks - 3 + e).
constexpr int kPlaneBack2 = 3;
__host__ __device__ constexpr int plane_cap2(int seg_rows) { return seg_rows + kPlaneBack2 + 3; }
template <int NV>
__device__ __forceinline__ float* plane_cache2(f2* ring_mem, int seg_rows)
{
    return reinterpret_cast<float*>(ring_mem + kRing * 4 * kThreads2) + (threadIdx.x >> 5) * plane_cap2(seg_rows) * NV;
}

// ---- batched ensemble: many independent boxes in one launch per sweep -----
// Each warp takes one work item (box, strip, first row of its segment); the
// warps of a block always belong to the same box.  Boxes step in
// lockstep (same sweep, same dt slot parity) but each has its own dt, time
// and state buffers.  Batches of up to kConstBoxes boxes read each box's
// coefficients from constant memory with a block-uniform index (no per-thread
// registers for them); larger batches stage them in shared memory.
__constant__ Coef<float> c_box[kConstBoxes];

__device__ __forceinline__ const BatchWork& batch_item(const BatchLaunch& L, SweepCtl& sc, const float*& in,
                                                       float*& out, int& box)
{
    const BatchWork& w = L.work[blockIdx.x * kWarpsX2 + (threadIdx.x >> 5)];
    box = L.work[blockIdx.x * kWarpsX2].box;
    const BoxDesc& B = L.boxes[box];
    sc.ctl = B.ctl;
    sc.slot_in = L.slot;
    sc.first = L.first;
    sc.last = L.last;
    sc.Delta = L.Delta;
    in = B.buf[L.cur];
    out = B.buf[L.cur ^ 1];
    return w;
}

constexpr size_t kRingBytes = (size_t)kRing * 4 * kThreads2 * sizeof(f2);


// ---- the two compiled forms of the 2D sweeps -----------------------------
namespace pkf {
constexpr bool kXL = false;
__device__ __forceinline__ f2 add2(f2 a, f2 b) { return add2f(a, b); }
__device__ __forceinline__ f2 mul2(f2 a, f2 b) { return mul2f(a, b); }
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) { return fma2f(a, b, c); }
__device__ __forceinline__ f2 sub2(f2 a, f2 b) { return sub2f(a, b); }
__device__ __forceinline__ f2 fnma2(f2 s, f2 b, f2 a) { return fnma2f(s, b, a); }
#include "sweep2d_x2_body.inc"
}  // namespace pkf

namespace pkx {
constexpr bool kXL = true;
// each packed operation one PTX instruction, rounded once, that the compiler
// cannot merge, split or re-associate
__device__ __forceinline__ unsigned long long pk(f2 a) { return *reinterpret_cast<unsigned long long*>(&a); }
__device__ __forceinline__ f2 upk(unsigned long long d) { return *reinterpret_cast<f2*>(&d); }
__device__ __forceinline__ f2 add2(f2 a, f2 b)
{
    unsigned long long d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(pk(a)), "l"(pk(b)));
    return upk(d);
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b)
{
    unsigned long long d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(pk(a)), "l"(pk(b)));
    return upk(d);
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c)
{
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(pk(a)), "l"(pk(b)), "l"(pk(c)));
    return upk(d);
}
__device__ __forceinline__ f2 sub2(f2 a, f2 b)
{
    unsigned long long d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(pk(a)), "l"(pk(b)));
    return upk(d);
}
__device__ __forceinline__ f2 fnma2(f2 s, f2 b, f2 a) { return fma2(make_float2(-s.x, -s.y), b, a); }
#include "sweep2d_x2_body.inc"
}  // namespace pkx

}  // namespace cm
