// FP32 instantiation of the kernels (state and stencil arithmetic in FP32,
// FMA contraction allowed; the dt rule and all reductions stay FP64).
#include "kernels_impl.cuh"
#include "sweep2d_x2.cuh"
#include "sweep3d_x2.cuh"

namespace cm {

template struct Launch<float>;

template <class K>
static int blocks_per_sm2(K kernel)
{
    int b = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, kernel, kThreads2, kRingBytes) != cudaSuccess || b < 1) {
        cudaGetLastError();
        b = 1;
    }
    return b;
}

cudaError_t launch_sweep_x2(int dir, const float* in, float* out, const float* zt, const Coef<float>& C,
                            const SweepCtl& sc, int seg_rows, cudaStream_t s)
{
    SweepIO2 io;
    io.in = in;
    io.out = out;
    io.zt = zt;
    io.nstrips = (C.nx + kOutW2 - 1) / kOutW2;
    using K = void (*)(SweepIO2, Coef<float>, SweepCtl);
    // [form][kernel]: z, x, x with dt, and the stretched-grid forms; form: the
    // default, the layout-exact one, the default for an odd nx
    static const K kern[3][6] = {
        {pkf::sweep_z2d_x2<false>, pkf::sweep_x2d_x2<false>, pkf::sweep_x2d_x2_dt<false>, pkf::sweep_z2d_x2s<false>,
         pkf::sweep_x2d_x2s<false>, pkf::sweep_x2d_x2s_dt<false>},
        {pkx::sweep_z2d_x2<false>, pkx::sweep_x2d_x2<false>, pkx::sweep_x2d_x2_dt<false>, pkx::sweep_z2d_x2s<false>,
         pkx::sweep_x2d_x2s<false>, pkx::sweep_x2d_x2s_dt<false>},
        {pkf::sweep_z2d_x2<true>, pkf::sweep_x2d_x2<true>, pkf::sweep_x2d_x2_dt<true>, pkf::sweep_z2d_x2s<true>,
         pkf::sweep_x2d_x2s<true>, pkf::sweep_x2d_x2s_dt<true>}};
    static int bz = 0, bx = 0;
    if (!bz) {
        for (int v = 0; v < 3; ++v)
            for (int q = 0; q < 6; ++q)  // stretched kernels: the ring plus the warps' plane caches
                cudaFuncSetAttribute(kern[v][q], cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)kRingBytes + (q >= 3 ? 96 * 1024 : 0));
        bz = blocks_per_sm2(pkf::sweep_z2d_x2<false>);
        bx = blocks_per_sm2(pkf::sweep_x2d_x2<false>);
    }
    const K* k = kern[(C.nx & 1) ? 2 : (C.layout_exact ? 1 : 0)];
    io.seg_rows = (seg_rows > 0 && !getenv("CM_SEG_ROWS")) ? seg_rows
                                                           : pick_segment(io.nstrips, C.nz, dir == 2 ? bz : bx, kWarpsX2, sm_count());
    const int nsegs = (C.nz + io.seg_rows - 1) / io.seg_rows;
    const long long warps = (long long)io.nstrips * nsegs;
    const int blocks = (int)((warps + kWarpsX2 - 1) / kWarpsX2);
    const dim3 g(blocks), b(kThreads2);
    const size_t cache = (size_t)kWarpsX2 * plane_cap2(io.seg_rows) * sizeof(float);
    if (dir == 2)
        return C.zp ? launch_pdl(true, k[3], g, b, kRingBytes + 5 * cache, s, io, C, sc)
                    : launch_pdl(true, k[0], g, b, kRingBytes, s, io, C, sc);
    if (dir == 0) {
        // the last sweep of a step also reduces the next dt (separate kernels, so
        // that the other x sweeps carry none of that code)
        if (C.zp)
            return sc.last ? launch_pdl(true, k[5], g, b, kRingBytes + 3 * cache, s, io, C, sc)
                           : launch_pdl(true, k[4], g, b, kRingBytes + 3 * cache, s, io, C, sc);
        return sc.last ? launch_pdl(true, k[2], g, b, kRingBytes, s, io, C, sc)
                       : launch_pdl(true, k[1], g, b, kRingBytes, s, io, C, sc);
    }
    return cudaErrorInvalidValue;
}

// segment lengths the block plane caches of the stretched kernels are sized for
constexpr int kSegMax3 = 256;

template <bool ODD>
static cudaError_t sweep3_x2(int dir, const Sweep3IO<float>& io, const Coef<float>& C, const SweepCtl& sc, dim3 grid,
                             cudaStream_t s)
{
    using K = void (*)(Sweep3IO<float>, Coef<float>, SweepCtl);
    // [stretched][kernel]: L_x, L_y, L_z, L_x with dt
    static const K kern[2][4] = {
        {sweep3d_x_x2<false, ODD, false>, sweep3d_march_x2<1, false, ODD>, sweep3d_march_x2<2, false, ODD>,
         sweep3d_x_x2<false, ODD, true>},
        {sweep3d_x_x2<true, ODD, false>, sweep3d_march_x2<1, true, ODD>, sweep3d_march_x2<2, true, ODD>,
         sweep3d_x_x2<true, ODD, true>}};
    // values per plane that the stretched kernels cache after the ring
    static const int per_plane[4] = {2, 0, 4, 2};
    const int q = dir == 0 && sc.last ? 3 : dir;
    auto bytes = [&](int seg) {
        return kRing3Bytes + (C.zp ? plane_cache_bytes<float>(seg, per_plane[q]) : 0);
    };
    const K k = kern[C.zp ? 1 : 0][q];
    static bool attr[2][4] = {};
    if (!attr[C.zp ? 1 : 0][q]) {
        cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes(kSegMax3));
        attr[C.zp ? 1 : 0][q] = true;
    }
    return launch_pdl(true, k, grid, dim3(kNW3p * 32), bytes(io.seg), s, io, C, sc);
}

cudaError_t launch_sweep3_x2(int dir, const float* in, float* out, const float* zt, const Coef<float>& C,
                             const SweepCtl& sc, int seg_rows, cudaStream_t s)
{
    if (dir < 0 || dir > 2) return cudaErrorInvalidValue;
    Sweep3IO<float> io;
    io.in = in;
    io.out = out;
    io.zt = zt;
    io.nstrips = (C.nx + kOutW2 - 1) / kOutW2;
    io.nmarch = (dir == 1) ? C.ny : C.nz;
    io.nw = (dir == 1) ? C.nz : C.ny;
    const int groups = (io.nw + kNW3p - 3) / (kNW3p - 2);
    io.seg = (seg_rows > 0 && !getenv("CM_SEG_ROWS"))
                 ? seg_rows
                 : pick_segment3((long long)io.nstrips * groups, io.nmarch, 1, sm_count());
    if (C.zp && io.seg > kSegMax3) io.seg = kSegMax3;
    const int nsegs = (io.nmarch + io.seg - 1) / io.seg;
    const dim3 grid(io.nstrips, groups, nsegs);
    return (C.nx & 1) ? sweep3_x2<true>(dir, io, C, sc, grid, s) : sweep3_x2<false>(dir, io, C, sc, grid, s);
}

cudaError_t launch_sweep_batch(int dir, const BatchLaunch& L, int nblocks, bool const_coefs, bool stretched,
                               bool layout_exact, cudaStream_t s)
{
    // stretched: per-warp plane caches of 5 (z) or 3 (x) values per plane after the ring
    constexpr size_t kCacheZ = kRingBytes + (size_t)kWarpsX2 * plane_cap2(kBatchSegMax) * 5 * sizeof(float);
    constexpr size_t kCacheX = kRingBytes + (size_t)kWarpsX2 * plane_cap2(kBatchSegMax) * 3 * sizeof(float);
    using K = void (*)(BatchLaunch);
    // [layout_exact][kernel][stretched][const coefficients]; kernel: z, x, x with dt
    static const K kern[2][3][2][2] = {
        {{{pkf::sweep_z2d_batch_smem<false>, pkf::sweep_z2d_batch<false>},
          {pkf::sweep_z2d_batch_smem<true>, pkf::sweep_z2d_batch<true>}},
         {{pkf::sweep_x2d_batch_smem<false, 0>, pkf::sweep_x2d_batch<false, 0>},
          {pkf::sweep_x2d_batch_smem<true, 0>, pkf::sweep_x2d_batch<true, 0>}},
         {{pkf::sweep_x2d_batch_smem<false, 1>, pkf::sweep_x2d_batch<false, 1>},
          {pkf::sweep_x2d_batch_smem<true, 1>, pkf::sweep_x2d_batch<true, 1>}}},
        {{{pkx::sweep_z2d_batch_smem<false>, pkx::sweep_z2d_batch<false>},
          {pkx::sweep_z2d_batch_smem<true>, pkx::sweep_z2d_batch<true>}},
         {{pkx::sweep_x2d_batch_smem<false, 0>, pkx::sweep_x2d_batch<false, 0>},
          {pkx::sweep_x2d_batch_smem<true, 0>, pkx::sweep_x2d_batch<true, 0>}},
         {{pkx::sweep_x2d_batch_smem<false, 1>, pkx::sweep_x2d_batch<false, 1>},
          {pkx::sweep_x2d_batch_smem<true, 1>, pkx::sweep_x2d_batch<true, 1>}}}};
    static bool init = false;
    if (!init) {
        for (int v = 0; v < 2; ++v)
            for (int d = 0; d < 3; ++d)
                for (int st = 0; st < 2; ++st)
                    for (int cc = 0; cc < 2; ++cc)
                        cudaFuncSetAttribute(kern[v][d][st][cc], cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)(st ? (d == 0 ? kCacheZ : kCacheX) : kRingBytes));
        init = true;
    }
    if (dir != 2 && dir != 0) return cudaErrorInvalidValue;
    const int d = dir == 2 ? 0 : (L.last ? 2 : 1);
    const size_t smem = stretched ? (d == 0 ? kCacheZ : kCacheX) : kRingBytes;
    kern[layout_exact ? 1 : 0][d][stretched ? 1 : 0][const_coefs ? 1 : 0]<<<nblocks, kThreads2, smem, s>>>(L);
    return cudaGetLastError();
}

cudaError_t set_batch_coefs(const Coef<float>* C, int n, cudaStream_t s)
{
    if (n < 1 || n > kConstBoxes) return cudaErrorInvalidValue;
    return cudaMemcpyToSymbolAsync(c_box, C, n * sizeof(Coef<float>), 0, cudaMemcpyHostToDevice, s);
}

}  // namespace cm
