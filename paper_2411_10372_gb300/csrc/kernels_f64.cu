// FP64 instantiation of the kernels.  Compiled with --fmad=false so that each
// FP64 operation rounds exactly as written (the FP64 path is the one checked
// against the CPU oracle at 1e-12).
#define CM_DEFINE_DIAG_FINAL
#include "kernels_impl.cuh"
#include "staged_f64.cuh"

namespace cm {

template struct Launch<double>;

// Chunks of about a million nodes (1.4e8 to 1.8e8 bytes): two thousand blocks
// a launch keep every SM busy to the end, and the chunk's intermediates are
// still mostly in L2 when the next stage reads them.  At least 16 planes, so
// that the planes recomputed around a chunk stay few.
long long staged_values(int nx, int ny, int nz, int ndim)
{
    const long long plane = (long long)nx * (ndim == 3 ? ny : 1);
    const long long rows = std::min<long long>(nz, std::max<long long>(16, ((1LL << 20) + plane - 1) / plane) + 4);
    return kStHead + (ndim == 3 ? StArrays<3>::kCount : StArrays<2>::kCount) * plane * rows;
}

bool staged_fits(const Coef<double>& C)
{
    if (!C.work) return false;
    const long long plane = (long long)C.nx * (C.ndim == 3 ? C.ny : 1);
    const int chunk = C.ndim == 3 ? st_chunk<3>(C) : st_chunk<2>(C);
    return chunk > 0 && plane * (chunk + 4) < (1LL << 31);
}

int sweep_launches(const Coef<double>& C)
{
    if (!staged_fits(C)) return 1;
    const int chunk = C.ndim == 3 ? st_chunk<3>(C) : st_chunk<2>(C);
    return 5 * ((C.nz + chunk - 1) / chunk);
}

template <int ND, int AL>
static cudaError_t staged_dir(const double* in, double* out, const double* zt, const Coef<double>& C, const SweepCtl& sc,
                              cudaStream_t s)
{
    return C.zp ? st_sweep<ND, AL, true>(in, out, zt, C, sc, s) : st_sweep<ND, AL, false>(in, out, zt, C, sc, s);
}

cudaError_t launch_sweep_staged(int dir, const double* in, double* out, const double* zt, const Coef<double>& C,
                                const SweepCtl& sc, cudaStream_t s)
{
    if (C.ndim == 3) {
        if (dir == 2) return staged_dir<3, 2>(in, out, zt, C, sc, s);
        if (dir == 1) return staged_dir<3, 1>(in, out, zt, C, sc, s);
        if (dir == 0) return staged_dir<3, 0>(in, out, zt, C, sc, s);
    } else {
        if (dir == 2) return staged_dir<2, 2>(in, out, zt, C, sc, s);
        if (dir == 0) return staged_dir<2, 0>(in, out, zt, C, sc, s);
    }
    return cudaErrorInvalidValue;
}

bool pdl_enabled()
{
    static int on = -1;
    if (on < 0) {
        const char* e = getenv("CM_PDL");
        on = (e && e[0] == '0') ? 0 : 1;
    }
    return on == 1;
}

cudaError_t launch_diag_final(const double* scratch, const double* zt, const DiagFinal& F, DevCtl* ctl, cm_diag* rec,
                              cudaStream_t s)
{
    diag_final<<<1, kDiagThreads, 0, s>>>(scratch, zt, F, ctl, rec);
    return cudaGetLastError();
}

}  // namespace cm
