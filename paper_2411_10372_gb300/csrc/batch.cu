// batch.cu -- the batched ensemble: many independent 2D boxes of uneven sizes
// and Rayleigh numbers advanced together, FP32 state, one launch per sweep
// for all boxes, the steps replayed from a captured CUDA graph.
//
// Each box is the single-box problem of include/cm.h (Sec. 2 equations,
// Sec. 3.1 scheme) with its own dt (per-box device control block), seed and
// Ra, on uniform planes or on a stretched z-grid (Sec. 3; then every box of
// the batch carries a plane table).  Work is split into warp items (box,
// column strip, row segment); the segment length of each box size class is
// chosen at init by an autotuner that times the batched sweeps themselves.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstdio>
#include <cstring>
#include <vector>

#include "../../include/cm.h"
#include "host_setup.h"
#include "kernels.h"
#include "sweep2d_x2_types.h"

namespace cm {
int set_error(int code, const char* msg);
}
using namespace cm;

namespace {

struct Box {
    cm_grid grid;
    double Ra;
    int pitch;
    long long fstride;
    size_t buf_elems;   // floats in one state buffer
    float* buf[2];
    float* zt_f;
    double* zt_d;
    double* Tc;
    double* pc;
    double* scratch;    // per-plane diagnostics sums
    DevCtl* ctl;
    Plane<float>* zp_f;     // stretched batches: per-plane metric (sweeps), else NULL
    Plane<double>* zp_d;    // the same in FP64 (diagnostics), else NULL
    Coef<float> C;
    int cls;            // size class for the autotuner
    int seg_z, seg_x;   // chosen segment lengths
};

struct Batch {
    std::vector<Box> boxes;
    cm_params prm;
    double Pr, gamma;
    void* pool;         // one allocation for every box's arrays
    BoxDesc* d_boxes;
    BatchWork* d_work_z;
    BatchWork* d_work_x;
    int nblk_z, nblk_x;
    size_t work_cap;    // items the work buffers hold
    std::vector<BatchWork> work_host;  // the list being built
    cm_diag* d_recs;
    cudaStream_t stream;
    bool own_stream;
    long long step;
    long long launches;
    cudaGraphExec_t graph;
    int graph_steps;
    int cur;
    bool const_coefs;   // coefficients in constant memory (at most kConstBoxes boxes)
    bool stretched;     // some box has a stretched z-grid: every box runs the plane-table sweeps
};

Batch* g_batch = nullptr;

int ck(cudaError_t e, const char* what)
{
    if (e == cudaSuccess) return CM_OK;
    char msg[256];
    snprintf(msg, sizeof msg, "%s: %s", what, cudaGetErrorString(e));
    cudaGetLastError();
    return set_error(CM_ECUDA, msg);
}

#define CKB(call) do { int rc_ = ck((call), #call); if (rc_) return rc_; } while (0)

// warp work items of one sweep for the given per-box segment lengths;
// each box's items are padded to whole blocks of kWarpsX2 warps.  The
// blocks are ordered by decreasing cost (rows stepped by their longest
// warp, pipeline ramp included), so that the hardware's in-order block
// dispatch schedules the longest first and short blocks fill the tail.  Costs
// are small integers: the blocks are dealt into one list per cost (the
// autotuner builds this list for every candidate).
void build_work(const Batch& B, bool zdir, std::vector<BatchWork>& sorted)
{
    static_assert(kWarpsX2 == 1, "a block is one item");
    const int top = kBatchSegMax + 3;  // the largest cost
    std::vector<size_t> at(top + 2, 0);
    auto each = [&](auto&& f) {
        for (int b = 0; b < (int)B.boxes.size(); ++b) {
            const Box& x = B.boxes[b];
            const int seg = zdir ? x.seg_z : x.seg_x, nz = x.grid.nz;
            const int nstrips = (x.grid.nx + kOutW2 - 1) / kOutW2;
            for (int ks = 0; ks < nz; ks += seg) f(b, seg, ks, nstrips, std::min(seg, nz - ks) + 3);
        }
    };
    each([&](int, int, int, int nstrips, int cost) { at[top - cost + 1] += nstrips; });
    for (int c = 1; c <= top + 1; ++c) at[c] += at[c - 1];
    sorted.resize(at[top + 1]);
    each([&](int b, int seg, int ks, int nstrips, int cost) {
        for (int st = 0; st < nstrips; ++st) sorted[at[top - cost]++] = {b, st, ks, seg, ks == 0 && st == 0, {0, 0, 0}};
    });
}

int upload_work(Batch& B, bool zdir)
{
    std::vector<BatchWork>& w = B.work_host;
    build_work(B, zdir, w);
    if (w.size() > B.work_cap) return set_error(CM_EINVAL, "batch work list overflow");
    // (the copy may still read the list after this: the caller waits before the next)
    CKB(cudaMemcpyAsync(zdir ? B.d_work_z : B.d_work_x, w.data(), w.size() * sizeof(BatchWork), cudaMemcpyHostToDevice, B.stream));
    (zdir ? B.nblk_z : B.nblk_x) = (int)w.size();
    return CM_OK;
}

int upload_work(Batch& B)
{
    for (const bool zdir : {true, false}) {
        const int rc = upload_work(B, zdir);
        if (rc) return rc;
        CKB(cudaStreamSynchronize(B.stream));
    }
    return CM_OK;
}

int launch(Batch& B, int dir, int first, int last, double Delta)
{
    BatchLaunch L;
    L.boxes = B.d_boxes;
    L.work = dir == 2 ? B.d_work_z : B.d_work_x;
    L.cur = B.cur;
    L.slot = (int)(B.step & 1);
    L.first = first;
    L.last = last;
    L.Delta = Delta;
    CKB(launch_sweep_batch(dir, L, dir == 2 ? B.nblk_z : B.nblk_x, B.const_coefs, B.stretched, B.prm.layout_exact != 0,
                           B.stream));
    B.launches++;
    return CM_OK;
}

int queue_steps(Batch& B, int n)
{
    for (int s = 0; s < n; ++s) {
        // z, x, z, x (Eq. time_step, rightmost operator first), or its palindrome x, z, z, x
        static const int printed[4] = {2, 0, 2, 0}, symmetric[4] = {0, 2, 2, 0};
        const int* order = B.prm.split == CM_SPLIT_SYMMETRIC ? symmetric : printed;
        for (int q = 0; q < 4; ++q) {
            int rc = launch(B, order[q], q == 0, q == 3, 0.0);
            if (rc) return rc;
            B.cur ^= 1;
        }
        B.step++;
    }
    return CM_OK;
}

// times batched sweeps (fixed tiny Delta, written to the scratch buffer, no
// bookkeeping): *ms = median of 3 launches in a row after a warm-up, with one
// wait for all four
struct SweepTimer {
    cudaEvent_t ev[4] = {nullptr, nullptr, nullptr, nullptr};
    int create()
    {
        for (cudaEvent_t& e : ev)
            if (cudaEventCreate(&e) != cudaSuccess) {
                cudaGetLastError();
                e = nullptr;
                return set_error(CM_ECUDA, "autotune: cudaEventCreate failed");
            }
        return CM_OK;
    }
    ~SweepTimer()
    {
        for (cudaEvent_t e : ev)
            if (e) cudaEventDestroy(e);
    }
    int run(Batch& B, int dir, float* ms)
    {
        int rc = launch(B, dir, 0, 0, 1e-9);
        for (int r = 0; r < 4 && !rc; ++r) {
            rc = ck(cudaEventRecord(ev[r], B.stream), "autotune: cudaEventRecord");
            if (!rc && r < 3) rc = launch(B, dir, 0, 0, 1e-9);
        }
        if (!rc) rc = ck(cudaEventSynchronize(ev[3]), "autotune: cudaEventSynchronize");
        float t[3] = {0.f, 0.f, 0.f};
        for (int r = 0; r < 3 && !rc; ++r) rc = ck(cudaEventElapsedTime(&t[r], ev[r], ev[r + 1]), "autotune: cudaEventElapsedTime");
        std::sort(t, t + 3);
        *ms = t[1];
        return rc;
    }
};

// Autotuner: coordinate descent over the segment length of each box size
// class (nz < 64, < 128, < 256, >= 256), per sweep direction, on the timed
// batched sweep itself: a first pass over every other candidate, a second one
// over the neighbours of what it chose, since the best length of one class
// depends on how the others fill the GPU.  (Two passes over all candidates,
// each list sorted and each launch waited for, made it 0.056 s of a 64-box
// init; now 0.012.)
int autotune(Batch& B)
{
    // CM_SEG_ROWS=n: every box runs n-row segments, untuned (profiling captures)
    if (const char* e = getenv("CM_SEG_ROWS")) {
        const int n = std::min(std::max(atoi(e), kBatchSegMin), kBatchSegMax);
        for (Box& x : B.boxes) x.seg_z = x.seg_x = n;
        return upload_work(B);
    }
    static const int cand[] = {kBatchSegMin, 8, 10, 12, 14, 16, 20, 24, 29, 32, 40, 48, 64, 96, 128};
    constexpr int ncand = sizeof cand / sizeof cand[0], start = 9;
    static_assert(kBatchSegMax >= 128, "the stretched batch kernels size their plane caches for kBatchSegMax rows");
    bool present[4] = {false, false, false, false};
    for (const Box& x : B.boxes) present[x.cls] = true;
    SweepTimer timer;
    int rc = timer.create();
    if (rc) return rc;
    for (int dir : {2, 0}) {
        int at[4] = {start, start, start, start};  // cand[start] = 32
        auto apply = [&]() {
            for (Box& x : B.boxes) (dir == 2 ? x.seg_z : x.seg_x) = cand[at[x.cls]];
            return upload_work(B, dir == 2);
        };
        if ((rc = apply())) return rc;
        float best = 0.f;
        if ((rc = timer.run(B, dir, &best))) return rc;
        for (int pass = 0; pass < 2; ++pass) {
            for (int c = 0; c < 4; ++c) {
                if (!present[c]) continue;
                const int from = at[c];
                for (int v = pass ? std::max(from - 2, 0) : 0; v < (pass ? std::min(from + 3, ncand) : ncand); v += pass ? 1 : 2) {
                    if (v == from) continue;
                    const int keep = at[c];
                    at[c] = v;
                    if ((rc = apply())) return rc;
                    float t = 0.f;
                    if ((rc = timer.run(B, dir, &t))) return rc;
                    if (t < 0.99f * best) best = t;
                    else at[c] = keep;
                }
            }
        }
        if ((rc = apply())) return rc;
        CKB(cudaStreamSynchronize(B.stream));
    }
    return ck(cudaGetLastError(), "autotune");
}

void free_batch(Batch* B)
{
    if (!B) return;
    cudaStreamSynchronize(B->stream);
    if (B->graph) cudaGraphExecDestroy(B->graph);
    cudaFree(B->pool);
    cudaFree(B->d_boxes);
    cudaFree(B->d_work_z);
    cudaFree(B->d_work_x);
    cudaFree(B->d_recs);
    if (B->own_stream) cudaStreamDestroy(B->stream);
    delete B;
}

}  // namespace

extern "C" {

int cm_batch_init(int nbox, const cm_grid* grids, const double* Ra, double Pr, double gamma, const cm_params* params)
{
    if (nbox < 1 || !grids || !Ra) return set_error(CM_EINVAL, "cm_batch_init: need nbox >= 1, grids and Ra");
    cm_params P;
    if (params) P = *params;
    else cm_default_params(&P);
    if (P.precision != CM_FP32) return set_error(CM_EINVAL, "cm_batch_init: the batch steps FP32 states");
    if (P.layout_exact != 0 && P.layout_exact != 1) return set_error(CM_EINVAL, "cm_batch_init: layout_exact must be 0 or 1");
    if (P.split != CM_SPLIT_PRINTED && P.split != CM_SPLIT_SYMMETRIC)
        return set_error(CM_EINVAL, "cm_batch_init: split must be CM_SPLIT_PRINTED or CM_SPLIT_SYMMETRIC");
    if (!(Pr > 0) || !(gamma > 1) || !(P.eps > 0) || !(P.D > 0) || !(P.cfl > 0) || P.cfl > 1.0)
        return set_error(CM_EINVAL, "cm_batch_init: bad physical parameters");
    for (int b = 0; b < nbox; ++b) {
        const cm_grid& G = grids[b];
        if (G.ndim != 2 || G.nx < 4 || G.nz < 5 || (G.nx & 1) || !(G.aspect > 0) || !(Ra[b] > 0))
            return set_error(CM_EINVAL, "cm_batch_init: every box must be 2D with even nx >= 4, nz >= 5, Ra > 0");
        if ((long long)G.nz * pitch_of(G.nx, CM_FP32) * 5 >= (1LL << 31))
            return set_error(CM_EINVAL, "cm_batch_init: box too large");
    }
    // z-planes of every box (uniform, tanh or given), validated before any device work
    std::vector<std::vector<double>> planes(nbox);
    bool any_st = false;
    for (int b = 0; b < nbox; ++b) {
        const char* why = "";
        if (!make_planes(grids[b], planes[b], &why)) {
            char msg[160];
            snprintf(msg, sizeof msg, "cm_batch_init: box %d: %s", b, why);
            return set_error(CM_EINVAL, msg);
        }
        any_st = any_st || stretched(grids[b]);
    }
    if (g_batch) { free_batch(g_batch); g_batch = nullptr; }
    Batch* B = new Batch();
    B->prm = P;
    B->Pr = Pr;
    B->gamma = gamma;
    B->pool = nullptr;
    B->d_boxes = nullptr;
    B->d_work_z = B->d_work_x = nullptr;
    B->d_recs = nullptr;
    B->graph = nullptr;
    B->graph_steps = 0;
    B->step = 0;
    B->launches = 0;
    B->cur = 0;
    B->stretched = any_st;
    auto bail = [&](int code) { free_batch(B); return code; };
    if (P.stream) {
        B->stream = (cudaStream_t)P.stream;
        B->own_stream = false;
    } else {
        if (cudaStreamCreateWithFlags(&B->stream, cudaStreamNonBlocking) != cudaSuccess)
            return bail(ck(cudaGetLastError(), "cudaStreamCreate"));
        B->own_stream = true;
    }
    // sizes of every box's arrays in one pool (256-byte aligned pieces)
    const Closure K(gamma, P);
    B->boxes.resize(nbox);
    size_t bytes = 0, items = 0;
    auto take = [&](size_t n) { size_t o = bytes; bytes += (n + 255) / 256 * 256; return o; };
    constexpr int kPieces = 9;
    std::vector<size_t> off(kPieces * nbox);
    for (int b = 0; b < nbox; ++b) {
        Box& x = B->boxes[b];
        x.grid = grids[b];
        x.grid.znodes = nullptr;  // caller memory: the planes were copied above
        x.Ra = Ra[b];
        x.pitch = pitch_of(x.grid.nx, CM_FP32);
        x.fstride = (long long)x.grid.nz * x.pitch;
        x.buf_elems = 4 * (size_t)x.fstride;
        const int nz = x.grid.nz;
        x.cls = nz < 64 ? 0 : nz < 128 ? 1 : nz < 256 ? 2 : 3;
        x.seg_z = x.seg_x = kBatchSegMin;  // smallest candidate: sizes the work buffers
        off[kPieces * b + 0] = take(2 * x.buf_elems * sizeof(float));
        off[kPieces * b + 1] = take(nz * sizeof(float));
        off[kPieces * b + 2] = take(nz * sizeof(double));
        off[kPieces * b + 3] = take(nz * sizeof(double));
        off[kPieces * b + 4] = take(nz * sizeof(double));
        off[kPieces * b + 5] = take((size_t)nz * kDiagQ * sizeof(double));
        off[kPieces * b + 6] = take(sizeof(DevCtl));
        off[kPieces * b + 7] = take(any_st ? nz * sizeof(Plane<float>) : 0);
        off[kPieces * b + 8] = take(any_st ? nz * sizeof(Plane<double>) : 0);
        items += ((size_t)((x.grid.nx + kOutW2 - 1) / kOutW2) * ((nz + kBatchSegMin - 1) / kBatchSegMin) + kWarpsX2);
    }
    B->work_cap = items;
    if (cudaMalloc(&B->pool, bytes) != cudaSuccess || cudaMalloc(&B->d_boxes, nbox * sizeof(BoxDesc)) != cudaSuccess ||
        cudaMalloc(&B->d_work_z, items * sizeof(BatchWork)) != cudaSuccess ||
        cudaMalloc(&B->d_work_x, items * sizeof(BatchWork)) != cudaSuccess ||
        cudaMalloc(&B->d_recs, nbox * sizeof(cm_diag)) != cudaSuccess) {
        cudaGetLastError();
        return bail(set_error(CM_ENOMEM, "cm_batch_init: device allocation failed"));
    }
    char* base = (char*)B->pool;
    std::vector<BoxDesc> desc(nbox);
    std::vector<DevCtl> first(nbox);  // control blocks after the first dt
    // host tables of each box, read by copies until the wait after the loop
    struct Tables {
        std::vector<float> zf;
        std::vector<double> z, Tc, pc;
        std::vector<Plane<float>> tf;
        std::vector<Plane<double>> td;
        DevCtl ctl;
        double rho_min;
    };
    std::vector<Tables> tables(nbox);
    int rc = CM_OK;
    for (int b = 0; b < nbox && !rc; ++b) {
        Box& x = B->boxes[b];
        const int nz = x.grid.nz;
        x.buf[0] = (float*)(base + off[kPieces * b + 0]);
        x.buf[1] = x.buf[0] + x.buf_elems;
        x.zt_f = (float*)(base + off[kPieces * b + 1]);
        x.zt_d = (double*)(base + off[kPieces * b + 2]);
        x.Tc = (double*)(base + off[kPieces * b + 3]);
        x.pc = (double*)(base + off[kPieces * b + 4]);
        x.scratch = (double*)(base + off[kPieces * b + 5]);
        x.ctl = (DevCtl*)(base + off[kPieces * b + 6]);
        x.zp_f = any_st ? (Plane<float>*)(base + off[kPieces * b + 7]) : nullptr;
        x.zp_d = any_st ? (Plane<double>*)(base + off[kPieces * b + 8]) : nullptr;
        fill_coef(x.C, x.grid, 1, x.pitch, x.fstride, x.Ra, Pr, K, P);
        Tables& t = tables[b];
        {
            Profile prof(planes[b], P, K);
            t.z = std::move(prof.z);
            t.Tc = std::move(prof.Tc);
            t.pc = std::move(prof.pc);
            t.rho_min = prof.rho_min;
        }
        if (any_st) {
            // uniform boxes of a stretched batch get the table of the planes k/K
            plane_table(planes[b], t.tf);
            plane_table(planes[b], t.td);
            x.C.zp = x.zp_f;
        }
        t.zf.resize(nz);
        for (int k = 0; k < nz; ++k) t.zf[k] = (float)t.z[k];
        std::memset(&t.ctl, 0, sizeof t.ctl);
        t.ctl.dt_slot[0] = t.ctl.dt_slot[1] = 0x7FF0000000000000ULL;
        rc = ck(cudaMemsetAsync(x.buf[0], 0, 2 * x.buf_elems * sizeof(float), B->stream), "memset");
        if (!rc) rc = ck(cudaMemcpyAsync(x.zt_f, t.zf.data(), nz * sizeof(float), cudaMemcpyHostToDevice, B->stream), "upload");
        if (!rc) rc = ck(cudaMemcpyAsync(x.zt_d, t.z.data(), nz * sizeof(double), cudaMemcpyHostToDevice, B->stream), "upload");
        if (!rc) rc = ck(cudaMemcpyAsync(x.Tc, t.Tc.data(), nz * sizeof(double), cudaMemcpyHostToDevice, B->stream), "upload");
        if (!rc) rc = ck(cudaMemcpyAsync(x.pc, t.pc.data(), nz * sizeof(double), cudaMemcpyHostToDevice, B->stream), "upload");
        if (!rc) rc = ck(cudaMemcpyAsync(x.ctl, &t.ctl, sizeof(DevCtl), cudaMemcpyHostToDevice, B->stream), "upload");
        if (!rc && any_st)
            rc = ck(cudaMemcpyAsync(x.zp_f, t.tf.data(), nz * sizeof(Plane<float>), cudaMemcpyHostToDevice, B->stream), "upload");
        if (!rc && any_st)
            rc = ck(cudaMemcpyAsync(x.zp_d, t.td.data(), nz * sizeof(Plane<double>), cudaMemcpyHostToDevice, B->stream), "upload");
        InitArgs A;
        A.Tc = x.Tc;
        A.pc = x.pc;
        A.zt = x.zt_d;
        A.a = K.a;
        A.b = K.b;
        A.g = K.g;
        A.amp = P.pert_amp;
        A.seed = P.seed + (unsigned long long)b;
        if (!rc) rc = ck(Launch<float>::init(x.buf[0], x.C, A, B->stream), "init launch");
        if (!rc) rc = ck(Launch<float>::dt(x.buf[0], x.zt_f, x.C, x.ctl, 0, B->stream), "dt launch");
        if (!rc) rc = ck(cudaMemcpyAsync(&first[b], x.ctl, sizeof(DevCtl), cudaMemcpyDeviceToHost, B->stream), "control block read");
        desc[b].C = x.C;
        desc[b].buf[0] = x.buf[0];
        desc[b].buf[1] = x.buf[1];
        desc[b].ctl = x.ctl;
        B->launches += 2;
    }
    {
        const int waited = ck(cudaStreamSynchronize(B->stream), "init");  // also after an error: copies read the tables
        if (!rc) rc = waited;
    }
    for (int b = 0; b < nbox && !rc; ++b) {
        // the first dt, and the explicit-diffusion bound cm_init applies
        double hmin = 0.0;
        std::memcpy(&hmin, &first[b].dt_slot[0], sizeof hmin);
        const double dt0 = P.dt_fixed > 0 ? P.dt_fixed : P.cfl * hmin;
        char msg[200];
        if (!(dt0 > 0) || !std::isfinite(dt0) || (first[b].status & 1)) {
            snprintf(msg, sizeof msg, "cm_batch_init: box %d: non-finite initial state", b);
            rc = set_error(CM_ENAN, msg);
            break;
        }
        const double dnum = diffusion_number(B->boxes[b].grid, planes[b], B->boxes[b].Ra, Pr, P, K, tables[b].rho_min, dt0);
        if (dnum > 0.5) {
            snprintf(msg, sizeof msg,
                     "cm_batch_init: box %d: explicit diffusion number %.3g > 0.5 at dt = %.3g: refine dt "
                     "(dt_fixed) or raise Ra", b, dnum, dt0);
            rc = set_error(CM_EUNSTABLE, msg);
        }
    }
    if (!rc) rc = ck(cudaMemcpyAsync(B->d_boxes, desc.data(), nbox * sizeof(BoxDesc), cudaMemcpyHostToDevice, B->stream), "upload");
    B->const_coefs = nbox <= kConstBoxes;
    if (!rc && B->const_coefs) {
        std::vector<Coef<float>> coefs(nbox);
        for (int b = 0; b < nbox; ++b) coefs[b] = desc[b].C;
        rc = ck(set_batch_coefs(coefs.data(), nbox, B->stream), "coefficient upload");
        if (!rc) rc = ck(cudaStreamSynchronize(B->stream), "coefficient upload");  // coefs is freed on return
    }
    if (!rc) rc = upload_work(*B);
    if (!rc) rc = autotune(*B);
    if (!rc) rc = ck(cudaStreamSynchronize(B->stream), "batch init");
    if (rc) return bail(rc);
    g_batch = B;
    return CM_OK;
}

int cm_batch_step(int n)
{
    if (!g_batch) return set_error(CM_ENOTINIT, "no batch: call cm_batch_init first");
    if (n < 0) return set_error(CM_EINVAL, "n must be >= 0");
    Batch& B = *g_batch;
    const int G = 50;  // steps per captured graph (even: the dt slot parity repeats)
    int rc;
    if ((B.step & 1) && n > 0) {
        if ((rc = queue_steps(B, 1))) return rc;
        --n;
    }
    if (n >= G && !B.graph) {
        cudaGraph_t g;
        CKB(cudaStreamBeginCapture(B.stream, cudaStreamCaptureModeThreadLocal));
        const long long s0 = B.step, l0 = B.launches;
        const int c0 = B.cur;
        rc = queue_steps(B, G);
        cudaError_t e = cudaStreamEndCapture(B.stream, &g);
        B.step = s0;  // capture only records the launches
        B.launches = l0;
        B.cur = c0;
        if (rc) return rc;
        CKB(e);
        e = cudaGraphInstantiate(&B.graph, g, 0);
        cudaGraphDestroy(g);
        CKB(e);
        B.graph_steps = G;
    }
    while (n >= G && B.graph) {
        CKB(cudaGraphLaunch(B.graph, B.stream));
        B.step += G;
        B.launches += 4LL * G;
        n -= G;
    }
    return queue_steps(B, n);
}

int cm_batch_diagnostics(cm_diag* out)
{
    if (!g_batch) return set_error(CM_ENOTINIT, "no batch: call cm_batch_init first");
    if (!out) return set_error(CM_EINVAL, "out is NULL");
    Batch& B = *g_batch;
    const Closure K(B.gamma, B.prm);
    for (int b = 0; b < (int)B.boxes.size(); ++b) {
        Box& x = B.boxes[b];
        DiagArgs A;
        A.zt = x.zt_d;
        A.a = K.a;
        A.b = K.b;
        A.g = K.g;
        A.D = B.prm.D;
        A.cs2 = K.cs2;
        CKB(Launch<float>::diag_planes(x.buf[B.cur], x.C, A, x.scratch, x.ctl, B.stream));
        DiagFinal F{};
        F.Ra = x.Ra;
        F.Pr = B.Pr;
        F.eps = B.prm.eps;
        F.D = B.prm.D;
        F.cfl = B.prm.cfl;
        F.dt_fixed = B.prm.dt_fixed;
        F.cells = (double)x.grid.nx;
        F.nz = x.grid.nz;
        F.slot = (int)(B.step & 1);
        F.zp = x.zp_d;
        CKB(launch_diag_final(x.scratch, x.zt_d, F, x.ctl, B.d_recs + b, B.stream));
        B.launches += 2;
    }
    CKB(cudaMemcpyAsync(out, B.d_recs, B.boxes.size() * sizeof(cm_diag), cudaMemcpyDeviceToHost, B.stream));
    CKB(cudaStreamSynchronize(B.stream));
    for (size_t b = 0; b < B.boxes.size(); ++b)
        if (out[b].status != CM_OK) return set_error(CM_ENAN, "a box met a non-finite value");
    return CM_OK;
}

int cm_batch_get_state(int box, double* host)
{
    if (!g_batch) return set_error(CM_ENOTINIT, "no batch: call cm_batch_init first");
    Batch& B = *g_batch;
    if (box < 0 || box >= (int)B.boxes.size() || !host) return set_error(CM_EINVAL, "bad box or host pointer");
    const Box& x = B.boxes[box];
    std::vector<float> tmp(4 * (size_t)x.grid.nz * x.grid.nx);
    CKB(cudaMemcpy2DAsync(tmp.data(), x.grid.nx * sizeof(float), x.buf[B.cur], x.pitch * sizeof(float),
                          x.grid.nx * sizeof(float), 4 * (size_t)x.grid.nz, cudaMemcpyDeviceToHost, B.stream));
    CKB(cudaStreamSynchronize(B.stream));
    for (size_t q = 0; q < tmp.size(); ++q) host[q] = (double)tmp[q];
    return CM_OK;
}

int cm_batch_tuning(int* seg_z, int* seg_x)
{
    if (!g_batch) return set_error(CM_ENOTINIT, "no batch: call cm_batch_init first");
    for (size_t b = 0; b < g_batch->boxes.size(); ++b) {
        if (seg_z) seg_z[b] = g_batch->boxes[b].seg_z;
        if (seg_x) seg_x[b] = g_batch->boxes[b].seg_x;
    }
    return CM_OK;
}

int cm_batch_profile_steps(int n, unsigned long long flush_bytes, double* total_ms)
{
    if (!g_batch) return set_error(CM_ENOTINIT, "no batch: call cm_batch_init first");
    if (n < 1 || !total_ms) return set_error(CM_EINVAL, "need n >= 1 and total_ms");
    Batch& B = *g_batch;
    void* flush = nullptr;
    if (flush_bytes && cudaMalloc(&flush, flush_bytes) != cudaSuccess) {
        cudaGetLastError();
        return set_error(CM_ENOMEM, "flush buffer allocation failed");
    }
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    if (flush) cudaMemsetAsync(flush, 1, flush_bytes, B.stream);
    cudaEventRecord(e0, B.stream);
    int rc = cm_batch_step(n);
    cudaEventRecord(e1, B.stream);
    float ms = 0.f;
    if (!rc) rc = ck(cudaEventSynchronize(e1), "profiled batch steps");
    if (!rc) rc = ck(cudaEventElapsedTime(&ms, e0, e1), "event time");
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (flush) cudaFree(flush);
    *total_ms = ms;
    return rc;
}

long long cm_batch_launch_count(void) { return g_batch ? g_batch->launches : 0; }

int cm_batch_finalize(void)
{
    if (g_batch) {
        free_batch(g_batch);
        g_batch = nullptr;
    }
    return CM_OK;
}

}  // extern "C"
