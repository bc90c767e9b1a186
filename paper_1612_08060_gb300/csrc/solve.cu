// solve.cu -- deterministic FP64 dot products, CG and CG with iterative
// refinement on top of the node-aware apply.
//
// Precision scheme: the matrix used inside the inner CG is the FP32 copy of
// A's values (FP32 products, FP64 sums); every vector, dot product and the
// outer residual r = b - A x stay FP64, the outer residual using the FP64
// values.  Each dot product sums over a fixed partition in a fixed order, so
// its value does not depend on scheduling.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <utility>

#include "internal.h"

namespace nap {
namespace {

constexpr int kDotBlocks = 1024;  // fixed grid: the partition of every dot product
constexpr int kThreads = 256;

struct Scal {
    double rr[2];  // r.r before the next iteration, by the parity of its number
    double bb, rnorm0;
    int err, pad;  // the workspace's error flag, as the last CG iteration saw it
};

// Sum of 256 values, one per thread of a group of 8 warps (group g of its CTA), in
// a fixed tree: lanes 16, 8, 4, 2, 1 apart within each warp, then the 8 warps' sums
// 4, 2, 1 apart; valid in the group's first warp.  GB300 issues an FP64 addition per
// warp every 84 cycles or so on a quarter of an SM, whatever its lanes hold, so the
// 248 additions of the tree are packed into full warps through shared memory: 13
// instructions, where a shuffle tree in every warp takes 45.  A CG iteration on 63^3
// fell from 36.7 to 31.8 us, a served one of 1.7M elements from 73 to 70.
constexpr int kSumDoubles = 256 + 128 + 64;  // shared memory of a group
__device__ __forceinline__ double group_sum(double v, double *sh, int g)
{
    double *a = sh + kSumDoubles * g, *b = a + 256, *c = b + 128;
    const int t = threadIdx.x % kThreads;
    a[t] = v;
    __syncthreads();
    if (t < 128) b[t] = a[32 * (t >> 4) + (t & 15)] + a[32 * (t >> 4) + (t & 15) + 16];
    __syncthreads();
    if (t < 64) c[t] = b[16 * (t >> 3) + (t & 7)] + b[16 * (t >> 3) + (t & 7) + 8];
    __syncthreads();
    if (t < 32) {
        v = c[8 * (t >> 2) + (t & 3)] + c[8 * (t >> 2) + (t & 3) + 4];
        v += __shfl_xor_sync(0xffffffffu, v, 2);
        v += __shfl_xor_sync(0xffffffffu, v, 1);
        v += 0.0;  // a sum of -0.0 counts as 0.0
        v += __shfl_xor_sync(0xffffffffu, v, 16);  // warps 4, 2, 1 apart
        v += __shfl_xor_sync(0xffffffffu, v, 8);
        v += __shfl_xor_sync(0xffffffffu, v, 4);
    }
    __syncthreads();
    return v;
}

// FP64 dot products over a fixed partition: partial b, of 1,024, sums the indices
// i = b*256 + t + q*1024*256 over the 256 threads t of a group, and the partials
// are added in a fixed order.  A CTA is four groups; partials past the vector's
// end are 0 and not launched.
constexpr int kDotGroups = 4;
// All threads of a CTA: f of the sum of the first nb partials (the others are 0),
// f taken by one thread: an FP64 division by every warp costs more than the sum.
template <class F>
__device__ __forceinline__ double sum_partials(const double *partial, int nb, double *sh, F f)
{
    __shared__ double total;
    const int g = threadIdx.x / kThreads, t = threadIdx.x % kThreads;
    double v = 0.0;
    if (g == 0)
        for (int q = t; q < kDotBlocks; q += kThreads) v += q < nb ? __ldcg(partial + q) : 0.0;
    v = group_sum(v, sh, g);
    if (threadIdx.x == 0) total = f(v);
    __syncthreads();
    return total;
}

// *result = x.y: the last CTA to finish adds the partials and resets the ticket.
__global__ void __launch_bounds__(kThreads *kDotGroups)
    k_dot(const double *x, const double *y, int64_t n, double *partial, unsigned *ticket,
          double *result)
{
    __shared__ double sh[kSumDoubles * kDotGroups];
    __shared__ bool last;
    griddep_wait();
    const int g = threadIdx.x / kThreads, t = threadIdx.x % kThreads;
    const int b = blockIdx.x * kDotGroups + g;
    double s = 0.0;
    for (int64_t i = (int64_t)b * kThreads + t; i < n; i += (int64_t)kDotBlocks * kThreads)
        s = fma(x[i], y[i], s);
    s = group_sum(s, sh, g);
    if (t == 0) partial[b] = s;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    __syncthreads();
    griddep_done();
    if (!last) return;
    __threadfence();
    const double v = sum_partials(partial, gridDim.x * kDotGroups, sh, [](double a) { return a; });
    if (threadIdx.x == 0) {
        *ticket = 0;
        *result = v;
    }
}

// A CG iteration after q = A p is three kernels, each CTA of the second and third
// adding the partials of the one before for itself (8 KB from L2), so that no sum
// and no scalar has a launch, a ticket or a last CTA of its own:
//   k_pq        partials of p.q
//   k_update    alpha = rr / p.q; x += alpha p, r -= alpha q, partials of r.r
//   k_next_p    beta = r.r / rr; p' = r + beta p into the other vector, and the
//               inter-node messages of p' (each sender's element is formed again
//               from p and r, the same operation), so that q = A p' is the windowed
//               SpMV alone
// Latency-bound at the sizes of a served solve.  Per iteration on 63^3 with FP32
// values (GB300): 31.8 us in four launches; 39 in five, the last CTA of a dot
// product summing and the messages in their own launch (with shuffle trees, 36.7
// against 39); 55 in ten.
struct CgIter {
    double *x, *r, *p, *p2, *q;
    int64_t n;
    double *pq, *rr;  // partials
    int nb;           // of them
    Scal *sc;
    int parity;
};
__global__ void __launch_bounds__(kThreads *kDotGroups) k_pq(const CgIter I)
{
    __shared__ double sh[kSumDoubles * kDotGroups];
    griddep_wait();
    const int g = threadIdx.x / kThreads, b = blockIdx.x * kDotGroups + g;
    double s = 0.0;
    for (int64_t i = (int64_t)b * kThreads + threadIdx.x % kThreads; i < I.n;
         i += (int64_t)kDotBlocks * kThreads)
        s = fma(I.p[i], I.q[i], s);
    s = group_sum(s, sh, g);
    if (threadIdx.x % kThreads == 0) I.pq[b] = s;
    griddep_done();
}
__global__ void __launch_bounds__(kThreads *kDotGroups) k_update(const CgIter I)
{
    __shared__ double sh[kSumDoubles * kDotGroups];
    griddep_wait();
    const double a = sum_partials(I.pq, I.nb, sh, [&](double pq) { return I.sc->rr[I.parity] / pq; });
    const int g = threadIdx.x / kThreads, b = blockIdx.x * kDotGroups + g;
    double s = 0.0;
    for (int64_t i = (int64_t)b * kThreads + threadIdx.x % kThreads; i < I.n;
         i += (int64_t)kDotBlocks * kThreads) {
        I.x[i] = fma(a, I.p[i], I.x[i]);
        const double r = fma(-a, I.q[i], I.r[i]);
        I.r[i] = r;
        s = fma(r, r, s);
    }
    s = group_sum(s, sh, g);
    if (threadIdx.x % kThreads == 0) I.rr[b] = s;
    griddep_done();
}
// The inter-node messages of r + beta p, by block `block` of `blocks` (see k_send).
template <class T>
__device__ __forceinline__ void send_next(const SendList &L, const double *p, const double *r,
                                          double beta, int block, int blocks)
{
    if (*(volatile const int *)L.err) return;
    const int lane = threadIdx.x & 31, warps = blockDim.x / 32;
    for (int g = block * warps + (threadIdx.x >> 5); g * kSendGroup < L.n; g += blocks * warps) {
        const int32_t shift = __ldg(L.shift + g);
#pragma unroll
        for (int u = 0; u < kSendGroup / 32; u++) {
            const int k = g * kSendGroup + 32 * u + lane;
            if (k >= L.n) continue;
            const int32_t j = __ldg(L.j + k), to = shift == kMixed ? __ldg(L.dst + k) : k + shift;
            const double v = fma(beta, p[j], r[j]);
            if constexpr (sizeof(T) == 4) static_cast<T *>(L.grecv)[to] = __double2float_rn(v);
            else static_cast<T *>(L.grecv)[to] = v;
        }
    }
}
// The first vec_blocks CTAs form p', the others send it (none where the product
// brings its own messages).
template <class T>
__global__ void __launch_bounds__(kThreads *kDotGroups)
    k_next_p(const CgIter I, const SendList L, int vec_blocks)
{
    __shared__ double sh[kSumDoubles * kDotGroups];
    griddep_wait();
    const double beta = sum_partials(I.rr, I.nb, sh, [&](double rr) {
        if (blockIdx.x == 0) {
            I.sc->rr[I.parity ^ 1] = rr;
            I.sc->err = *(volatile const int *)L.err;
        }
        return rr / I.sc->rr[I.parity];
    });
    if ((int)blockIdx.x < vec_blocks) {
        for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < I.n;
             i += (int64_t)vec_blocks * blockDim.x)
            I.p2[i] = fma(beta, I.p[i], I.r[i]);
    } else {
        send_next<T>(L, I.p, I.r, beta, (int)blockIdx.x - vec_blocks, (int)gridDim.x - vec_blocks);
    }
    griddep_done();
}
// Launch as a programmatic dependent of the stream's last kernel.
template <typename... KArgs, typename... Args>
int launch_dependent(void (*kern)(KArgs...), dim3 grid, int threads, cudaStream_t s, Args &&...args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)threads);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    NAP_CUDA(cudaLaunchKernelEx(&cfg, kern, std::forward<Args>(args)...));
    count_launch(1);
    return NAPSPMV_OK;
}
// r = b - q ; p = r
__global__ void k_resid(double *r, double *p, const double *b, const double *q, int64_t n)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const double v = b[i] - q[i];
        r[i] = v;
        if (p) p[i] = v;
    }
}
// x += d
__global__ void k_add(double *x, const double *d, int64_t n)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        x[i] += d[i];
}

struct DotScratch {
    double *partial = nullptr;
    unsigned *ticket = nullptr;
};

dim3 dot_grid(int64_t n)
{
    const int64_t per = kThreads * kDotGroups;
    return dim3((unsigned)std::max<int64_t>(1, std::min<int64_t>((n + per - 1) / per,
                                                                 kDotBlocks / kDotGroups)));
}
int dot_launch(const double *x, const double *y, int64_t n, double *result, DotScratch &ds,
               cudaStream_t s)
{
    return launch_dependent(k_dot, dot_grid(n), kThreads * kDotGroups, s, x, y, n, ds.partial, ds.ticket,
                            result);
}

struct CgBuffers {
    double *r = nullptr, *p = nullptr, *p2 = nullptr, *q = nullptr, *d = nullptr;
    Scal *sc = nullptr;
    DotScratch ds;
    cudaStream_t s = 0;
    ~CgBuffers()
    {
        void *ptrs[] = {r, p, p2, q, d, sc, ds.partial, ds.ticket};
        for (void *x : ptrs)
            if (x) cudaFreeAsync(x, s);
    }
};

int cg_alloc(CgBuffers &B, int64_t n, cudaStream_t s)
{
    B.s = s;
    NAP_CUDA(cudaMallocAsync(&B.r, sizeof(double) * n, s));
    NAP_CUDA(cudaMallocAsync(&B.p, sizeof(double) * n, s));
    NAP_CUDA(cudaMallocAsync(&B.p2, sizeof(double) * n, s));
    NAP_CUDA(cudaMallocAsync(&B.q, sizeof(double) * n, s));
    NAP_CUDA(cudaMallocAsync(&B.d, sizeof(double) * n, s));
    NAP_CUDA(cudaMallocAsync(&B.sc, sizeof(Scal), s));
    NAP_CUDA(cudaMallocAsync(&B.ds.partial, sizeof(double) * 2 * kDotBlocks, s));
    NAP_CUDA(cudaMallocAsync(&B.ds.ticket, sizeof(unsigned), s));
    NAP_CUDA(cudaMemsetAsync(B.ds.ticket, 0, sizeof(unsigned), s));
    NAP_CUDA(cudaMemsetAsync(B.sc, 0, sizeof(Scal), s));
    return NAPSPMV_OK;
}

// q <- A p with the plan's default options.  keep: the caller's last apply, whose
// receives napspmv_spmv_step may ask for.
int apply_one(napspmv_plan_t *P, const double *p, double *q, int32_t precision, bool keep,
              cudaStream_t s)
{
    napspmv_opts o{};
    o.precision = precision;
    const int32_t reps = 1;
    const double scale = 1.0;
    return apply_batch(1, &P, nullptr, &p, &q, &reps, &scale, &o, s, keep);
}

int grid_for(const napspmv_plan_t *P, int64_t n)
{
    return (int)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, (int64_t)P->num_sms * 8));
}

// CG on A x = b from the x given, products at `precision`.  Stops when the
// recursive residual satisfies ||r|| <= rtol * ||b|| or after max_it
// iterations (checked on the host every `poll` iterations).  x, b: device.
int cg_core(napspmv_plan_t *P, const double *b, double *x, double rtol, int max_it,
            int32_t precision, CgBuffers &B, int *iters)
{
    cudaStream_t s = B.s;
    const int64_t n = P->n;
    const int g = grid_for(P, n);
    int rc;
    if ((rc = apply_one(P, x, B.q, precision, false, s))) return rc;
    k_resid<<<g, 256, 0, s>>>(B.r, B.p, b, B.q, n);
    count_launch(1);
    if ((rc = dot_launch(b, b, n, &B.sc->bb, B.ds, s))) return rc;
    if ((rc = dot_launch(B.r, B.r, n, &B.sc->rr[0], B.ds, s))) return rc;
    Scal h{};
    NAP_CUDA(cudaMemcpyAsync(&h, B.sc, sizeof(Scal), cudaMemcpyDeviceToHost, s));
    NAP_CUDA(cudaStreamSynchronize(s));
    const double bn = h.bb > 0 ? std::sqrt(h.bb) : 1.0;
    int it = 0;
    const int poll = 8;
    // on staged windows the iteration sends p itself, the first time from here
    const bool windows = runs_on_windows(P, precision), f32 = precision == NAPSPMV_PREC_F32;
    const SendList sends = send_list(P, P->ws);
    const int64_t groups = (sends.n + kSendGroup - 1) / kSendGroup;
    const int send_blocks =
        windows ? (int)std::min<int64_t>((groups + kThreads * kDotGroups / 32 - 1) / (kThreads * kDotGroups / 32),
                                     (int64_t)P->num_sms)
                : 0;
    const dim3 dg = dot_grid(n);
    if (windows && (rc = send_alone(1, &P, &P->ws, precision, &B.p, s))) return rc;
    bool done = std::sqrt(h.rr[0]) <= rtol * bn;
    while (!done && it < max_it) {
        for (int q = 0; q < poll && it < max_it; q++, it++) {
            if (windows) rc = window_alone(1, &P, &P->ws, precision, &B.p, &B.q, s);
            else rc = apply_one(P, B.p, B.q, precision, false, s);
            if (rc) return rc;
            const CgIter I{x, B.r, B.p, B.p2, B.q, n, B.ds.partial, B.ds.partial + kDotBlocks,
                           (int)dg.x * kDotGroups, B.sc, it & 1};
            if ((rc = launch_dependent(k_pq, dg, kThreads * kDotGroups, s, I))) return rc;
            if ((rc = launch_dependent(k_update, dg, kThreads * kDotGroups, s, I))) return rc;
            if ((rc = launch_dependent(f32 ? k_next_p<float> : k_next_p<double>,
                                       dim3(dg.x + (unsigned)send_blocks), kThreads * kDotGroups, s, I, sends,
                                       (int)dg.x)))
                return rc;
            std::swap(B.p, B.p2);
        }
        NAP_CUDA(cudaMemcpyAsync(&h, B.sc, sizeof(Scal), cudaMemcpyDeviceToHost, s));
        NAP_CUDA(cudaStreamSynchronize(s));
        // (a flag set by the last product itself is read here too: it was set
        // before the update kernel read it)
        if (h.err && (rc = napspmv_ws_status(P->ws, s))) return rc;
        if (!std::isfinite(h.rr[it & 1])) break;
        done = std::sqrt(h.rr[it & 1]) <= rtol * bn;
    }
    *iters = it;
    return NAPSPMV_OK;
}

// ||b - A x|| / ||b|| in FP64 with the FP64 apply; leaves r = b - A x in B.r.
int true_relres(napspmv_plan_t *P, const double *b, const double *x, CgBuffers &B, double *out)
{
    cudaStream_t s = B.s;
    int rc;
    if ((rc = apply_one(P, x, B.q, NAPSPMV_PREC_F64, true, s))) return rc;
    k_resid<<<grid_for(P, P->n), 256, 0, s>>>(B.r, nullptr, b, B.q, P->n);
    count_launch(1);
    if ((rc = dot_launch(B.r, B.r, P->n, &B.sc->rnorm0, B.ds, s))) return rc;
    if ((rc = dot_launch(b, b, P->n, &B.sc->bb, B.ds, s))) return rc;
    Scal h{};
    NAP_CUDA(cudaMemcpyAsync(&h, B.sc, sizeof(Scal), cudaMemcpyDeviceToHost, s));
    NAP_CUDA(cudaStreamSynchronize(s));
    if ((rc = napspmv_ws_status(P->ws, s))) return rc;
    *out = std::sqrt(h.rnorm0) / (h.bb > 0 ? std::sqrt(h.bb) : 1.0);
    return NAPSPMV_OK;
}

}  // namespace
}  // namespace nap

using namespace nap;

extern "C" {

int napspmv_dot(const double *x, const double *y, int64_t n, double *result, void *stream)
{
    if ((n > 0 && (!x || !y)) || !result || n < 0) {
        set_error(NAPSPMV_ERR_ARG, "NULL vector or result, or n < 0");
        return NAPSPMV_ERR_ARG;
    }
    cudaStream_t s = (cudaStream_t)stream;
    DotScratch ds;
    NAP_CUDA(cudaMallocAsync(&ds.partial, sizeof(double) * kDotBlocks, s));
    NAP_CUDA(cudaMallocAsync(&ds.ticket, sizeof(unsigned), s));
    NAP_CUDA(cudaMemsetAsync(ds.ticket, 0, sizeof(unsigned), s));
    int rc = dot_launch(x, y, n, result, ds, s);
    cudaFreeAsync(ds.partial, s);
    cudaFreeAsync(ds.ticket, s);
    return rc;
}

int napspmv_cg(napspmv_plan_t *P, const double *b, double *x, double rtol, int32_t max_it,
               napspmv_cg_info *info, void *stream)
{
    if (!P || !b || !x || max_it < 0 || !(rtol > 0)) {
        set_error(NAPSPMV_ERR_ARG, "NULL plan or vector, max_it < 0 or rtol <= 0");
        return NAPSPMV_ERR_ARG;
    }
    CgBuffers B;
    int rc = cg_alloc(B, P->n, (cudaStream_t)stream);
    if (rc) return rc;
    int it = 0;
    if ((rc = cg_core(P, b, x, rtol, max_it, NAPSPMV_PREC_F64, B, &it))) return rc;
    double rr = 0;
    if ((rc = true_relres(P, b, x, B, &rr))) return rc;
    if (info) {
        info->outer_iters = 1;
        info->inner_iters = it;
        info->relres = rr;
        info->converged = rr <= rtol;
    }
    return NAPSPMV_OK;
}

int napspmv_cg_ir(napspmv_plan_t *P, const double *b, double *x, double rtol, double inner_rtol,
                  int32_t max_outer, int32_t inner_max, napspmv_cg_info *info, void *stream)
{
    if (!P || !b || !x || max_outer < 1 || inner_max < 1 || !(rtol > 0) || !(inner_rtol > 0)) {
        set_error(NAPSPMV_ERR_ARG, "bad arguments to napspmv_cg_ir");
        return NAPSPMV_ERR_ARG;
    }
    if (!P->d_val32) {
        set_error(NAPSPMV_ERR_STATE, "plan was built without NAPSPMV_F32_VALUES");
        return NAPSPMV_ERR_STATE;
    }
    cudaStream_t s = (cudaStream_t)stream;
    CgBuffers B, I;
    int rc = cg_alloc(B, P->n, s);
    if (rc) return rc;
    if ((rc = cg_alloc(I, P->n, s))) return rc;
    int outer = 0, inner_total = 0;
    double rr = 0;
    for (;;) {
        if ((rc = true_relres(P, b, x, B, &rr))) return rc;  // B.r = b - A x (FP64)
        if (rr <= rtol || outer >= max_outer || !std::isfinite(rr)) break;
        // inner solve A d = r with FP32-stored values, d_0 = 0
        NAP_CUDA(cudaMemsetAsync(I.d, 0, sizeof(double) * P->n, s));
        int it = 0;
        if ((rc = cg_core(P, B.r, I.d, inner_rtol, inner_max, NAPSPMV_PREC_F32, I, &it))) return rc;
        k_add<<<grid_for(P, P->n), 256, 0, s>>>(x, I.d, P->n);
        count_launch(1);
        NAP_CUDA(cudaGetLastError());
        inner_total += it;
        outer++;
    }
    if (info) {
        info->outer_iters = outer;
        info->inner_iters = inner_total;
        info->relres = rr;
        info->converged = rr <= rtol;
    }
    return NAPSPMV_OK;
}

}  // extern "C"

// ===================================================================
// Batched CG steps over independent requests (the request server).
//
// Every slot is one CG solve with its own plan, vectors and scalars.  A dot
// product of slot i uses slot_blocks(n_i) blocks over a fixed strided
// partition of its own vectors and a fixed-order final sum: a function of its
// own length only, so its value does not depend on which other slots share
// the launch.  One block per 1,024 elements, at most 4,096; the final sum is
// one warp's, lanes over a fixed stride and a fixed shuffle tree.  A fixed 64
// blocks left a 1.7M-element solve latency-bound on its vector kernels (about
// 330 us per CG iteration on GB300).
namespace nap {
namespace {

constexpr int kMaxSlots = 64;
constexpr int kSlotBlocksMax = 4096;
constexpr int64_t kSlotChunk = 4 * 256;

__host__ __device__ __forceinline__ int slot_blocks(int64_t n)
{
    const int64_t b = (n + kSlotChunk - 1) / kSlotChunk;
    return (int)(b < 1 ? 1 : (b > kSlotBlocksMax ? kSlotBlocksMax : b));
}

enum Scl { S_RR = 0, S_PQ = 1, S_ALPHA = 2, S_BETA = 3, S_RRNEW = 4, S_BB = 5 };

struct SlotVecs {
    int32_t count;
    int64_t n[kMaxSlots];
    const double *b[kMaxSlots];
    double *x[kMaxSlots], *r[kMaxSlots], *p[kMaxSlots], *q[kMaxSlots], *scal[kMaxSlots];
};

// mode 0: r = b - q, p = r, partial(r.r) and partial(b.b)
// mode 1: partial(p.q)
// mode 2: x += alpha p, r -= alpha q, partial(r.r)
// mode 3: p = r + beta p
// mode 4: r = b, p = b, partial(r.r), partial(b.b)   (x = 0)
// The slot's last block to finish adds its partials in a fixed order (lane l of a
// warp adds partials l, l + 32, ... in order, then a fixed shuffle tree), applies
// the scalar recurrences of CG and resets the slot's ticket.  It brings the
// partials into shared memory first: a warp that read them from L2 one by one, in
// a launch of its own, took 15 us per sum of a 1.7M-element slot (GB300; its CG
// iteration falls from 96 to 73 us, bound by the FP64 pipe and HBM in turn).
constexpr int kSumRound = 2048;  // partials in shared memory at a time
template <int MODE>
__global__ void __launch_bounds__(kThreads)
    k_slot_vec(const __grid_constant__ SlotVecs S, double *partial, unsigned *ticket)
{
    constexpr bool both = MODE == 0 || MODE == 4;
    __shared__ double sh[kSumDoubles];
    __shared__ double part[MODE == 3 ? 1 : kSumRound];
    __shared__ bool last;
    griddep_wait();
    const int i = blockIdx.y;
    const int64_t n = S.n[i];
    const int nb = slot_blocks(n);
    if ((int)blockIdx.x >= nb) return;  // the whole block: this slot needs fewer
    const double *b = S.b[i];
    double *x = S.x[i], *r = S.r[i], *p = S.p[i], *q = S.q[i];
    const double alpha = MODE == 2 ? S.scal[i][S_ALPHA] : 0.0;
    const double beta = MODE == 3 ? S.scal[i][S_BETA] : 0.0;
    double s1 = 0.0, s2 = 0.0;
    for (int64_t k = (int64_t)blockIdx.x * kThreads + threadIdx.x; k < n;
         k += (int64_t)nb * kThreads) {
        if (both) {
            const double v = MODE == 0 ? b[k] - q[k] : b[k];
            r[k] = v;
            p[k] = v;
            if (MODE == 4) x[k] = 0.0;
            s1 = fma(v, v, s1);
            s2 = fma(b[k], b[k], s2);
        } else if (MODE == 1) {
            s1 = fma(p[k], q[k], s1);
        } else if (MODE == 2) {
            x[k] = fma(alpha, p[k], x[k]);
            const double v = fma(-alpha, q[k], r[k]);
            r[k] = v;
            s1 = fma(v, v, s1);
        } else {
            p[k] = fma(beta, p[k], r[k]);
        }
    }
    if (MODE == 3) {
        griddep_done();
        return;
    }
    double *mine = partial + (int64_t)i * 2 * kSlotBlocksMax;  // r.r or p.q, then b.b
    s1 = group_sum(s1, sh, 0);
    if (both) s2 = group_sum(s2, sh, 0);
    if (threadIdx.x == 0) {
        mine[blockIdx.x] = s1;
        if (both) mine[kSlotBlocksMax + blockIdx.x] = s2;
        __threadfence();
        last = atomicAdd(ticket + i, 1u) == (unsigned)nb - 1;
    }
    __syncthreads();
    griddep_done();
    if (!last) return;
    __threadfence();
    double sum[2] = {0.0, 0.0};
    for (int w = 0; w < (both ? 2 : 1); w++) {
        double a = 0.0;
        for (int q0 = 0; q0 < nb; q0 += kSumRound) {
            const int m = min(kSumRound, nb - q0);
            __syncthreads();
            for (int k = threadIdx.x; k < m; k += kThreads)
                part[k] = __ldcg(mine + w * kSlotBlocksMax + q0 + k);
            __syncthreads();
            if (threadIdx.x < 32)
                for (int k = threadIdx.x; k < m; k += 32) a += part[k];
        }
        if (threadIdx.x < 32)
            for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        sum[w] = a;
    }
    if (threadIdx.x != 0) return;
    ticket[i] = 0;
    double *s = S.scal[i];
    if (both) {
        s[S_RR] = sum[0];
        s[S_BB] = sum[1];
    } else if (MODE == 1) {
        s[S_PQ] = sum[0];
        s[S_ALPHA] = s[S_RR] / sum[0];
    } else {
        s[S_RRNEW] = sum[0];
        s[S_BETA] = sum[0] / s[S_RR];
        s[S_RR] = sum[0];
    }
}

// The direction update of slots whose products run on staged windows: p' = r +
// beta p into the slot's other vector, and the inter-node messages of p' in further
// blocks (none after the last iteration of a call, whose product's receives stay).
struct SlotNext {
    int64_t n[kMaxSlots];
    const double *p[kMaxSlots], *r[kMaxSlots], *scal[kMaxSlots];
    double *p2[kMaxSlots];
    SendList sends[kMaxSlots];
    int *state[kMaxSlots];  // set to 1 after the last iteration
    int32_t last;
};
__host__ __device__ __forceinline__ int slot_send_blocks(int n)
{
    const int g = (n + kSendGroup * (kThreads / 32) - 1) / (kSendGroup * (kThreads / 32));
    return g < 304 ? g : 304;
}
template <class T>
__global__ void __launch_bounds__(kThreads) k_slot_next(const __grid_constant__ SlotNext S)
{
    griddep_wait();
    const int i = blockIdx.y, nb = slot_blocks(S.n[i]), ns = S.last ? 0 : slot_send_blocks(S.sends[i].n);
    const int block = (int)blockIdx.x;
    if (block >= nb + ns) return;
    const double *p = S.p[i], *r = S.r[i], beta = S.scal[i][S_BETA];
    if (block < nb) {
        if (S.last && block == 0 && threadIdx.x == 0) *S.state[i] = 1;
        for (int64_t k = (int64_t)block * kThreads + threadIdx.x; k < S.n[i]; k += (int64_t)nb * kThreads)
            S.p2[i][k] = fma(beta, p[k], r[k]);
    } else {
        send_next<T>(S.sends[i], p, r, beta, block - nb, ns);
    }
    griddep_done();
}

struct Partials {
    double *p = nullptr;
    unsigned *ticket = nullptr;
    cudaStream_t s = 0;
    ~Partials()
    {
        if (p) cudaFreeAsync(p, s);
    }
    int alloc(int count, cudaStream_t st)
    {
        s = st;
        const size_t sums = sizeof(double) * 2 * kSlotBlocksMax * count;
        NAP_CUDA(cudaMallocAsync(&p, sums + sizeof(unsigned) * count, st));
        ticket = reinterpret_cast<unsigned *>(reinterpret_cast<char *>(p) + sums);
        NAP_CUDA(cudaMemsetAsync(ticket, 0, sizeof(unsigned) * count, st));
        return NAPSPMV_OK;
    }
};

template <int MODE>
int slot_vec(const SlotVecs &S, const Partials &P)
{
    int gx = 1;
    for (int i = 0; i < S.count; i++) gx = std::max(gx, slot_blocks(S.n[i]));
    return launch_dependent(k_slot_vec<MODE>, dim3(gx, S.count), kThreads, P.s, S, P.p, P.ticket);
}

int slot_setup(int32_t count, const napspmv_cg_slot *slots, SlotVecs &S)
{
    if (count < 1 || count > kMaxSlots || !slots) {
        set_error(NAPSPMV_ERR_ARG, "need 1..64 CG slots");
        return NAPSPMV_ERR_ARG;
    }
    memset(&S, 0, sizeof(S));
    S.count = count;
    for (int i = 0; i < count; i++) {
        const napspmv_cg_slot &c = slots[i];
        if (!c.plan || !c.b || !c.x || !c.r || !c.p || !c.q || !c.scal) {
            set_error(NAPSPMV_ERR_ARG, "CG slot with a NULL pointer");
            return NAPSPMV_ERR_ARG;
        }
        S.n[i] = c.plan->n;
        S.b[i] = c.b;
        S.x[i] = c.x;
        S.r[i] = c.r;
        S.p[i] = c.p;
        S.q[i] = c.q;
        S.scal[i] = c.scal;
    }
    return NAPSPMV_OK;
}

int slot_apply(int32_t count, const napspmv_cg_slot *slots, bool from_x, int32_t precision,
               bool keep, cudaStream_t st)
{
    napspmv_plan_t *plans[kMaxSlots];
    napspmv_ws_t *wss[kMaxSlots];
    const double *vs[kMaxSlots];
    double *ws_[kMaxSlots];
    int32_t reps[kMaxSlots];
    double sc[kMaxSlots];
    for (int i = 0; i < count; i++) {
        plans[i] = slots[i].plan;
        wss[i] = slots[i].ws;
        vs[i] = from_x ? slots[i].x : slots[i].p;
        ws_[i] = slots[i].q;
        reps[i] = 1;
        sc[i] = 1.0;
    }
    // A slot whose matrix holds NAPSPMV_SOLO_NNZ or more stored entries gets an
    // apply of its own (staged windows or the phased engine); the others share
    // launches: the windows' two per apply, or the persistent one of the plans
    // without windows.  Measured on GB300 (FP32 mode, one apply): a 2.0M-row 7-point
    // plan takes 77 us phased against 191 us in the persistent launch, a
    // 0.4M-row one 33 against 70 us; below about half a million entries the
    // shared launch costs less than a call per slot.  The choice depends on the
    // slot's own matrix only, and every slot runs with its own plan's default
    // options (slots whose defaults differ go into separate fused launches), so
    // a slot's bits do not depend on the batch.
    int nb = 0;
    for (int i = 0; i < count; i++) {
        if (plans[i]->nnz >= NAPSPMV_SOLO_NNZ) {
            napspmv_opts o{};  // unset fields: the plan's defaults
            o.precision = precision;
            o.engine = NAPSPMV_ENGINE_PHASED;
            if (int rc = apply_batch(1, &plans[i], &wss[i], &vs[i], &ws_[i], &reps[i], &sc[i], &o, st, keep))
                return rc;
        } else {
            plans[nb] = plans[i];
            wss[nb] = wss[i];
            vs[nb] = vs[i];
            ws_[nb] = ws_[i];
            nb++;
        }
    }
    if (nb == 0) return NAPSPMV_OK;
    napspmv_opts o{};  // unset fields: each slot's own plan defaults
    o.precision = precision;
    return apply_batch(nb, plans, wss, vs, ws_, reps, sc, &o, st, keep, true);
}

// An even number of CG iterations of slots that all run on short-row staged windows
// of their own workspaces: one windowed launch for all products, and the direction
// alternates between the slot's p and the workspace's vector, which so ends as the
// last product's source (what napspmv_spmv_step asks for) with p current.  Four
// launches an iteration; with the messages in their own, a slot of 1.7M elements took
// 70.6 us per iteration against 68.9, 16 small ones 33 against 29 (GB300).
bool slots_on_windows(int32_t count, const napspmv_cg_slot *slots, int32_t precision, cudaStream_t st)
{
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    int dev = -1;
    if (cudaStreamIsCapturing(st, &cs) != cudaSuccess || cs != cudaStreamCaptureStatusNone ||
        cudaGetDevice(&dev) != cudaSuccess ||
        (precision != NAPSPMV_PREC_F64 && precision != NAPSPMV_PREC_F32))
        return false;
    for (int i = 0; i < count; i++) {
        const napspmv_cg_slot &c = slots[i];
        const napspmv_ws_t *W = c.ws ? c.ws : c.plan->ws;
        if (!runs_on_windows(c.plan, precision) || c.plan->device != dev || W->plan != c.plan ||
            c.p == c.q || (precision == NAPSPMV_PREC_F32 && !c.plan->d_val32))
            return false;
        for (int q = 0; q < i; q++)
            if (W == (slots[q].ws ? slots[q].ws : slots[q].plan->ws)) return false;
    }
    return true;
}
int slots_iterate(int32_t count, const napspmv_cg_slot *slots, SlotVecs &S, int32_t precision,
                  int32_t iters, const Partials &P, cudaStream_t st)
{
    const bool f32 = precision == NAPSPMV_PREC_F32;
    napspmv_plan_t *plans[kMaxSlots];
    napspmv_ws_t *ws[kMaxSlots];
    const double *in[kMaxSlots];
    double *q[kMaxSlots];
    SlotNext N;
    int gv = 1, gs = 1;
    for (int i = 0; i < count; i++) {
        plans[i] = slots[i].plan;
        ws[i] = slots[i].ws ? slots[i].ws : plans[i]->ws;
        in[i] = slots[i].p;
        q[i] = slots[i].q;
        N.n[i] = S.n[i];
        N.r[i] = S.r[i];
        N.scal[i] = S.scal[i];
        N.sends[i] = send_list(plans[i], ws[i]);
        N.state[i] = ws[i]->state;
        gv = std::max(gv, slot_blocks(S.n[i]));
        gs = std::max(gs, slot_blocks(S.n[i]) + slot_send_blocks(N.sends[i].n));
    }
    int rc = send_alone(count, plans, ws, precision, in, st);
    for (int it = 0; it < iters && !rc; it++) {
        N.last = it + 1 == iters;
        for (int i = 0; i < count; i++) {
            double *own = slots[i].p, *other = ws[i]->xtmp;
            S.p[i] = it & 1 ? other : own;
            in[i] = N.p[i] = S.p[i];
            N.p2[i] = it & 1 ? own : other;
        }
        if ((rc = window_alone(count, plans, ws, precision, in, q, st))) break;
        if ((rc = slot_vec<1>(S, P))) break;
        if ((rc = slot_vec<2>(S, P))) break;
        rc = launch_dependent(f32 ? k_slot_next<float> : k_slot_next<double>,
                              dim3((unsigned)(N.last ? gv : gs), (unsigned)count), kThreads, st, N);
    }
    for (int i = 0; i < count; i++) {
        S.p[i] = slots[i].p;
        ws[i]->recv_vector = true;
        // (as the engines that served a slot of its size leave the buffers)
        ws[i]->buf_f32 = f32 && plans[i]->nnz >= NAPSPMV_SOLO_NNZ;
    }
    return rc;
}

}  // namespace
}  // namespace nap

extern "C" {

int napspmv_cg_batch_init(int32_t count, const napspmv_cg_slot *slots, int32_t precision,
                          int32_t x_is_zero, void *stream)
{
    SlotVecs S;
    int rc = slot_setup(count, slots, S);
    if (rc) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    Partials P;
    if ((rc = P.alloc(count, st))) return rc;
    if (x_is_zero) return slot_vec<4>(S, P);
    if ((rc = slot_apply(count, slots, true, precision, true, st))) return rc;
    return slot_vec<0>(S, P);
}

int napspmv_cg_batch_iterate(int32_t count, const napspmv_cg_slot *slots, int32_t precision,
                             int32_t iters, void *stream)
{
    SlotVecs S;
    int rc = slot_setup(count, slots, S);
    if (rc) return rc;
    if (iters < 0) {
        set_error(NAPSPMV_ERR_ARG, "iters < 0");
        return NAPSPMV_ERR_ARG;
    }
    cudaStream_t st = (cudaStream_t)stream;
    Partials P;
    if ((rc = P.alloc(count, st))) return rc;
    int it = 0;
    if (iters >= 2 && slots_on_windows(count, slots, precision, st)) {
        it = iters & ~1;
        if ((rc = slots_iterate(count, slots, S, precision, it, P, st))) return rc;
    }
    for (; it < iters; it++) {
        if ((rc = slot_apply(count, slots, false, precision, it + 1 == iters, st))) return rc;
        if ((rc = slot_vec<1>(S, P))) return rc;
        if ((rc = slot_vec<2>(S, P))) return rc;
        if ((rc = slot_vec<3>(S, P))) return rc;
    }
    return NAPSPMV_OK;
}

}  // extern "C"

namespace nap {
namespace {
struct AddVecs {
    int32_t count;
    int64_t n[kMaxSlots];
    double *y[kMaxSlots];
    const double *x[kMaxSlots];
};
__global__ void k_slot_add(const __grid_constant__ AddVecs A)
{
    const int i = blockIdx.y;
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < A.n[i];
         k += (int64_t)gridDim.x * blockDim.x)
        A.y[i][k] += A.x[i][k];
}
}  // namespace
}  // namespace nap

extern "C" int napspmv_batch_add(int32_t count, double *const *y, const double *const *x,
                                 const int64_t *n, void *stream)
{
    if (count < 1 || count > kMaxSlots || !y || !x || !n) {
        set_error(NAPSPMV_ERR_ARG, "need 1..64 vector pairs");
        return NAPSPMV_ERR_ARG;
    }
    AddVecs A;
    memset(&A, 0, sizeof(A));
    A.count = count;
    for (int i = 0; i < count; i++) {
        if (!y[i] || !x[i] || n[i] < 0) {
            set_error(NAPSPMV_ERR_ARG, "NULL vector or n < 0");
            return NAPSPMV_ERR_ARG;
        }
        A.y[i] = y[i];
        A.x[i] = x[i];
        A.n[i] = n[i];
    }
    int gx = 1;
    for (int i = 0; i < count; i++) gx = std::max(gx, slot_blocks(n[i]));
    k_slot_add<<<dim3(gx, count), kThreads, 0, (cudaStream_t)stream>>>(A);
    count_launch(1);
    NAP_CUDA(cudaGetLastError());
    return NAPSPMV_OK;
}
