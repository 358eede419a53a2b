// Loss at the final step and its seed, gradient finalisation, macroscopic
// fields, Darcy permeability and the Adam update (arXiv 2310.00810:
// compute_loss of section 2.2, Eq. 7, Eq. 15, Eq. 12, Eq. 9, section 3.4).
//
// All sums over nodes are FP64: per-block partials (warp shuffles, then
// shared memory) followed by one fixed-order pass, so results are
// deterministic run to run.
#include <cooperative_groups.h>
#include <cuda.h>

#include <algorithm>

#include <mutex>

#include "device.cuh"

namespace lbm {

// The passes over a finished state are bound by FP64 arithmetic (about two
// lanes per SM and clock), which a warp pays for in full while one of its
// lanes works.  They take chunks of kChunk nodes, list the chunk's fluid nodes
// in shared memory, in node order, and run the arithmetic on full warps.
constexpr int kChunk = 1024;
constexpr int kChunkThreads = 256;
constexpr int kChunkBlocks = 912;  // at most: six per SM

// Nodes per chunk: shorter ones where whole ones would leave SMs idle.
int chunk_nodes(long long N)
{
    int c = kChunk;
    while (c > 128 && N / c < kChunkBlocks) c /= 2;
    return c;
}

unsigned chunk_grid(long long N)
{
    const int c = chunk_nodes(N);
    const long long chunks = (N + c - 1) / c;
    return (unsigned)(chunks < kChunkBlocks ? chunks : kChunkBlocks);
}

// Lists the nodes base <= n < end (at most kChunk) for which active(n) holds;
// idle(n) is called for the others.  Returns their number (every thread).
template <class A, class I>
__device__ __forceinline__ int chunk_list(unsigned short* list, long long base, long long end, A active, I idle)
{
    __shared__ int s_cnt[kChunk / 32 + 1];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int R = kChunk / kChunkThreads;
    bool on[R];
    unsigned bal[R];
    __syncthreads();  // the list of the chunk before is done with
#pragma unroll
    for (int j = 0; j < R; ++j) {
        const long long n = base + j * kChunkThreads + threadIdx.x;
        on[j] = n < end && active(n);
        if (n < end && !on[j]) idle(n);
        bal[j] = __ballot_sync(0xffffffffu, on[j]);
        if (lane == 0) s_cnt[j * (kChunkThreads / 32) + warp] = __popc(bal[j]);
    }
    __syncthreads();
    if (warp == 0) {  // exclusive scan of the kChunk / 32 = 32 counts
        int v = s_cnt[lane], inc = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += t;
        }
        s_cnt[lane] = inc - v;
        if (lane == 31) s_cnt[32] = inc;
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < R; ++j)
        if (on[j])
            list[s_cnt[j * (kChunkThreads / 32) + warp] + __popc(bal[j] & ((1u << lane) - 1u))] =
                (unsigned short)(j * kChunkThreads + threadIdx.x);
    __syncthreads();
    return s_cnt[32];
}

// -------------------------------------------------------------- loss

__global__ void __launch_bounds__(kChunkThreads) k_count_roi(Geo g, const uint8_t* __restrict__ roi,
                                                             double* __restrict__ partial)
{
    int c = 0;
    for (long long n = (long long)blockIdx.x * kChunkThreads + threadIdx.x; n < g.N; n += (long long)gridDim.x * kChunkThreads)
        if (!(g.link[n] & kLinkSolid) && (!roi || roi[n])) ++c;
    const double bs = block_sum((double)c, threadIdx.x, blockDim.x);
    if (threadIdx.x == 0) partial[blockIdx.x] = bs;
}

// weight = 1 / count (mean over ROI fluid nodes)
__global__ void k_loss_weight(const double* __restrict__ partial, int nb, double* __restrict__ scalars)
{
    const double c = block_reduce_array(partial, nb);
    if (threadIdx.x == 0) {
        scalars[0] = c;
        scalars[1] = c > 0.0 ? 1.0 / c : 0.0;
    }
}

// Per node: u from shifted f^T; loss term; lambda^T_k = sum_a dL/du_a (c_ka - u_a) / rho.
// MEAN: the terms carry *weight, else 1.  One FP64 partial per block.  Bound by
// FP64 on lattices in cache (128x64x64 D3Q19 FP32: 18 us, 24 without the list)
// and by memory on large ones (512x256x256: 1584 us with a block sum per 128
// nodes, 1400 so, for 6.0 GB).
template <int Q, typename T, int KIND, bool MEAN>
__global__ void __launch_bounds__(kChunkThreads)
    k_loss(const T* __restrict__ f, const double* __restrict__ ut, const uint8_t* __restrict__ roi, Geo g,
           const double* __restrict__ weight, T* __restrict__ lam, double* __restrict__ partial, int chunk)
{
    using L = Lattice<Q>;
    __shared__ unsigned short list[kChunk];
    const long long N = g.N;
    const double wgt = MEAN ? *weight : 1.0;
    double term = 0.0;
    auto node = [&](long long n) {
        T v[Q];
#pragma unroll
        for (int j = 0; j < Q; ++j) v[j] = f[(long long)j * N + n];
        double t[3] = {0.0, 0.0, 0.0};
#pragma unroll
        for (int a = 0; a < L::D; ++a) t[a] = ut[(long long)a * N + n];
        T drho, rho, u[3];
        moments<Q, T>(v, drho, rho, u);
        double du[3] = {0.0, 0.0, 0.0};
        if (KIND == LBM_LOSS_VEC) {
#pragma unroll
            for (int a = 0; a < L::D; ++a) {
                const double e = (double)u[a] - t[a];
                term += MEAN ? wgt * e * e : e * e;
                du[a] = MEAN ? 2.0 * wgt * e : e;
            }
        } else {
            double uu = 0.0, tt = 0.0;
#pragma unroll
            for (int a = 0; a < L::D; ++a) {
                uu += (double)u[a] * (double)u[a];
                tt += t[a] * t[a];
            }
            const double un = sqrt(uu);
            const double e = un - sqrt(tt);
            term += MEAN ? wgt * e * e : e * e;
            if (uu != 0.0)
#pragma unroll
                for (int a = 0; a < L::D; ++a) du[a] = (MEAN ? 2.0 * wgt : 1.0) * e * (double)u[a] / un;
        }
        T dv[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) dv[a] = MEAN ? T(du[a]) : T(2) * T(du[a]);  // doubling is exact
        const T inv = T(1) / rho;
#pragma unroll
        for (int k = 0; k < Q; ++k) {
            T s = 0;
#pragma unroll
            for (int a = 0; a < L::D; ++a) s += dv[a] * (T(L::c(k, a)) - u[a]);
            lam[(long long)k * N + n] = s * inv;
        }
    };
    auto active = [&](long long n) { return !(g.link[n] & kLinkSolid) && (!roi || roi[n]); };
    auto idle = [&](long long n) {
#pragma unroll
        for (int k = 0; k < Q; ++k) lam[(long long)k * N + n] = T(0);
    };
    for (long long base = (long long)blockIdx.x * chunk; base < N; base += (long long)gridDim.x * chunk) {
        const long long end = base + chunk < N ? base + chunk : N;
        const int cnt = chunk_list(list, base, end, active, idle);
        for (int i = threadIdx.x; i < cnt; i += kChunkThreads) node(base + list[i]);
    }
    const double bs = block_sum(term, threadIdx.x, blockDim.x);
    if (threadIdx.x == 0) partial[blockIdx.x] = bs;
}

// Density probes, a second loss term (w sum_p (rho(x_p) - rho_p)^2) for the
// joint inversion of the head and tau, whose velocity field alone fixes only
// their ratio in the Stokes regime.  Adds the term to *d_loss and its seed
// 2 w (rho(x_p) - rho_p) to every direction of lambda^T at x_p (drho/df_k = 1,
// Eq. 1).  One block: the loss is summed in a fixed order; a node listed twice
// gets both seeds through atomics (their order, so the last bit, may vary).
// An out-of-range node latches LBM_ERR_INVALID_ARG and is skipped; a solid
// node contributes nothing.
template <int Q, typename T>
__global__ void __launch_bounds__(kReduceThreads)
    k_probe_loss(const T* __restrict__ f, Geo g, long long n_probe, const int64_t* __restrict__ node,
                 const double* __restrict__ rho_t, double w, double* __restrict__ d_loss, T* __restrict__ lam,
                 uint32_t* __restrict__ status)
{
    const long long N = g.N;
    double term = 0.0;
    for (long long p = threadIdx.x; p < n_probe; p += blockDim.x) {
        const long long n = node[p];
        if (n < 0 || n >= N) {
            atomicOr(status, 1u << LBM_ERR_INVALID_ARG);
            continue;
        }
        if (g.link[n] & kLinkSolid) continue;
        T s = 0;
#pragma unroll
        for (int i = 0; i < Q; ++i) s += f[(long long)i * N + n];
        const double e = (1.0 + (double)s) - rho_t[p];
        term += w * e * e;
        const T seed = T(2.0 * w * e);
#pragma unroll
        for (int k = 0; k < Q; ++k) atomicAdd(lam + (long long)k * N + n, seed);
    }
    const double bs = block_sum(term, threadIdx.x, blockDim.x);
    if (threadIdx.x == 0) {
        *d_loss += bs;
        if (!isfinite(*d_loss)) atomicOr(status, 1u << LBM_ERR_NONFINITE);
    }
}

lbm_status probe_launch(const PlanInfo& p, const void* f, long long n_probe, const int64_t* node,
                        const double* rho_target, double weight, double* d_loss, void* lambda, uint32_t* status,
                        cudaStream_t s)
{
    const dim3 grid(1), block(kReduceThreads);
    if (p.q == 9 && p.prec == 4)
        k_probe_loss<9, float><<<grid, block, 0, s>>>(static_cast<const float*>(f), p.geo, n_probe, node, rho_target,
                                                      weight, d_loss, static_cast<float*>(lambda), status);
    else if (p.q == 9)
        k_probe_loss<9, double><<<grid, block, 0, s>>>(static_cast<const double*>(f), p.geo, n_probe, node,
                                                       rho_target, weight, d_loss, static_cast<double*>(lambda),
                                                       status);
    else if (p.prec == 4)
        k_probe_loss<19, float><<<grid, block, 0, s>>>(static_cast<const float*>(f), p.geo, n_probe, node, rho_target,
                                                       weight, d_loss, static_cast<float*>(lambda), status);
    else
        k_probe_loss<19, double><<<grid, block, 0, s>>>(static_cast<const double*>(f), p.geo, n_probe, node,
                                                        rho_target, weight, d_loss, static_cast<double*>(lambda),
                                                        status);
    return cuda_status(cudaGetLastError());
}

__global__ void k_loss_final(const double* __restrict__ partial, int nb, double* __restrict__ d_loss,
                             uint32_t* __restrict__ status)
{
    const double L = block_reduce_array(partial, nb);
    if (threadIdx.x == 0) {
        *d_loss = L;
        if (status && !isfinite(L)) atomicOr(status, 1u << LBM_ERR_NONFINITE);
    }
}

// The loss's launches on partial (one double per block of the grid) and
// scalars (two doubles).  The ROI count is only taken where the mean needs it.
template <int Q, typename T>
static void launch_loss(const PlanInfo& p, const void* f, const double* ut, const uint8_t* roi, int kind, int norm,
                        double* d_loss, void* lambda, double* scalars, double* partial, uint32_t* status,
                        cudaStream_t s)
{
    const unsigned nb = chunk_grid(p.geo.N);
    const T* fp = static_cast<const T*>(f);
    T* lp = static_cast<T*>(lambda);
    auto go = [&](auto kernel) { kernel<<<nb, kChunkThreads, 0, s>>>(fp, ut, roi, p.geo, scalars + 1, lp, partial, chunk_nodes(p.geo.N)); };
    if (norm == LBM_NORM_MEAN_FLUID) {
        k_count_roi<<<nb, kChunkThreads, 0, s>>>(p.geo, roi, partial);
        k_loss_weight<<<1, kReduceThreads, 0, s>>>(partial, (int)nb, scalars);
        if (kind == LBM_LOSS_VEC) go(k_loss<Q, T, LBM_LOSS_VEC, true>);
        else go(k_loss<Q, T, LBM_LOSS_NORM, true>);
    } else {
        if (kind == LBM_LOSS_VEC) go(k_loss<Q, T, LBM_LOSS_VEC, false>);
        else go(k_loss<Q, T, LBM_LOSS_NORM, false>);
    }
    k_loss_final<<<1, kReduceThreads, 0, s>>>(partial, (int)nb, d_loss, status);
}

template <int Q, typename T>
static void loss_impl(const PlanInfo& p, const void* f, const double* ut, const uint8_t* roi, int kind, int norm,
                      double* d_loss, void* lambda, unsigned char* ws, const Workspace& w, cudaStream_t s)
{
    launch_loss<Q, T>(p, f, ut, roi, kind, norm, d_loss, lambda,
                      reinterpret_cast<double*>(ws + w.status + kScalarCount),
                      reinterpret_cast<double*>(ws + w.partial2), reinterpret_cast<uint32_t*>(ws + w.status), s);
}

lbm_status loss_launch(const PlanInfo& p, const void* f, const double* u_target, const uint8_t* roi, int kind,
                       int norm, double* d_loss, void* lambda, unsigned char* ws, const Workspace& w,
                       cudaStream_t s)
{
    if (p.q == 9 && p.prec == 4) loss_impl<9, float>(p, f, u_target, roi, kind, norm, d_loss, lambda, ws, w, s);
    else if (p.q == 9 && p.prec == 8) loss_impl<9, double>(p, f, u_target, roi, kind, norm, d_loss, lambda, ws, w, s);
    else if (p.q == 19 && p.prec == 4) loss_impl<19, float>(p, f, u_target, roi, kind, norm, d_loss, lambda, ws, w, s);
    else if (p.q == 19 && p.prec == 8)
        loss_impl<19, double>(p, f, u_target, roi, kind, norm, d_loss, lambda, ws, w, s);
    else return LBM_ERR_UNSUPPORTED;
    return cuda_status(cudaGetLastError());
}

// ------------------------------------------- loss without a workspace

// Scratch of lbm_loss_grad_noalloc: two scalars, then one FP64 partial per
// thread block of the loss grid.  Every GPU that loads the library holds this
// array until the process exits.
constexpr int kNoallocHead = 32;  // doubles before the partials (count, weight, padding)
static __device__ __align__(256) double g_noalloc_scratch[kNoallocHead + LBM_NOALLOC_MAX_BLOCKS];

namespace {
constexpr int kMaxDevices = 64;

// The array's device address is looked up once per device and context: a
// device reset (cudaDeviceReset) or a new primary context loads the module
// again, possibly at another address, so the cached address is kept with the
// id of the context it was taken in and looked up again when that id changes.
struct NoallocAddr {
    unsigned long long ctx_id = 0;
    double* addr = nullptr;
};
NoallocAddr g_noalloc_addr[kMaxDevices];
std::mutex g_noalloc_mu;

using PfnCtxGetCurrent = CUresult (*)(CUcontext*);
using PfnCtxGetId = CUresult (*)(CUcontext, unsigned long long*);

// Id of the calling thread's current context (driver entry points fetched
// through the runtime, so the library does not link the driver library).
bool current_context_id(unsigned long long* id)
{
    static PfnCtxGetCurrent get_current = nullptr;
    static PfnCtxGetId get_id = nullptr;
    if (!get_current || !get_id) {
        void* a = nullptr;
        void* b = nullptr;
        cudaDriverEntryPointQueryResult qa, qb;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &a, 12000, cudaEnableDefault, &qa) != cudaSuccess ||
            qa != cudaDriverEntryPointSuccess || !a)
            return false;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &b, 12000, cudaEnableDefault, &qb) != cudaSuccess ||
            qb != cudaDriverEntryPointSuccess || !b)
            return false;
        get_current = reinterpret_cast<PfnCtxGetCurrent>(a);
        get_id = reinterpret_cast<PfnCtxGetId>(b);
    }
    CUcontext ctx = nullptr;
    if (get_current(&ctx) != CUDA_SUCCESS || !ctx) return false;
    return get_id(ctx, id) == CUDA_SUCCESS;
}
}  // namespace

lbm_status loss_launch_noalloc(const PlanInfo& p, const void* f, const double* u_target, const uint8_t* roi, int kind,
                               int norm, double* d_loss, void* lambda, cudaStream_t s)
{
    if (p.n_blocks > LBM_NOALLOC_MAX_BLOCKS) return LBM_ERR_INVALID_ARG;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return LBM_ERR_CUDA;
    if (dev < 0 || dev >= kMaxDevices) return LBM_ERR_UNSUPPORTED;
    // makes the device's primary context current on this thread (the runtime
    // initialises it here), so that its id can be read; allocates nothing
    if (cudaSetDevice(dev) != cudaSuccess) return LBM_ERR_CUDA;
    unsigned long long ctx_id = 0;
    if (!current_context_id(&ctx_id)) return LBM_ERR_CUDA;
    double* base = nullptr;
    {
        // set-up per device and context (with that device current): the
        // host-side name of the array is not a device address, so ask the
        // runtime for it
        std::lock_guard<std::mutex> lock(g_noalloc_mu);
        NoallocAddr& a = g_noalloc_addr[dev];
        if (!a.addr || a.ctx_id != ctx_id) {
            void* ptr = nullptr;
            if (cudaGetSymbolAddress(&ptr, g_noalloc_scratch) != cudaSuccess || !ptr) return LBM_ERR_CUDA;
            a.addr = static_cast<double*>(ptr);
            a.ctx_id = ctx_id;
        }
        base = a.addr;
    }
    double* scalars = base;  // [0] ROI fluid count, [1] loss weight
    double* partial = base + kNoallocHead;
    // the scalars and the partials are fully overwritten before they are read
    // (no status word on this path: a non-finite loss shows as NaN/Inf in d_loss)
    if (p.q == 9 && p.prec == 4)
        launch_loss<9, float>(p, f, u_target, roi, kind, norm, d_loss, lambda, scalars, partial, nullptr, s);
    else if (p.q == 9 && p.prec == 8)
        launch_loss<9, double>(p, f, u_target, roi, kind, norm, d_loss, lambda, scalars, partial, nullptr, s);
    else if (p.q == 19 && p.prec == 4)
        launch_loss<19, float>(p, f, u_target, roi, kind, norm, d_loss, lambda, scalars, partial, nullptr, s);
    else if (p.q == 19 && p.prec == 8)
        launch_loss<19, double>(p, f, u_target, roi, kind, norm, d_loss, lambda, scalars, partial, nullptr, s);
    else return LBM_ERR_UNSUPPORTED;
    return cuda_status(cudaGetLastError());
}

// ------------------------------------------- sums of a time-window loss

__global__ void k_accumulate(double* __restrict__ dst, const double* __restrict__ src) { *dst += *src; }

template <typename T>
__global__ void k_add_state(T* __restrict__ dst, const T* __restrict__ src, long long n)
{
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        dst[i] += src[i];
}

lbm_status accumulate_launch(double* dst, const double* src, cudaStream_t s)
{
    k_accumulate<<<1, 1, 0, s>>>(dst, src);
    return cuda_status(cudaGetLastError());
}

// dst += src over a dense state (Q N values of the plan's precision).
lbm_status add_state_launch(const PlanInfo& p, void* dst, const void* src, cudaStream_t s)
{
    const long long n = (long long)p.q * p.geo.N;
    const unsigned grid = (unsigned)std::min<long long>((n + 255) / 256, 4096);
    if (p.prec == 4) k_add_state<float><<<grid, 256, 0, s>>>(static_cast<float*>(dst), static_cast<const float*>(src), n);
    else k_add_state<double><<<grid, 256, 0, s>>>(static_cast<double*>(dst), static_cast<const double*>(src), n);
    return cuda_status(cudaGetLastError());
}

// ----------------------------------------------------- gradient finalise

// dL/dtau = -(sum of dL/domega partials) / tau^2 ; dL/drho_in from the
// per-inlet-node accumulators (summed for a constant head).
__global__ void k_finish_gradients(const double* __restrict__ grad_acc, int n_acc, int profile,
                                   const double* __restrict__ partial, int nb, const double* __restrict__ tau,
                                   double* __restrict__ g_rho_in, double* __restrict__ g_tau,
                                   uint32_t* __restrict__ status)
{
    const double gw = block_reduce_array(partial, nb);
    double gsum = 0.0;
    if (!profile) gsum = block_reduce_array(grad_acc, n_acc);
    bool bad = false;
    if (profile)
        for (int i = threadIdx.x; i < n_acc; i += blockDim.x) {
            g_rho_in[i] = grad_acc[i];
            bad |= !isfinite(grad_acc[i]);
        }
    if (threadIdx.x == 0) {
        const double t = *tau;
        *g_tau = -gw / (t * t);
        if (!profile) g_rho_in[0] = gsum;
        bad |= !isfinite(gw) || !isfinite(gsum);
    }
    if (bad) atomicOr(status, 1u << LBM_ERR_NONFINITE);
}

lbm_status finish_gradients_launch(const PlanInfo& p, const double* grad_acc, const double* partial,
                                   const double* tau, double* d_grad_rho_in, double* d_grad_tau, uint32_t* status,
                                   cudaStream_t s)
{
    k_finish_gradients<<<1, kReduceThreads, 0, s>>>(grad_acc, p.n_acc, p.n_in > 1 ? 1 : 0, partial, p.n_partial, tau,
                                                    d_grad_rho_in, d_grad_tau, status);
    return cuda_status(cudaGetLastError());
}

// ------------------------------------------------------- macroscopic

// FP64 moments; bound by FP64 (128x64x64 D3Q19, half of it solid: 115 us
// without the list, 56 with it).  A component's quotient is its product with the reciprocal and
// one step of Markstein's correction (IBM J. Res. Dev. 34, 1990), within an ulp
// of the division; the ends of the exponent range take the division itself.
template <int Q, typename T>
__global__ void __launch_bounds__(kChunkThreads)
    k_macroscopic(const T* __restrict__ f, Geo g, double* __restrict__ rho_out, double* __restrict__ u_out, int chunk)
{
    using L = Lattice<Q>;
    __shared__ unsigned short list[kChunk];
    const long long N = g.N;
    for (long long base = (long long)blockIdx.x * chunk; base < N; base += (long long)gridDim.x * chunk) {
        const int cnt = chunk_list(
            list, base, base + chunk < N ? base + chunk : N, [&](long long n) { return !(g.link[n] & kLinkSolid); },
            [&](long long n) {
                if (rho_out) rho_out[n] = 0.0;
#pragma unroll
                for (int a = 0; a < L::D; ++a) u_out[(long long)a * N + n] = 0.0;
            });
        for (int i = threadIdx.x; i < cnt; i += kChunkThreads) {
            const long long n = base + list[i];
            T v[Q];
#pragma unroll
            for (int d = 0; d < Q; ++d) v[d] = f[(long long)d * N + n];
            double s = 0.0, j[3] = {0.0, 0.0, 0.0};
#pragma unroll
            for (int d = 0; d < Q; ++d) {
                const double w = (double)v[d];
                s += w;
#pragma unroll
                for (int a = 0; a < L::D; ++a)
                    if (L::c(d, a) != 0) j[a] += L::c(d, a) > 0 ? w : -w;
            }
            const double r = 1.0 + s, inv = 1.0 / r;
            const bool plain = fabs(r) > 1e-100 && fabs(r) < 1e100 && fabs(j[0]) < 1e100 && fabs(j[1]) < 1e100 &&
                               fabs(j[2]) < 1e100;  // false for a NaN
            if (rho_out) rho_out[n] = r;
#pragma unroll
            for (int a = 0; a < L::D; ++a) {
                const double q = j[a] * inv;
                u_out[(long long)a * N + n] = plain ? fma(fma(-q, r, j[a]), inv, q) : j[a] / r;
            }
        }
    }
}

lbm_status macroscopic_launch(const PlanInfo& p, const void* f, double* rho, double* u, cudaStream_t s)
{
    const unsigned nb = chunk_grid(p.geo.N);
    auto go = [&](auto kernel, auto* fp) { kernel<<<nb, kChunkThreads, 0, s>>>(fp, p.geo, rho, u, chunk_nodes(p.geo.N)); };
    if (p.q == 9 && p.prec == 4) go(k_macroscopic<9, float>, static_cast<const float*>(f));
    else if (p.q == 9 && p.prec == 8) go(k_macroscopic<9, double>, static_cast<const double*>(f));
    else if (p.q == 19 && p.prec == 4) go(k_macroscopic<19, float>, static_cast<const float*>(f));
    else if (p.q == 19 && p.prec == 8) go(k_macroscopic<19, double>, static_cast<const double*>(f));
    else return LBM_ERR_UNSUPPORTED;
    return cuda_status(cudaGetLastError());
}

// ------------------------------------------------------------- Darcy

// k = nu J / (dp/dx), J = section mean of rho u_x, nu = (tau - 1/2)/3 (Eq. 9),
// dp/dx = (mean rho_in - rho_out) / (3 nx)  (Eq. 12).
// One cluster of up to eight blocks: each sums its cells, the first adds the
// blocks' sums in order through their shared memory (a single block took 31 us
// for the 64x64 section of a D3Q19 lattice).
constexpr int kDarcyCtas = 8;
template <int Q, typename T>
__global__ void __launch_bounds__(kReduceThreads)
    k_darcy(const T* __restrict__ f, Geo g, const double* __restrict__ rho_in, int n_in,
            const double* __restrict__ tau, double rho_out, int xs, double* __restrict__ k, double* __restrict__ flux)
{
    using L = Lattice<Q>;
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    __shared__ double s_j;
    const long long N = g.N;
    const long long cells = (long long)g.ny * g.nz;
    double J = 0.0;
    for (long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x; c < cells; c += (long long)gridDim.x * blockDim.x) {
        const long long n = c * g.nx + xs;  // c = z * ny + y
        if (g.link[n] & kLinkSolid) continue;
        double jx = 0.0;
#pragma unroll
        for (int i = 0; i < Q; ++i)
            if (L::c(i, 0) != 0) jx += L::c(i, 0) * (double)f[(long long)i * N + n];
        J += jx;  // rho u_x = sum_i c_ix f_i (the rest shift has zero momentum)
    }
    J = block_sum(J, threadIdx.x, blockDim.x);
    if (threadIdx.x == 0) s_j = J;
    cluster.sync();
    if (blockIdx.x == 0) {
        const double rin = block_reduce_array(rho_in, n_in);
        if (threadIdx.x == 0) {
            J = 0.0;
            for (unsigned b = 0; b < gridDim.x; ++b) J += *cluster.map_shared_rank(&s_j, b);
            J /= (double)cells;
            const double nu = (*tau - 0.5) / 3.0;
            const double dpdx = (rin / n_in - rho_out) / (3.0 * g.nx);
            *k = nu * J / dpdx;
            if (flux) *flux = J;
        }
    }
    cluster.sync();  // the blocks' shared memory stays until it has been read
}

template <int Q, typename T>
static lbm_status launch_darcy(const PlanInfo& p, const void* f, const double* rho_in, int n_in, const double* tau,
                               double rho_out, int xs, double* k, double* flux, cudaStream_t s)
{
    const long long cells = (long long)p.geo.ny * p.geo.nz;
    unsigned ctas = 1;
    while (ctas < kDarcyCtas && (long long)ctas * kReduceThreads < cells) ctas *= 2;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(ctas);
    cfg.blockDim = dim3(kReduceThreads);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = ctas;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cuda_status(cudaLaunchKernelEx(&cfg, k_darcy<Q, T>, static_cast<const T*>(f), p.geo, rho_in, n_in, tau,
                                          rho_out, xs, k, flux));
}

lbm_status darcy_launch(const PlanInfo& p, const void* f, const double* rho_in, int n_in, const double* tau,
                        double rho_out, int xs, double* k, double* flux, cudaStream_t s)
{
    if (p.q == 9 && p.prec == 4) return launch_darcy<9, float>(p, f, rho_in, n_in, tau, rho_out, xs, k, flux, s);
    if (p.q == 9 && p.prec == 8) return launch_darcy<9, double>(p, f, rho_in, n_in, tau, rho_out, xs, k, flux, s);
    if (p.q == 19 && p.prec == 4) return launch_darcy<19, float>(p, f, rho_in, n_in, tau, rho_out, xs, k, flux, s);
    if (p.q == 19 && p.prec == 8) return launch_darcy<19, double>(p, f, rho_in, n_in, tau, rho_out, xs, k, flux, s);
    return LBM_ERR_UNSUPPORTED;
}

// -------------------------------------------------------------- Adam

__global__ void k_adam(int n, double* __restrict__ theta, double* __restrict__ m, double* __restrict__ v,
                       const double* __restrict__ grad_p, double* __restrict__ p, double off, double scale, double bc1,
                       double bc2, double lr, double b1, double b2, double eps)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double g = grad_p[i] * scale;  // dL/dtheta = dL/dp * dp/dtheta
    const double mi = b1 * m[i] + (1.0 - b1) * g;
    const double vi = b2 * v[i] + (1.0 - b2) * g * g;
    m[i] = mi;
    v[i] = vi;
    const double th = theta[i] - lr * (mi / bc1) / (sqrt(vi / bc2) + eps);
    theta[i] = th;
    p[i] = off + scale * th;
}

lbm_status adam_launch(int n, double* theta, double* m, double* v, const double* grad_p, double* p, double off,
                       double scale, int t, double lr, double b1, double b2, double eps, cudaStream_t s)
{
    const double bc1 = 1.0 - pow(b1, (double)t), bc2 = 1.0 - pow(b2, (double)t);
    k_adam<<<(n + 255) / 256, 256, 0, s>>>(n, theta, m, v, grad_p, p, off, scale, bc1, bc2, lr, b1, b2, eps);
    return cuda_status(cudaGetLastError());
}

}  // namespace lbm
