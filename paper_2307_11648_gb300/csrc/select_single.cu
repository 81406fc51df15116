// Directed Gaussian-process selection for one target over n training points
// (Section 3; the selection step of the directed regression algorithm).
//
// The training points are rows spread over the blocks of one cooperative launch (thread =
// row, rows beyond the grid strided); the partial Cholesky factor of the candidates is kept
// in the caller's workspace, column-major [k][n] (a thread touches its row of every column,
// neighbouring threads neighbouring addresses).  The conditional variances and covariances
// with the target, var[n] and cov[n], sit in the workspace too.  Per step: score cov^2/var
// (eq. obj_gp), block argmax (ties: lowest training index), one grid barrier, every block
// reduces the blocks' bests, stages the pivot's row in shared memory, and every thread
// appends u_j = (Theta_{jq} - F_j . F_q)/sqrt(var_q) and downdates var and cov
// (eq. cond_select).  out_var traces the target's conditional variance.
//
// Bound: the FP64 pipe (n k (k/2 + 17) operations; the factor, 8 n k bytes, stays in L2) plus
// a barrier and three dependent L2 round trips per step.  One block on one SM was the whole
// kernel before: 98.3 ms for
// n = 65,536, k = 64 in FP64 (3-D, Matern 5/2); spread over the grid 1.16 ms.
#include "sic_internal.cuh"

namespace {

constexpr int NT_MAX = 256;
constexpr int NW_MAX = NT_MAX / 32;
constexpr int WAIT_POLLS = 1 << 24;  // a grid barrier gives up after this many polls

template <typename T>
__device__ __forceinline__ bool better(T s, long long i, T bs, long long bi) {
    return s > bs || (s == bs && i < bi);
}

// a block's best candidate of a step
template <typename T>
struct Best {
    T score, var, cov;
    long long idx;
};

constexpr long long NONE = 0x7fffffffffffffffLL;

// The blocks' scratch -- the barrier's arrival count, then one Best per block and step parity --
// lies in the factor's last column, which nothing reads (and which is not written then): with
// 64 or more rows per block a column always holds it.
template <typename T>
inline unsigned* scratch_of(T* ws, long long n, long long k) {
    return reinterpret_cast<unsigned*>((reinterpret_cast<uintptr_t>(ws + (k - 1) * n) + 15) / 16 * 16);
}
template <typename T>
constexpr long long scratch_bytes(long long blocks) {
    return 16 + 2 * (long long)sizeof(Best<T>) * blocks;
}
static_assert(scratch_bytes<float>(2) + 12 <= 65 * 4 && 2 * sizeof(Best<float>) <= 64 * 4, "scratch of the blocks");
static_assert(scratch_bytes<double>(2) + 8 <= 65 * 8 && 2 * sizeof(Best<double>) <= 64 * 8, "scratch of the blocks");

// Arrival of every block, `target` arrivals in all; false when the wait gave up.  The launch is
// cooperative, so the blocks run at the same time.
__device__ __forceinline__ bool grid_wait(unsigned* count, unsigned target) {
    __threadfence();
    atomicAdd(count, 1u);
    for (int i = 0; i < WAIT_POLLS; ++i) {
        unsigned c;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(c) : "l"(count) : "memory");
        if (c >= target) return true;
    }
    return false;
}

template <typename T>
__global__ void __launch_bounds__(NT_MAX) k_select_single(const double* __restrict__ xtr, long long n, int dim,
                                                          const double* __restrict__ xt, KP<T> kp, T floor_, int k,
                                                          int32_t* __restrict__ out_idx,
                                                          double* __restrict__ out_var,
                                                          int32_t* __restrict__ out_count, T* ws, unsigned* count,
                                                          DevStatus* st) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* piv = reinterpret_cast<T*>(smem_raw);  // k
    __shared__ Best<T> wbest[NW_MAX];
    __shared__ Best<T> gbest;
    __shared__ int s_ok;
    __shared__ double tab[sizeof(T) == 8 ? EXP_TAB : 1];  // s2 2^(j/256): the FP64 Matern's exp
    T* F = ws;
    T* var = F + (long long)k * n;
    T* cov = var + n;
    Best<T>* bests = reinterpret_cast<Best<T>*>(count + 4);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
    const long long j0 = blockIdx.x * (long long)blockDim.x + tid, jstep = (long long)gridDim.x * blockDim.x;
    const T NEG = -INFINITY;
    double org[3] = {0.0, 0.0, 0.0};
    for (int d = 0; d < dim; ++d) org[d] = xt[d];
    auto coord = [&](long long j, int d) -> T {
        if constexpr (sizeof(T) == 8) return (T)xtr[j * dim + d];
        return (T)(xtr[j * dim + d] - org[d]);
    };
    // Theta at squared distance d2 (no nugget): in FP64 the table-driven exp and the Newton
    // square root (few FP64-pipe operations, about 2 ulp)
    auto theta = [&](T d2) -> T {
        if constexpr (sizeof(T) == 8)
            return matern_d2_fast(kp, d2, tab);
        else
            return matern<T>(kp, sic_sqrt(d2));
    };
    if constexpr (sizeof(T) == 8) {
        exp_table_fill(tab, kp.s2);
        __syncthreads();
    }
    for (long long j = j0; j < n; j += jstep) {
        T d2 = (T)0;
        for (int d = 0; d < dim; ++d) {
            T df = (T)(xtr[j * dim + d] - org[d]);
            d2 += df * df;
        }
        var[j] = kp.s2 + kp.nugget;
        cov[j] = theta(d2);
    }
    double vt = (double)(kp.s2 + kp.nugget);
    if (j0 == 0) out_var[0] = vt;
    int t = 0;
    for (; t < k; ++t) {
        Best<T> b;
        b.score = NEG;
        b.idx = NONE;
        b.var = b.cov = (T)0;
        auto take = [&](const Best<T>& o) {
            if (better(o.score, o.idx, b.score, b.idx)) b = o;
        };
        for (long long j = j0; j < n; j += jstep) {
            const T v = var[j];
            if (v >= floor_) {
                const T c = cov[j];
                take(Best<T>{c * c / v, v, c, j});
            }
        }
        auto block_best = [&]() {  // b of every thread -> the block's best in gbest
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) {
                Best<T> o;
                o.score = __shfl_xor_sync(0xffffffffu, b.score, off);
                o.var = __shfl_xor_sync(0xffffffffu, b.var, off);
                o.cov = __shfl_xor_sync(0xffffffffu, b.cov, off);
                o.idx = __shfl_xor_sync(0xffffffffu, b.idx, off);
                take(o);
            }
            if (lane == 0) wbest[warp] = b;
            __syncthreads();
            if (tid == 0) {
                for (int w = 1; w < nw; ++w) take(wbest[w]);
                gbest = b;
            }
        };
        block_best();
        if (gridDim.x > 1) {
            Best<T>* mine = bests + (t & 1) * gridDim.x;
            if (tid == 0) {
                mine[blockIdx.x] = gbest;
                s_ok = grid_wait(count, (unsigned)gridDim.x * (unsigned)(t + 1));
            }
            __syncthreads();
            if (!s_ok) {
                if (tid == 0) record_error(st, SIC_ERR_TIMEOUT, -1);
                break;
            }
            b.score = NEG;
            b.idx = NONE;
            for (int i = tid; i < (int)gridDim.x; i += blockDim.x) {
                Best<T> o;
                o.score = __ldcg(&mine[i].score);
                o.var = __ldcg(&mine[i].var);
                o.cov = __ldcg(&mine[i].cov);
                o.idx = __ldcg(&mine[i].idx);
                take(o);
            }
            block_best();
        }
        __syncthreads();
        const long long q = gbest.idx;
        if (q == NONE || !(gbest.score > (T)0)) break;
        const T vq = gbest.var, cq = gbest.cov;
        T qx[3] = {(T)0, (T)0, (T)0};
        for (int d = 0; d < dim; ++d) qx[d] = coord(q, d);
        for (int tau = tid; tau < t; tau += blockDim.x) piv[tau] = __ldcg(&F[(long long)tau * n + q]);
        __syncthreads();
        T rs;
        if constexpr (sizeof(T) == 8)
            rs = rsqrt_newton(vq);
        else
            rs = (T)1 / sic_sqrt(vq);
        const T ut = cq * rs;
        for (long long j = j0; j < n; j += jstep) {
            const T vj = var[j];
            if (vj == NEG) continue;
            T d2 = (T)0;
            for (int d = 0; d < dim; ++d) {
                T df = coord(j, d) - qx[d];
                d2 += df * df;
            }
            T num = theta(d2);
            if (j == q) num += kp.nugget;
            const T* Fj = F + j;
            int tau = 0;
            for (; tau + 8 <= t; tau += 8) {  // eight loads in flight, the sum in order
                T f[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) f[i] = Fj[(long long)(tau + i) * n];
#pragma unroll
                for (int i = 0; i < 8; ++i) num = fma(-f[i], piv[tau + i], num);
            }
            for (; tau < t; ++tau) num = fma(-Fj[(long long)tau * n], piv[tau], num);
            const T u = num * rs;
            if (t + 1 < k) F[(long long)t * n + j] = u;  // the last column has no reader
            if (j == q) {
                var[j] = NEG;
            } else {
                var[j] = fma(-u, u, vj);
                cov[j] = fma(-u, ut, cov[j]);
            }
        }
        vt -= (double)ut * (double)ut;
        if (j0 == 0) {
            out_idx[t] = (int32_t)q;
            out_var[t + 1] = vt;
        }
    }
    if (blockIdx.x == 0) {
        if (tid == 0) *out_count = t;
        for (int q = t + tid; q < k; q += blockDim.x) out_idx[q] = -1;
    }
}

// Rows per block: the step chain (barrier, reduction, pivot row) costs the same at any block
// size, so small n spreads over the SMs in blocks of 64 rows; from 152 x 256 rows on two blocks of
// 256 share an SM and further rows are strided.
template <typename T>
sic_status launch_single(sic_handle* h, const double* x_train, int64_t n, const double* x_target,
                         const sic_kernel* kp, int32_t k, int32_t* out_idx, double* out_var, int32_t* out_count,
                         void* ws, cudaStream_t s) {
    auto kern = k_select_single<T>;
    const size_t smem = sizeof(T) * (size_t)k;
    if (smem > 40 * 1024)
        SIC_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    const long long per = (n + h->num_sms - 1) / h->num_sms;
    const int nt = per <= 64 ? 64 : (per <= 128 ? 128 : 256);
    int grid = persistent_grid(h, kern, nt, smem, (n + nt - 1) / nt);
    if (grid > 2 * h->num_sms) grid = 2 * h->num_sms;
    T* w = (T*)ws;
    int dim = kp->dim;
    long long nn = n;
    KP<T> kpt = make_kp<T>(*kp);
    T fl = (T)sic_floor_of(kp);
    unsigned* count = scratch_of<T>(w, n, k);
    if (grid > 1) SIC_CUDA_TRY(cudaMemsetAsync(count, 0, 16, s));
    for (;;) {
        if (grid == 1) {
            kern<<<1, nt, smem, s>>>(x_train, nn, dim, x_target, kpt, fl, k, out_idx, out_var, out_count, w, count,
                                 h->d_status);
            break;
        }
        void* args[] = {&x_train, &nn, &dim, &x_target, &kpt, &fl, &k, &out_idx, &out_var, &out_count, &w, &count,
                        &h->d_status};
        cudaError_t e = cudaLaunchCooperativeKernel((const void*)kern, dim3((unsigned)grid), dim3((unsigned)nt), args, smem, s);
        if (e != cudaErrorCooperativeLaunchTooLarge) break;
        cudaGetLastError();  // fewer SMs than the device reports (a partitioned context): fewer blocks
        grid /= 2;
    }
    SIC_CUDA_TRY(cudaGetLastError());
    return SIC_OK;
}

}  // namespace

extern "C" sic_status sic_select_single_workspace(int64_t n, int32_t k, sic_precision prec, size_t* bytes) {
    if (!bytes || n < 1 || k < 1) return SIC_ERR_INVALID;
    size_t el = (prec == SIC_FP64) ? 8 : 4;
    *bytes = el * ((size_t)k * (size_t)n + 2 * (size_t)n);
    return SIC_OK;
}

extern "C" sic_status sic_select_single(sic_handle* h, const double* x_train, int64_t n, const double* x_target,
                                        const sic_kernel* kp, int32_t k, sic_precision prec, int32_t* out_idx,
                                        double* out_var, int32_t* out_count, void* ws, size_t ws_bytes,
                                        void* stream) {
    if (!h || !x_train || !x_target || !sic_valid_kernel(kp) || n < 1 || k < 1 || !out_idx || !out_var ||
        !out_count)
        return SIC_ERR_INVALID;
    if (n > 0x7fffffffLL) return SIC_ERR_UNSUPPORTED;
    size_t need = 0;
    sic_select_single_workspace(n, k, prec, &need);
    if (!ws || ws_bytes < need) return SIC_ERR_INVALID;
    SIC_CUDA_TRY(cudaSetDevice(h->device));
    cudaStream_t s = (cudaStream_t)stream;
    if (prec == SIC_FP64)
        return launch_single<double>(h, x_train, n, x_target, kp, k, out_idx, out_var, out_count, ws, s);
    if (prec == SIC_FP32_MIXED)
        return launch_single<float>(h, x_train, n, x_target, kp, k, out_idx, out_var, out_count, ws, s);
    return SIC_ERR_INVALID;
}
