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
// Between two barriers no block reads what another one writes: a block publishes its best row's variance and
// covariance with the score (var[q] and cov[q] themselves change in the same step), in slots of two alternating
// parities, and the pivot's row has only columns of earlier steps.
//
// In FP64 the factor is held in fixed point (fx.cuh, select_fx.cu): exact integer dot products instead of FP64
// multiply-adds, and scores in FP32 first, the FP64 quotient only where a row is within 2^-18 of its block's largest.
//
// (A best covariance below 2^-30 of the variance starts over with the rows in FP64, as in select_fx.cu.)
//
// Bound: a barrier and three dependent L2 round trips per step (slots; the pivot's coordinates and row), then the factor's L2
// traffic (4 n k^2 bytes) and the FP64 pipe.  One block on one SM was the whole kernel: 98.3 ms for n = 65,536, k = 64 in FP64 (3-D, Matern 5/2); over
// the grid with FP64 multiply-adds and divisions 1.16 ms, in fixed point 0.86 ms.
// Error of out_var against 128-bit arithmetic over 48 problems (n 700 .. 65,536, k 30 .. 64, nugget 1e-8 .. 1e-2; variance 1):
// 1.7e-16 on average, 9e-16 at most; with the library exponential and FP64 sums 2.0e-16 and 1.5e-15.  Either is a
// few roundings of out_var itself; single problems go either way.
#include "fx.cuh"

namespace {

constexpr int NT_MAX = 512;
constexpr int NW_MAX = NT_MAX / 32;
constexpr int WAIT_POLLS = 1 << 24;  // a grid barrier gives up after this many polls

template <typename T>
__device__ __forceinline__ bool better(T s, long long i, T bs, long long bi) {
    return s > bs || (s == bs && i < bi);
}

// a block's best candidate of a step, with what the others need of its state
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
                                                          const double* __restrict__ xt, KP<T> kp, T floor_, int e,
                                                          int k, int32_t* __restrict__ out_idx,
                                                          double* __restrict__ out_var,
                                                          int32_t* __restrict__ out_count, T* ws, unsigned* count,
                                                          DevStatus* st) {
    constexpr bool F64 = sizeof(T) == 8;
    constexpr unsigned FULL = 0xffffffffu;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* piv = reinterpret_cast<T*>(smem_raw);         // k: the pivot's row (FP64: fixed point, int2)
    __shared__ unsigned wkey[NW_MAX];
    __shared__ Best<T> wbest[NW_MAX];
    __shared__ long long s_q;
    __shared__ T s_rs, s_ut;
    __shared__ int s_ok, s_small;
    __shared__ double tab[F64 ? EXP_TAB : 1];  // s2 2^(j/256): the FP64 Matern's exp
    T* F = ws;
    T* var = F + (long long)k * n;
    T* cov = var + n;
    int2* Fx = reinterpret_cast<int2*>(ws);
    const int2* px = reinterpret_cast<const int2*>(piv);
    Best<T>* bests = reinterpret_cast<Best<T>*>(count + 4);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
    const long long j0 = blockIdx.x * (long long)blockDim.x + tid, jstep = (long long)gridDim.x * blockDim.x;
    const T NEG = -INFINITY;
    double org[3] = {0.0, 0.0, 0.0};
    for (int d = 0; d < dim; ++d) org[d] = xt[d];
    auto coord = [&](long long j, int d) -> T {
        if constexpr (F64) return (T)xtr[j * dim + d];
        return (T)(xtr[j * dim + d] - org[d]);
    };
    // Theta at squared distance d2 (no nugget): in FP64 the table-driven exp and the Newton
    // square root (few FP64-pipe operations, about 2 ulp)
    auto theta = [&](T d2) -> T {
        if constexpr (F64)
            return matern_d2_fast(kp, d2, tab);
        else
            return matern<T>(kp, sic_sqrt(d2));
    };
    if constexpr (F64) {
        exp_table_fill(tab, kp.s2);
        __syncthreads();
    }
    auto unconditional = [&]() {
        for (long long j = j0; j < n; j += jstep) {
            T d2 = (T)0;
            for (int d = 0; d < dim; ++d) {
                T df = (T)(xtr[j * dim + d] - org[d]);
                d2 += df * df;
            }
            var[j] = kp.s2 + kp.nugget;
            cov[j] = theta(d2);
        }
    };
    unconditional();
    double vt = (double)(kp.s2 + kp.nugget);
    if (j0 == 0) out_var[0] = vt;
    // FP32 score key of a row (0: not a candidate)
    auto key_of = [&](long long j) -> unsigned {
        const T v = var[j];
        if (!(v >= floor_)) return 0u;
        const float c = fx_f32(fabs((double)cov[j]), 2 * e);
        return __float_as_uint(__fdividef(c * c, fx_f32((double)v, 2 * e))) + 1u;
    };
    auto warp_best = [&](Best<T>& b) {
        T s = b.score;
        long long i = b.idx;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            const T os = __shfl_xor_sync(FULL, s, off);
            const long long oi = __shfl_xor_sync(FULL, i, off);
            if (better(os, oi, s, i)) {
                s = os;
                i = oi;
            }
        }
        const int src = __ffs(__ballot_sync(FULL, b.idx == i)) - 1;
        b = Best<T>{s, __shfl_sync(FULL, b.var, src), __shfl_sync(FULL, b.cov, src), i};
    };
    bool rows64 = false;  // (FP64) from the start once more, the factor's rows in FP64
    int t = 0, round = 0;
    for (; t < k; ++t, ++round) {
        Best<T> b{NEG, (T)0, (T)0, NONE};
        unsigned lim = 1u, mine = 0u;
        if constexpr (F64) {
            for (long long j = j0; j < n; j += jstep) mine = max(mine, key_of(j));
            const unsigned m = __reduce_max_sync(FULL, mine);
            if (lane == 0) wkey[warp] = m;
            __syncthreads();
            const unsigned gk = __reduce_max_sync(FULL, lane < nw ? wkey[lane] : 0u);
            // within 2^-18 of the block's largest, or every live row where FP32 cannot tell (or it is not finite)
            if (gk > 0x0da24260u && gk < 0x7f000000u) lim = gk - 32u;  // 1e-30
        }
        // the exact scores (FP64: of those rows only), the block's best
        if (!F64 || __any_sync(FULL, mine >= lim)) {
            if (!F64 || mine >= lim)
                for (long long j = j0; j < n; j += jstep) {
                    const T v = var[j];
                    if (v >= floor_ && (!F64 || key_of(j) >= lim)) {
                        const T c = cov[j];
                        const T s = c * c / v;
                        if (better(s, j, b.score, b.idx)) b = Best<T>{s, v, c, j};
                    }
                }
            __syncwarp();
            warp_best(b);
        }
        if (lane == 0) wbest[warp] = b;
        __syncthreads();
        if (warp == 0) {
            b = lane < nw ? wbest[lane] : Best<T>{NEG, (T)0, (T)0, NONE};
            warp_best(b);
            int ok = 1;
            if (gridDim.x > 1) {
                Best<T>* all = bests + (round & 1) * gridDim.x;
                if (lane == 0) {
                    all[blockIdx.x] = b;
                    ok = grid_wait(count, (unsigned)gridDim.x * (unsigned)(round + 1));
                }
                ok = __shfl_sync(FULL, ok, 0);
                b = Best<T>{NEG, (T)0, (T)0, NONE};
                for (int i = lane; ok && i < (int)gridDim.x; i += 32) {
                    const Best<T> o{__ldcg(&all[i].score), __ldcg(&all[i].var), __ldcg(&all[i].cov), __ldcg(&all[i].idx)};
                    if (better(o.score, o.idx, b.score, b.idx)) b = o;
                }
                warp_best(b);
            }
            if (lane == 0) {
                s_ok = ok;
                const bool go = ok && b.idx != NONE && b.score > (T)0;
                s_q = go ? b.idx : NONE;
                s_small = F64 && go && !rows64 && exponent_of((double)b.cov) < 2 * e - FX_COV_BITS;
                if (go) {
                    if constexpr (F64)
                        s_rs = rsqrt_newton(b.var);
                    else
                        s_rs = (T)1 / sic_sqrt(b.var);
                    s_ut = b.cov * s_rs;
                }
            }
        }
        __syncthreads();
        if (!s_ok) {
            if (tid == 0) record_error(st, SIC_ERR_TIMEOUT, -1);
            break;
        }
        const long long q = s_q;
        if (q == NONE) break;
        if (F64 && s_small) {  // every block decides the same from the same best
            rows64 = true;
            unconditional();
            vt = (double)(kp.s2 + kp.nugget);
            t = -1;
            continue;
        }
        const T rs = s_rs, ut = s_ut;
        T qx[3] = {(T)0, (T)0, (T)0};
        for (int d = 0; d < dim; ++d) qx[d] = coord(q, d);
        for (int tau = tid; tau < t; tau += blockDim.x) piv[tau] = __ldcg(&F[(long long)tau * n + q]);
        __syncthreads();
        long long M = 0;
        int h = 0;
        if constexpr (F64) fx_factor(rs, e, M, h);
        for (long long j = j0; j < n; j += jstep) {
            const T vj = var[j];
            if (!(vj != NEG)) continue;
            T d2 = (T)0;
            for (int d = 0; d < dim; ++d) {
                T df = coord(j, d) - qx[d];
                d2 += df * df;
            }
            T num = theta(d2);
            if (j == q) num += kp.nugget;
            T u;
            if (F64 && rows64) {
                for (int tau = 0; tau < t; ++tau) num = fma(-F[(long long)tau * n + j], piv[tau], num);
                u = num * rs;
                if (t + 1 < k) F[(long long)t * n + j] = u;
            } else if constexpr (F64) {
                long long sum = 0, ux = 0;
                for (int c0 = 0; c0 < t; c0 += 256) {  // (the cross sums stay in 64 bits over 256 columns)
                    const int c1 = min(t, c0 + 256);
                    FxSum a{0, 0};
                    for (int c = c0; c < c1; c += 8) {  // eight loads in flight
                        int2 f[8];
#pragma unroll
                        for (int i = 0; i < 8; ++i) f[i] = Fx[(long long)min(c + i, c1 - 1) * n + j];
#pragma unroll
                        for (int i = 0; i < 8; ++i)
                            if (c + i < c1) a.add(f[i], px[c + i]);
                    }
                    sum += a.value();
                }
                if (!not_finite(num)) ux = fx_mul(fx_of_positive(num, FXS - 2 * e) - sum, M, h);
                if (t + 1 < k) Fx[(long long)t * n + j] = fx_split(ux);  // the last column has no reader
                u = not_finite(num) ? NAN : fx_to_double(ux, e - FXS);   // (never a candidate again)
            } else {
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
                u = num * rs;
                if (t + 1 < k) F[(long long)t * n + j] = u;  // the last column has no reader
            }
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
// size, so small n spreads over the SMs in blocks of 64 rows; from 152 x 512 rows on further rows are
// strided.
template <typename T>
sic_status launch_single(sic_handle* h, const double* x_train, int64_t n, const double* x_target,
                         const sic_kernel* kp, int32_t k, int32_t* out_idx, double* out_var, int32_t* out_count,
                         void* ws, cudaStream_t s) {
    auto kern = k_select_single<T>;
    const size_t smem = sizeof(T) * (size_t)k;
    if (smem > 40 * 1024)
        SIC_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    const long long per = (n + h->num_sms - 1) / h->num_sms;
    const int nt = per <= 64 ? 64 : (per <= 128 ? 128 : (per <= 256 ? 256 : 512));
    int grid = persistent_grid(h, kern, nt, smem, (n + nt - 1) / nt);
    if (grid > h->num_sms) grid = h->num_sms;
    T* w = (T*)ws;
    int dim = kp->dim;
    long long nn = n;
    KP<T> kpt = make_kp<T>(*kp);
    T fl = (T)sic_floor_of(kp);
    int e = fx_exponent(kp);
    unsigned* count = scratch_of<T>(w, n, k);
    if (grid > 1) SIC_CUDA_TRY(cudaMemsetAsync(count, 0, 16, s));
    for (;;) {
        if (grid == 1) {
            kern<<<1, nt, smem, s>>>(x_train, nn, dim, x_target, kpt, fl, e, k, out_idx, out_var, out_count, w, count,
                                 h->d_status);
            break;
        }
        void* args[] = {&x_train, &nn, &dim, &x_target, &kpt, &fl, &e, &k, &out_idx, &out_var, &out_count, &w, &count,
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
