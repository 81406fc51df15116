// Preconditioned conjugate gradients on (Theta + shift I) x = b with the sparse factor
// as preconditioner M^{-1} = L L^T (the use of the factor studied in Section 6.4).
//
// FP32 mode, up to two right-hand sides and many points (k_matvec_f32; else matvec_tc.cu): y = (Theta + shift I) x without
// forming Theta.  The kernel entries are FP32 (a fixed, symmetric rounding of Theta: K(|x_i - x_j|) is evaluated
// identically for (i, j) and (j, i)); x is carried as an unevaluated sum of two FP32 numbers (hi + lo) and the
// products are summed as a double-FP32 pair with the error-free transformations TwoProduct (by fma) and
// TwoSum (Knuth), 256 terms at a time, then in FP64 -- so the product is accurate to a few 1e-15 of sum |K x| (typically) and
// CG can reach small residuals.  k_matvec_f64 is FP64 throughout (reference mode; the kernel entries by the fill's table-driven exp
// and Newton square root, about 2 ulp).  The diagonal adds the nugget and the shift in FP64.
// The CG vector updates and dot products are fused kernels with fixed-order reductions
// (bit-reproducible); the scalars alpha and beta are formed on the device per RHS.
// The iteration loop runs on the host (C++), reading back the residual norms each step.
#include <math.h>

#include <vector>

#include "matvec_f32.cuh"

namespace {

constexpr int MV_NT = 128;   // FP64: target rows per CTA
constexpr int RED_TILE = 4096;

// One or two right-hand sides (matvec_f32.cuh)
template <int NR>
__global__ void __launch_bounds__(32 * MVF_WARPS, 2) k_matvec_f32(const double* __restrict__ pts, long long n, int dim,
                                                                  KP<float> kp, double diag_extra,
                                                                  const double* __restrict__ x, double* __restrict__ y,
                                                                  int nrhs) {
    __shared__ MvfSmem<NR> sm;
    const long long row0 = blockIdx.x * (long long)MVF_ROWS;
    mvf_tile<NR>(
        sm, pts, n, dim, x, nrhs, row0,
        [&](float2 d2) { return make_float2(matern<float>(kp, sqrtf(d2.x)), matern<float>(kp, sqrtf(d2.y))); },
        [](int) { return 1.0; });
    for (int e = threadIdx.x; e < MVF_ROWS * nrhs; e += 32 * MVF_WARPS) {
        const int row = e / nrhs, r = e - row * nrhs;
        const long long i = row0 + row;
        if (i < n) y[i * nrhs + r] = sm.sum(row, r) + diag_extra * x[i * nrhs + r];
    }
}

template <int NR>
__global__ void __launch_bounds__(MV_NT) k_matvec_f64(const double* __restrict__ pts, long long n, int dim,
                                                      KP<double> kp, double diag_extra, const double* __restrict__ x,
                                                      double* __restrict__ y, int nrhs) {
    __shared__ double sx[MV_TILE], sy[MV_TILE], sz[MV_TILE];
    __shared__ double sv[MV_TILE * NR];
    __shared__ double tab[EXP_TAB];  // s2 2^(j/256) for the table-driven exp
    exp_table_fill(tab, kp.s2);      // ordered before use by the tile loop's barrier
    const long long i = blockIdx.x * (long long)MV_NT + threadIdx.x;
    const bool live = i < n;
    double xi = 0, yi = 0, zi = 0;
    if (live) {
        xi = pts[i * dim];
        if (dim > 1) yi = pts[i * dim + 1];
        if (dim > 2) zi = pts[i * dim + 2];
    }
    double acc[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r) acc[r] = 0.0;
    for (long long j0 = 0; j0 < n; j0 += MV_TILE) {
        __syncthreads();
        for (int t = threadIdx.x; t < MV_TILE; t += MV_NT) {
            const long long j = j0 + t;
            const bool ok = j < n;
            sx[t] = ok ? pts[j * dim] : 0.0;
            sy[t] = (ok && dim > 1) ? pts[j * dim + 1] : 0.0;
            sz[t] = (ok && dim > 2) ? pts[j * dim + 2] : 0.0;
#pragma unroll
            for (int r = 0; r < NR; ++r) sv[t * NR + r] = (ok && r < nrhs) ? x[j * nrhs + r] : 0.0;
        }
        __syncthreads();
        const int cnt = (int)min((long long)MV_TILE, n - j0);
        double part[NR];
#pragma unroll
        for (int r = 0; r < NR; ++r) part[r] = 0.0;
        for (int t = 0; t < cnt; ++t) {
            const double dx = xi - sx[t], dy = yi - sy[t], dz = zi - sz[t];
            const double kv = matern_d2_fast(kp, fma(dz, dz, fma(dy, dy, dx * dx)), tab);
#pragma unroll
            for (int r = 0; r < NR; ++r) part[r] = fma(kv, sv[t * NR + r], part[r]);
        }
#pragma unroll
        for (int r = 0; r < NR; ++r) acc[r] += part[r];
    }
    if (live) {
#pragma unroll
        for (int r = 0; r < NR; ++r)
            if (r < nrhs) y[i * nrhs + r] = acc[r] + diag_extra * x[i * nrhs + r];
    }
}

// partial[b * nrhs + r] = sum over rows of tile b of a[row][r] * c[row][r]
__global__ void __launch_bounds__(256) k_dot_tiles(const double* __restrict__ a, const double* __restrict__ c,
                                                   long long n, int nrhs, double* __restrict__ partial) {
    __shared__ double s[256];
    const long long base = blockIdx.x * (long long)RED_TILE;
    for (int r = 0; r < nrhs; ++r) {
        double acc = 0.0;
        for (int t = threadIdx.x; t < RED_TILE; t += 256) {
            const long long i = base + t;
            if (i < n) acc = fma(a[i * nrhs + r], c[i * nrhs + r], acc);
        }
        s[threadIdx.x] = acc;
        __syncthreads();
        for (int off = 128; off > 0; off >>= 1) {
            if (threadIdx.x < off) s[threadIdx.x] += s[threadIdx.x + off];
            __syncthreads();
        }
        if (threadIdx.x == 0) partial[blockIdx.x * nrhs + r] = s[0];
        __syncthreads();
    }
}

__global__ void k_dot_final(const double* __restrict__ partial, long long nb, int nrhs, double* __restrict__ out) {
    const int r = threadIdx.x;
    if (r >= nrhs) return;
    double s = 0.0;
    for (long long b = 0; b < nb; ++b) s += partial[b * nrhs + r];
    out[r] = s;
}

// x += alpha p, r -= alpha q with alpha = rz / pq (0 for converged right-hand sides)
__global__ void k_cg_xr(double* __restrict__ x, double* __restrict__ res, const double* __restrict__ p,
                        const double* __restrict__ q, const double* __restrict__ rz, const double* __restrict__ pq,
                        const int* __restrict__ active, long long n, int nrhs) {
    const long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (e >= n * nrhs) return;
    const int r = (int)(e % nrhs);
    if (!active[r]) return;
    const double alpha = rz[r] / pq[r];
    x[e] = fma(alpha, p[e], x[e]);
    res[e] = fma(-alpha, q[e], res[e]);
}

// p = z + beta p with beta = rz_new / rz; then rz = rz_new
__global__ void k_cg_p(double* __restrict__ p, const double* __restrict__ z, const double* __restrict__ rz_new,
                       const double* __restrict__ rz, const int* __restrict__ active, long long n, int nrhs) {
    const long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (e >= n * nrhs) return;
    const int r = (int)(e % nrhs);
    if (!active[r]) return;
    p[e] = fma(rz_new[r] / rz[r], p[e], z[e]);
}

__global__ void k_copy_rz(double* __restrict__ rz, const double* __restrict__ rz_new, int nrhs) {
    if (threadIdx.x < nrhs) rz[threadIdx.x] = rz_new[threadIdx.x];
}

template <int NR>
void matvec_f64(cudaStream_t s, const double* pts, long long n, int dim, const sic_kernel* kp, double shift,
                const double* x, double* y, int nrhs) {
    k_matvec_f64<NR><<<(unsigned)((n + MV_NT - 1) / MV_NT), MV_NT, 0, s>>>(pts, n, dim, make_kp<double>(*kp),
                                                                         kp->nugget + shift, x, y, nrhs);
}

sic_status matvec_any(sic_handle* h, cudaStream_t s, const double* pts, long long n, int dim, const sic_kernel* kp,
                      double shift, sic_precision prec, const double* x, double* y, int nrhs) {
    if (prec == SIC_FP64) {
        if (nrhs == 1) matvec_f64<1>(s, pts, n, dim, kp, shift, x, y, nrhs);
        else if (nrhs <= 2) matvec_f64<2>(s, pts, n, dim, kp, shift, x, y, nrhs);
        else if (nrhs <= 4) matvec_f64<4>(s, pts, n, dim, kp, shift, x, y, nrhs);
        else matvec_f64<8>(s, pts, n, dim, kp, shift, x, y, nrhs);
        return SIC_OK;
    }
    // The tensor-core kernel's time does not depend on the right-hand sides (N = 50,001: 7.8 ms for 3, 8.0 for 8),
    // this one's does (5.2 ms for 1 or 2); at few rows the former also spreads a row tile over more CTAs (one right-hand
    // side: N = 4096 0.116 against 0.138 ms, 8192 0.260 against 0.268, 10,000 0.476 against 0.417) and takes any
    // scale of x.
    if (nrhs > 2 || n < 12288) return matvec_tc(h, pts, n, kp, shift, x, y, nrhs, s);
    k_matvec_f32<2><<<(unsigned)((n + MVF_ROWS - 1) / MVF_ROWS), 32 * MVF_WARPS, 0, s>>>(
        pts, n, dim, make_kp<float>(*kp), kp->nugget + shift, x, y, nrhs);
    return SIC_OK;
}

void dots(cudaStream_t s, const double* a, const double* c, long long n, int nrhs, double* partial, double* out) {
    long long nb = (n + RED_TILE - 1) / RED_TILE;
    k_dot_tiles<<<(unsigned)nb, 256, 0, s>>>(a, c, n, nrhs, partial);
    k_dot_final<<<1, 32, 0, s>>>(partial, nb, nrhs, out);
}

// workspace layout (doubles): r, z, p, q (n x nrhs each), partial (nb x nrhs), scalars
struct PcgWs {
    long long n;
    int nrhs;
    long long nb() const { return (n + RED_TILE - 1) / RED_TILE; }
    long long vec() const { return n * nrhs; }
    long long size() const { return 4 * vec() + nb() * nrhs + 8 * 8 + n * nrhs /* LL^T intermediate */ + 8; }
};

}  // namespace

extern "C" sic_status sic_matern_matvec(sic_handle* h, const double* pts, int64_t n, const sic_kernel* kp,
                                        double shift, sic_precision prec, const double* x, double* y, int32_t nrhs,
                                        void* stream) {
    if (!h || !pts || n < 1 || !sic_valid_kernel(kp) || !x || !y || nrhs < 1) return SIC_ERR_INVALID;
    if (prec != SIC_FP64 && prec != SIC_FP32_MIXED) return SIC_ERR_INVALID;
    if (nrhs > 8) return SIC_ERR_UNSUPPORTED;
    SIC_CUDA_TRY(cudaSetDevice(h->device));
    const sic_status e = matvec_any(h, (cudaStream_t)stream, pts, n, kp->dim, kp, shift, prec, x, y, nrhs);
    if (e != SIC_OK) return e;
    SIC_CUDA_TRY(cudaGetLastError());
    return SIC_OK;
}

extern "C" sic_status sic_pcg_workspace(int64_t n, int32_t nrhs, size_t* bytes) {
    if (!bytes || n < 1 || nrhs < 1) return SIC_ERR_INVALID;
    PcgWs W{n, nrhs};
    *bytes = sizeof(double) * (size_t)W.size() + 64;
    return SIC_OK;
}

extern "C" sic_status sic_apply_factor(sic_handle* h, int64_t n, const int64_t* col_ptr, const int32_t* row_idx,
                                       const double* val, sic_op op, const double* x, double* y, int32_t nrhs,
                                       void* ws, size_t ws_bytes, void* stream);

extern "C" sic_status sic_pcg_solve(sic_handle* h, const double* pts, int64_t n, const sic_kernel* kp, double shift,
                                    sic_precision prec, const int64_t* col_ptr, const int32_t* row_idx, const double* val,
                                    const double* b, double* x, int32_t nrhs, double tol, int32_t max_iter,
                                    int32_t* iters, double* relres, void* ws, size_t ws_bytes, void* stream) {
    if (!h || !pts || n < 1 || !sic_valid_kernel(kp) || !b || !x || nrhs < 1 || !(tol > 0) || max_iter < 0 ||
        !iters || !relres || !ws)
        return SIC_ERR_INVALID;
    if (prec != SIC_FP64 && prec != SIC_FP32_MIXED) return SIC_ERR_INVALID;
    if (nrhs > 8) return SIC_ERR_UNSUPPORTED;
    if ((col_ptr != nullptr) != (row_idx != nullptr) || (col_ptr != nullptr) != (val != nullptr))
        return SIC_ERR_INVALID;
    PcgWs W{n, nrhs};
    if (ws_bytes < sizeof(double) * (size_t)W.size()) return SIC_ERR_INVALID;
    SIC_CUDA_TRY(cudaSetDevice(h->device));
    cudaStream_t s = (cudaStream_t)stream;
    double* base = (double*)ws;
    double* r = base;
    double* z = r + W.vec();
    double* p = z + W.vec();
    double* q = p + W.vec();
    double* partial = q + W.vec();
    double* sc = partial + W.nb() * nrhs;  // 8 x 8 scalars
    double* rz = sc, *pq = sc + 8, *rzn = sc + 16, *rr = sc + 24, *bb = sc + 32;
    int* active = (int*)(sc + 40);
    double* llt = sc + 64;  // n x nrhs intermediate of L L^T
    const size_t vb = sizeof(double) * (size_t)W.vec();
    const unsigned eb = (unsigned)((W.vec() + 255) / 256);
    auto precond = [&](const double* in, double* out) -> sic_status {
        if (!col_ptr) return cudaMemcpyAsync(out, in, vb, cudaMemcpyDeviceToDevice, s) == cudaSuccess ? SIC_OK
                                                                                                  : SIC_ERR_CUDA;
        return sic_apply_factor(h, n, col_ptr, row_idx, val, SIC_OP_LLT, in, out, nrhs, llt, vb, stream);
    };
    // x = 0, r = b
    SIC_CUDA_TRY(cudaMemsetAsync(x, 0, vb, s));
    SIC_CUDA_TRY(cudaMemcpyAsync(r, b, vb, cudaMemcpyDeviceToDevice, s));
    dots(s, b, b, n, nrhs, partial, bb);
    sic_status e = precond(r, z);
    if (e != SIC_OK) return e;
    SIC_CUDA_TRY(cudaMemcpyAsync(p, z, vb, cudaMemcpyDeviceToDevice, s));
    dots(s, r, z, n, nrhs, partial, rz);
    std::vector<int> act(nrhs, 1);
    std::vector<double> hbb(nrhs), hrr(nrhs);
    SIC_CUDA_TRY(cudaMemcpyAsync(hbb.data(), bb, sizeof(double) * nrhs, cudaMemcpyDeviceToHost, s));
    SIC_CUDA_TRY(cudaStreamSynchronize(s));
    for (int c = 0; c < nrhs; ++c) {
        iters[c] = 0;
        relres[c] = hbb[c] > 0 ? 1.0 : 0.0;
        if (!(hbb[c] > 0)) act[c] = 0;
    }
    for (int it = 1; it <= max_iter; ++it) {
        bool any = false;
        for (int c = 0; c < nrhs; ++c) any |= act[c] != 0;
        if (!any) break;
        SIC_CUDA_TRY(cudaMemcpyAsync(active, act.data(), sizeof(int) * nrhs, cudaMemcpyHostToDevice, s));
        e = matvec_any(h, s, pts, n, kp->dim, kp, shift, prec, p, q, nrhs);
        if (e != SIC_OK) return e;
        dots(s, p, q, n, nrhs, partial, pq);
        k_cg_xr<<<eb, 256, 0, s>>>(x, r, p, q, rz, pq, active, n, nrhs);
        dots(s, r, r, n, nrhs, partial, rr);
        SIC_CUDA_TRY(cudaMemcpyAsync(hrr.data(), rr, sizeof(double) * nrhs, cudaMemcpyDeviceToHost, s));
        SIC_CUDA_TRY(cudaStreamSynchronize(s));
        for (int c = 0; c < nrhs; ++c) {
            if (!act[c]) continue;
            iters[c] = it;
            relres[c] = sqrt(hrr[c] / hbb[c]);
            if (relres[c] < tol) act[c] = 0;
        }
        SIC_CUDA_TRY(cudaMemcpyAsync(active, act.data(), sizeof(int) * nrhs, cudaMemcpyHostToDevice, s));
        e = precond(r, z);
        if (e != SIC_OK) return e;
        dots(s, r, z, n, nrhs, partial, rzn);
        k_cg_p<<<eb, 256, 0, s>>>(p, z, rzn, rz, active, n, nrhs);
        k_copy_rz<<<1, 32, 0, s>>>(rz, rzn, nrhs);
    }
    SIC_CUDA_TRY(cudaGetLastError());
    SIC_CUDA_TRY(cudaStreamSynchronize(s));
    return SIC_OK;
}
