// KL-optimal fill of single columns (eq. L_col) with at most 48 picks: one warp per column.
//
// The picks, latest first, and the target last are factored Theta = F F^T by a left-looking Cholesky in
// fixed point (as select_fx.cu's rows, with two more bits, since here the factor itself is the result: entries
// round(F 2^(60 - e)) = H 2^30 + L, sums of H H', H L' and L H' in three 64-bit words, quotients by the full
// 128-bit product).  Against 128-bit arithmetic on the same Theta the columns' values are off by (rms, of their
// largest) 1.7e-13 at nugget 1e-8, k = 16 and 1.4e-16 at nugget 1e-6, k = 32 in 3-D, where the FP64 panels of k_fill are off
// by 5.9e-12 and 2.8e-15; what remains of either is Theta's own rounding.  Lane i owns the picks i and i + 32; the lower triangle of the picks lies in shared memory as
// [pair of columns][row] of int4, triangular; the target's row is spread over the lanes by column, its products
// added by warp reductions (three redux of 26-bit limbs).  The column is x = F^-T e_last: a back substitution in
// FP64, b_i -= F_li x_l, lane = entry; log v = log of the target's pivot, 32 columns' logarithms at a time.
//
// The fixed point is absolute: a kernel entry below 2^-36 of the variance would keep fewer than 24 bits, one below 2^-60
// none (points many length scales apart).  A column with such an entry is formed in FP64 by the same steps.
//
// The CTA-wide fill (k_fill) spends 5 warps and two barriers per panel on a 33 x 33 block: 65,536 columns of 32 picks
// 4.19 ms; here 2.3 ms.  Bound: the FP64 pipe (Theta's 8
// operations per entry, the substitution: about 300 warp instructions per column of 32 picks).
#include <limits.h>

#include "fx.cuh"

namespace {

constexpr int WARPS = 4;
constexpr unsigned FULL = 0xffffffffu;

// pair p of columns holds rows 2p .. N - 1
__host__ __device__ __forceinline__ int pair_base(int p, int N) { return p * N - p * (p - 1); }

// 8-byte words of one warp: the triangle (int4), coordinates, sorted positions
__host__ __device__ inline int warp_words(int k) {
    const int pairs = (k + 1) / 2;
    return 2 * pair_base(pairs, k + (k & 1)) + 3 * (k + 1) + (k + 2) / 2 + 1;
}

// sum over the warp of 64-bit values (below 2^63 itself)
__device__ __forceinline__ long long warp_sum(long long v) {
    const unsigned a = (unsigned)v & 0x3ffffffu, b = (unsigned)(v >> 26) & 0x3ffffffu;
    const int c = (int)(v >> 52);
    return (long long)__reduce_add_sync(FULL, a) + ((long long)__reduce_add_sync(FULL, b) << 26) +
           ((long long)__reduce_add_sync(FULL, c) << 52);
}

// S sets of 32 picks
template <int S>
__global__ void __launch_bounds__(32 * WARPS, S == 1 ? 9 : 5) k_fill_columns(
    const double* __restrict__ pts, int dim, KP<double> kp, int e, const int32_t* __restrict__ sel_idx,
    const int32_t* __restrict__ sel_count, int k, long long n, long long col0, long long n_cols,
    const long long* __restrict__ col_ptr, long long base, int32_t* __restrict__ row_idx, double* __restrict__ val,
    double* __restrict__ logv, int words, DevStatus* st) {
    extern __shared__ __align__(16) long long sm64[];
    double* tab = reinterpret_cast<double*>(sm64);  // s2 2^(j/256)
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int N = k + (k & 1);
    long long* mine = sm64 + EXP_TAB + (long long)warp * words;
    int4* F = reinterpret_cast<int4*>(mine);
    long long* xf = mine + 2 * pair_base((k + 1) / 2, N);  // 3 x (k + 1) coordinates, fixed point
    int* pos = reinterpret_cast<int*>(xf + 3 * (k + 1));   // k + 1 positions in the order
    exp_table_fill(tab, kp.s2);
    __syncthreads();
    // entry of column j, row i >= j
    auto entry = [&](int j, int i) -> int2* {
        return reinterpret_cast<int2*>(F + pair_base(j >> 1, N) + i - 2 * (j >> 1)) + (j & 1);
    };
    const long long diag_x = fx_of_positive(kp.s2 + kp.nugget, FCS - 2 * e);
    const long long nw = (long long)gridDim.x * WARPS;
    double pend = 1.0;          // a column's target pivot, held by one lane
    long long pend_col = -1;
    int held = 0;
    auto flush = [&]() {
        if (pend_col >= 0) logv[pend_col] = log(pend);
        pend_col = -1;
        held = 0;
    };
    for (long long c = blockIdx.x * (long long)WARPS + warp; c < n_cols; c += nw) {
        const long long tgt = col0 + c;
        const int cnt = sel_count[c];
        if (cnt < 0 || cnt > k || tgt >= n) {
            if (lane == 0) record_error(st, SIC_ERR_INVALID, c);
            continue;
        }
        // ---- the picks latest first, the target last; distinct positions after the target ----
        __syncwarp();
        bool bad = lane == 0 && col_ptr[c + 1] - col_ptr[c] != (long long)cnt + 1;
        int v[S];
#pragma unroll
        for (int s = 0; s < S; ++s) {
            v[s] = lane + 32 * s < cnt ? sel_idx[c * k + lane + 32 * s] : 0x7fffffff;
            if (lane + 32 * s < cnt && (v[s] <= tgt || v[s] >= n)) bad = true;
        }
        int later[S];
#pragma unroll
        for (int s = 0; s < S; ++s) later[s] = 0;
#pragma unroll
        for (int q = 0; q < S; ++q)
            for (int l = 0; l < min(32, cnt - 32 * q); ++l) {
                const int w = __shfl_sync(FULL, v[q], l);
#pragma unroll
                for (int s = 0; s < S; ++s) {
                    later[s] += w > v[s];
                    if (w == v[s] && l + 32 * q != lane + 32 * s) bad = true;
                }
            }
        if (__any_sync(FULL, bad)) {
            if (lane == 0) record_error(st, SIC_ERR_INVALID, c);
            continue;
        }
#pragma unroll
        for (int s = 0; s < S; ++s)
            if (lane + 32 * s < cnt) pos[later[s]] = v[s];
        if (lane == 0) pos[cnt] = (int)tgt;
        __syncwarp();
        // ---- coordinates in fixed point at the largest exponent per dimension ----
        int E[3] = {0, 0, 0};
        for (int d = 0; d < dim; ++d) {
            int m = 0;
            for (int i = lane; i <= cnt; i += 32) m = max(m, (__double2hiint(pts[(long long)pos[i] * dim + d]) >> 20) & 0x7ff);
            E[d] = __reduce_max_sync(FULL, m);
            for (int i = lane; i <= cnt; i += 32) xf[d * (k + 1) + i] = fx_coord(pts[(long long)pos[i] * dim + d], E[d]);
        }
        __syncwarp();
        bool small_ = false;  // an entry that the fixed point holds to fewer than 24 bits
        auto theta64 = [&](int i, int j) -> double {
            return matern_d2_fast(kp, fx_dist2(xf, k + 1, dim, i, j, E[0], E[1], E[2]), tab);
        };
        auto theta = [&](int i, int j) -> long long {
            const double d2 = fx_dist2(xf, k + 1, dim, i, j, E[0], E[1], E[2]);
            const double th = matern_d2_fast(kp, d2, tab);
            small_ = small_ || (exponent_of(th) < 2 * e - 36 && __double_as_longlong(th) != 0LL);
            // (without a nugget coincident points make Theta singular, whatever the factorisation's rounding)
            return not_finite(th) || (d2 == 0.0 && !(kp.nugget > 0.0)) ? LLONG_MIN : fx_of_positive(th, FCS - 2 * e);
        };
        // ---- Theta of the picks into the triangle (flat), the target's row into the lanes ----
        bool nan_ = false;
        {
            int i = (int)((sqrtf(8.0f * (float)lane + 1.0f) - 1.0f) * 0.5f);
            while (i * (i + 1) / 2 > lane) --i;
            while ((i + 1) * (i + 2) / 2 <= lane) ++i;
            int j = lane - i * (i + 1) / 2;
            while (i < cnt) {
                const long long t = i == j ? diag_x : theta(i, j);
                nan_ = nan_ || t == LLONG_MIN;
                *reinterpret_cast<long long*>(entry(j, i)) = t;
                j += 32;
                while (j > i) {
                    j -= i + 1;
                    ++i;
                }
            }
        }
        long long tr[S];  // the target's row: Theta, then F, by column
        double rsd[S];    // 1 / F_jj of the own columns
#pragma unroll
        for (int s = 0; s < S; ++s) {
            tr[s] = lane + 32 * s < cnt ? theta(cnt, lane + 32 * s) : 0;
            nan_ = nan_ || tr[s] == LLONG_MIN;
            rsd[s] = 0.0;
        }
        bool npd = __any_sync(FULL, nan_);
        const bool wide = __any_sync(FULL, small_);
        double b[S];  // the target's row in FP64, then the column
        double d = 0.0;
        if (wide) {
            // ---- the same in FP64 (points many length scales apart): factor entries as doubles in the same words ----
            auto at = [&](int j, int i) -> double& { return *reinterpret_cast<double*>(entry(j, i)); };
            __syncwarp();
            int i = (int)((sqrtf(8.0f * (float)lane + 1.0f) - 1.0f) * 0.5f);
            while (i * (i + 1) / 2 > lane) --i;
            while ((i + 1) * (i + 2) / 2 <= lane) ++i;
            int j = lane - i * (i + 1) / 2;
            while (i < cnt) {
                at(j, i) = i == j ? kp.s2 + kp.nugget : theta64(i, j);
                j += 32;
                while (j > i) {
                    j -= i + 1;
                    ++i;
                }
            }
#pragma unroll
            for (int s = 0; s < S; ++s) b[s] = lane + 32 * s < cnt ? theta64(cnt, lane + 32 * s) : 0.0;
            __syncwarp();
            auto sum64 = [&](double v) {
#pragma unroll
                for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(FULL, v, off);
                return v;
            };
            for (int c = 0; c < cnt && !npd; ++c) {
                double num[S], part = 0.0;
#pragma unroll
                for (int s = 0; s < S; ++s) {
                    const int r = lane + 32 * s;
                    const bool own = r >= c && r < cnt;
                    num[s] = own ? at(c, r) : 0.0;
                    for (int p = 0; p < c; ++p) num[s] = fma(-at(p, own ? r : c), at(p, c), num[s]);
                    if (r < c) part = fma(b[s], at(r, c), part);
                }
                const double dot = sum64(part);
                double dc = num[0];
#pragma unroll
                for (int s = 1; s < S; ++s) dc = (c >> 5) == s ? num[s] : dc;
                dc = __shfl_sync(FULL, dc, c & 31);
                npd = !(dc > 0.0);
                const double rs = rsqrt_newton(npd ? 1.0 : dc);
                __syncwarp();
#pragma unroll
                for (int s = 0; s < S; ++s) {
                    const int r = lane + 32 * s;
                    if (r >= c && r < cnt) at(c, r) = num[s] * rs;
                    if (r == c) {
                        rsd[s] = rs;
                        b[s] = (b[s] - dot) * rs;
                    }
                }
                __syncwarp();
            }
            double part = 0.0;
#pragma unroll
            for (int s = 0; s < S; ++s) part = fma(b[s], b[s], part);
            d = kp.s2 + kp.nugget - sum64(part);
            npd = npd || !(d > 0.0);
        }
        __syncwarp();
        // ---- left-looking Cholesky ----
        for (int j = 0; j < cnt && !npd && !wide; ++j) {
            const int pairs = j >> 1;
            FcSum a[S];
#pragma unroll
            for (int s = 0; s < S; ++s) a[s].hh = a[s].c1 = a[s].c2 = 0;
            long long num[S];
            const int s0 = j >> 5;  // sets below have no rows left
            for (int p = 0; p < pairs; ++p) {
                const int4* Fp = F + pair_base(p, N) - 2 * p;
                const int4 q = Fp[j];
#pragma unroll
                for (int s = 0; s < S; ++s)
                    if (s >= s0) {
                        const int i = lane + 32 * s;
                        a[s].add2(Fp[i >= j && i < cnt ? i : j], q);
                    }
            }
            if (j & 1) {  // the column before, alone in its pair
                const int2 q = *entry(j - 1, j);
#pragma unroll
                for (int s = 0; s < S; ++s)
                    if (s >= s0) {
                        const int i = lane + 32 * s;
                        a[s].add(*entry(j - 1, i >= j && i < cnt ? i : j), q);
                    }
            }
            // the target's products with row j, one column per lane
            long long part = 0;
#pragma unroll
            for (int s = 0; s < S; ++s) {
                const int t = lane + 32 * s;
                if (t < j) {
                    FcSum b{0, 0, 0};
                    b.add(fc_split(tr[s]), *entry(t, j));
                    part += b.hh * 2 + ((b.c1 + b.c2) >> 29);  // one more bit for the sum
                }
            }
            const long long dot = warp_sum(part);
#pragma unroll
            for (int s = 0; s < S; ++s) {
                const int i = lane + 32 * s;
                num[s] = (i >= j && i < cnt) ? *reinterpret_cast<const long long*>(entry(j, i)) - a[s].value() : 0;
            }
            // the pivot, from the lane that owns row j
            long long dj = num[0];
#pragma unroll
            for (int s = 1; s < S; ++s) dj = s0 == s ? num[s] : dj;
            dj = __shfl_sync(FULL, dj, j & 31);
            if (dj <= 0) {
                npd = true;
                break;
            }
            long long M;
            int h;
            fc_pivot(dj, M, h);
            const double rs = fx_to_double(M, h - FCS - e);
            __syncwarp();
#pragma unroll
            for (int s = 0; s < S; ++s) {
                const int i = lane + 32 * s;
                if (i >= j && i < cnt) *entry(j, i) = fc_split(fc_mul(num[s], M, h));
                if (i == j) {
                    rsd[s] = rs;
                    tr[s] = fc_mul(tr[s] - ((dot + 1) >> 1), M, h);
                }
            }
            __syncwarp();
        }
        long long part = 0;
#pragma unroll
        for (int s = 0; s < S; ++s) {
            FcSum b{0, 0, 0};
            const int2 f = lane + 32 * s < cnt ? fc_split(tr[s]) : make_int2(0, 0);
            b.add(f, f);
            part += b.hh * 2 + ((b.c1 + b.c2) >> 29);
        }
        const long long dt = diag_x - ((warp_sum(part) + 1) >> 1);
        if (npd || (!wide && dt <= 0)) {
            if (lane == 0) record_error(st, SIC_ERR_NOT_PD, c);
            continue;
        }
        // ---- x = F^-T e_last ----
        if (!wide) {
            d = fx_to_double(dt, 2 * e - FCS);
#pragma unroll
            for (int s = 0; s < S; ++s) b[s] = lane + 32 * s < cnt ? fx_to_double(tr[s], e - FCS) : 0.0;
        }
        const double xt = rsqrt_newton(d);
#pragma unroll
        for (int s = 0; s < S; ++s) b[s] *= -xt;
#pragma unroll
        for (int q = S - 1; q >= 0; --q)
            for (int l = min(31, cnt - 1 - 32 * q); l >= 0; --l) {
                const int r = l + 32 * q;
                if (lane == l) b[q] *= rsd[q];
                const double x = __shfl_sync(FULL, b[q], l);
#pragma unroll
                for (int s = 0; s <= q; ++s) {
                    const int i = lane + 32 * s;
                    if (i < r) {
                        const int2 f = *entry(i, r);
                        const double v = wide ? *reinterpret_cast<const double*>(&f)
                                              : fx_to_double(((long long)f.x << 30) + f.y, e - FCS);
                        b[s] = fma(-v, x, b[s]);
                    }
                }
            }
        const long long e0 = col_ptr[c] - base;
        if (lane == 0) {
            row_idx[e0] = (int32_t)tgt;
            val[e0] = xt;
        }
#pragma unroll
        for (int s = 0; s < S; ++s) {
            const int i = lane + 32 * s;
            if (i < cnt) {
                row_idx[e0 + cnt - i] = pos[i];
                val[e0 + cnt - i] = b[s];
            }
        }
        if (lane == held) {
            pend = d;
            pend_col = c;
        }
        if (++held == 32) flush();
    }
    flush();
}

template <int S>
sic_status launch(sic_handle* h, const double* pts, long long n, const sic_kernel* kp, const int32_t* sel_idx,
                  const int32_t* sel_count, int k, long long col0, long long n_cols, const int64_t* col_ptr,
                  long long base, int32_t* row_idx, double* val, double* logv, cudaStream_t s) {
    auto kern = k_fill_columns<S>;
    const int words = (warp_words(k) + 1) / 2 * 2;
    const size_t smem = 8 * ((size_t)EXP_TAB + (size_t)WARPS * words);
    SIC_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    const int grid = persistent_grid(h, kern, 32 * WARPS, smem, (n_cols + WARPS - 1) / WARPS);
    kern<<<grid, 32 * WARPS, smem, s>>>(pts, kp->dim, make_kp<double>(*kp), fx_exponent(kp), sel_idx, sel_count, k, n,
                                        col0, n_cols, (const long long*)col_ptr, base, row_idx, val, logv, words,
                                        h->d_status);
    SIC_CUDA_TRY(cudaGetLastError());
    return SIC_OK;
}

}  // namespace

// 16,384 columns: k = 32 0.66 against 1.07 ms, k = 48 1.57 against 1.76, k = 64 3.6 against 2.8 (few warps fit an SM then)
bool fill_columns_applies(int k) { return k >= 1 && k <= 48; }

sic_status launch_fill_columns(sic_handle* h, const double* pts, long long n, const sic_kernel* kp,
                               const int32_t* sel_idx, const int32_t* sel_count, int k, long long col0,
                               long long n_cols, const int64_t* col_ptr, long long base, int32_t* row_idx, double* val,
                               double* logv, cudaStream_t s) {
    if (k <= 32)
        return launch<1>(h, pts, n, kp, sel_idx, sel_count, k, col0, n_cols, col_ptr, base, row_idx, val, logv, s);
    return launch<2>(h, pts, n, kp, sel_idx, sel_count, k, col0, n_cols, col_ptr, base, row_idx, val, logv, s);
}
