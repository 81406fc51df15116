// Greedy conditional selection in double precision: single columns (Section 3.1 / Section 4) and
// supernodes (Section 5.2, the two partial factors of Appendix C.2), with the factor rows in
// fixed point.
//
// This GPU retires 1.6 FP64 multiply-adds per clock and SM, so the left-looking dot products
// F_j . F_q (one multiply-add per candidate, step and earlier column) are taken off the FP64 pipe:
// with 1.9 2^(2e) >= variance + nugget >= F_jt^2 an entry is held as the integer round(F 2^(58 - e)),
// split as H 2^29 + L (|H| < 2^29.5, |L| <= 2^28), and a product sum is two exact 64-bit sums of 32 x 32-bit
// products, sum H H' and sum (H L' + L H') (no overflow: the rows' norms are at most 2^(e + 0.47), so the
// first stays below 2^59 and the second below 2^62.3 up to 192 columns); sum L L' is left out, about
// 2^-57 of 2^(2e).  A double of magnitude near 2^e is held exactly; FP64 multiply-adds would round each
// term at 2^-53 of the running sum.  Theta_jq goes to the same fixed point, the numerator
// n = Theta_jq - sum is exact there, u = n / sqrt(var_q) one 64 x 64-bit high product.  What stays
// FP64 per candidate and step: Theta (distance, Newton square root, table-driven exp) and the
// downdates of the conditional variances (and covariance), which keep their range and rounding.
//
// One CTA owns one unit at a time.  State of a unit, columns of Cm int2 entries (a thread
// reads its own rows, neighbouring threads neighbouring words): F2 (the m targets' columns by
// forward substitution with chol(Theta_PP), then the picks conditioned on targets and picks), then F1
// (the picks conditioned on picks only; single columns have F1 alone).  The first NC columns
// in this order are in shared memory -- the targets' columns are read at every step --, the others in a
// per-CTA slab of the workspace.
//
// Step: every row's score -- var_j / var_j|P (eq. greedy_mult), or cov_j^2 / var_j (eq. obj_gp) -- in
// FP32 from the FP64 state (good to 2^-20); the block's largest; the rows within 2^-18 of it (one, as
// a rule) go to a list, and of several the FP64 quotient decides, ties to the lowest candidate index;
// the pivot's rows are staged, every row gets its new entries and its variances are downdated.
//
// Single columns are scored by their covariance with the target, which may be far below the variance (points many
// length scales apart) and is then down to products of entries below the fixed point's resolution.  When the best
// candidate's covariance falls below 2^-30 of the variance -- what the format still resolves to 2^-28 -- the column
// starts over with its rows in FP64 (same storage).  Variances ratios (supernodes) lose nothing: an entry below the
// resolution changes no variance.
//
// Bound: latency of the step's phases (with 1024 candidates per supernode 44 % of the issue slots and
// 35 % of the FP64 pipe are busy, L2 delivers 30 bytes per clock and SM); half of each scheduler's warps therefore
// evaluate Theta while the others sum.  N = 2^16 with 1024 candidates, k = 64 (2,811 supernodes): 61.3 ms with FP64
// multiply-adds over FP64 rows, 19.2 ms now; 4096 columns of 256 candidates, k = 16: 2.30 -> 0.83 ms.  One row per thread
// at 64 registers (1024 threads per SM) is faster than two rows per thread at 128 (26.2 ms).
#include "fx.cuh"

namespace {

constexpr int FX_THREADS = 1024;  // threads per SM: 64 registers each
constexpr int SMEM_SM = 227 * 1024;
constexpr int STATIC_ROOM = 5 * 1024;  // static arrays, and the system's 1 KB per CTA

// Columns lie in pairs, [pair][row] of int4, so that one 16-byte load brings a row's entries of two columns;
// counts of columns below are even.
struct FxLayout {
    int Cm;     // rows per column: max_cand rounded up to 32
    int mm, k;  // largest group, picks
    int fb;     // first column of F1 (columns of F2)
    int cols;   // columns of the state
    int nc;     // columns in shared memory
    __host__ __device__ size_t words(int c) const { return (size_t)c * Cm; }  // 8-byte words of c columns
};

// start of row i of chol(Theta_PP) (i + 1 entries): rows 2s and 2s + 1 have 2s + 2 slots, so that every row
// starts on a 16-byte boundary
__host__ __device__ constexpr int tri_row(int i) {
    const int s = i >> 1;
    return 2 * s * (s + 1) + (i & 1) * (2 * s + 2);
}

// dynamic shared memory besides the columns, in 8-byte words: pivot rows, chol(Theta_PP) with its
// reciprocal diagonal (multiplier, shift), coordinates, variances, the exp table, and the list (ints)
template <bool ONE>
__host__ __device__ inline size_t fx_fixed_words(const FxLayout& L, int dim) {
    return (size_t)L.cols + (ONE ? 0 : (size_t)tri_row((L.mm + 1) / 2 * 2) + 2 * L.mm) +
           (size_t)dim * (L.Cm + (ONE ? 0 : L.mm)) + 2 * (size_t)L.Cm + EXP_TAB + (size_t)(L.Cm + 1) / 2;
}

template <bool ONE>
inline FxLayout fx_layout(int max_cand, int mm, int k) {
    FxLayout L;
    L.Cm = max_cand <= 32 ? 32 : (max_cand + 31) / 32 * 32;
    L.mm = mm;
    L.k = k;
    L.fb = ONE ? 0 : (mm + k + 1) / 2 * 2;
    L.cols = L.fb + (k + 1) / 2 * 2;
    L.nc = 0;
    return L;
}

// row of the packed lower triangle (row i has i + 1 entries) that holds flat entry f
__device__ __forceinline__ int tri_of(int f) {
    int i = (int)((sqrtf(8.0f * (float)f + 1.0f) - 1.0f) * 0.5f);
    while (i * (i + 1) / 2 > f) --i;
    while ((i + 1) * (i + 2) / 2 <= f) ++i;
    return i;
}

template <int NT, bool ONE>
__global__ void __launch_bounds__(NT, FX_THREADS / NT) k_select_fx(
    const double* __restrict__ pts, long long n, int dim, KP<double> kp, double floor_, int e,
    const int32_t* __restrict__ targets, const long long* __restrict__ grp_ptr, long long n_units,
    const long long* __restrict__ cand_ptr, const int32_t* __restrict__ cand_idx, int max_cand, int k,
    int32_t* __restrict__ sel_idx, int32_t* __restrict__ sel_count, int4* __restrict__ ws, FxLayout L,
    double* __restrict__ gain, double vfloor, DevStatus* st) {
    constexpr int NW = NT / 32, UNROLL = 4;
    constexpr unsigned FULL = 0xffffffffu;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    int4* S = reinterpret_cast<int4*>(smem_raw);
    int2* p2 = reinterpret_cast<int2*>(smem_raw + 8 * L.words(L.nc));  // pivot's row of F2 (targets, picks)
    int2* p1 = p2 + L.fb;                                              // pivot's row of F1
    double* T = reinterpret_cast<double*>(p2 + L.cols);  // Theta_PP, then its factor (off-diagonal as int2)
    long long* rM = reinterpret_cast<long long*>(T + (ONE ? 0 : tri_row((L.mm + 1) / 2 * 2)));
    int* rS = reinterpret_cast<int*>(rM + (ONE ? 0 : L.mm));
    // coordinates: as read, then in fixed point at the unit's largest exponent per dimension (fx_coord)
    // where that is exact (a point near zero or far out leaves no room for all bits), else in FP64
    double* X = reinterpret_cast<double*>(rS + (ONE ? 0 : 2 * L.mm));
    const long long* Xf = reinterpret_cast<const long long*>(X);
    const int ldx = L.Cm + (ONE ? 0 : L.mm);
    double* VA = X + dim * ldx;  // var_j given the picks
    double* VB = VA + L.Cm;      // supernodes: var_j given targets and picks; columns: cov with the target
    double* tab = VB + L.Cm;
    int* list = reinterpret_cast<int*>(tab + EXP_TAB);
    __shared__ unsigned wkey[NW];
    __shared__ int s_cnt[2];
    __shared__ int s_q, s_go, s_fail;
    __shared__ int s_ex[3];  // largest biased exponent of the coordinates per dimension
    __shared__ double s_r[2];
    __shared__ double gv1[129], gv2[128];  // the picks' variances (gains only)
    __shared__ int qs[128];                // the picks' candidate rows, translated after the steps

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int Cm = L.Cm, nc = L.nc;
    const double NEG = -INFINITY;
    const double diag = kp.s2 + kp.nugget;
    // column c >= nc at W + (c / 2) Cm
    int4* W = ws + (size_t)blockIdx.x * (L.words(L.cols - nc) / 2) - L.words(nc) / 2;
    exp_table_fill(tab, kp.s2);
    const int fb = L.fb;

    auto entry = [&](int c, int r) -> int2* {  // entry of column c, row r
        return reinterpret_cast<int2*>((c < nc ? S : W) + (c >> 1) * Cm + r) + (c & 1);
    };
    bool plain = false;  // the unit's coordinates stay in FP64
    auto theta = [&](int i, int j) -> double {
        double d2;
        if (plain) {
            d2 = 0.0;
            for (int d = 0; d < dim; ++d) {
                const double df = X[d * ldx + i] - X[d * ldx + j];
                d2 = fma(df, df, d2);
            }
        } else {
            d2 = fx_dist2(Xf, ldx, dim, i, j, s_ex[0], s_ex[1], s_ex[2]);
        }
        return matern_d2_fast(kp, d2, tab);
    };
    // sum over columns c0 .. c0 + len (c0 even) of row r with the pivot's entries p; where len is odd the
    // pivot's next entry is zero (the column's may be anything)
    auto dot = [&](int c0, int len, int r, const int2* __restrict__ p) -> long long {
        FxSum a{0, 0};
        const int4* __restrict__ p4 = reinterpret_cast<const int4*>(p);
        auto range = [&](const int4* __restrict__ F, int from, int to) {
            int c = from;
            for (; c + UNROLL <= to; c += UNROLL) {
                int4 v[UNROLL];
#pragma unroll
                for (int i = 0; i < UNROLL; ++i) v[i] = F[(c + i) * Cm + r];
#pragma unroll
                for (int i = 0; i < UNROLL; ++i) a.add2(v[i], p4[c + i]);
            }
            if (c < to) {  // the last ones, their loads in flight together too
                int4 v[UNROLL - 1];
#pragma unroll
                for (int i = 0; i < UNROLL - 1; ++i) v[i] = F[min(c + i, to - 1) * Cm + r];
#pragma unroll
                for (int i = 0; i < UNROLL - 1; ++i)
                    if (c + i < to) a.add2(v[i], p4[c + i]);
            }
        };
        const int pairs = (len + 1) >> 1, in = min(max(nc - c0, 0) >> 1, pairs);  // of these, in shared memory
        range(S + (c0 >> 1) * Cm, 0, in);
        range(W + (c0 >> 1) * Cm, in, pairs);
        return a.value();
    };

    bool rows64 = false;  // (columns) the unit once more, its factor rows in FP64
    for (long long g = blockIdx.x; g < n_units; g += rows64 ? 0LL : (long long)gridDim.x) {
        const long long g0 = ONE ? (targets ? (long long)targets[g] : g) : grp_ptr[g];
        const int m = ONE ? 1 : (int)(grp_ptr[g + 1] - g0);
        const long long b0 = cand_ptr[g];
        const int C = (int)(cand_ptr[g + 1] - b0);
        if (m < 1 || m > (ONE ? 1 : L.mm) || C < 0 || C > max_cand || g0 < 0 || g0 + m > n) {
            if (tid == 0) {
                record_error(st, SIC_ERR_INVALID, g);
                sel_count[g] = 0;
            }
            for (int q = tid; q < k; q += NT) sel_idx[g * k + q] = -1;
            continue;
        }
        const int mt = ONE ? 0 : m;  // target columns
        // ---- coordinates, variances, (columns) the covariances with the target ----
        if (tid < 2) s_cnt[tid] = 0;
        if (tid < 3) s_ex[tid] = 0;
        if (tid == 0) s_fail = 0;
        __syncthreads();
        int ex[3] = {0, 0, 0};
        for (int i = tid; i < C + mt; i += NT) {
            const bool cnd = i < C;
            long long p = cnd ? (long long)cand_idx[b0 + i] : g0 + (i - C);
            const int xi = cnd ? i : Cm + (i - C);
            bool ok = true;
            if (cnd && (p < g0 + m || p >= n)) {  // candidates must lie after the unit
                record_error(st, SIC_ERR_INVALID, g);
                p = g0;
                ok = false;
            }
            double d2 = 0.0;
            bool fin = true;
            for (int d = 0; d < dim; ++d) fin = fin && !not_finite(pts[p * dim + d]);
            if (!fin && !cnd) s_fail = 1;  // Theta_PP has no factor
            for (int d = 0; d < dim; ++d) {
                const double v = pts[p * dim + d];
                X[d * ldx + xi] = fin ? v : 0.0;
                const int b = fin ? (__double2hiint(v) >> 20) & 0x7ff : 0;
                if (d == 0) ex[0] = max(ex[0], b);
                if (d == 1) ex[1] = max(ex[1], b);
                if (d == 2) ex[2] = max(ex[2], b);
                if (ONE) {
                    const double df = v - pts[g0 * dim + d];
                    d2 = fma(df, df, d2);
                }
            }
            if (cnd) {
                const double v0 = !ok ? NEG : (fin ? diag : NAN);  // neither is ever a candidate
                VA[i] = v0;
                VB[i] = ONE ? d2 : v0;  // (columns: the covariance follows the table's barrier)
            }
        }
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const int b = __reduce_max_sync(FULL, ex[d]);
            if (lane == 0 && b > 0) atomicMax(&s_ex[d], b);
        }
        __syncthreads();
        bool cut = false;
        for (int i = tid; i < C + mt; i += NT)
            for (int d = 0; d < dim; ++d) cut = cut || !fx_coord_exact(X[d * ldx + (i < C ? i : Cm + (i - C))], s_ex[d]);
        plain = __syncthreads_or(cut);
        if (!plain)
            for (int i = tid; i < C + mt; i += NT) {
                const int xi = i < C ? i : Cm + (i - C);
                for (int d = 0; d < dim; ++d)
                    reinterpret_cast<long long*>(X)[d * ldx + xi] = fx_coord(X[d * ldx + xi], s_ex[d]);
            }
        if (!ONE) __syncthreads();
        if constexpr (ONE) {
            for (int i = tid; i < C; i += NT) VB[i] = matern_d2_fast(kp, VB[i], tab);
        } else {
            // ---- chol(Theta_PP): right-looking over all threads, packed rows ----
            for (int f = tid; f < m * (m + 1) / 2; f += NT) {
                const int i = tri_of(f), j = f - i * (i + 1) / 2;
                T[tri_row(i) + j] = i == j ? diag : theta(Cm + i, Cm + j);
            }
            __syncthreads();
            for (int a = 0; a < m; ++a) {
                if (warp == 0) {
                    const double d = T[tri_row(a) + a];
                    if (s_fail || !(d > 0.0)) {
                        if (lane == 0) {
                            record_error(st, SIC_ERR_NOT_PD, g);
                            s_fail = 1;
                        }
                    } else {
                        const double rs = rsqrt_newton(d);
                        if (lane == 0) {
                            s_r[0] = rs;
                            fx_factor(rs, e, rM[a], rS[a]);
                        }
                    }
                }
                __syncthreads();
                if (s_fail) break;
                const double rs = s_r[0];
                for (int i = a + 1 + tid; i < m; i += NT) T[tri_row(i) + a] *= rs;
                __syncthreads();
                const int w = m - a - 1;  // the trailing triangle, rows a + 1 .. m - 1
                for (int f = tid; f < w * (w + 1) / 2; f += NT) {
                    const int i0 = tri_of(f), j = f - i0 * (i0 + 1) / 2 + a + 1;
                    double* Ti = T + tri_row(i0 + a + 1);
                    Ti[j] = fma(-Ti[a], T[tri_row(j) + a], Ti[j]);
                }
                __syncthreads();
            }
            if (!s_fail) {
                for (int f = tid; f < m * (m + 1) / 2; f += NT) {  // to fixed point, in place; 0 on the diagonal
                    const int i = tri_of(f), j = f - i * (i + 1) / 2;
                    const double t = T[tri_row(i) + j];
                    const long long x = i == j ? 0LL : fx_of_positive(fabs(t), FXS - e);
                    reinterpret_cast<int2*>(T)[tri_row(i) + j] = fx_split(t < 0.0 ? -x : x);
                }
                __syncthreads();
                // ---- the targets' columns of F2: every row by forward substitution ----
                for (int r = tid; r < C; r += NT) {
                    double v = VB[r];  // (an invalid candidate's stays -inf)
                    for (int a = 0; a < m; ++a) {
                        const double th = theta(r, Cm + a);
                        if (not_finite(th)) v = NAN;
                        const long long n2 = fx_of_positive(th, FXS - 2 * e) -
                                             dot(0, a, r, reinterpret_cast<const int2*>(T) + tri_row(a));
                        const long long u = fx_mul(n2, rM[a], rS[a]);
                        *entry(a, r) = fx_split(u);
                        const double ud = fx_to_double(u, e - FXS);
                        v = fma(-ud, ud, v);
                    }
                    VB[r] = v;
                }
            }
        }
        __syncthreads();
        // ---- the steps ----
        double vt = diag;  // columns: the target's variance (thread 0, gains only)
        int t = 0;
        bool again = false;
        if (!s_fail) {
            for (; t < k; ++t) {
                int* cnt = &s_cnt[t & 1];
                // FP32 score key of a row (0: not a candidate); positive scores, so the bits are monotone
                auto key_of = [&](int r) -> unsigned {
                    const double va = VA[r], vb = VB[r];
                    if (!((ONE ? va : vb) >= floor_)) return 0u;
                    float s;
                    if (ONE) {
                        const float c = fx_f32(fabs(vb), 2 * e);
                        s = __fdividef(c * c, fx_f32(va, 2 * e));
                    } else {
                        s = __fdividef(fx_f32(va, 2 * e), fx_f32(vb, 2 * e));
                    }
                    return __float_as_uint(s) + 1u;
                };
                const unsigned mine = tid < C ? key_of(tid) : 0u;
                unsigned bk = mine;
                for (int r = tid + NT; r < C; r += NT) bk = max(bk, key_of(r));
                bk = __reduce_max_sync(FULL, bk);
                if (lane == 0) wkey[warp] = bk;
                __syncthreads();
                const unsigned gk = __reduce_max_sync(FULL, lane < NW ? wkey[lane] : 0u);
                if (gk == 0u) break;
                // rows that may hold the largest score: within 2^-18 of the FP32 maximum, or every live row
                // where the maximum is too small for FP32 to tell (or is not finite)
                const bool clear_ = gk > 0x0da24260u && gk < 0x7f000000u;  // 1e-30
                const unsigned lim = clear_ ? gk - 32u : 1u;
                if (mine >= lim) list[atomicAdd(cnt, 1)] = tid;
                for (int r = tid + NT; r < C; r += NT)
                    if (key_of(r) >= lim) list[atomicAdd(cnt, 1)] = r;
                __syncthreads();
                const int nl = *cnt;
                int q;
                if (nl == 1 && clear_) {
                    q = list[0];
                } else {  // FP64 quotients, ties to the lowest index
                    if (warp == 0) {
                        double bs = NEG;
                        int bi = 0x7fffffff;
                        for (int i = lane; i < nl; i += 32) {
                            const int r = list[i];
                            const double va = VA[r], vb = VB[r];
                            const double s = ONE ? vb * vb / va : va / vb;
                            if (s > bs || (s == bs && r < bi)) { bs = s; bi = r; }
                        }
#pragma unroll
                        for (int off = 16; off > 0; off >>= 1) {
                            const double os = __shfl_xor_sync(FULL, bs, off);
                            const int oi = __shfl_xor_sync(FULL, bi, off);
                            if (os > bs || (os == bs && oi < bi)) { bs = os; bi = oi; }
                        }
                        if (lane == 0) {
                            s_q = bi;
                            s_go = bi != 0x7fffffff && (!ONE || bs > 0.0);
                        }
                    }
                    __syncthreads();
                    if (!s_go) break;
                    q = s_q;
                }
                if (ONE && !rows64 && exponent_of(VB[q]) < 2 * e - FX_COV_BITS) {
                    again = true;
                    break;
                }
                // ---- stage the pivot: its rows, and 1/sqrt of its variances by the last warp ----
                if (warp == NW - 1) {
                    const double v = (!ONE && lane == 1) ? VB[q] : VA[q];
                    const double r = rsqrt_newton(v);
                    if (lane < 2) s_r[lane] = r;
                }
                for (int c = tid; c <= t; c += NT) p1[c] = c < t ? *entry(fb + c, q) : make_int2(0, 0);
                if constexpr (!ONE)
                    for (int c = tid; c <= mt + t; c += NT) p2[c] = c < mt + t ? *entry(c, q) : make_int2(0, 0);
                const double vaq = VA[q], vbq = VB[q];
                if (tid == 0) {
                    s_cnt[(t + 1) & 1] = 0;
                    qs[t] = q;  // no global load on the step chain
                    if (gain) {
                        if (ONE) {
                            gv1[t] = vt;
                        } else {
                            gv1[t] = vaq;
                            gv2[t] = vbq;
                        }
                    }
                }
                __syncthreads();
                long long M1, M2 = 0;
                int h1, h2 = 0;
                fx_factor(s_r[0], e, M1, h1);
                if (!ONE) fx_factor(s_r[1], e, M2, h2);
                const double ut = ONE ? vbq * s_r[0] : 0.0;
                if (ONE && rows64) {
                    const double2* p = reinterpret_cast<const double2*>(p1);
                    for (int r = tid; r < C; r += NT) {
                        const double va = VA[r];
                        if (!(va >= -1e300)) continue;
                        double num = theta(r, q);
                        if (r == q) num += kp.nugget;
                        const double2* F = reinterpret_cast<const double2*>(S) + r;
                        for (int c = 0; c < t >> 1; ++c) num = fma(-F[c * Cm].y, p[c].y, fma(-F[c * Cm].x, p[c].x, num));
                        if (t & 1) num = fma(-F[(t >> 1) * Cm].x, p[t >> 1].x, num);
                        const double u = num * s_r[0];
                        *reinterpret_cast<double*>(entry(t, r)) = u;
                        VA[r] = r == q ? NEG : fma(-u, u, va);  // (NaN: never a candidate again)
                        VB[r] = fma(-u, ut, VB[r]);
                    }
                } else {
                    for (int r = tid; r < C; r += NT) {
                        const double va = VA[r];
                        if (!(va >= -1e300)) continue;  // picked, invalid (-inf) or NaN
                        // half of each scheduler's warps evaluate Theta (FP64 pipe) before the sums (integer
                        // pipes and loads), the other half after them
                        double th = 0.0;
                        long long s1 = 0, s2 = 0;
#pragma unroll 1
                        for (int ph = 0; ph < 2; ++ph) {
                            if (ph == ((warp >> 2) & 1)) {
                                th = theta(r, q);
                            } else {
                                if constexpr (!ONE) s2 = dot(0, mt + t, r, p2);
                                s1 = dot(fb, t, r, p1);
                            }
                        }
                        if (r == q) th += kp.nugget;
                        if (not_finite(th)) {  // never a candidate again
                            VA[r] = VB[r] = NAN;
                            continue;
                        }
                        const long long tx = fx_of_positive(th, FXS - 2 * e);
                        if constexpr (!ONE) {
                            const long long u2 = fx_mul(tx - s2, M2, h2);
                            *entry(mt + t, r) = fx_split(u2);
                            const double d2 = fx_to_double(u2, e - FXS);
                            VB[r] = r == q ? NEG : fma(-d2, d2, VB[r]);
                        }
                        const long long u1 = fx_mul(tx - s1, M1, h1);
                        *entry(fb + t, r) = fx_split(u1);
                        const double d1 = fx_to_double(u1, e - FXS);
                        VA[r] = r == q ? NEG : fma(-d1, d1, va);
                        if constexpr (ONE) VB[r] = fma(-d1, ut, VB[r]);
                    }
                }
                if (ONE && gain && tid == 0) {
                    vt = fmax(vt - ut * ut, vfloor);
                    gv1[t + 1] = vt;
                }
            }
        }
        // the picks' global indices and (with gain) the decreases of 2 KL per nonzero (Section 5.4), off the
        // step chain
        __syncthreads();
        if (ONE && again) {
            rows64 = true;
            continue;
        }
        rows64 = false;
        for (int q = tid; q < t; q += NT) {
            sel_idx[g * k + q] = cand_idx[b0 + qs[q]];
            if (gain) gain[g * k + q] = ONE ? log(gv1[q] / gv1[q + 1]) : log(gv1[q] / gv2[q]) / m;
        }
        if (tid == 0) sel_count[g] = t;
        for (int q = t + tid; q < k; q += NT) sel_idx[g * k + q] = -1;
        __syncthreads();
    }
}

template <int NT, bool ONE>
int fx_grid(sic_handle* h, size_t smem, long long units) {
    auto kern = k_select_fx<NT, ONE>;
    // (one limit for every plan: calls of several threads do not disturb each other's)
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_SM - 3 * 1024);
    return persistent_grid(h, kern, NT, smem, units);
}

// Threads: a row per thread up to 1024 rows (strided beyond); smaller units share an SM and its shared
// memory.
template <bool ONE>
FxPlan fx_plan(sic_handle* h, long long units, int dim, int max_cand, int mm, int k, int nt) {
    FxPlan P;
    FxLayout L = fx_layout<ONE>(max_cand, mm, k);
    if (nt != 128 && nt != 256 && nt != 512 && nt != 1024)
        nt = max_cand <= 128 ? 128 : (max_cand <= 256 ? 256 : (max_cand <= 512 ? 512 : 1024));
    const size_t fixed = 8 * fx_fixed_words<ONE>(L, dim);
    // 1024 threads per SM; fewer where the fixed part or, without a workspace (single columns), the whole
    // state needs more of the SM's shared memory.  The largest fixed part, 4096 candidates with 64 targets
    // and 128 picks, is 204 KB, the largest single-column state with its fixed part 171 KB.
    const size_t must = fixed + (ONE ? 8 * L.words(L.cols) : 0);
    size_t room = 0;
    for (int ctas = FX_THREADS / nt; ctas >= 1 && room < must; ctas /= 2) room = (size_t)SMEM_SM / ctas - STATIC_ROOM;
    const size_t fit = (room - fixed) / (8 * L.words(2)) * 2;
    L.nc = fit < (size_t)L.cols ? (int)fit : L.cols;
    P.nt = nt;
    P.nc = L.nc;
    P.smem = fixed + 8 * L.words(L.nc);
    const long long work = units > 0 ? units : 1;
    P.grid = nt == 128   ? fx_grid<128, ONE>(h, P.smem, work)
             : nt == 256 ? fx_grid<256, ONE>(h, P.smem, work)
             : nt == 512 ? fx_grid<512, ONE>(h, P.smem, work)
                         : fx_grid<1024, ONE>(h, P.smem, work);
    // (16 more: the slabs start at the next 16-byte boundary of a workspace of any alignment)
    P.ws_bytes = L.nc < L.cols ? 8 * L.words(L.cols - L.nc) * (size_t)P.grid + 16 : 0;
    return P;
}

template <bool ONE>
sic_status fx_launch(sic_handle* h, const FxPlan& P, const double* pts, long long n, const sic_kernel* kp,
                     const int32_t* targets, const int64_t* grp_ptr, long long units, const int64_t* cand_ptr,
                     const int32_t* cand_idx, int max_cand, int mm, int k, int32_t* sel_idx, int32_t* sel_count,
                     double* gain, void* ws, cudaStream_t s) {
    if (P.ws_bytes > 0 && !ws) return SIC_ERR_INVALID;
    int4* slabs = reinterpret_cast<int4*>((reinterpret_cast<uintptr_t>(ws) + 15) / 16 * 16);
    FxLayout L = fx_layout<ONE>(max_cand, mm, k);
    L.nc = P.nc;
    const int e = fx_exponent(kp);
    const KP<double> p = make_kp<double>(*kp);
    const double fl = sic_floor_of(kp);
#define SIC_FX_LAUNCH(NTV)                                                                                      \
    k_select_fx<NTV, ONE><<<P.grid, NTV, P.smem, s>>>(pts, n, kp->dim, p, fl, e, targets, (const long long*)grp_ptr, \
                                                      units, (const long long*)cand_ptr, cand_idx, max_cand, k, \
                                                      sel_idx, sel_count, slabs, L, gain, fl, h->d_status)
    if (P.nt == 128)
        SIC_FX_LAUNCH(128);
    else if (P.nt == 256)
        SIC_FX_LAUNCH(256);
    else if (P.nt == 512)
        SIC_FX_LAUNCH(512);
    else
        SIC_FX_LAUNCH(1024);
#undef SIC_FX_LAUNCH
    SIC_CUDA_TRY(cudaGetLastError());
    return SIC_OK;
}

}  // namespace

FxPlan fx_plan_groups(sic_handle* h, long long n_grp, int max_cand, int max_m, int k, int nt) {
    return fx_plan<false>(h, n_grp, 3, max_cand, max_m, k, nt);
}

sic_status launch_fx_groups(sic_handle* h, const FxPlan& P, const double* pts, long long n, const sic_kernel* kp,
                            const int64_t* grp_ptr, int64_t n_grp, const int64_t* cand_ptr, const int32_t* cand_idx,
                            int max_cand, int max_m, int k, int32_t* sel_idx, int32_t* sel_count, double* gain,
                            void* ws, cudaStream_t s) {
    return fx_launch<false>(h, P, pts, n, kp, nullptr, grp_ptr, n_grp, cand_ptr, cand_idx, max_cand, max_m, k, sel_idx,
                            sel_count, gain, ws, s);
}

sic_status launch_fx_columns(sic_handle* h, const double* pts, long long n, const sic_kernel* kp,
                             const int32_t* targets, int64_t n_cols, const int64_t* cand_ptr, const int32_t* cand_idx,
                             int max_cand, int k, int32_t* sel_idx, int32_t* sel_count, double* gain, cudaStream_t s) {
    const FxPlan P = fx_plan<true>(h, n_cols, kp->dim, max_cand, 1, k, 0);
    return fx_launch<true>(h, P, pts, n, kp, targets, nullptr, n_cols, cand_ptr, cand_idx, max_cand, 1, k, sel_idx,
                           sel_count, gain, nullptr, s);
}
