// y = (Theta + shift I) x for several right-hand sides, the sums on the 5th-generation tensor cores.
//
// The kernel entries are evaluated in FP32 (the same fixed, symmetric rounding of Theta as in pcg.cu's
// kernel for few right-hand sides); what cost most was summing their products to far below FP32, 11
// operations per entry and right-hand side.  Here both factors are cut into 8-bit digits, which BF16
// holds exactly, and the digits' products are summed exactly (after Ozaki et al., Numer. Algorithms 59 (2012)):
//   Theta_ij / 2^E = sum_a A_a 2^-(7 + 8a), a = 0..7 (2^E >= variance),
//   x_jr / 2^X_r   = sum_b B_b 2^-(7 + 8b), b = 0..7 (2^X_r > max_j |x_jr|), |A_a|, |B_b| <= 128,
// with A_0 = round(128 Theta / 2^E), the remainder times 256, and so on (exact FP32 operations).  Products of
// level a + b = l <= 8 go to one accumulator: 128 sources x 8 pairs x 2^14 <= 2^24, so FP32 holds every partial
// sum exactly; after 128 sources the levels are added to three 64-bit integers per row and right-hand
// side.  The integers do not depend on the order of the sum.
//
// Accuracy.  An FP32 entry is held exactly from 2^-40 of the variance on, an x from 2^-10 of max|x| on; the digits cut off
// below that and the levels left out come to about sqrt(n) 2^-68 variance max|x| in a row (their signs are random).
// A row must be as good as its own sum S_i = sum_j |Theta_ij x_j|, not as max|x|: a row far from a large x_j, or one
// with a wide range of x, has a small S_i.  So one more MMA per step sums A_0 times the leading 15 bits of |x|, a
// lower bound of S_i (to its rounding), and where it stays below sqrt(n) 2^-20 variance max|x| the entry of y is marked (a
// NaN with a payload of its own) and k_matvec_rows, launched behind, forms it in double-FP32.  The others are within
// 2^-48 of S_i, as far as such sums go.  (With six digits and no check, rows beside a spike of 1e12 were off by 1e-3 S_i,
// and rows of a unit vector's product lost entries below 2^-47.)
//
// A CTA takes 128 rows (TMEM lanes) and, in a cluster, a share of the sources; 256 threads = row and half of a step's
// 16 sources.  Per step the threads write the eight digit tiles of Theta (128 x 16 BF16, K-major core matrices) into
// one of two buffers and one thread issues the MMAs, digit a against B_0 .. B_(8-a) into the columns from level a on (N a
// multiple of 16; where that is one digit more than needed it lands in level 9, which is not read).  The MMAs run under the next step's evaluation; the accumulators (two sets) are read one chunk late.
//
// Bound: FP32 issue of the kernel evaluation and the digits, about 50 operations per entry whatever the
// number of right-hand sides.  N = 50,001 with 8 of them: 16.6 ms with double-FP32 sums on the CUDA cores, 8.0 ms
// now (N = 4096: 1.04 -> 0.125 ms); 6.8 ms with six digits and no check; with sqrtf and a run-time smoothness, whose branches
// keep the evaluations from overlapping, half as much again.
#include "matvec_f32.cuh"
#include "tc_common.cuh"

namespace {

constexpr int ROWS = 128, CH = 128, SUB = 16, NT = 256;
constexpr int KD = 8, XD = 8;    // digits of Theta and of x
constexpr int BR = XD * 8 + 16;  // rows of an x tile: the digits, then the leading 7 and the next 8 bits of |x|
constexpr int A_TILE = ROWS * SUB * 2;       // one digit tile
constexpr int SA = 0;                        // [2 buffers][KD] tiles
constexpr int SB = SA + 2 * KD * A_TILE;     // [2 chunks] x: BR rows x CH, K-major
constexpr int B_TILE = BR * CH * 2;
constexpr int B_GROUP = (CH / 8) * 128;      // 8 rows of it
constexpr int SC = SB + 2 * B_TILE;          // [2 chunks][3][CH] negated coordinates
constexpr int SX = SC + 2 * 3 * CH * 4;      // largest biased exponent per right-hand side, a flag
constexpr int SBAR = SX + 16 * 4;            // two mbarriers, TMEM address
constexpr int SMEM_MV = SBAR + 32;
constexpr int SACC = SA;                     // [ROWS][8][4] 64-bit sums for the cluster (after the last MMA)
static_assert(ROWS * 8 * 4 * 8 <= SB, "the sums fit in the digit tiles");
// two CTAs per SM: all 512 TMEM columns, none waits for them
constexpr unsigned TMEM_COLS = 256;
constexpr uint32_t T_SET = 128;              // columns of an accumulator set: 8 per level 0 .. 9, then S
constexpr uint32_t T_S = 80;
constexpr int S_BITS = 20;                   // marked below sqrt(n) 2^-S_BITS

// an entry of y that k_matvec_rows has to form; the low bits hold the biased exponent of max|x|
constexpr unsigned long long MARK = 0x7ff85ac000000000ULL;
__device__ __forceinline__ bool is_marked(double v) {
    return ((unsigned long long)__double_as_longlong(v) & ~0x7ffULL) == MARK;
}

__device__ __forceinline__ void tmem_ld4(uint32_t taddr, float (&v)[4]) {
    uint32_t r[4];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(taddr));
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_sync_all() {
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ long long ld_cluster_s64(uint32_t addr, uint32_t rank) {
    long long v;
    asm volatile(
        "{\n.reg .u32 a;\nmapa.shared::cluster.u32 a, %1, %2;\nld.shared::cluster.s64 %0, [a];\n}\n"
        : "=l"(v)
        : "r"(addr), "r"(rank)
        : "memory");
    return v;
}

// The square roots of a pair by fused operations after Markstein (IBM J. Res. Dev. 34 (1990)), without branches, so that
// the evaluations overlap.  From an approximate reciprocal root y: g = x y and h = y / 2, both brought on by their
// common error e = 1/2 - g h (g += g e, h += h e), then g += h (x - g^2) with the residual exact: correctly rounded,
// equal to sqrtf for every significand (sic_selftest_sqrt_f32).  Below 2^-100 (distances that leave every kernel at
// its value at 0) the last bits may differ; infinity stays infinite.
__device__ __forceinline__ float2 sqrt_f2(float2 x) {
    float ya, yb;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(ya) : "f"(fmaxf(x.x, 1.2e-38f)));
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(yb) : "f"(fmaxf(x.y, 1.2e-38f)));
    const float2 neg1 = make_float2(-1.f, -1.f), half2 = make_float2(0.5f, 0.5f);
    const float2 y = make_float2(ya, yb);
    const float2 g = __fmul2_rn(x, y), h = __fmul2_rn(y, half2);
    const float2 e = __ffma2_rn(__fmul2_rn(g, neg1), h, half2);
    const float2 g1 = __ffma2_rn(g, e, g), h1 = __ffma2_rn(h, e, h);
    const float2 r = __ffma2_rn(__ffma2_rn(__fmul2_rn(g1, neg1), g1, x), h1, g1);
    return make_float2(x.x < INFINITY ? r.x : x.x, x.y < INFINITY ? r.y : x.y);
}

// matern<float> (the same operations) with the smoothness a constant
template <int NU>
__device__ __forceinline__ float matern_nu(const KP<float>& k, float r) {
    const float t = k.c_over_ell * r;
    const float e = sic_exp(-t);
    if (NU == 1) return k.s2 * e;
    if (NU == 3) return k.s2 * (1.f + t) * e;
    return k.s2 * (1.f + t + t * t * (float)(1.0 / 3.0)) * e;
}

__device__ __forceinline__ int ld_cluster_s32(uint32_t addr, uint32_t rank) {
    int v;
    asm volatile(
        "{\n.reg .u32 a;\nmapa.shared::cluster.u32 a, %1, %2;\nld.shared::cluster.s32 %0, [a];\n}\n"
        : "=r"(v)
        : "r"(addr), "r"(rank)
        : "memory");
    return v;
}

// whether x at a sampled source comes near the largest of its right-hand side
__device__ __noinline__ bool sample_large(const double* x, long long n, int nrhs, const int* sx) {
    const long long j = (long long)threadIdx.x * n / NT;
    bool large = false;
    for (int r = 0; r < nrhs; ++r)
        large = large || (sx[r] > 0 && ((__double2hiint(x[j * nrhs + r]) >> 20) & 0x7ff) > sx[r] - 12);
    return large;
}

template <int NU>
__global__ void __launch_bounds__(NT, 2) k_matvec_tc(const double* __restrict__ pts, long long n, int dim, KP<float> kp,
                                                     float to_unit, int E, double diag_extra,
                                                     const double* __restrict__ x, double* __restrict__ y, int nrhs,
                                                     int parts, float least, DevStatus* st) {
    extern __shared__ __align__(1024) unsigned char sm[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int row = (warp & 3) * 32 + lane, half = warp >> 2;
    int* sx = reinterpret_cast<int*>(sm + SX);  // [0..7] exponents, [9] whether digits are formed
    uint64_t* bars = reinterpret_cast<uint64_t*>(sm + SBAR);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(sm + SBAR + 16);
    const uint32_t bar[2] = {smem_u32(bars), smem_u32(bars + 1)};
    const uint32_t aA = smem_u32(sm + SA), aB = smem_u32(sm + SB);

    if (tid == 0) {
        for (int b = 0; b < 2; ++b) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar[b]) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (tid < 16) sx[tid] = 0;
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tmem_slot;
    const uint32_t lane_addr = tmem + ((uint32_t)((warp & 3) * 32) << 16);

    // the largest exponent of every right-hand side (by its bits), the cluster's CTAs a share each
    const uint32_t cluster_part = parts > 1 ? cluster_rank() : 0u;
    {
        int ex[8];
#pragma unroll
        for (int r = 0; r < 8; ++r) ex[r] = 0;
        for (long long j = (long long)cluster_part * NT + tid; j < n; j += (long long)parts * NT) {
#pragma unroll
            for (int r = 0; r < 8; ++r)
                if (r < nrhs) ex[r] = max(ex[r], (__double2hiint(x[j * nrhs + r]) >> 20) & 0x7ff);
        }
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const int m = __reduce_max_sync(0xffffffffu, ex[r]);
            if (lane == 0) atomicMax(&sx[r], m);
        }
    }
    // rows, and this CTA's chunks of sources
    const long long tile = blockIdx.x / parts;
    const uint32_t rank = cluster_part;
    const long long i = tile * ROWS + row;
    float rc[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) rc[d] = (i < n && d < dim) ? (float)pts[i * dim + d] : 0.f;
    long long hi[4] = {0, 0, 0, 0}, mid[4] = {0, 0, 0, 0}, lo[4] = {0, 0, 0, 0};
    float S[4] = {0.f, 0.f, 0.f, 0.f};
    float chk = 0.f;  // NaN once a kernel entry is
    bool failed = false;
    uint32_t par[2] = {0u, 0u};
    bool used[2] = {false, false};
    // adds the levels of accumulator set `set` to the sums
    auto take = [&](int set) {
        const uint32_t at = lane_addr + set * T_SET + 4 * half;
        auto three = [&](int l, long long(&sum)[4]) {
            float v[3][4];
#pragma unroll
            for (int i = 0; i < 3; ++i) tmem_ld4(at + 8 * (l + i), v[i]);
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
            for (int r = 0; r < 4; ++r)
                sum[r] += ((long long)__float2int_rn(v[0][r]) << 16) + (__float2int_rn(v[1][r]) * 256LL) +
                          __float2int_rn(v[2][r]);
        };
        three(0, hi);
        three(3, mid);
        three(6, lo);
        float v[2][4];
#pragma unroll
        for (int i = 0; i < 2; ++i) tmem_ld4(at + T_S + 8 * i, v[i]);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
        for (int r = 0; r < 4; ++r) S[r] -= fmaf(v[0][r], 256.f, v[1][r]);  // (Theta's digits have the minus sign)
    };
    __syncthreads();
    if (parts > 1) {
        cluster_sync_all();
        int m = 0;
        if (tid < 8)
            for (int q = 0; q < parts; ++q) m = max(m, ld_cluster_s32(smem_u32(sx + tid), q));
        cluster_sync_all();
        if (tid < 8) sx[tid] = m;
        __syncthreads();
    }
    // Where next to no x comes near its right-hand side's largest (256 sources, the same for every CTA), nearly all rows
    // would be marked: no digits then, the sums stay zero and all rows are (a unit vector at N = 50,001: 20.9 -> 13.7 ms,
    // 2048: 0.21 -> 0.17; fewer points keep the digits, whose sums are exact).
    // The decision goes through shared memory: as the barrier's result it made the loop below 7 % slower.
    sx[9] = 8 * __syncthreads_count(n < 2048 || sample_large(x, n, nrhs, sx)) >= NT;
    __syncthreads();
    const long long chunks = (n + CH - 1) / CH;
    const long long c_lo = chunks * rank / parts, c_hi = chunks * (rank + 1) / parts;
    for (long long c = sx[9] ? c_lo : c_hi; c < c_hi && !failed; ++c) {
        const int set = (int)((c - c_lo) & 1);
        // ---- the chunk's coordinates and the digits of its x ----
        float* nc = reinterpret_cast<float*>(sm + SC) + set * 3 * CH;
        for (int e = tid; e < 3 * CH; e += NT) {
            const int d = e / CH, t = e % CH;
            const long long j = c * CH + t;
            const float v = (j < n && d < dim) ? (float)pts[j * dim + d] : 0.f;
            nc[d * CH + t] = -v;
        }
#pragma unroll
        for (int q = 0; q < CH * 8 / NT; ++q) {
            const int t = (tid >> 3) + q * (NT / 8), r = tid & 7;
            const long long j = c * CH + t;
            long long I = 0;    // round(x 2^(63 - X)), |I| < 2^63
            unsigned top = 0u;  // the leading 15 bits of |x| 2^-X
            if (j < n && r < nrhs) {
                const long long u = __double_as_longlong(x[j * nrhs + r]);
                const int e = (int)((u >> 52) & 0x7ff);
                const long long mant = (u & 0xfffffffffffffLL) | 0x10000000000000LL;
                const int sh = sx[r] - e - 10;  // X = sx[r] - 1022
                if (e > 0) I = sh <= 0 ? mant << -sh : (sh < 55 ? ((mant >> (sh - 1)) + 1) >> 1 : 0LL);
                top = (unsigned)(I >> 48);
                if (u < 0) I = -I;
            }
            unsigned char* Bt = sm + SB + set * B_TILE;
#pragma unroll
            for (int b = XD - 1; b >= 0; --b) {
                const int dgt = b > 0 ? (int)(signed char)(I & 255) : (int)I;
                I = (I - dgt) >> 8;
                *reinterpret_cast<__nv_bfloat16*>(Bt + core_off(b * 8 + r, t, CH)) = __float2bfloat16_rn((float)dgt);
            }
            *reinterpret_cast<__nv_bfloat16*>(Bt + core_off(XD * 8 + r, t, CH)) = __float2bfloat16_rn((float)(top >> 8));
            *reinterpret_cast<__nv_bfloat16*>(Bt + core_off(XD * 8 + 8 + r, t, CH)) =
                __float2bfloat16_rn((float)(top & 255u));
        }
        __syncthreads();
        for (int s = 0; s < CH / SUB; ++s) {
            const int buf = s & 1;
            if (used[buf]) {  // the MMAs that read this buffer last
                if (!bar_wait(bar[buf], par[buf])) failed = true;
                par[buf] ^= 1u;
            }
            used[buf] = true;
            // ---- eight kernel entries, two at a time, and their digits ----
            uint32_t dg[KD][4];
            const float* cx = nc + s * SUB + half * 8;
#pragma unroll
            for (int p = 0; p < 4; ++p) {
                const float2 dx = __fadd2_rn(make_float2(rc[0], rc[0]), *reinterpret_cast<const float2*>(cx + 2 * p));
                const float2 dy =
                    __fadd2_rn(make_float2(rc[1], rc[1]), *reinterpret_cast<const float2*>(cx + CH + 2 * p));
                float2 d2 = __ffma2_rn(dx, dx, __fmul2_rn(dy, dy));
                if (dim > 2) {
                    const float2 dz =
                        __fadd2_rn(make_float2(rc[2], rc[2]), *reinterpret_cast<const float2*>(cx + 2 * CH + 2 * p));
                    d2 = __ffma2_rn(dz, dz, d2);
                }
                const float2 dist = sqrt_f2(d2);
                const float2 k = make_float2(matern_nu<NU>(kp, dist.x), matern_nu<NU>(kp, dist.y));
                float2 r = __fmul2_rn(k, make_float2(to_unit, to_unit));
                const float2 M = make_float2(12582912.f, 12582912.f);  // 1.5 2^23: adding it rounds to an integer
                const float2 neg1 = make_float2(-1.f, -1.f);
#pragma unroll
                for (int a = 0; a < KD; ++a) {
                    const float f = a == 0 ? 128.f : 256.f;
                    const float2 f2 = make_float2(f, f);
                    const float2 nd = __ffma2_rn(__ffma2_rn(r, f2, M), neg1, M);  // minus the digit
                    if (a == 0) chk += nd.x + nd.y;
                    if (a + 1 < KD) r = __ffma2_rn(r, f2, nd);  // exact
                    dg[a][p] = pack2(nd.x, nd.y);
                }
            }
#pragma unroll
            for (int a = 0; a < KD; ++a)
                *reinterpret_cast<uint4*>(sm + SA + (buf * KD + a) * A_TILE + core_off(row, half * 8, SUB)) =
                    make_uint4(dg[a][0], dg[a][1], dg[a][2], dg[a][3]);
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            if (__syncthreads_or(failed)) {
                failed = true;
                break;
            }
            if (tid == 0) {
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                // `digits` digits of x from b on, against digit a, into the columns from `col` on
                auto mma = [&](int a, int b, int digits, uint32_t col, uint32_t acc) {
                    mma_f16(tmem + set * T_SET + col, smem_desc(aA + (buf * KD + a) * A_TILE, 128, 256),
                            smem_desc(aB + set * B_TILE + b * B_GROUP + s * (SUB / 8) * 128, 128, B_GROUP), acc,
                            idesc_bf16(8 * digits, 0, 0));
                };
                // a chunk's first MMAs set the columns: 16 .. 79 by digit 2, 0 .. 15 by digit 0, then S
                const uint32_t acc = s > 0 ? 1u : 0u;
                mma(2, 0, 8, 16, acc);
                mma(0, 0, 2, 0, acc);
                mma(0, 2, 6, 16, 1u);
                mma(0, XD, 2, T_S, acc);
                mma(1, 0, 8, 8, 1u);
#pragma unroll
                for (int a = 3; a < KD; ++a) mma(a, 0, (10 - a) / 2 * 2, 8 * a, 1u);
                mma_commit(bar[buf]);
            }
            // the previous chunk's last MMAs were waited for in this chunk's first two steps
            if (s == 2 && c > c_lo) {
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                take(set ^ 1);
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            }
        }
    }
    for (int b = 0; b < 2; ++b)
        if (used[b] && !failed)
            if (!bar_wait(bar[b], par[b])) failed = true;
    if (__syncthreads_or(failed)) failed = true;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (!failed && c_hi > c_lo && sx[9]) take((int)((c_hi - 1 - c_lo) & 1));
    if (failed && tid == 0) record_error(st, SIC_ERR_TIMEOUT, blockIdx.x);
    // a kernel entry that is not a number in either half of the row: the row's result is NaN
    int* flag = reinterpret_cast<int*>(sm + SC);
    if (half == 0) flag[row] = 0;
    __syncthreads();
    if (!(fabsf(chk) < INFINITY)) flag[row] = 1;
    __syncthreads();
    bool nan_row = flag[row] != 0;
    // ---- the cluster's sums to its first CTA, the result ----
    long long* acc = reinterpret_cast<long long*>(sm + SACC);
    constexpr long long NOT_A_NUMBER = (long long)0x8000000000000000ULL;
    if (parts > 1) {
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            long long* at = acc + (row * 8 + 4 * half + r) * 4;
            at[0] = nan_row ? NOT_A_NUMBER : hi[r];
            at[1] = mid[r];
            at[2] = lo[r];
            at[3] = (long long)S[r];
        }
        cluster_sync_all();
        if (rank == 0) {
            for (int q = 1; q < parts; ++q) {
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const uint32_t at = smem_u32(acc + (row * 8 + 4 * half + r) * 4);
                    const long long h = ld_cluster_s64(at, q);
                    if (h == NOT_A_NUMBER) nan_row = true;
                    hi[r] += h;
                    mid[r] += ld_cluster_s64(at + 8, q);
                    lo[r] += ld_cluster_s64(at + 16, q);
                    S[r] += (float)ld_cluster_s64(at + 24, q);
                }
            }
        }
        cluster_sync_all();
    }
    if (rank == 0 && i < n && !failed) {
#pragma unroll
        for (int r0 = 0; r0 < 4; ++r0) {
            const int r = 4 * half + r0;
            if (r >= nrhs) continue;
            // (the sums have the minus sign of Theta's digits)
            double v = -(ldexp((double)hi[r0], -30) + (ldexp((double)mid[r0], -54) + ldexp((double)lo[r0], -78)));
            v = ldexp(v, E + sx[r] - 1022);
            if (nan_row || sx[r] == 0x7ff) v = NAN;
            v += diag_extra * x[i * nrhs + r];
            // (S in units of 2^-22; sx 0: the right-hand side is zero)
            if (!nan_row && sx[r] != 0x7ff && sx[r] > 0 && !(S[r0] >= least))
                v = __longlong_as_double((long long)(MARK | (unsigned)sx[r]));
            y[i * nrhs + r] = v;
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
    }
}

// The marked entries of y in double-FP32 (matvec_f32.cuh), a CTA per 64 rows.  Up to ROW_FEW marked rows go two at a time,
// thread = every 256th source (a tile's chain over all sources takes far longer than that); more of them by
// the whole tile.  Right-hand sides beyond FP32's range are scaled by a power of two.
constexpr int ROW_FEW = 6;

template <int NU>
__global__ void __launch_bounds__(NT, 2) k_matvec_rows(const double* __restrict__ pts, long long n, int dim, KP<float> kp,
                                                       double diag_extra, const double* __restrict__ x,
                                                       double* __restrict__ y, int nrhs) {
    static_assert(NT == 32 * MVF_WARPS, "the tile's threads");
    __shared__ MvfSmem<8> sm;
    __shared__ unsigned mask[MVF_ROWS];  // marked right-hand sides of a row
    __shared__ int list[MVF_ROWS], expo[8];
    __shared__ int count;
    __shared__ double up[8];  // scale of a right-hand side
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const long long row0 = blockIdx.x * (long long)MVF_ROWS;
    if (tid < MVF_ROWS) mask[tid] = 0u;
    if (tid < 8) expo[tid] = 1022;
    if (tid == 0) count = 0;
    __syncthreads();
    bool any = false;
    for (int e = tid; e < MVF_ROWS * nrhs; e += NT) {
        const int row = e / nrhs, r = e - row * nrhs;
        if (row0 + row >= n) break;
        const double v = y[(row0 + row) * nrhs + r];
        if (is_marked(v)) {
            atomicOr(&mask[row], 1u << r);
            expo[r] = (int)(__double_as_longlong(v) & 0x7ffLL);
            any = true;
        }
    }
    if (!__syncthreads_or(any)) return;
    if (tid < MVF_ROWS && mask[tid]) list[atomicAdd(&count, 1)] = tid;
    if (tid < 8) {
        const int X = expo[tid] - 1022;
        up[tid] = X > 120 || X < -100 ? ldexp(1.0, min(max(-X, -1000), 1000)) : 1.0;
    }
    __syncthreads();
    const int rows = count;
    auto entry = [&](float2 d2) {
        const float2 r = sqrt_f2(d2);
        return make_float2(matern_nu<NU>(kp, r.x), matern_nu<NU>(kp, r.y));
    };
    auto put = [&](int row, int r, double sum) {
        const long long i = row0 + row;
        if (mask[row] >> r & 1u) y[i * nrhs + r] = sum / up[r] + diag_extra * x[i * nrhs + r];
    };
    if (rows > ROW_FEW) {
        mvf_tile<8>(sm, pts, n, dim, x, nrhs, row0, entry, [&](int r) { return up[r]; });
        for (int e = tid; e < MVF_ROWS * 8; e += NT) put(e >> 3, e & 7, sm.sum(e >> 3, e & 7));
        return;
    }
    auto coord = [&](long long i, int d) { return d < dim ? (float)pts[i * dim + d] : 0.f; };
    for (int p = 0; p < rows; p += 2) {
        const int ra = list[p], rb = list[min(p + 1, rows - 1)];
        const long long ia = row0 + ra, ib = row0 + rb;
        const float2 rx = make_float2(coord(ia, 0), coord(ib, 0)), ry = make_float2(coord(ia, 1), coord(ib, 1)),
                     rz = make_float2(coord(ia, 2), coord(ib, 2));
        float2 S[2][4], lo[2][4];
        double acc[2][8];
#pragma unroll
        for (int q = 0; q < 2; ++q)
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                S[q][r] = lo[q][r] = make_float2(0.f, 0.f);
                acc[q][2 * r] = acc[q][2 * r + 1] = 0.0;
            }
        int terms = 0;
        for (long long j = tid; j < n; j += NT) {
            const float cx = coord(j, 0), cy = coord(j, 1), cz = coord(j, 2);
            const float2 dx = __fadd2_rn(rx, make_float2(-cx, -cx)), dy = __fadd2_rn(ry, make_float2(-cy, -cy)),
                         dz = __fadd2_rn(rz, make_float2(-cz, -cz));
            const float2 k = entry(__ffma2_rn(dz, dz, __ffma2_rn(dx, dx, __fmul2_rn(dy, dy))));
            float2 xh[4], xl[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                xh[r] = xl[r] = make_float2(0.f, 0.f);
                if (2 * r < nrhs) split_f64(x[j * nrhs + 2 * r] * up[2 * r], xh[r].x, xl[r].x);
                if (2 * r + 1 < nrhs) split_f64(x[j * nrhs + 2 * r + 1] * up[2 * r + 1], xh[r].y, xl[r].y);
            }
            mvf_add<4>(k.x, k.y, xh, xl, S, lo);
            if (++terms == 32 * MVF_FLUSH) {
                mvf_flush<4>(S, lo, acc);
                terms = 0;
            }
        }
        mvf_flush<4>(S, lo, acc);
#pragma unroll
        for (int q = 0; q < 2; ++q)
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                double a = acc[q][r];
#pragma unroll
                for (int off = 16; off > 0; off >>= 1) a += __shfl_xor_sync(0xffffffffu, a, off);
                if (lane == 0) sm.acc[warp][r][q] = a;
            }
        __syncthreads();
        if (tid < 16) put(tid < 8 ? ra : rb, tid & 7, sm.sum(tid >> 3, tid & 7));
        __syncthreads();
    }
}

}  // namespace

__global__ void k_sqrt_f32(const float* __restrict__ x, long long n, float* __restrict__ root, float* __restrict__ ref) {
    const long long step = 2LL * gridDim.x * blockDim.x;
    for (long long i = 2 * (blockIdx.x * (long long)blockDim.x + threadIdx.x); i < n; i += step) {
        const bool two = i + 1 < n;
        const float2 v = make_float2(x[i], two ? x[i + 1] : 1.f), r = sqrt_f2(v);
        root[i] = r.x;
        ref[i] = sqrtf(v.x);
        if (two) {
            root[i + 1] = r.y;
            ref[i + 1] = sqrtf(v.y);
        }
    }
}

extern "C" sic_status sic_selftest_sqrt_f32(sic_handle* h, const float* x, int64_t n, float* root, float* ref,
                                            void* stream) {
    if (!h || n < 0 || (n > 0 && (!x || !root || !ref))) return SIC_ERR_INVALID;
    if (n == 0) return SIC_OK;
    SIC_CUDA_TRY(cudaSetDevice(h->device));
    long long blocks = (n + 511) / 512;
    if (blocks > 8LL * h->num_sms) blocks = 8LL * h->num_sms;
    k_sqrt_f32<<<(unsigned)blocks, 256, 0, (cudaStream_t)stream>>>(x, n, root, ref);
    SIC_CUDA_TRY(cudaGetLastError());
    return SIC_OK;
}

template <int NU>
static sic_status launch_matvec_tc(sic_handle* h, const double* pts, long long n, const sic_kernel* kp, double shift,
                                   const double* x, double* y, int nrhs, cudaStream_t s) {
    auto kern = k_matvec_tc<NU>;
    SIC_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_MV));
    const long long tiles = (n + ROWS - 1) / ROWS, slots = 2LL * h->num_sms;
    // CTAs per row tile (a cluster, at least two chunks of sources each): the number that leaves the last wave of two
    // CTAs per SM fullest -- N = 50,001: 391 tiles are 1.3 waves, eight parts 10.3
    int parts = 1;
    double best = 0.0;
    for (int p = 1; p <= 8 && (p == 1 || 2 * p <= tiles); p *= 2) {
        const long long waves = (tiles * p + slots - 1) / slots;
        const double full = (double)(tiles * p) / (double)(waves * slots);
        if (full > best + 0.02) {
            best = full;
            parts = p;
        }
    }
    int E = 0;
    const float s2 = (float)kp->variance;
    if (frexpf(s2, &E) == 0.5f) --E;  // variance <= 2^E
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(tiles * parts));
    cfg.blockDim = dim3(NT);
    cfg.dynamicSmemBytes = SMEM_MV;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)parts;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = parts > 1 ? 1 : 0;
    SIC_CUDA_TRY(cudaLaunchKernelEx(&cfg, kern, pts, n, (int)kp->dim, make_kp<float>(*kp), ldexpf(1.f, -E), E,
                                    kp->nugget + shift, x, y, nrhs, parts,
                                    (float)(sqrt((double)n) * ldexp(1.0, 22 - S_BITS)), h->d_status));
    k_matvec_rows<NU><<<(unsigned)((n + MVF_ROWS - 1) / MVF_ROWS), NT, 0, s>>>(
        pts, n, kp->dim, make_kp<float>(*kp), kp->nugget + shift, x, y, nrhs);
    SIC_CUDA_TRY(cudaGetLastError());
    return SIC_OK;
}

sic_status matvec_tc(sic_handle* h, const double* pts, long long n, const sic_kernel* kp, double shift, const double* x,
                     double* y, int nrhs, cudaStream_t s) {
    if (kp->nu_x2 == 1) return launch_matvec_tc<1>(h, pts, n, kp, shift, x, y, nrhs, s);
    if (kp->nu_x2 == 3) return launch_matvec_tc<3>(h, pts, n, kp, shift, x, y, nrhs, s);
    return launch_matvec_tc<5>(h, pts, n, kp, shift, x, y, nrhs, s);
}
