// FP64 side state of a selection: the picks' conditional variances in FP64.
//
// For the picks q_0, q_1, ... (in pick order) of a unit with targets P (a supernode's m
// members, or one column's target),
//   var1_t = Theta_{q_t q_t | q_0..q_t-1}      the pivot's conditional variance given the
//                                              earlier picks,
//   var2_t = Theta_{q_t q_t | P, q_0..q_t-1}   the same given the targets as well,
// and the pick's decrease of logdet Theta_{PP|I} per nonzero, log(var1_t / var2_t) / m
// (eq. greedy_mult; for one target it is log(v_t / v_t+1), eq. global_obj).  The pivots
// of a left-to-right factorisation are the conditional variances given what precedes
// them (eq. cond_select), so var1 is the diagonal D of the LDL^T of Theta_SS (S in pick
// order) and var2 the diagonal of the LDL^T of Theta over [P; S] at the picks' rows.
//
// One CTA per unit (persistent): the two factorisations one after the other, each by the fill's blocked LDL^T
// (ldl.cuh: panels of four columns, the trailing update as integer dot products of fixed-point rows).
// Bound: the panels' barriers and their FP64 chains, as in the fill; N = 2^16 (2,786 supernodes of 23 members, k =
// 64): 1.7 ms; 2.0 ms by flat FP64 updates, two barriers per pivot.
#include "ldl.cuh"

namespace {

// doubles: exp table, scratch, packed triangle, pivots' reciprocals, the first factorisation's pivots; then positions
struct SideLayout {
    int nmax, k;
    __host__ __device__ int xyz() const { return EXP_TAB; }
    __host__ __device__ int G() const { return xyz() + fill_scratch_doubles(nmax); }
    __host__ __device__ int piv() const { return G() + nmax * (nmax + 1) / 2; }
    __host__ __device__ int v1() const { return piv() + 4; }
    __host__ __device__ int size() const { return v1() + k; }
    __host__ __device__ size_t bytes() const { return sizeof(double) * (size_t)size() + sizeof(int) * (size_t)nmax; }
};

constexpr int side_min_ctas(int nt) { return nt == 128 ? 5 : 3; }
constexpr int SIDE_M_SPLIT = 32;  // units of at most this size run in their own launch

template <int NT>
__global__ void __launch_bounds__(NT + 32, side_min_ctas(NT)) k_side(
    const double* __restrict__ pts, long long n, int dim, KP<double> kp, const long long* __restrict__ grp_ptr,
    const int32_t* __restrict__ targets, long long n_units, const int32_t* __restrict__ sel_idx,
    const int32_t* __restrict__ sel_count, int k, int max_m, int m_lo, int m_hi, SideLayout L, double* __restrict__ pvar,
    double* __restrict__ pvar_p, double* __restrict__ gain, DevStatus* st) {
    extern __shared__ double sm[];
    double* tab = sm;
    double* xyz = sm + L.xyz();
    int* fx = reinterpret_cast<int*>(xyz);
    double* G = sm + L.G();
    double* piv = sm + L.piv();
    double* v1s = sm + L.v1();
    int* pos = reinterpret_cast<int*>(sm + L.size());
    __shared__ ClassDeal<NT + 32> deal;
    __shared__ int s_bad, s_npd;  // invalid unit or pick; a pivot not positive
    const int tid = threadIdx.x, NMAX = L.nmax;
    const bool worker = tid < NT;
    const double NaN = __longlong_as_double(0x7ff8000000000000LL);
    exp_table_fill(tab, kp.s2);

    // this launch's units (the invalid ones are the first class's to report)
    auto in_class = [&](long long u) {
        const long long m = grp_ptr ? grp_ptr[u + 1] - grp_ptr[u] : 1;
        return m < 1 || m > max_m ? m_lo == 1 : m >= m_lo && m <= m_hi;
    };
    deal.start();
    for (long long u = deal.next(n_units, in_class); u >= 0; u = deal.next(n_units, in_class)) {
        long long p0;
        int m;
        if (grp_ptr) {
            p0 = grp_ptr[u];
            m = (int)(grp_ptr[u + 1] - p0);
        } else {
            p0 = targets ? (long long)targets[u] : u;
            m = 1;
        }
        const int cnt_raw = sel_count[u];
        const bool bad_unit = m < 1 || m > max_m || p0 < 0 || p0 + m > n || cnt_raw < 0 || cnt_raw > k;
        const int cnt = bad_unit ? 0 : cnt_raw;
        if (tid == 0) {
            s_bad = bad_unit ? 1 : 0;
            s_npd = 0;
        }
        __syncthreads();
        for (int i = tid; i < cnt; i += NT + 32) {
            const long long p = sel_idx[u * k + i];
            if (p < 0 || p >= n) s_bad = 1;
        }
        __syncthreads();
        if (!s_bad && cnt > 0) {
            // Theta_SS in pick order, then Theta over [P; S]: the pivots of the picks' rows
            for (int pass = 0; pass < 2; ++pass) {
                const int m0 = pass == 0 ? 0 : m, nn = m0 + cnt;
                for (int i = worker ? tid : nn; i < nn; i += NT)
                    pos[i] = i < m0 ? (int)(p0 + i) : sel_idx[u * k + (i - m0)];
                __syncthreads();
                unit_theta<NT, true>(pts, dim, kp, tab, pos, nn, NMAX, xyz, G, nullptr, &s_npd,
                                     !(kp.nugget > 0.0));
                ldl_panels<NT, true>(G, fx, piv, nn, NMAX, &s_npd);
                if (pass == 0) {
                    for (int t = tid; t < cnt; t += NT + 32) v1s[t] = G[pk(t, t)];
                    __syncthreads();
                }
            }
        }
        const int bad = s_bad ? 1 : (s_npd ? 2 : 0);
        if (bad && tid == 0) record_error(st, bad == 2 ? SIC_ERR_NOT_PD : SIC_ERR_INVALID, u);
        const int nout = bad_unit ? ((cnt_raw > 0 && cnt_raw <= k) ? cnt_raw : 0) : cnt;
        for (int t = tid; t < nout; t += NT + 32) {
            double v1 = NaN, v2 = NaN, g = NaN;
            if (!bad) {
                v1 = v1s[t];
                v2 = G[pk(m + t, m + t)];
                g = log(v1 / v2) / m;
            }
            if (pvar) pvar[u * k + t] = v1;
            if (pvar_p) pvar_p[u * k + t] = v2;
            if (gain) gain[u * k + t] = g;
        }
        __syncthreads();
    }
}

// ---- few or small units ----
//
// Both factorisations of a unit at once, right-looking over all 256 threads, two barriers per pivot.  It takes more
// work than the panels, but a unit's chain is shorter and there is one launch of one class: with few units per SM, or
// few picks, that is the time.  Few units, k = 55: 262 260 us against 451 by the panels, 857 589 against 636; 1,121 with k = 64
// 910 against 949, 1,410 1,177 against 1,042.  2,816 units of up to 64 members: k = 16 377 us against 442, 32 694 against 722,
// 40 971 against 915, 64 1,994 against 1,884; of up to 24: 40 745 against 772, 48 990 each, 64 1,730 against 1,569;
// 32,768 columns: k = 32 2.47 ms against 3.31, 64 9.98 against 10.12.
constexpr int FLAT_NT = 256;

struct FlatLayout {
    int nmax, k;
    int dec;  // 1: the packed-triangle decode table follows the doubles (when it fits)
    __host__ __device__ int tab() const { return 0; }
    __host__ __device__ int A() const { return EXP_TAB; }
    __host__ __device__ int B() const { return A() + nmax * (nmax + 1) / 2; }
    __host__ __device__ int xyz() const { return B() + k * (k + 1) / 2; }
    __host__ __device__ int clA() const { return xyz() + 3 * nmax; }
    __host__ __device__ int clB() const { return clA() + nmax; }
    __host__ __device__ int rdA() const { return clB() + k; }
    __host__ __device__ int rdB() const { return rdA() + nmax; }
    __host__ __device__ int size() const { return rdB() + k; }  // doubles
    // then the decode table of the packed triangle: entry e -> (row << 8) | column
    __host__ __device__ int tri() const { return nmax * (nmax + 1) / 2; }
    __host__ __device__ size_t bytes() const {
        return sizeof(double) * (size_t)size() + (dec ? sizeof(uint16_t) * (size_t)tri() : 0);
    }
};

__global__ void __launch_bounds__(FLAT_NT) k_side_flat(const double* __restrict__ pts, long long n, int dim,
                                                  KP<double> kp, const long long* __restrict__ grp_ptr,
                                                  const int32_t* __restrict__ targets, long long n_units,
                                                  const int32_t* __restrict__ sel_idx,
                                                  const int32_t* __restrict__ sel_count, int k, int max_m,
                                                  FlatLayout L, double* __restrict__ pvar,
                                                  double* __restrict__ pvar_p, double* __restrict__ gain,
                                                  DevStatus* st) {
    extern __shared__ double sm[];
    double* tab = sm + L.tab();
    double* A = sm + L.A();
    double* B = sm + L.B();
    double* xyz = sm + L.xyz();
    double* clA = sm + L.clA();
    double* clB = sm + L.clB();
    double* rdA = sm + L.rdA();
    double* rdB = sm + L.rdB();
    uint16_t* dec = reinterpret_cast<uint16_t*>(sm + L.size());  // packed-triangle decode table
    __shared__ int s_bad;  // 1: invalid unit or pick, 2: a pivot not positive
    const int tid = threadIdx.x, NMAX = L.nmax;
    const double diag = kp.s2 + kp.nugget;
    const bool singular = !(kp.nugget > 0.0);
    const double NaN = __longlong_as_double(0x7ff8000000000000LL);
    exp_table_fill(tab, kp.s2);
    if (L.dec)
        for (int e = threadIdx.x; e < L.tri(); e += blockDim.x) {
            const int r = pk_row(e);
            dec[e] = (uint16_t)((r << 8) | (e - r * (r + 1) / 2));
        }
    // row and column of packed-triangle element e: from the table, else by the square root
    auto decode = [&](int e, int& r, int& c) {
        if (L.dec) {
            const unsigned v = dec[e];
            r = (int)(v >> 8);
            c = (int)(v & 255u);
        } else {
            r = pk_row(e);
            c = e - r * (r + 1) / 2;
        }
    };

    for (long long u = blockIdx.x; u < n_units; u += gridDim.x) {
        long long p0;
        int m;
        if (grp_ptr) {
            p0 = grp_ptr[u];
            m = (int)(grp_ptr[u + 1] - p0);
        } else {
            p0 = targets ? (long long)targets[u] : u;
            m = 1;
        }
        const int cnt_raw = sel_count[u];
        const bool bad_unit = m < 1 || m > max_m || p0 < 0 || p0 + m > n || cnt_raw < 0 || cnt_raw > k;
        const int cnt = bad_unit ? 0 : cnt_raw;
        const int nn = m + cnt;
        if (tid == 0) s_bad = bad_unit ? 1 : 0;
        __syncthreads();
        for (int i = tid; i < (bad_unit ? 0 : nn); i += FLAT_NT) {
            long long p = i < m ? p0 + i : (long long)sel_idx[u * k + (i - m)];
            if (p < 0 || p >= n) {
                s_bad = 1;
                p = p0;
            }
#pragma unroll
            for (int d = 0; d < 3; ++d) xyz[d * NMAX + i] = (d < dim) ? pts[p * dim + d] : 0.0;
        }
        __syncthreads();
        if (!s_bad && cnt > 0) {
            // Theta over [P; S] (packed lower) and a copy of its S block
            const int tri = nn * (nn + 1) / 2;
            if (singular)  // coincident points without a nugget, whatever rounding would leave of the pivot
                for (int e = tid; e < tri; e += FLAT_NT) {
                    int a, b;
                    decode(e, a, b);
                    const double dx = xyz[a] - xyz[b], dy = xyz[NMAX + a] - xyz[NMAX + b],
                                 dz = xyz[2 * NMAX + a] - xyz[2 * NMAX + b];
                    if (a != b && __double_as_longlong(fma(dz, dz, fma(dy, dy, dx * dx))) == 0LL) s_bad = 2;
                }
            for (int e = tid; e < tri; e += FLAT_NT) {
                int a, b;
                decode(e, a, b);
                double v = diag;
                if (a != b) {
                    const double dx = xyz[a] - xyz[b], dy = xyz[NMAX + a] - xyz[NMAX + b],
                                 dz = xyz[2 * NMAX + a] - xyz[2 * NMAX + b];
                    v = matern_d2_fast(kp, fma(dz, dz, fma(dy, dy, dx * dx)), tab);
                }
                A[e] = v;
                if (b >= m) B[pk(a - m, b - m)] = v;
            }
            if (tid == 0) {
                rdA[0] = 1.0 / diag;
                rdB[0] = 1.0 / diag;
            }
            __syncthreads();
            for (int j = 0; j < nn; ++j) {
                const bool jb = j < cnt;
                const double ra = rdA[j], rb = jb ? rdB[j] : 0.0;
                for (int a = j + 1 + tid; a < nn; a += FLAT_NT) clA[a] = A[pk(a, j)] * ra;
                if (jb)
                    for (int a = j + 1 + tid; a < cnt; a += FLAT_NT) clB[a] = B[pk(a, j)] * rb;
                __syncthreads();
                const int TA = nn - j - 1, TB = jb ? cnt - j - 1 : 0;
                const int eA = TA * (TA + 1) / 2, eB = TB * (TB + 1) / 2;
                for (int e = tid; e < eA + eB; e += FLAT_NT) {
                    const bool inA = e < eA;
                    const int f = inA ? e : e - eA;
                    int r, c;
                    decode(f, r, c);
                    const int a = j + 1 + r, b = j + 1 + c;
                    double* M = inA ? A : B;
                    const double* cl = inA ? clA : clB;
                    const double v = fma(-cl[a], M[pk(b, j)], M[pk(a, b)]);
                    M[pk(a, b)] = v;
                    if (r == 0) {  // the next pivot (a = b = j + 1)
                        if (!(v > 0.0)) s_bad = 2;
                        (inA ? rdA : rdB)[j + 1] = 1.0 / v;
                    }
                }
                __syncthreads();
            }
        }
        const int bad = s_bad;
        if (bad && tid == 0) record_error(st, bad == 2 ? SIC_ERR_NOT_PD : SIC_ERR_INVALID, u);
        const int nout = bad_unit ? ((cnt_raw > 0 && cnt_raw <= k) ? cnt_raw : 0) : cnt;
        for (int t = tid; t < nout; t += FLAT_NT) {
            double v1 = NaN, v2 = NaN, g = NaN;
            if (!bad) {
                v1 = B[pk(t, t)];
                v2 = A[pk(m + t, m + t)];
                g = log(v1 / v2) / m;
            }
            if (pvar) pvar[u * k + t] = v1;
            if (pvar_p) pvar_p[u * k + t] = v2;
            if (gain) gain[u * k + t] = g;
        }
        __syncthreads();
    }
}

constexpr int FLAT_UNITS_PER_SM = 8;
constexpr int PANELS_K = 40, PANELS_ROWS = 72;  // least picks, and least rows of the largest unit, for the panels

}  // namespace

extern "C" sic_status sic_side_state_fp64(sic_handle* h, const double* pts, int64_t n, const sic_kernel* kp,
                                          const int64_t* grp_ptr, const int32_t* targets, int64_t n_units,
                                          int32_t max_m, const int32_t* sel_idx, const int32_t* sel_count,
                                          int32_t k, double* pvar, double* pvar_p, double* gain, void* stream) {
    if (!h || !pts || !sic_valid_kernel(kp) || n < 1 || n_units < 0 || k < 1 || max_m < 1) return SIC_ERR_INVALID;
    if (!grp_ptr && max_m != 1) return SIC_ERR_INVALID;
    if (k > 128 || max_m > 64) return SIC_ERR_UNSUPPORTED;
    if (!pvar && !pvar_p && !gain) return SIC_ERR_INVALID;
    if (n_units == 0) return SIC_OK;
    if (!sel_idx || !sel_count) return SIC_ERR_INVALID;
    if (n_units > 0x7fffffffLL) return SIC_ERR_UNSUPPORTED;
    SIC_CUDA_TRY(cudaSetDevice(h->device));
    FlatLayout F;
    F.nmax = max_m + k;
    F.k = k;
    F.dec = 1;
    if (F.bytes() > 227 * 1024 - 1024) F.dec = 0;
    const bool panels = n_units > (int64_t)FLAT_UNITS_PER_SM * h->num_sms && k >= PANELS_K && max_m + k >= PANELS_ROWS;
    if (!panels && F.bytes() <= 227 * 1024 - 1024) {
        const size_t smem = F.bytes();
        SIC_CUDA_TRY(cudaFuncSetAttribute(k_side_flat, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        const int grid = persistent_grid(h, k_side_flat, FLAT_NT, smem, n_units);
        k_side_flat<<<grid, FLAT_NT, smem, (cudaStream_t)stream>>>(pts, n, kp->dim, make_kp<double>(*kp),
                                                                   (const long long*)grp_ptr, targets, n_units, sel_idx,
                                                                   sel_count, k, max_m, F, pvar, pvar_p, gain,
                                                                   h->d_status);
        SIC_CUDA_TRY(cudaGetLastError());
        return SIC_OK;
    }
    // two size classes, as in the fill: the shared memory (and so the CTAs per SM) of each launch fits its own
    // largest unit
    const int split = max_m < SIDE_M_SPLIT ? max_m : SIDE_M_SPLIT;
    for (int c = 0; c < 2; ++c) {
        const int lo = c == 0 ? 1 : split + 1, hi = c == 0 ? split : max_m;
        if (lo > hi) break;
        SideLayout L;
        L.nmax = hi + k;
        L.k = k;
        const size_t smem = L.bytes();
        const int nt = L.nmax <= 128 && c == 0 ? 128 : 256;  // a worker thread per row
        auto kern = nt == 128 ? k_side<128> : k_side<256>;
        // opt in at any size: the static arrays count against the 48 KB default as well
        SIC_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        const int grid = persistent_grid(h, kern, nt + 32, smem, n_units);
        kern<<<grid, nt + 32, smem, (cudaStream_t)stream>>>(pts, n, kp->dim, make_kp<double>(*kp),
                                                            (const long long*)grp_ptr, targets, n_units, sel_idx,
                                                            sel_count, k, max_m, lo, hi, L, pvar, pvar_p, gain,
                                                            h->d_status);
    }
    SIC_CUDA_TRY(cudaGetLastError());
    return SIC_OK;
}
