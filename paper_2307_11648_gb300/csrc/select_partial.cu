// Partial selection for nonadjacent groups (Section 5.1.1; Section 5.2 "Partial selection";
// Appendix C.3).
//
// A group's targets P (positions i_1 < ... < i_m, not consecutive) share one selection, but a
// candidate j conditions only the targets before it (i < j).  Objective: the log-determinant
// of the partially conditioned target covariance, sum_i log Theta_{ii | s_i \ i} (eq.
// partial_kl), greedily minimised.  The state is the Cholesky factor L of the joint
// covariance of the targets and picks, columns ordered from the latest position to the
// earliest (a column's pivot is then conditioned on exactly the later points), with a row for
// every candidate and target:
//   score    thread = candidate row j: walk the columns carrying v = Theta_{jj | columns so
//            far}; a target column e with e < j gets the factor (v - L_jc^2) / v -- its
//            variance ratio after conditioning on j (eq. obj_partial) -- and v -= L_jc^2 (eq.
//            partial_induct).  The product of the factors is the exponential of minus the
//            objective's decrease; it never falls below v_last / v_0, so it cannot underflow;
//            the least product wins (ties: the earliest candidate).  A candidate whose v after
//            the last column is below the floor is exhausted.
//   insert   the pick q goes to its place p (the number of columns of later points): the
//            columns before p stay; the new column is Theta_{:,q | first p} / sqrt(Theta_{qq |
//            first p}) by left-looking; the columns from p on are downdated in place by it
//            column by column (eq. chol_partial_update): one warp forms the rotations in order
//            from the pivot rows (the targets and picks), the candidate rows apply them.
// Columns live in physical slots in insertion order; `pk/opos` map the logical (latest-first)
// order to the pivot row and slot and to the target position (INT_MAX for a pick).  One CTA per
// group (persistent, two size classes), L in shared memory, rows spread over the threads of all warps but the first.
//
// A step walks each candidate row's columns twice: the left-looking product over the first p, then
// one walk that applies the rotations and takes the next step's score as it goes.  The first warp
// runs the rotations' serial chain at the same time -- its rows' downdate values in registers, a pivot's value
// by shuffle, the entries of the next column loaded ahead -- and hands them over 16 columns at a time through
// named barriers; the target block is factored once, before the candidates' rows, which need no barrier then.
// Bound: that chain, about 200 cycles per column in one warp's instructions (a chain without the
// shuffle took as long), with the walk of two warps per scheduler behind it.  N = 2^16, 256 candidates, k = 64 (2,811
// groups): 16.1 ms with score, columns and rotations one after the other, 9.0 ms with one CTA per SM, 7.1 ms now that
// the smaller groups run two to an SM.
#include <limits.h>

#include "sic_internal.cuh"

namespace {

constexpr int PT_NT = 512;     // one CTA per SM
constexpr int PT_NT_2 = 288;   // groups whose state fits an SM twice: a row per thread up to 256 candidates

__device__ __forceinline__ float pt_div(float a, float b) { return __fdividef(a, b); }
__device__ __forceinline__ double pt_div(double a, double b) { return a / b; }

// A column's rotation from its pivot entry lee and downdate value xe: the new pivot
// rr = sqrt(lee^2 - xe^2), cos = rr / lee, sin = xe / lee and 1 / cos = lee / rr.  Only xe is on the
// insertion's serial chain; a = lee^2 and, in FP32, ilee = 1 / lee come from the pivot's own lane.  FP32
// takes one fast reciprocal and one reciprocal square root; FP64 divides exactly.
__device__ __forceinline__ float pt_inv(float lee) { return __fdividef(1.f, lee); }
__device__ __forceinline__ double pt_inv(double) { return 0.0; }
__device__ __forceinline__ bool pt_rot(float lee, float a, float ilee, float xe, float& rr, float& cth, float& sth,
                                       float& icth) {
    const float rr2 = fmaf(-xe, xe, a);
    const float irr = rsqrtf(rr2);
    rr = rr2 * irr;
    cth = rr * ilee;
    sth = xe * ilee;
    icth = lee * irr;
    return rr2 > 0.f && lee > 0.f;
}
__device__ __forceinline__ bool pt_rot(double lee, double a, double, double xe, double& rr, double& cth, double& sth,
                                       double& icth) {
    const double rr2 = fma(-xe, xe, a);
    rr = sqrt(rr2 > 0.0 ? rr2 : 0.0);
    cth = rr / lee;
    sth = xe / lee;
    icth = lee / rr;
    return rr2 > 0.0 && lee > 0.0;
}

struct PtLayout {
    int R, W, P;  // rows (candidates + targets), columns (targets + picks), row pitch (odd)
    __host__ __device__ size_t bytes(size_t tsz) const {
        return tsz * ((size_t)R * P + 4 * (size_t)R + 3 * (size_t)W) + sizeof(int) * ((size_t)R + 4 * (size_t)W);
    }
    // the size that decides which problems are taken (the state's size with two more integers per row)
    size_t limit_bytes(size_t tsz) const {
        return tsz * ((size_t)R * P + 4 * (size_t)R + 3 * (size_t)W) + sizeof(int) * (2 * (size_t)R + 3 * (size_t)W);
    }
};

constexpr int PT_STATIC = 4096;  // static shared memory and what the system keeps of a CTA's share, at most
constexpr int PT_MIN_CLASS = 4;
constexpr int PT_CHUNK = 16;  // columns handed over per named barrier
constexpr int PT_EL = 6;      // element rows per lane of the first warp: 32 * PT_EL = 192 columns

template <int NT>
__device__ __forceinline__ void pt_arrive(int id) {
    asm volatile("barrier.arrive %0, %1;" ::"r"(id), "n"(NT) : "memory");
}
template <int NT>
__device__ __forceinline__ void pt_sync(int id) {
    asm volatile("barrier.sync %0, %1;" ::"r"(id), "n"(NT) : "memory");
}

// The least (key, index) over the warp, key INFINITY where there is none
__device__ __forceinline__ void pt_warp_min(float& key, int& idx) {
    const unsigned b = __float_as_uint(key);
    const unsigned o = (b & 0x80000000u) ? ~b : (b | 0x80000000u);  // monotone in the key (-0 < +0 apart)
    const unsigned lo = __reduce_min_sync(0xffffffffu, o);
    idx = (int)__reduce_min_sync(0xffffffffu, o == lo ? (unsigned)idx : (unsigned)INT_MAX);
    key = __uint_as_float((lo & 0x80000000u) ? (lo & 0x7fffffffu) : ~lo);
}
__device__ __forceinline__ void pt_warp_min(double& key, int& idx) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const double ok = __shfl_xor_sync(0xffffffffu, key, off);
        const int oi = __shfl_xor_sync(0xffffffffu, idx, off);
        if (ok < key || (ok == key && oi < idx)) {
            key = ok;
            idx = oi;
        }
    }
}

// Rotations j0 .. min(j0 + 32, ne) of a downdate, by the first warp: lane = pivot row of rotation j0 + lane
// (block 0) and of j0 + 32 i + lane (block i < NA, to which the rotations are applied), with each row's downdate
// value x, its offset in Lm, its entry L in the current column and its pivot entry lee.  pc: (row << 8 | slot) of
// the columns from the first rotation on.  Rotations go to rc / rsn / ric and are handed over per chunk.
template <int NT, int NA, typename T>
__device__ __forceinline__ bool pt_chain(T* __restrict__ Lm, const int* __restrict__ pc, T* __restrict__ rc,
                                         T* __restrict__ rsn, T* __restrict__ ric, int j0, int ne, int lane,
                                         const int (&row)[PT_EL], const T (&lee)[PT_EL], T (&x)[PT_EL], T (&L)[PT_EL]) {
    constexpr unsigned FULL = 0xffffffffu;
    bool ok = true;
    const T a0 = lee[0] * lee[0], i0 = pt_inv(lee[0]);
    int s = pc[j0] & 255, s1 = pc[min(j0 + 1, ne - 1)] & 255;
    const int n = min(32, ne - j0);
    for (int cc = 0; cc < n; ++cc) {
        const int j = j0 + cc;
        const T le = __shfl_sync(FULL, lee[0], cc), la = __shfl_sync(FULL, a0, cc), li = __shfl_sync(FULL, i0, cc);
        const T xe = __shfl_sync(FULL, x[0], cc);
        const int s2 = pc[min(j + 2, ne - 1)] & 255;
        T ln[NA];
#pragma unroll
        for (int i = 0; i < NA; ++i) ln[i] = Lm[row[i] + s1];
        T rr, cth, sth, icth;
        ok = pt_rot(le, la, li, xe, rr, cth, sth, icth) && ok;
        if (lane == 0) {
            rc[j] = cth;
            rsn[j] = sth;
            ric[j] = icth;
        }
#pragma unroll
        for (int i = 0; i < NA; ++i) {
            const T xr = x[i];
            const T nl = (L[i] - sth * xr) * icth;
            const T xn = cth * xr - sth * nl;
            const bool act = i == 0 ? (lane > cc && lane < n) : (j0 + 32 * i + lane < ne);
            if (act) {
                Lm[row[i] + s] = nl;
                x[i] = xn;
            }
            L[i] = ln[i];
        }
        if (lane == cc) Lm[row[0] + s] = rr;
        s = s1;
        s1 = s2;
        if ((j & (PT_CHUNK - 1)) == PT_CHUNK - 1 || j == ne - 1) pt_arrive<NT>(1 + j / PT_CHUNK);
    }
    return ok;
}

// groups of m_lo .. m_hi members
template <typename T, int NT>
__global__ void __launch_bounds__(NT, NT == PT_NT ? 1 : 2) k_select_partial(
    const double* __restrict__ pts, long long n, int dim, KP<T> kp, T floor_, const long long* __restrict__ grp_ptr,
    const long long* __restrict__ members, long long n_grp, const long long* __restrict__ cand_ptr,
    const int32_t* __restrict__ cand_idx, int max_cand, int max_m, int m_lo, int m_hi, int k, int32_t* __restrict__ sel_idx,
    int32_t* __restrict__ sel_count, double* __restrict__ gain, PtLayout Lay, DevStatus* st) {
    extern __shared__ __align__(16) unsigned char smraw[];
    T* Lm = reinterpret_cast<T*>(smraw);              // [R][P]
    T* X = Lm + (size_t)Lay.R * Lay.P;                // [3][R] coordinates
    T* xv = X + 3 * Lay.R;                            // [R] downdate vector
    T* rc = xv + Lay.R;                               // [W] rotation of logical column c: cos,
    T* rsn = rc + Lay.W;                              //     sin,
    T* ric = rsn + Lay.W;                             //     1 / cos
    int* pos = reinterpret_cast<int*>(ric + Lay.W);   // [R] positions; ~position once the row is a pivot
    int* pk = pos + Lay.R;                            // 2 x [W] (pivot row << 8 | slot) of logical column c
    int* opos = pk + 2 * Lay.W;                       // 2 x [W] target position of column c (INT_MAX: a pick)
    __shared__ T s_rs, s_d;
    __shared__ int s_fail;
    __shared__ T wkey[NT / 32];
    __shared__ int widx[NT / 32];
    __shared__ double gprod[128];
    __shared__ int gcnd[128];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int WT = NT - 32;  // threads of the walking warps
    constexpr unsigned FULL = 0xffffffffu;
    const int wt = tid - 32;
    const int PP = Lay.P, RR = Lay.R;
    const T diag = kp.s2 + kp.nugget;
    const T INF = (T)INFINITY;

    __shared__ ClassDeal<NT> deal;
    // this launch's groups (the invalid ones are the first class's to report)
    auto in_class = [&](long long g) {
        const long long m = grp_ptr[g + 1] - grp_ptr[g];
        return m < 1 || m > max_m ? m_lo == 1 : m >= m_lo && m <= m_hi;
    };
    deal.start();
    for (long long g = deal.next(n_grp, in_class); g >= 0; g = deal.next(n_grp, in_class)) {
        const long long a0 = grp_ptr[g];
        const int m = (int)(grp_ptr[g + 1] - a0);
        const long long b0 = cand_ptr[g];
        const int C = (int)(cand_ptr[g + 1] - b0);
        if (m < 1 || m > max_m || C < 0 || C > max_cand) {
            if (tid == 0) {
                record_error(st, SIC_ERR_INVALID, g);
                sel_count[g] = 0;
            }
            for (int q = tid; q < k; q += NT) sel_idx[g * k + q] = -1;
            continue;
        }
        const int R = C + m;
        const long long first = members[a0];
        if (tid == 0) s_fail = (first < 0 || first >= n) ? 1 : 0;
        double org[3] = {0.0, 0.0, 0.0};
        if constexpr (sizeof(T) == 4)
            if (first >= 0 && first < n)
                for (int d = 0; d < dim; ++d) org[d] = pts[first * dim + d];
        __syncthreads();
        for (int r = tid; r < R; r += NT) {
            long long p = r < C ? (long long)cand_idx[b0 + r] : members[a0 + (r - C)];
            const bool bad = p < 0 || p >= n || (r < C && p <= first) ||
                             (r > C && p <= members[a0 + (r - C) - 1]);
            if (bad) {
                s_fail = 1;
                p = 0;
            }
            pos[r] = (int)p;
#pragma unroll
            for (int d = 0; d < 3; ++d) X[d * RR + r] = (d < dim) ? (T)(pts[p * dim + d] - org[d]) : (T)0;
        }
        __syncthreads();
        if (s_fail) {
            if (tid == 0) {
                record_error(st, SIC_ERR_INVALID, g);
                sel_count[g] = 0;
            }
            for (int q = tid; q < k; q += NT) sel_idx[g * k + q] = -1;
            __syncthreads();
            continue;
        }
        int cur = 0;  // which half of pk / opos holds the current maps
        auto theta = [&](int r, T qx, T qy, T qz) -> T {
            const T dx = X[r] - qx, dy = X[RR + r] - qy, dz = X[2 * RR + r] - qz;
            return matern<T>(kp, sic_sqrt(dx * dx + dy * dy + dz * dz));
        };
        // by the first warp: Theta_{qq | first p} and 1 / its root to s_d, s_rs, from row q's entries
        auto pivot = [&](int q, int p, const int* __restrict__ cols) {
            T part = (T)0;
            for (int c = lane; c < p; c += 32) {
                const T l = Lm[q * PP + (cols ? (cols[c] & 255) : c)];
                part = fma(l, l, part);
            }
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) part += __shfl_xor_sync(FULL, part, off);
            if (lane == 0) {
                const T d = diag - part;  // Theta_{qq | first p}
                s_d = d;
                if (!(d > (T)0)) s_fail = 2;
                s_rs = (d > (T)0) ? (T)1 / sic_sqrt(d) : (T)0;
            }
        };

        // ---- the targets, latest first: column c = slot c = row C + m - 1 - c, no downdates ----
        bool ok = true;
        for (int c = 0; c < m; ++c) {
            const int q = C + m - 1 - c;
            if (warp == 0) pivot(q, c, nullptr);
            __syncthreads();
            if (s_fail) {
                ok = false;
                break;
            }
            const T rs = s_rs;
            if (tid == 0) {
                Lm[q * PP + c] = s_d * rs;  // sqrt(d)
                ric[c] = rs;                // (for the candidates' rows below)
                pk[c] = (q << 8) | c;
                opos[c] = pos[q];
            }
            const int r = C + wt;  // the targets still to come
            if (wt >= 0 && r < q) {
                T num = theta(r, X[q], X[RR + q], X[2 * RR + q]);
                for (int c1 = 0; c1 < c; ++c1) num = fma(-Lm[r * PP + c1], Lm[q * PP + c1], num);
                Lm[r * PP + c] = num * rs;
            }
            __syncthreads();
        }
        T bk = INF;  // this thread's best candidate
        int bi = INT_MAX;
        if (ok) {
            for (int r = wt; wt >= 0 && r < C; r += WT) {
                const int pj = pos[r];
                T v = diag, pr = (T)1;
                for (int c = 0; c < m; ++c) {
                    const int q = C + m - 1 - c;
                    T num = theta(r, X[q], X[RR + q], X[2 * RR + q]);
#pragma unroll 4
                    for (int c1 = 0; c1 < c; ++c1) num = fma(-Lm[r * PP + c1], Lm[q * PP + c1], num);
                    const T l = num * ric[c];
                    Lm[r * PP + c] = l;
                    const T vn = fma(-l, l, v);
                    if (opos[c] < pj) pr = pt_div(pr * vn, v);  // a target j conditions (eq. obj_partial)
                    v = vn;                                     // eq. partial_induct
                }
                if (v >= floor_ && (pr < bk || (pr == bk && r < bi))) {
                    bk = pr;
                    bi = r;
                }
            }
            __syncthreads();
            for (int r = C + tid; r < R; r += NT) pos[r] = ~pos[r];
            // (visible after the first step's barriers)
        }
        int ncol = m, t = 0;
        for (; t < k && ok; ++t) {
            pt_warp_min(bk, bi);
            if (lane == 0) {
                wkey[warp] = bk;
                widx[warp] = bi;
            }
            __syncthreads();
            T gk = lane < NT / 32 ? wkey[lane] : INF;
            int q = lane < NT / 32 ? widx[lane] : INT_MAX;
            pt_warp_min(gk, q);
            if (q == INT_MAX) break;
            const int pq = pos[q];
            const int* __restrict__ pc = pk + cur * Lay.W;
            const int* __restrict__ oc = opos + cur * Lay.W;
            // its place, and the targets it conditions (its nonzeros)
            int p = 0, nc = 0;
            for (int c0 = 0; c0 < ncol; c0 += 32) {
                const int c = c0 + lane;
                p += __popc(__ballot_sync(FULL, c < ncol && ~pos[pc[c < ncol ? c : 0] >> 8] > pq));
                nc += __popc(__ballot_sync(FULL, c < ncol && oc[c < ncol ? c : 0] < pq));
            }
            if (tid == 0) {
                gprod[t] = (double)gk;
                gcnd[t] = nc;
                sel_idx[g * k + t] = pq;
            }
            // ---- the new column, left-looking (candidates, and pivots at earlier positions) ----
            if (warp == 0) {
                pivot(q, p, pc);
            } else {
                const T qx = X[q], qy = X[RR + q], qz = X[2 * RR + q];
                const T* __restrict__ Lq = Lm + q * PP;
                for (int r = wt; r < R; r += WT) {
                    const int ps = pos[r];
                    if (r == q || (ps < 0 && ~ps > pq)) continue;
                    const T* __restrict__ Lr = Lm + r * PP;
                    T num = theta(r, qx, qy, qz);
#pragma unroll 8
                    for (int c = 0; c < p; ++c) {
                        const int s = pc[c] & 255;
                        num = fma(-Lr[s], Lq[s], num);
                    }
                    xv[r] = num;
                }
            }
            __syncthreads();
            if (s_fail) {
                ok = false;
                break;
            }
            const T rs = s_rs;
            for (int r = wt; wt >= 0 && r < R; r += WT) {
                const int ps = pos[r];
                if (r == q) {
                    Lm[r * PP + ncol] = s_d * rs;  // sqrt(d)
                    pos[r] = ~pq;
                } else if (ps >= 0 || ~ps < pq) {
                    const T u = xv[r] * rs;
                    Lm[r * PP + ncol] = u;
                    xv[r] = u;
                }
            }
            __syncthreads();
            const int ne = ncol - p;  // columns to downdate: the rotations are numbered 0 .. ne - 1 from p
            if (warp == 0) {
                // the rotations, in order, from the pivot rows alone -- the rows of the targets and picks
                // at earlier positions than q, which are the pivots of those same columns
                int row[PT_EL];
                T lee[PT_EL], x[PT_EL], L[PT_EL];
                const int s = ne > 0 ? (pc[p] & 255) : 0;
#pragma unroll
                for (int i = 0; i < PT_EL; ++i) {
                    const int c2 = lane + 32 * i;
                    row[i] = q * PP;  // (rows beyond the last: read, not written)
                    lee[i] = x[i] = L[i] = (T)0;
                    if (c2 < ne) {
                        const int e = pc[p + c2];
                        row[i] = (e >> 8) * PP;
                        lee[i] = Lm[row[i] + (e & 255)];
                        x[i] = xv[e >> 8];
                        L[i] = Lm[row[i] + s];
                    }
                }
                bool good = true;
                for (int j0 = 0; j0 < ne; j0 += 32) {
                    const int na = (ne - j0 + 31) >> 5;
                    const int* pj = pc + p;
                    T *c_ = rc + p, *s_ = rsn + p, *i_ = ric + p;
                    const bool g1 = na == 1   ? pt_chain<NT, 1>(Lm, pj, c_, s_, i_, j0, ne, lane, row, lee, x, L)
                                    : na == 2 ? pt_chain<NT, 2>(Lm, pj, c_, s_, i_, j0, ne, lane, row, lee, x, L)
                                    : na == 3 ? pt_chain<NT, 3>(Lm, pj, c_, s_, i_, j0, ne, lane, row, lee, x, L)
                                              : pt_chain<NT, PT_EL>(Lm, pj, c_, s_, i_, j0, ne, lane, row, lee, x, L);
                    good = good && g1;
#pragma unroll
                    for (int i = 0; i + 1 < PT_EL; ++i) {  // the next block of pivot rows
                        row[i] = row[i + 1];
                        lee[i] = lee[i + 1];
                        x[i] = x[i + 1];
                        L[i] = L[i + 1];
                    }
                }
                if (!good && lane == 0) s_fail = 2;
                bk = INF;
                bi = INT_MAX;
            } else {
                // the maps with the new column in its place, for the next step
                if (wt <= ncol) {
                    int e, o;
                    if (wt == p) {
                        e = (q << 8) | ncol;
                        o = INT_MAX;
                    } else {
                        e = pc[wt < p ? wt : wt - 1];
                        o = oc[wt < p ? wt : wt - 1];
                    }
                    pk[(cur ^ 1) * Lay.W + wt] = e;
                    opos[(cur ^ 1) * Lay.W + wt] = o;
                }
                bk = INF;
                bi = INT_MAX;
                bool wait = true;  // the first rows wait for the rotations
                int r = wt;
                do {
                    const bool live = r < C && pos[r < C ? r : 0] >= 0;
                    T* __restrict__ Lr = Lm + (live ? r : 0) * PP;
                    const int pj = live ? pos[r] : 0;
                    T v = diag, pr = (T)1, xr = (T)0;
                    auto take = [&](T l, int o) {
                        const T vn = fma(-l, l, v);
                        if (o < pj) pr = pt_div(pr * vn, v);  // a target j conditions (eq. obj_partial)
                        v = vn;                               // eq. partial_induct
                    };
                    if (live) {
                        xr = xv[r];
#pragma unroll 4
                        for (int c = 0; c < p; ++c) take(Lr[pc[c] & 255], oc[c]);
                        take(xr, INT_MAX);
                    }
                    for (int j0 = 0; j0 < ne; j0 += PT_CHUNK) {
                        if (wait) {
                            __syncwarp();
                            pt_sync<NT>(1 + j0 / PT_CHUNK);
                        }
                        if (live) {
                            const int c1 = p + min(j0 + PT_CHUNK, ne);
#pragma unroll 4
                            for (int c = p + j0; c < c1; ++c) {
                                const int s = pc[c] & 255;
                                const T nl = (Lr[s] - rsn[c] * xr) * ric[c];
                                Lr[s] = nl;
                                xr = rc[c] * xr - rsn[c] * nl;
                                take(nl, oc[c]);
                            }
                        }
                    }
                    if (live && v >= floor_ && (pr < bk || (pr == bk && r < bi))) {
                        bk = pr;
                        bi = r;
                    }
                    wait = false;
                    r += WT;
                } while (r - wt < C);
            }
            __syncthreads();
            if (s_fail) {
                ok = false;
                break;
            }
            cur ^= 1;
            ++ncol;
        }
        if (!ok && tid == 0) record_error(st, SIC_ERR_NOT_PD, g);
        if (tid == 0) sel_count[g] = t;
        for (int q = t + tid; q < k; q += NT) sel_idx[g * k + q] = -1;
        if (gain) {
            __syncthreads();
            // decrease of the objective per nonzero (the targets the pick conditions)
            for (int q = tid; q < t; q += NT) gain[g * k + q] = -log(gprod[q]) / (gcnd[q] > 0 ? gcnd[q] : 1);
        }
        __syncthreads();
    }
}

// Per-column selection lists of nonadjacent groups for the fill: member i's column holds the
// later members and the picks after i (Section 5.1.1); one warp per group.
__global__ void k_partial_columns(long long n, const long long* __restrict__ grp_ptr,
                                  const long long* __restrict__ members, long long n_grp,
                                  const int32_t* __restrict__ sel_idx, const int32_t* __restrict__ sel_count, int k,
                                  int kc, int32_t* __restrict__ col_sel, int32_t* __restrict__ col_count,
                                  DevStatus* st) {
    const int lane = threadIdx.x & 31;
    const long long nw = (long long)gridDim.x * (blockDim.x >> 5);
    for (long long g = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; g < n_grp; g += nw) {
        const long long a0 = grp_ptr[g], a1 = grp_ptr[g + 1];
        int cnt = sel_count[g];
        if (cnt < 0 || cnt > k) {
            if (lane == 0) record_error(st, SIC_ERR_INVALID, g);
            cnt = 0;
        }
        for (long long a = a0 + lane; a < a1; a += 32) {
            const long long i = members[a];
            if (i < 0 || i >= n) {
                record_error(st, SIC_ERR_INVALID, g);
                continue;
            }
            if (!col_sel) {  // counts only
                int w = (int)(a1 - a - 1);
                for (int t = 0; t < cnt; ++t) w += sel_idx[g * k + t] > i;
                col_count[i] = w;
                continue;
            }
            int w = 0;
            int32_t* out = col_sel + i * kc;
            for (long long b = a + 1; b < a1 && w < kc; ++b) out[w++] = (int32_t)members[b];
            for (int t = 0; t < cnt && w < kc; ++t) {
                const int32_t q = sel_idx[g * k + t];
                if (q > i) out[w++] = q;
            }
            if ((a1 - a - 1) + cnt > kc && w == kc) record_error(st, SIC_ERR_INVALID, g);
            col_count[i] = w;
        }
    }
}

}  // namespace

extern "C" sic_status sic_select_partial(sic_handle* h, const double* pts, int64_t n, const sic_kernel* kp,
                                         const int64_t* grp_ptr, const int64_t* members, int64_t n_grp,
                                         const int64_t* cand_ptr, const int32_t* cand_idx, int32_t max_cand,
                                         int32_t max_m, int32_t k, sic_precision prec, int32_t* sel_idx,
                                         int32_t* sel_count, double* gain, void* stream) {
    if (!h || !pts || !sic_valid_kernel(kp) || !grp_ptr || !members || !cand_ptr || !sel_idx || !sel_count ||
        n < 1 || n_grp < 0 || max_cand < 0 || max_m < 1 || k < 1)
        return SIC_ERR_INVALID;
    if (k > 128 || max_m > 64 || n > INT_MAX) return SIC_ERR_UNSUPPORTED;
    if (n_grp == 0) return SIC_OK;
    if (max_cand > 0 && !cand_idx) return SIC_ERR_INVALID;
    const size_t tsz = prec == SIC_FP64 ? sizeof(double) : sizeof(float);
    auto layout = [&](int m) {
        PtLayout L;
        L.R = max_cand + m;
        L.W = m + k;
        L.P = L.W | 1;
        return L;
    };
    if (layout(max_m).limit_bytes(tsz) > 227 * 1024 - 4096) return SIC_ERR_UNSUPPORTED;
    if (prec != SIC_FP64 && prec != SIC_FP32_MIXED) return SIC_ERR_INVALID;
    if (n_grp > INT_MAX) return SIC_ERR_UNSUPPORTED;
    SIC_CUDA_TRY(cudaSetDevice(h->device));
    cudaStream_t s = (cudaStream_t)stream;
    // Two size classes: a step's time is its chain of dependent operations, so two groups on an SM take little longer than
    // one.  Up to `two` members the state fits twice (256 candidates, k = 64 in FP32: 25 members).  N = 2^16, 2,811
    // groups: 9.0 ms as one class, 7.1 as two.  But the two launches follow one another, so with few groups per SM one launch
    // of one group per SM is shorter.  FP32, 256 candidates, k = 64: 88 groups 0.81 ms against 1.29, 173 1.42
    // against 1.33, 342 1.87 against 1.42.  FP64, where two groups share the pipe they are bound by, 100 candidates, k = 20: 117 groups
    // 3.1 ms against 5.6, 747 7.0 against 8.1, 989 9.7 against 9.0.
    int two = max_m;
    while (two > 0 && layout(two).bytes(tsz) > 227 * 1024 / 2 - PT_STATIC) --two;
    if (two < max_m && (two < PT_MIN_CLASS || n_grp <= (prec == SIC_FP64 ? 5LL : 1LL) * h->num_sms)) two = 0;
    for (int c = 0; c < 2; ++c) {
        const int lo = c == 0 ? 1 : two + 1, hi = c == 0 ? two : max_m;
        if (lo > hi) continue;
        const PtLayout L = layout(hi);
        const size_t smem = L.bytes(tsz);
        const int nt = c == 0 ? PT_NT_2 : PT_NT;
        auto launch = [&](auto kern, auto kpt, auto floor_) -> sic_status {
            SIC_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
            const int grid = persistent_grid(h, kern, nt, smem, n_grp);
            kern<<<grid, nt, smem, s>>>(pts, n, kp->dim, kpt, floor_, (const long long*)grp_ptr,
                                        (const long long*)members, n_grp, (const long long*)cand_ptr, cand_idx, max_cand,
                                        max_m, lo, hi, k, sel_idx, sel_count, gain, L, h->d_status);
            return SIC_OK;
        };
        const double fl = sic_floor_of(kp);
        const sic_status e =
            prec == SIC_FP64
                ? launch(c == 0 ? k_select_partial<double, PT_NT_2> : k_select_partial<double, PT_NT>, make_kp<double>(*kp), fl)
                : launch(c == 0 ? k_select_partial<float, PT_NT_2> : k_select_partial<float, PT_NT>, make_kp<float>(*kp), (float)fl);
        if (e != SIC_OK) return e;
    }
    SIC_CUDA_TRY(cudaGetLastError());
    return SIC_OK;
}

extern "C" sic_status sic_partial_columns(sic_handle* h, int64_t n, const int64_t* grp_ptr, const int64_t* members,
                                          int64_t n_grp, const int32_t* sel_idx, const int32_t* sel_count, int32_t k,
                                          int32_t kc, int32_t* col_sel, int32_t* col_count, void* stream) {
    if (!h || n < 1 || n_grp < 0 || k < 1 || kc < 1 || !grp_ptr || !members || !sel_idx || !sel_count || !col_count)
        return SIC_ERR_INVALID;
    if (n_grp == 0) return SIC_OK;
    SIC_CUDA_TRY(cudaSetDevice(h->device));
    const int grid = persistent_grid(h, k_partial_columns, 256, 0, (n_grp + 7) / 8);
    k_partial_columns<<<grid, 256, 0, (cudaStream_t)stream>>>(n, (const long long*)grp_ptr,
                                                              (const long long*)members, n_grp, sel_idx, sel_count, k,
                                                              kc, col_sel, col_count, h->d_status);
    SIC_CUDA_TRY(cudaGetLastError());
    return SIC_OK;
}
