// The blocked LDL^T of the kernel matrix of a small point set in shared memory (one CTA: NT worker threads and
// a pivot warp), shared by the fills (fill.cu, consecutive and nonadjacent groups) and the FP64 side state
// (side.cu): Theta by unit_theta, the factorisation by ldl_panels.
//
// F64 (nonadjacent groups and side state): nothing is held in fewer bits than FP64 -- distances from FP64
// differences, panel rows in 58 bits and rounded, L kept in FP64.  Consecutive groups: coordinates in fixed point,
// panel rows truncated to 53 bits of the row's largest entry, L as double-float pairs of 48 bits.
#pragma once

#include "sic_internal.cuh"

constexpr int FILL_B = 4;         // panel width of the blocked LDL^T (integer trailing update)


// doubles of the scratch region: the points' coordinates while Theta is formed, then the
// panel's rows in fixed point ((2 FILL_B + 1) ints per row); even, so what follows stays
// 16-byte aligned
__host__ __device__ constexpr int fill_scratch_doubles(int nmax) {
    return ((3 * nmax > ((2 * FILL_B + 1) * nmax + 1) / 2 ? 3 * nmax : ((2 * FILL_B + 1) * nmax + 1) / 2) + 1) & ~1;
}

// Packed lower-triangle index (nn <= 192, so every index fits in 32 bits; 32-bit integer
// arithmetic and int-to-float conversions stay off the FP64 pipe).
__device__ __forceinline__ int pk(int i, int j) { return i * (i + 1) / 2 + j; }

// row i of the packed lower triangle that holds flat entry e (i(i+1)/2 <= e < (i+1)(i+2)/2)
__device__ __forceinline__ int pk_row(int e) {
    int i = (int)((sqrtf(8.0f * (float)e + 1.0f) - 1.0f) * 0.5f);
    while (i * (i + 1) / 2 > e) --i;
    while ((i + 1) * (i + 2) / 2 <= e) ++i;
    return i;
}

// Pivot of column c of the LDL^T factorisation from its final Schur complement v: D_cc = v
// (kept on the diagonal) and d^(-1/2) by rsqrt_newton (five FP64 operations with the
// diagonal's update) into piv slot c & 3 (the panel's columns); the column is then scaled as
// G_ic = U_ic d^(-1/2) and L_ic = G_ic d^(-1/2).  A non-positive pivot raises *bad.  The range
// test reads the bits (no FP64 compare).
__device__ __forceinline__ void fill_pivot(double v, int c, double* G, double* piv, int* bad) {
    const long long vb = __double_as_longlong(v);
    if (vb <= 0 || vb >= 0x7ff0000000000000LL) {  // not in (+0, +inf): non-positive, infinite or NaN
        *bad = 1;
        return;
    }
    G[pk(c, c)] = v;
    piv[c & 3] = rsqrt_newton(v);
}

// ---- the integer update of a panel ----
//
// A row of a panel, its FILL_B values g_j (entries of G = L D^(1/2)), is held in fixed point:
// g_j = M_j 2^(E - 1075) with E the largest biased exponent among them and M_j the 53-bit
// significands shifted to E and truncated (signed; zero and subnormal values count as 0), split
// as M_j = Mh_j 2^26 + Ml_j (Mh signed, 0 <= Ml < 2^26).  Layout (B = 4, ld rows, fx 16-byte
// aligned): the Mh of a row as one int4 at fx[4 row], its Ml at fx[4 (ld + row)], E at
// fx[8 ld + row] (a warp reading consecutive rows reads consecutive 16-byte words).
// The dot product of two rows is formed from exact 32 x 32-bit products (fx_dot).  Truncating
// to the row's exponent costs each value at most 2^-52 of the row's largest, and fx_dot's own
// truncations stay below 2^-51 of the largest product: with G's rows (|G_ij| <= sqrt(A_ii)) the
// error of an entry's update stays within a few B 2^-52 sqrt(A_ii A_ll), the order of the FP64
// Cholesky's own backward error bound.
//
// F64: M_j has five more bits (g_j = M_j 2^(E - 1080)) and is rounded, split at 2^29.  An entry is then held exactly
// while its exponent is within 5 of E, else to 2^-59 of the row's largest, and what fx_dot leaves out is below 5 units of
// 2^-58 of the largest product: the FP64 rounding of the sum and of the subtraction are what remains.
template <int B, bool F64>
__device__ __forceinline__ void fx_row_store(const double (&g)[B], int* __restrict__ fx, int ld, int row) {
    static_assert(B == 4, "the fixed-point rows are stored as int4");
    int e[B];
    int E = 0;
#pragma unroll
    for (int j = 0; j < B; ++j) {
        e[j] = (__double2hiint(g[j]) >> 20) & 0x7ff;
        E = max(E, e[j]);
    }
    int mh[B], ml[B];
#pragma unroll
    for (int j = 0; j < B; ++j) {
        const long long u = __double_as_longlong(g[j]);
        long long m = e[j] ? ((u & 0xfffffffffffffLL) | 0x10000000000000LL) : 0LL;
        const int sh = E - e[j];
        if constexpr (F64)
            m = sh < 60 ? (((m << 6) >> sh) + 1) >> 1 : 0LL;
        else
            m = sh < 63 ? (m >> sh) : 0LL;
        if (u < 0) m = -m;
        mh[j] = (int)(m >> (F64 ? 29 : 26));
        ml[j] = (int)(m & (F64 ? 0x1fffffffLL : 0x3ffffffLL));
    }
    reinterpret_cast<int4*>(fx)[row] = make_int4(mh[0], mh[1], mh[2], mh[3]);
    reinterpret_cast<int4*>(fx)[ld + row] = make_int4(ml[0], ml[1], ml[2], ml[3]);
    fx[8 * ld + row] = E;
}

// s 2^e2 as FP64 by integer operations, the significand truncated (relative error < 2^-52) or, with ROUND, to nearest;
// 0 for s = 0 and below FP64's normal range
template <bool ROUND>
__device__ __forceinline__ double i64_scaled(long long s, int e2) {
    if (s == 0) return 0.0;
    const unsigned long long sg = (unsigned long long)s & (1ULL << 63);
    const unsigned long long mag = s < 0 ? 0ULL - (unsigned long long)s : (unsigned long long)s;
    const int z = __clzll((long long)mag);
    const int be = e2 + 63 - z + 1023;
    if (be <= 0) return 0.0;
    if constexpr (ROUND) {  // the significand's leading bit (or the carry to 2^53) adds to the exponent field
        const unsigned long long m = (((mag << z) >> 10) + 1ULL) >> 1;
        return __longlong_as_double((long long)(sg | (((unsigned long long)(be - 1) << 52) + m)));
    }
    return __longlong_as_double((long long)(sg | ((unsigned long long)be << 52) | (((mag << z) >> 11) & 0xfffffffffffffULL)));
}

// sum_j g_ij g_lj of rows i and l: 2^52 sum Mh Mh + 2^26 sum (Mh Ml + Ml Mh) exactly in two 64-bit
// sums of 32 x 32-bit products, scaled down by 2^52 into one 64-bit integer (the dropped fraction
// and the omitted sum Ml Ml are below 5 units of 2^(Ei + El - 2098)), converted to FP64.  (F64: 2^58 and 2^29, units of
// 2^(Ei + El - 2102), the sums below 2^61.)
template <int B, bool F64>
__device__ __forceinline__ double fx_dot(const int* __restrict__ fx, int ld, int i, int l) {
    static_assert(B == 4, "the fixed-point rows are stored as int4");
    const int4 hi4 = reinterpret_cast<const int4*>(fx)[i], li4 = reinterpret_cast<const int4*>(fx)[ld + i];
    const int4 hl4 = reinterpret_cast<const int4*>(fx)[l], ll4 = reinterpret_cast<const int4*>(fx)[ld + l];
    const int hi_[4] = {hi4.x, hi4.y, hi4.z, hi4.w}, li[4] = {li4.x, li4.y, li4.z, li4.w};
    const int hl[4] = {hl4.x, hl4.y, hl4.z, hl4.w}, ll[4] = {ll4.x, ll4.y, ll4.z, ll4.w};
    long long a2 = 0, a1 = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        a2 += (long long)hi_[j] * hl[j];
        a1 += (long long)hi_[j] * ll[j] + (long long)li[j] * hl[j];
    }
    return i64_scaled<F64>(a2 + (a1 >> (F64 ? 29 : 26)), fx[8 * ld + i] + fx[8 * ld + l] - (F64 ? 2102 : 2098));
}

// Theta over the nn points pos[0 .. nn) into G (packed lower): the coordinates go to fixed point at the
// unit's largest exponent in each dimension (fx_coord), so that differences and squared distances are exact integer
// arithmetic (fx_dist2); the Matern in FP64 (matern_d2_fast; the all-double-float Matern of dfloat.cuh would
// spare the FP64 pipe entirely, but its ~1e-14 of the variance per entry is amplified by 1/v in the Schur
// complements, v ~ 2 nugget on the finest groups: factor columns then miss the oracle's by more than 1e-8).
// F64: FP64 differences, which keep every pair's own precision whatever else is in the unit (a point far out
// takes bits from the others' fixed-point coordinates); a non-finite entry raises *bad.
// pos[i] is written by thread i mod NT; emax: three words, zero; ends with a barrier.  NT workers and one more warp.
// Coincident points without a nugget (`singular`) make Theta singular: *bad is raised then, whatever the
// factorisation's rounding would leave of the pivot.
template <int NT, bool F64>
__device__ __forceinline__ void unit_theta(const double* __restrict__ pts, int dim, const KP<double>& kp,
                                           const double* __restrict__ tab, const int* pos, int nn, int nmax, double* xyz,
                                           double* G, unsigned* emax, int* bad, bool singular) {
    const int tid = threadIdx.x, lane = tid & 31;
    const bool worker = tid < NT;
    {
        unsigned em[3] = {0u, 0u, 0u};
        for (int i = worker ? tid : nn; i < nn; i += NT) {
            const int p = pos[i];
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                const double x = (d < dim) ? pts[(long long)p * dim + d] : 0.0;
                xyz[d * nmax + i] = x;
                if (!F64) em[d] = max(em[d], ((unsigned)__double2hiint(x) >> 20) & 0x7ffu);
            }
        }
        if constexpr (!F64) {
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                em[d] = __reduce_max_sync(0xffffffffu, em[d]);
                if (lane == 0 && em[d]) atomicMax(&emax[d], em[d]);
            }
        }
    }
    __syncthreads();
    int E0 = 0, E1 = 0, E2 = 0;
    long long* xf = reinterpret_cast<long long*>(xyz);
    if constexpr (!F64) {
        E0 = (int)emax[0], E1 = (int)emax[1], E2 = (int)emax[2];
        for (int i = worker ? tid : nn; i < nn; i += NT)
            for (int d = 0; d < dim; ++d)
                xf[d * nmax + i] = fx_coord(xyz[d * nmax + i], d == 0 ? E0 : (d == 1 ? E1 : E2));
        __syncthreads();
    }
    auto dist2 = [&](int i, int j) -> double {
        if constexpr (F64) {
            const double dx = xyz[i] - xyz[j], dy = xyz[nmax + i] - xyz[nmax + j],
                         dz = xyz[2 * nmax + i] - xyz[2 * nmax + j];
            return fma(dz, dz, fma(dy, dy, dx * dx));
        } else {
            return fx_dist2(xf, nmax, dim, i, j, E0, E1, E2);
        }
    };
    if (singular)  // (a pass of its own: in the loop below the test took 1.5 % of the fill)
        for (int e = tid; e < nn * (nn - 1) / 2; e += NT + 32) {
            const int i = pk_row(e);
            if (__double_as_longlong(dist2(i + 1, e - i * (i + 1) / 2)) == 0LL) *bad = 2;
        }
    // entry e = i (i + 1) / 2 + j, stepped by NT
    for (int i = worker ? pk_row(tid) : nn, j = worker ? tid - i * (i + 1) / 2 : 0; i < nn;) {
        double v = matern_d2_fast(kp, dist2(i, j), tab);
        if (F64 && i != j && ((unsigned)__double2hiint(v) & 0x7ff00000u) == 0x7ff00000u) *bad = 2;
        if (i == j) v = F64 ? kp.s2 + kp.nugget : v + kp.nugget;
        G[pk(i, j)] = v;
        j += NT;
        while (j > i) {
            j -= i + 1;
            ++i;
        }
    }
    __syncthreads();
}

// blocked right-looking LDL^T factorisation Theta_RR = L D L^T in place on the packed
// lower triangle, in panels of FILL_B columns, in FP64: d_j = A_jj, L_ij = A_ij / d_j and
// A_il -= L_ij U_lj within the panel (U_lj = A_lj, the panel's entries unscaled).  The
// rows below the panel keep G_ij = U_ij d_j^(-1/2) (G = L D^(1/2)) in fixed point; the
// trailing matrix then takes the panel's whole rank-FILL_B update as one integer dot
// product of two G rows per entry (exact products), subtracted in FP64 (fx_dot): FILL_B
// FP64 FMAs become one FP64 addition, the products going to the integer multiply-add
// units.  The FP64 units are per SM sub-partition and charge a warp instruction whatever
// its active lanes, so the flat loops keep full warps.
// The panel's diagonal block (at most FILL_B x FILL_B) is factored by the pivot warp, lane
// r owning the block's row r (its pivots and their reciprocal square roots are a chain of
// dependent FP64 operations, warp-synchronous): the next panel's block takes the current
// panel's update and is factored while the workers update the rest of the trailing matrix.
// Every worker row below the block then applies the block's columns to its own panel
// entries in registers (A_il -= L_ij U_lj reads the block's unscaled entries, which stay
// in place until the block's L entries are written back in the next phase), so that a
// panel costs two barriers.  Worker thread i owns row i (nn <= NT, the launcher's
// choice).  Same operations, in the same order, as a column-by-column elimination.
// (*bad becomes 1 where a pivot is not positive; piv: four doubles, fx: the scratch of fill_scratch_doubles; G's
// off-diagonal entries end as L, as double-float pairs or (F64) in FP64; ends with a barrier.)
template <int NT, bool F64>
__device__ __forceinline__ void ldl_panels(double* G, int* fx, double* piv, int nn, int nmax, int* bad) {
    const int tid = threadIdx.x, lane = tid & 31;
    const bool worker = tid < NT;
    const int i = tid;
    const int rowi = pk(i, 0);
    double lb[FILL_B];  // pivot warp: L of the block's row `lane` (columns below it)
    auto store_l = [&](int at, double v) {
        if constexpr (F64) {
            G[at] = v;
        } else {
            float h, l;
            f64_split(v, h, l);
            reinterpret_cast<float2*>(G)[at] = make_float2(h, l);
        }
    };
    // the block [J, J + bs) (its entries final): lane r owns row J + r
    auto factor_block = [&](int J, int bs) {
        const int r = lane;
        const int ib = J + r;
        if (r == 0) fill_pivot(G[pk(J, J)], J, G, piv, bad);
        __syncwarp();
#pragma unroll
        for (int jj = 0; jj < FILL_B - 1; ++jj) {
            if (jj >= bs - 1) break;
            const int j = J + jj;
            if (r > jj && r < bs) {
                const double rsd = piv[j & 3];
                const double uv = G[pk(ib, j)];
                const double g = uv * rsd;
                const double l = g * rsd;
                lb[jj] = l;
#pragma unroll
                for (int c2 = jj + 1; c2 < FILL_B; ++c2)
                    if (c2 <= r) G[pk(ib, J + c2)] = fma(-l, G[pk(J + c2, j)], G[pk(ib, J + c2)]);
                if (r == jj + 1) fill_pivot(G[pk(ib, ib)], ib, G, piv, bad);
            }
            __syncwarp();
        }
    };
    if (!worker) factor_block(0, min(FILL_B, nn));
    __syncthreads();
    for (int J = 0; J < nn && !*bad; J += FILL_B) {
        const int je = min(J + FILL_B, nn);  // je < nn implies a full panel
        // the own row's panel entries (rows below the block): L and G by the block's columns
        if (worker && i >= je && i < nn) {
            double u[FILL_B], gv[FILL_B], lv[FILL_B];
#pragma unroll
            for (int c = 0; c < FILL_B; ++c) u[c] = G[rowi + J + c];
#pragma unroll
            for (int jj = 0; jj < FILL_B; ++jj) {
                const double rsd = piv[jj];  // (J + jj) & 3
                const double g = u[jj] * rsd;
                const double l = g * rsd;
                gv[jj] = g;
                lv[jj] = l;
#pragma unroll
                for (int c2 = jj + 1; c2 < FILL_B; ++c2) u[c2] = fma(-l, G[pk(J + c2, J + jj)], u[c2]);
            }
            fx_row_store<FILL_B, F64>(gv, fx, nmax, i);
            // the L entries as double-float pairs (hi, lo) in their 8-byte slots (f64_split: 48
            // significant bits; only the member solves read them)
#pragma unroll
            for (int c = 0; c < FILL_B; ++c) store_l(rowi + J + c, lv[c]);
        }
        __syncthreads();
        if (worker) {
            // the trailing matrix, entries (i, l) with je <= l <= i < nn, takes the panel's
            // update, but for the next panel's block (the first nbt flat entries)
            if (je < nn) {
                const int nt = nn - je;
                const int bs2 = min(FILL_B, nt), nbt = bs2 * (bs2 + 1) / 2;
                // entry e = ii (ii + 1) / 2 + ll of the trailing triangle, stepped by NT
                int ii = pk_row(tid + nbt), ll = tid + nbt - ii * (ii + 1) / 2;
                while (ii < nt) {
                    const int i = je + ii, l = je + ll;
                    G[pk(i, l)] -= fx_dot<FILL_B, F64>(fx, nmax, i, l);
                    ll += NT;
                    while (ll > ii) {
                        ll -= ii + 1;
                        ++ii;
                    }
                }
            }
        } else {
            // the block's L entries, now that the workers have read its
            // unscaled entries; then the next block: its update, and its factorisation
            const int bs = je - J;
            if (lane < bs) {
#pragma unroll
                for (int c = 0; c < FILL_B - 1; ++c)
                    if (c < lane) store_l(pk(J + lane, J + c), lb[c]);
            }
            if (je < nn) {
                const int bs2 = min(FILL_B, nn - je);
                if (lane < bs2 * (bs2 + 1) / 2) {
                    const int ii = pk_row(lane), ll = lane - ii * (ii + 1) / 2;
                    G[pk(je + ii, je + ll)] -= fx_dot<FILL_B, F64>(fx, nmax, je + ii, je + ll);
                }
                __syncwarp();
                factor_block(je, bs2);
            }
        }
        __syncthreads();
    }
    __syncthreads();
}
