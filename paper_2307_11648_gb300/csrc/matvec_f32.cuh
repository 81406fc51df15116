// The double-FP32 sums of the product with Theta over 64 target rows, for a CTA of 8 warps: the kernel for one or two
// right-hand sides (pcg.cu) and the rows that the digits' product leaves (matvec_tc.cu).
//
// Two rows per lane, so that a source's values are read once for both and the kernel evaluation runs in packed
// FP32 pairs; the warps share the staged source tile, 32 sources each, and their sums are added in order at the end.
// With one thread per row over all sources, N = 50,001 left an SM ten warps.  Bound: FP32 lanes (11 operations per
// source, row and right-hand side, about 22 per entry).  N = 50,001, one right-hand side: 6.0 ms with a thread per row,
// 5.2 ms now (two: 8.0 and 5.3).
#pragma once

#include "sic_internal.cuh"

constexpr int MV_TILE = 256;  // source points per shared-memory tile
constexpr int MVF_WARPS = 8, MVF_ROWS = 64;
constexpr int MVF_FLUSH = 8;  // tiles between FP64 additions: 256 terms (1024 left three times the error)

template <int NR>
union MvfSmem {
    static constexpr int NP = (NR + 1) / 2;  // right-hand sides in pairs
    struct {
        float4 c[MV_TILE];        // coordinates
        float2 h[MV_TILE][NP];    // high parts of x
        float2 l[MV_TILE][NP];    // low parts
    } t;
    double acc[MVF_WARPS][2 * NP][MVF_ROWS];
    __device__ __forceinline__ double sum(int row, int r) const {  // the warps' sums in order
        double a = acc[0][r][row];
#pragma unroll
        for (int w = 1; w < MVF_WARPS; ++w) a += acc[w][r][row];
        return a;
    }
};

// One source's products k x for two rows, added to S + lo: TwoProduct, TwoSum (packed operations: lane-wise the scalar
// roundings)
template <int NP>
__device__ __forceinline__ void mvf_add(float k0, float k1, const float2 (&xh)[NP], const float2 (&xl)[NP],
                                        float2 (&S)[2][NP], float2 (&lo)[2][NP]) {
    const float2 neg1 = make_float2(-1.f, -1.f);
#pragma unroll
    for (int r = 0; r < NP; ++r) {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const float2 k = q == 0 ? make_float2(k0, k0) : make_float2(k1, k1);
            const float2 p = __fmul2_rn(k, xh[r]);
            const float2 pe = __ffma2_rn(k, xl[r], __ffma2_rn(k, xh[r], __fmul2_rn(p, neg1)));
            const float2 s = __fadd2_rn(S[q][r], p);
            const float2 nb = __ffma2_rn(s, neg1, S[q][r]);                  // -(s - S)
            const float2 ea = __ffma2_rn(__fadd2_rn(s, nb), neg1, S[q][r]);  // S - (s - (s - S))
            lo[q][r] = __fadd2_rn(lo[q][r], __fadd2_rn(__fadd2_rn(ea, __fadd2_rn(p, nb)), pe));
            S[q][r] = s;
        }
    }
}

// S + lo to the FP64 sums, S = lo = 0
template <int NP>
__device__ __forceinline__ void mvf_flush(float2 (&S)[2][NP], float2 (&lo)[2][NP], double (&acc)[2][2 * NP]) {
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int r = 0; r < NP; ++r) {
            acc[q][2 * r] += (double)S[q][r].x + (double)lo[q][r].x;
            acc[q][2 * r + 1] += (double)S[q][r].y + (double)lo[q][r].y;
            S[q][r] = lo[q][r] = make_float2(0.f, 0.f);
        }
}

// The rows row0 .. row0 + 63 (those before n) into sm.acc; entry(d2): the kernel entries at a pair of squared distances;
// scale(r): factor of right-hand side r.  All 256 threads; ends with a barrier.
template <int NR, typename Entry, typename Scale>
__device__ __forceinline__ void mvf_tile(MvfSmem<NR>& sm, const double* __restrict__ pts, long long n, int dim,
                                         const double* __restrict__ x, int nrhs, long long row0, Entry entry,
                                         Scale scale) {
    constexpr int NP = MvfSmem<NR>::NP, NT = 32 * MVF_WARPS;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const long long i0 = row0 + lane, i1 = i0 + 32;
    auto coord = [&](long long i, int d) { return i < n && d < dim ? (float)pts[i * dim + d] : 0.f; };
    const float2 rx = make_float2(coord(i0, 0), coord(i1, 0)), ry = make_float2(coord(i0, 1), coord(i1, 1)),
                 rz = make_float2(coord(i0, 2), coord(i1, 2));
    float2 S[2][NP], lo[2][NP];
    double acc[2][2 * NP];
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int r = 0; r < NP; ++r) {
            S[q][r] = lo[q][r] = make_float2(0.f, 0.f);
            acc[q][2 * r] = acc[q][2 * r + 1] = 0.0;
        }
    int tiles = 0;
    for (long long j0 = 0; j0 < n; j0 += MV_TILE) {
        __syncthreads();
        for (int t = tid; t < MV_TILE; t += NT) {
            const long long j = j0 + t;
            sm.t.c[t] = make_float4(coord(j, 0), coord(j, 1), coord(j, 2), 0.f);
#pragma unroll
            for (int r = 0; r < NP; ++r) {
                float2 h = make_float2(0.f, 0.f), l = h;
                if (j < n) {
                    if (2 * r < nrhs) split_f64(x[j * nrhs + 2 * r] * scale(2 * r), h.x, l.x);
                    if (2 * r + 1 < nrhs) split_f64(x[j * nrhs + 2 * r + 1] * scale(2 * r + 1), h.y, l.y);
                }
                sm.t.h[t][r] = h;
                sm.t.l[t][r] = l;
            }
        }
        __syncthreads();
        const int t0 = warp * (MV_TILE / MVF_WARPS);
        const int t1 = (int)min((long long)(t0 + MV_TILE / MVF_WARPS), n - j0);
        for (int t = t0; t < t1; ++t) {
            const float4 c = sm.t.c[t];
            const float2 dx = __fadd2_rn(rx, make_float2(-c.x, -c.x)), dy = __fadd2_rn(ry, make_float2(-c.y, -c.y)),
                         dz = __fadd2_rn(rz, make_float2(-c.z, -c.z));
            const float2 k = entry(__ffma2_rn(dz, dz, __ffma2_rn(dx, dx, __fmul2_rn(dy, dy))));
            float2 xh[NP], xl[NP];
#pragma unroll
            for (int r = 0; r < NP; ++r) {
                xh[r] = sm.t.h[t][r];
                xl[r] = sm.t.l[t][r];
            }
            mvf_add<NP>(k.x, k.y, xh, xl, S, lo);
        }
        if (++tiles == MVF_FLUSH) {
            mvf_flush<NP>(S, lo, acc);
            tiles = 0;
        }
    }
    mvf_flush<NP>(S, lo, acc);
    __syncthreads();
#pragma unroll
    for (int r = 0; r < 2 * NP; ++r) {
        sm.acc[warp][r][lane] = acc[0][r];
        sm.acc[warp][r][lane + 32] = acc[1][r];
    }
    __syncthreads();
}
