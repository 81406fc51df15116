// One training step of the proposal network (8 -> 128 -> 128 -> 1, erf GELU, weighted binary
// cross-entropy) with BF16 operands on the 5th-generation tensor cores, forward and backward
// of a row tile in one visit.
//
// A CTA of 256 threads takes tiles of 128 rows (thread = row and one half of the 128 hidden
// columns) and keeps its weight gradients in TMEM and registers over all of them:
//   Z1 = X W1            K-major x K-major, N = 128, K = 16 (8 features, 8 zeros)
//   H1 = bf16(gelu(Z1 + b1))             -> shared memory, the next A operand
//   Z2 = H1 W2           K = 128
//   s = gelu(Z2 + b2) . w3 + b3, loss, dS, dZ2 = dS w3 gelu'(Z2) -> shared memory (BF16)
//   dH1 = dZ2 W2^T       A K-major, B = the same W2 tile read MN-major
//   dW2 += H1^T dZ2      both operands the tiles above read MN-major, accumulated in TMEM
//   dZ1 = dH1 gelu'(Z1 + b1)             -> shared memory (BF16)
//   dW1 += dZ1^T X       N = 16, accumulated in TMEM (transposed: 128 hidden x 8 features)
// dw3 is an FP32 column sum (a 32 x 32 exchange over the warp, lane = column).  db1, db2 and db3 have
// the rounding of one running FP32 sum down the rows of the batch, which is what these gradients
// have always had (it is up to 2e-5 of them at 65536 rows): dZ1, dZ2 and dS go to the workspace
// with each tile's column sums, k_train_bias runs chunks of 512 rows in parallel, each from the
// total of the tiles before it, and the chunks' increments are added in order.  k_train_sum adds the
// CTAs' partial gradients in a fixed order.  The products' operands never leave the SM: they are the tiles
// themselves, whose core matrices (8 rows x 16 bytes) serve as K-major for products along
// the hidden dimension and as MN-major for products along the rows.
//
// TMEM (512 columns, one CTA per SM): Z1 at 0, Z2 and then dH1 at 128, dW2 at 256, dW1 at 384.
// Bound: FP32 issue of the erf GELU and its derivative (three evaluations per row and hidden
// column).  65,536 rows with the AdamW step: 175 us; 6.9 ms as separate GEMM,
// elementwise and one-thread-per-column kernels over activations in memory.
#include "tc_common.cuh"

namespace {

constexpr int NF = 8, HID = 128;
constexpr int OFF_B1 = NF * HID, OFF_W2 = OFF_B1 + HID, OFF_B2 = OFF_W2 + HID * HID, OFF_W3 = OFF_B2 + HID,
              OFF_B3 = OFF_W3 + HID, NPARAM = OFF_B3 + 1;
constexpr int PART = (NPARAM + 1 + 3) / 4 * 4;  // one CTA's gradients, its loss sum at NPARAM
constexpr int NT = 256, ROWS = 128;
constexpr int NB = 2 * HID;       // bias columns 0..127 (dZ1) and 128..255 (dZ2); dS is column NB
constexpr int MAX_CTAS = 152;     // one per SM
constexpr int CHUNK = 4;          // tiles per running sum of k_train_bias

// Workspace of one step (floats): the CTAs' partial gradients, per tile the column sums of dZ1, dZ2
// and dS, per chunk its increments, then dZ [tile][NB][128 rows] and dS [rows].
struct TrainTc {
    long long rows, tiles, ctas;
    __host__ __device__ long long chunks() const { return (tiles + CHUNK - 1) / CHUNK; }
    __host__ __device__ long long part() const { return 0; }
    __host__ __device__ long long tsum() const { return ctas * PART; }
    __host__ __device__ long long delta() const { return tsum() + tiles * (NB + 4); }
    __host__ __device__ long long dz() const { return delta() + chunks() * (NB + 4); }
    __host__ __device__ long long ds() const { return dz() + tiles * ROWS * NB; }
    __host__ __device__ long long size() const { return ds() + rows; }
};

constexpr unsigned TMEM_COLS = 512;
constexpr uint32_t T_Z1 = 0, T_Z2 = 128, T_DW2 = 256, T_DW1 = 384;

constexpr int SX = 0;                      // two X tiles, 128 x 16 bf16 each
constexpr int SX_SZ = ROWS * 16 * 2;
constexpr int SW1 = SX + 2 * SX_SZ;        // W1^T, 128 x 16
constexpr int SW2 = SW1 + HID * 16 * 2;    // W2^T, 128 x 128
constexpr int SH1 = SW2 + HID * HID * 2;   // H1
constexpr int SDZ = SH1 + ROWS * HID * 2;  // dZ2, then dZ1
constexpr int SVEC = SDZ + ROWS * HID * 2; // b1, b2, w3
constexpr int SRED = SVEC + 3 * HID * 4;   // the two halves' partial logits
constexpr int SCOL = SRED + 2 * ROWS * 4;  // column sums of the four row groups: dZ1, dZ2, dw3
constexpr int SDS = SCOL + 3 * 4 * HID * 4;  // dS of the tile's rows
constexpr int SBAR = SDS + ROWS * 4;
// padded above half an SM's shared memory: one CTA per SM holds all 512 TMEM columns, so none waits
// for them
constexpr int SMEM_TR = 140 * 1024;
static_assert(SBAR + 16 <= SMEM_TR, "shared memory of the training step");

__device__ __forceinline__ float gelu_f(float z) { return 0.5f * z * (1.0f + erff(z * 0.70710678118654752f)); }
__device__ __forceinline__ float dgelu_f(float z) {
    return 0.5f * (1.0f + erff(z * 0.70710678118654752f)) + z * expf(-0.5f * z * z) * 0.39894228040143268f;
}
__device__ __forceinline__ float bf16_round(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }

// v[j] of every lane -> lane j: the sum over the warp's lanes of their v[j] (31 exchanges)
__device__ __forceinline__ float column_sum(float (&v)[32], int lane) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const bool up = lane & off;
#pragma unroll
        for (int i = 0; i < off; ++i) {
            const float send = up ? v[i] : v[i + off], keep = up ? v[i + off] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
        }
    }
    return v[0];
}

// 32 values of one row at column c0 into a K-major tile of 128 columns, rounded to BF16
__device__ __forceinline__ void store_row(unsigned char* tile, int row, int c0, const float (&v)[32]) {
#pragma unroll
    for (int g = 0; g < 4; ++g)
        *reinterpret_cast<uint4*>(tile + core_off(row, c0 + 8 * g, HID)) =
            make_uint4(pack2(v[8 * g], v[8 * g + 1]), pack2(v[8 * g + 2], v[8 * g + 3]),
                       pack2(v[8 * g + 4], v[8 * g + 5]), pack2(v[8 * g + 6], v[8 * g + 7]));
}

// 32 values of one row at column c0 into dZ, laid out [tile][column][row of the tile]: a warp's 32 rows
// of a column are one 128-byte line
__device__ __forceinline__ void store_cols(float* dZ, long long tile, int c0, int row, const float (&v)[32]) {
    float* p = dZ + (tile * NB + c0) * ROWS + row;
#pragma unroll
    for (int j = 0; j < 32; ++j) p[j * ROWS] = v[j];
}

__global__ void __launch_bounds__(NT, 1) k_train_tc(const float* __restrict__ X, const float* __restrict__ label,
                                                    long long rows, const float* __restrict__ params, float pw,
                                                    float* __restrict__ score, float* __restrict__ ws, TrainTc L,
                                                    DevStatus* st) {
    extern __shared__ __align__(1024) unsigned char sm[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int row = (warp & 3) * 32 + lane;  // TMEM lane: a warp reads the 32 lanes of its rank mod 4
    const int half = warp >> 2, c0 = half * 64;
    float* b1 = reinterpret_cast<float*>(sm + SVEC);
    float* b2 = b1 + HID;
    float* w3 = b2 + HID;
    float* red = reinterpret_cast<float*>(sm + SRED);
    float* cs = reinterpret_cast<float*>(sm + SCOL);  // [3][4][128]
    float* sds = reinterpret_cast<float*>(sm + SDS);
    float* tsum = ws + L.tsum();
    float* dZ = ws + L.dz();
    float* dSg = ws + L.ds();
    uint64_t* bar = reinterpret_cast<uint64_t*>(sm + SBAR);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(sm + SBAR + 8);
    const uint32_t bar_a = smem_u32(bar);

    for (int e = tid; e < HID * 16; e += NT) {
        const int n = e % HID, k = e / HID;
        *reinterpret_cast<__nv_bfloat16*>(sm + SW1 + core_off(n, k, 16)) =
            __float2bfloat16_rn(k < NF ? params[k * HID + n] : 0.f);
    }
    for (int e = tid; e < HID * HID; e += NT) {
        const int n = e % HID, k = e / HID;
        *reinterpret_cast<__nv_bfloat16*>(sm + SW2 + core_off(n, k, HID)) =
            __float2bfloat16_rn(params[OFF_W2 + k * HID + n]);
    }
    for (int i = tid; i < HID; i += NT) {
        b1[i] = bf16_round(params[OFF_B1 + i]);
        b2[i] = bf16_round(params[OFF_B2 + i]);
        w3[i] = bf16_round(params[OFF_W3 + i]);
    }
    const float b3 = bf16_round(params[OFF_B3]);
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar_a) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
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
    const uint32_t aW1 = smem_u32(sm + SW1), aW2 = smem_u32(sm + SW2), aH1 = smem_u32(sm + SH1),
                   aDZ = smem_u32(sm + SDZ), aX = smem_u32(sm + SX);
    uint32_t parity = 0;
    bool failed = false;
    float dw3[2] = {0.f, 0.f}, loss = 0.f;
    int buf = 0;
    uint32_t any = 0;  // weight gradients: accumulate from the second tile on

    // the tiles written before this are visible to the MMAs issued after it by thread 0
    auto staged = [&]() {
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
        if (tid == 0) asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    };
    // waits for the MMAs committed last; false when the wait gave up
    auto done = [&]() {
        if (!bar_wait(bar_a, parity)) failed = true;
        parity ^= 1u;
        if (__syncthreads_or(failed)) failed = true;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        return !failed;
    };

    const long long ntiles = (rows + ROWS - 1) / ROWS;
    for (long long tile = blockIdx.x; tile < ntiles; tile += gridDim.x, buf ^= 1, any = 1u) {
        const long long r = tile * ROWS + row;
        const bool live = r < rows;
        // the last tile's dW1 product may still read the other X buffer
        if (half == 0) {
            float4 f0 = make_float4(0.f, 0.f, 0.f, 0.f), f1 = f0;
            if (live) {
                f0 = make_float4(X[r * NF], X[r * NF + 1], X[r * NF + 2], X[r * NF + 3]);
                f1 = make_float4(X[r * NF + 4], X[r * NF + 5], X[r * NF + 6], X[r * NF + 7]);
            }
            *reinterpret_cast<uint4*>(sm + SX + buf * SX_SZ + core_off(row, 0, 16)) =
                make_uint4(pack2(f0.x, f0.y), pack2(f0.z, f0.w), pack2(f1.x, f1.y), pack2(f1.z, f1.w));
            *reinterpret_cast<uint4*>(sm + SX + buf * SX_SZ + core_off(row, 8, 16)) = make_uint4(0u, 0u, 0u, 0u);
        }
        const float yy = live ? label[r] : 0.f;
        staged();
        if (tid == 0) {
            mma_f16(tmem + T_Z1, smem_desc(aX + buf * SX_SZ, 128, 256), smem_desc(aW1, 128, 256), 0u);
            mma_commit(bar_a);
        }
        if (!done()) break;
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            float v[32];
            tmem_ld32(lane_addr + T_Z1 + c0 + c * 32, v);
#pragma unroll
            for (int j = 0; j < 32; ++j) v[j] = gelu_f(v[j] + b1[c0 + c * 32 + j]);
            store_row(sm + SH1, row, c0 + c * 32, v);
        }
        staged();
        if (tid == 0) {
#pragma unroll
            for (int kk = 0; kk < 8; ++kk)
                mma_f16(tmem + T_Z2, smem_desc(aH1 + kk * 256, 128, 2048), smem_desc(aW2 + kk * 256, 128, 2048),
                        kk > 0 ? 1u : 0u);
            mma_commit(bar_a);
        }
        if (!done()) break;
        // the head: this half's part of the logit; h2 and w3 gelu'(z2) stay in registers
        float h2[2][32], g2[2][32], s = 0.f;
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            tmem_ld32(lane_addr + T_Z2 + c0 + c * 32, h2[c]);
#pragma unroll
            for (int j = 0; j < 32; ++j) {
                const float z = h2[c][j] + b2[c0 + c * 32 + j];
                h2[c][j] = gelu_f(z);
                g2[c][j] = dgelu_f(z);
                s = fmaf(h2[c][j], w3[c0 + c * 32 + j], s);
            }
        }
        red[half * ROWS + row] = s;
        __syncthreads();
        s = red[row] + red[ROWS + row] + b3;
        float dS = 0.f;
        if (live) {
            const float sig = 1.f / (1.f + expf(-s));
            dS = (pw * yy * (sig - 1.f) + (1.f - yy) * sig) / (float)rows;
            if (half == 0) {
                // softplus(x) = max(x, 0) + log1p(exp(-|x|))
                const float l1 = log1pf(expf(-fabsf(s)));
                loss += pw * yy * (fmaxf(-s, 0.f) + l1) + (1.f - yy) * (fmaxf(s, 0.f) + l1);
                dSg[r] = dS;
                if (score) score[r] = s;
            }
        }
        if (half == 0) sds[row] = dS;
#pragma unroll
        for (int c = 0; c < 2; ++c) {
#pragma unroll
            for (int j = 0; j < 32; ++j) {
                h2[c][j] *= dS;
                g2[c][j] = dS * w3[c0 + c * 32 + j] * g2[c][j];
            }
            store_row(sm + SDZ, row, c0 + c * 32, g2[c]);
            store_cols(dZ, tile, HID + c0 + c * 32, row, g2[c]);
            dw3[c] += column_sum(h2[c], lane);
            cs[(4 + (warp & 3)) * HID + c0 + c * 32 + lane] = column_sum(g2[c], lane);
        }
        staged();
        if (tid == 0) {
#pragma unroll
            for (int kk = 0; kk < 8; ++kk)
                mma_f16(tmem + T_Z2, smem_desc(aDZ + kk * 256, 128, 2048), smem_desc(aW2 + kk * 4096, 2048, 128),
                        kk > 0 ? 1u : 0u, idesc_bf16(HID, 0, 1));
#pragma unroll
            for (int kk = 0; kk < 8; ++kk)
                mma_f16(tmem + T_DW2, smem_desc(aH1 + kk * 4096, 2048, 128), smem_desc(aDZ + kk * 4096, 2048, 128),
                        kk > 0 ? 1u : any, idesc_bf16(HID, 1, 1));
            mma_commit(bar_a);
        }
        if (!done()) break;
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            float v[32], z[32];
            tmem_ld32(lane_addr + T_Z1 + c0 + c * 32, z);
            tmem_ld32(lane_addr + T_Z2 + c0 + c * 32, v);
#pragma unroll
            for (int j = 0; j < 32; ++j) v[j] *= dgelu_f(z[j] + b1[c0 + c * 32 + j]);
            store_row(sm + SDZ, row, c0 + c * 32, v);
            store_cols(dZ, tile, c0 + c * 32, row, v);
            cs[(warp & 3) * HID + c0 + c * 32 + lane] = column_sum(v, lane);
        }
        staged();
        {  // the tile's column sums (cs and sds are next written after the barriers of the next tile)
            const float* q = cs + half * 4 * HID + (tid & (HID - 1));
            tsum[tile * (NB + 4) + tid] = (q[0] + q[HID]) + (q[2 * HID] + q[3 * HID]);
            if (warp == 0) {
                float a = (sds[lane] + sds[lane + 32]) + (sds[lane + 64] + sds[lane + 96]);
#pragma unroll
                for (int off = 16; off > 0; off >>= 1) a += __shfl_xor_sync(0xffffffffu, a, off);
                if (lane == 0) tsum[tile * (NB + 4) + NB] = a;
            }
        }
        if (tid == 0) {
#pragma unroll
            for (int kk = 0; kk < 8; ++kk)
                mma_f16(tmem + T_DW1, smem_desc(aDZ + kk * 4096, 2048, 128),
                        smem_desc(aX + buf * SX_SZ + kk * 512, 256, 128), kk > 0 ? 1u : any, idesc_bf16(16, 1, 1));
            // the next tile's first commit covers these; after the last tile they get their own
            if (tile + gridDim.x >= ntiles) mma_commit(bar_a);
        }
    }
    if (!failed) done();  // the last dW1 product
    if (!failed) {
        float* P = ws + L.part() + (long long)blockIdx.x * PART;
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            float v[32];
            tmem_ld32(lane_addr + T_DW2 + c0 + c * 32, v);
#pragma unroll
            for (int j = 0; j < 32; j += 4)
                *reinterpret_cast<float4*>(P + OFF_W2 + row * HID + c0 + c * 32 + j) =
                    make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
        }
        if (half == 0) {  // (32 columns read, the 16 of dW1 and 16 unused ones)
            float v[32];
            tmem_ld32(lane_addr + T_DW1, v);
#pragma unroll
            for (int f = 0; f < NF; ++f) P[f * HID + row] = v[f];
        }
        // dw3 and the loss over the row groups, in order
#pragma unroll
        for (int c = 0; c < 2; ++c) cs[(8 + (warp & 3)) * HID + c0 + c * 32 + lane] = dw3[c];
        if (half == 0) sds[row] = loss;
        __syncthreads();
        if (tid < HID) {
            const float* q = cs + 8 * HID + tid;
            P[OFF_W3 + tid] = (q[0] + q[HID]) + (q[2 * HID] + q[3 * HID]);
        }
        if (warp == 0) {
            float a = (sds[lane] + sds[lane + 32]) + (sds[lane + 64] + sds[lane + 96]);
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) a += __shfl_xor_sync(0xffffffffu, a, off);
            if (lane == 0) P[NPARAM] = a;
        }
    } else if (tid == 0) {
        record_error(st, SIC_ERR_TIMEOUT, blockIdx.x);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
    }
}

// Increment of one chunk's running FP32 sum of a column of dZ (blockIdx.y 0: dZ1, 1: dZ2; one thread per
// column, 32 rows at a time through shared memory) or of dS (2), from the total of the earlier tiles.
// Rows beyond the batch hold zeros in dZ and are left out of dS.
__global__ void __launch_bounds__(HID) k_train_bias(float* __restrict__ ws, TrainTc L) {
    __shared__ float sv[HID][33];
    const long long t0 = (long long)blockIdx.x * CHUNK, t1 = t0 + CHUNK < L.tiles ? t0 + CHUNK : L.tiles;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int col = blockIdx.y < 2 ? (int)blockIdx.y * HID + tid : NB;
    const float* tsum = ws + L.tsum() + col;
    float s0 = 0.f;
    if (blockIdx.y < 2 || tid == 0) {
        long long t = 0;
        for (; t + 8 <= t0; t += 8) {
            float v[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) v[i] = tsum[(t + i) * (NB + 4)];
#pragma unroll
            for (int i = 0; i < 8; ++i) s0 += v[i];
        }
        for (; t < t0; ++t) s0 += tsum[t * (NB + 4)];
    }
    float s = s0;
    if (blockIdx.y < 2) {
        const float* dZ = ws + L.dz();
        float v[32];  // this warp's 32 columns of the next 32 rows, lane = row
        auto load = [&](long long i) {
            const float* p = dZ + ((t0 + (i >> 2)) * NB + blockIdx.y * HID + warp * 32) * ROWS + (i & 3) * 32 + lane;
#pragma unroll
            for (int j = 0; j < 32; ++j) v[j] = p[j * ROWS];
        };
        load(0);
        for (long long i = 0; i < 4 * (t1 - t0); ++i) {
            __syncwarp();  // a warp stages and sums its own columns
#pragma unroll
            for (int j = 0; j < 32; ++j) sv[warp * 32 + j][lane] = v[j];
            __syncwarp();
            if (i + 1 < 4 * (t1 - t0)) load(i + 1);
#pragma unroll
            for (int j = 0; j < 32; ++j) s += sv[tid][j];
        }
    } else {
        const float* dS = ws + L.ds();
        for (long long r = t0 * ROWS; r < t1 * ROWS; r += ROWS) {
            __syncthreads();
            sv[0][tid] = r + tid < L.rows ? dS[r + tid] : 0.f;  // (row 0 of sv runs on into the next rows)
            __syncthreads();
            if (tid == 0)
                for (int j = 0; j < ROWS; ++j) s += (&sv[0][0])[j];
        }
    }
    if (blockIdx.y < 2 || tid == 0) ws[L.delta() + blockIdx.x * (NB + 4) + col] = s - s0;
}

// grads[i] = sum over the CTAs of part[cta][i] -- for a bias, over the chunks of its increments --, loss =
// the loss sums / rows, in a fixed order: 8 threads per value take every eighth term, their sums
// added in order
__global__ void __launch_bounds__(256) k_train_sum(const float* __restrict__ ws, TrainTc L, float* __restrict__ grads,
                                                   float* __restrict__ loss) {
    __shared__ float s[8][32];
    const int i = blockIdx.x * 32 + (threadIdx.x & 31), z = threadIdx.x >> 5;
    const int bias = (i >= OFF_B1 && i < OFF_W2)   ? i - OFF_B1
                     : (i >= OFF_B2 && i < OFF_W3) ? HID + i - OFF_B2
                     : i == OFF_B3                 ? NB
                                                   : -1;
    const float* p = bias >= 0 ? ws + L.delta() + bias : ws + L.part() + i;
    const long long step = bias >= 0 ? NB + 4 : PART, terms = bias >= 0 ? L.chunks() : L.ctas;
    float a = 0.f;
    if (i <= NPARAM)
        for (long long c = z; c < terms; c += 8) a += p[c * step];
    s[z][threadIdx.x & 31] = a;
    __syncthreads();
    if (z == 0 && i <= NPARAM) {
#pragma unroll
        for (int q = 1; q < 8; ++q) a += s[q][threadIdx.x];
        if (i < NPARAM)
            grads[i] = a;
        else
            *loss = a / (float)L.rows;
    }
}

inline TrainTc train_layout(long long batch) {
    TrainTc L;
    L.rows = batch;
    L.tiles = (batch + ROWS - 1) / ROWS;
    L.ctas = L.tiles < MAX_CTAS ? L.tiles : MAX_CTAS;
    return L;
}

}  // namespace

long long train_tc_floats(long long batch) { return train_layout(batch).size(); }

sic_status train_tc(sic_handle* h, const float* params, const float* feat, const float* label, long long batch,
                    float pos_weight, float* grads, float* loss, float* score, float* ws, cudaStream_t s) {
    SIC_CUDA_TRY(cudaFuncSetAttribute(k_train_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_TR));
    const TrainTc L = train_layout(batch);
    k_train_tc<<<(unsigned)L.ctas, NT, SMEM_TR, s>>>(feat, label, batch, params, pos_weight, score, ws, L, h->d_status);
    k_train_bias<<<dim3((unsigned)L.chunks(), 3), HID, 0, s>>>(ws, L);
    k_train_sum<<<(NPARAM + 1 + 31) / 32, 256, 0, s>>>(ws, L, grads, loss);
    SIC_CUDA_TRY(cudaGetLastError());
    return SIC_OK;
}
