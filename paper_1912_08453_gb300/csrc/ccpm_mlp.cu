// ccpm_mlp.cu -- the constraint-ordering network: a 3-layer perceptron
// (16 -> 64 -> 64 -> 1, ReLU) with BF16 tensor-core forward and backward
// kernels (mma.sync m16n8k16, FP32 accumulate), FP32 master weights and an
// Adam update.  It scores non-local constraints; the pruning pipeline runs
// the best-scored remaining constraint next (every constraint still runs).
//
// Numerics (both here and in the CPU reference the tests compare against):
// inputs X, weights W1/W2 and the hidden activations H1 are rounded to BF16
// before each tensor-core product; products accumulate in FP32; biases, the
// last layer (64 -> 1 dot product), the loss and all gradient reductions
// across the batch are FP32.  The backward products (dW2 = H1^T dZ2,
// dZ1 = dZ2 W2^T, dW1 = X^T dZ1) round their operands (H1, dZ2, W2, X, dZ1)
// to BF16 the same way.
#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <mutex>
#include <cstring>
#include <new>
#include <string>
#include <thread>
#include <vector>

#include "ccpm_internal.h"

namespace ccpm {

constexpr int IN = CCPM_MLP_IN, HID = CCPM_MLP_HIDDEN;
constexpr int OFF_W1 = 0, OFF_B1 = OFF_W1 + IN * HID, OFF_W2 = OFF_B1 + HID, OFF_B2 = OFF_W2 + HID * HID,
              OFF_W3 = OFF_B2 + HID, OFF_B3 = OFF_W3 + HID, NPARAM = OFF_B3 + 1;
static_assert(NPARAM == CCPM_MLP_PARAMS, "parameter layout");
constexpr int ROWS = 64;          // batch rows per CTA
constexpr int THREADS = 128;      // 4 warps

// ---------------------------------------------------------------- mma core

__device__ __forceinline__ uint32_t pack2(__nv_bfloat16 lo, __nv_bfloat16 hi) {
    uint32_t l = (uint32_t)__bfloat16_as_ushort(lo), h = (uint32_t)__bfloat16_as_ushort(hi);
    return l | (h << 16);
}

// Strided view of a BF16 matrix in shared memory: element (r, c) at
// base[r * rs + c * cs] (a transposed view swaps the strides).
struct View {
    const __nv_bfloat16 *p;
    int rs, cs;
    __device__ __forceinline__ __nv_bfloat16 at(int r, int c) const { return p[r * rs + c * cs]; }
};

// C[M x N] (+)= A[M x K] B[K x N] with all operands in shared memory; the
// CTA's warps share the 16 x 8 output tiles.  C is FP32 with row stride ldc.
__device__ void cta_gemm(View A, View B, float *C, int ldc, int M, int N, int K, bool accumulate) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int g = lane >> 2, tq = lane & 3;
    const int tiles = (M / 16) * (N / 8);
    for (int t = warp; t < tiles; t += nw) {
        const int m0 = (t / (N / 8)) * 16, n0 = (t % (N / 8)) * 8;
        float c[4];
        if (accumulate) {
            c[0] = C[(m0 + g) * ldc + n0 + tq * 2];
            c[1] = C[(m0 + g) * ldc + n0 + tq * 2 + 1];
            c[2] = C[(m0 + g + 8) * ldc + n0 + tq * 2];
            c[3] = C[(m0 + g + 8) * ldc + n0 + tq * 2 + 1];
        } else {
            c[0] = c[1] = c[2] = c[3] = 0.f;
        }
        for (int k0 = 0; k0 < K; k0 += 16) {
            const uint32_t a0 = pack2(A.at(m0 + g, k0 + tq * 2), A.at(m0 + g, k0 + tq * 2 + 1));
            const uint32_t a1 = pack2(A.at(m0 + g + 8, k0 + tq * 2), A.at(m0 + g + 8, k0 + tq * 2 + 1));
            const uint32_t a2 = pack2(A.at(m0 + g, k0 + tq * 2 + 8), A.at(m0 + g, k0 + tq * 2 + 9));
            const uint32_t a3 = pack2(A.at(m0 + g + 8, k0 + tq * 2 + 8), A.at(m0 + g + 8, k0 + tq * 2 + 9));
            const uint32_t b0 = pack2(B.at(k0 + tq * 2, n0 + g), B.at(k0 + tq * 2 + 1, n0 + g));
            const uint32_t b1 = pack2(B.at(k0 + tq * 2 + 8, n0 + g), B.at(k0 + tq * 2 + 9, n0 + g));
            asm volatile(
                "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 "
                "{%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
                : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
        }
        C[(m0 + g) * ldc + n0 + tq * 2] = c[0];
        C[(m0 + g) * ldc + n0 + tq * 2 + 1] = c[1];
        C[(m0 + g + 8) * ldc + n0 + tq * 2] = c[2];
        C[(m0 + g + 8) * ldc + n0 + tq * 2 + 1] = c[3];
    }
}

// ------------------------------------------------------------- forward

struct FwdSmem {
    __nv_bfloat16 x[ROWS * IN];
    __nv_bfloat16 w1[IN * HID];
    __nv_bfloat16 w2[HID * HID];
    __nv_bfloat16 h1b[ROWS * HID];
    float z1[ROWS * HID];
    float z2[ROWS * HID];
};

// Forward pass of one 64-row tile: z1 = X W1 + b1, h1 = relu(z1),
// z2 = h1 W2 + b2, h2 = relu(z2), y = h2 . w3 + b3.
__device__ void forward_tile(const float *__restrict__ prm, const float *__restrict__ X, int B, int row0,
                             FwdSmem &S) {
    for (int i = threadIdx.x; i < ROWS * IN; i += blockDim.x) {
        const int r = i / IN;
        S.x[i] = __float2bfloat16_rn(row0 + r < B ? X[(size_t)(row0 + r) * IN + (i % IN)] : 0.f);
    }
    for (int i = threadIdx.x; i < IN * HID; i += blockDim.x) S.w1[i] = __float2bfloat16_rn(prm[OFF_W1 + i]);
    for (int i = threadIdx.x; i < HID * HID; i += blockDim.x) S.w2[i] = __float2bfloat16_rn(prm[OFF_W2 + i]);
    __syncthreads();
    cta_gemm(View{S.x, IN, 1}, View{S.w1, HID, 1}, S.z1, HID, ROWS, HID, IN, false);
    __syncthreads();
    for (int i = threadIdx.x; i < ROWS * HID; i += blockDim.x) {
        const float z = S.z1[i] + prm[OFF_B1 + (i % HID)];
        S.z1[i] = z;
        S.h1b[i] = __float2bfloat16_rn(z > 0.f ? z : 0.f);
    }
    __syncthreads();
    cta_gemm(View{S.h1b, HID, 1}, View{S.w2, HID, 1}, S.z2, HID, ROWS, HID, HID, false);
    __syncthreads();
    for (int i = threadIdx.x; i < ROWS * HID; i += blockDim.x) S.z2[i] += prm[OFF_B2 + (i % HID)];
    __syncthreads();
}

__device__ float out_row(const float *__restrict__ prm, const FwdSmem &S, int r) {
    float y = prm[OFF_B3];
    for (int j = 0; j < HID; j++) {
        const float h = S.z2[r * HID + j];
        y += (h > 0.f ? h : 0.f) * prm[OFF_W3 + j];
    }
    return y;
}

__global__ void __launch_bounds__(THREADS) k_mlp_forward(const float *prm, const float *X, int B, float *Y) {
    extern __shared__ __align__(16) unsigned char smem[];
    FwdSmem &S = *reinterpret_cast<FwdSmem *>(smem);
    for (int row0 = blockIdx.x * ROWS; row0 < B; row0 += gridDim.x * ROWS) {
        forward_tile(prm, X, B, row0, S);
        for (int r = threadIdx.x; r < ROWS; r += blockDim.x)
            if (row0 + r < B) Y[row0 + r] = out_row(prm, S, r);
        __syncthreads();
    }
}

// ------------------------------------------------------------- backward

struct BwdSmem {
    FwdSmem f;
    __nv_bfloat16 dz2b[ROWS * HID];
    __nv_bfloat16 dz1b[ROWS * HID];
    float dz2[ROWS * HID];
    float dz1[ROWS * HID];
    float gw2[HID * HID];
    float gw1[IN * HID];
    float dy[ROWS];
};

// Loss 0.5 * mean((y - t)^2) over the rows idx[0..B): gradients of every
// parameter are added (FP32 atomics) into grad, the summed squared error into
// *sse.  idx may be NULL (rows 0..B-1).
__global__ void __launch_bounds__(THREADS)
k_mlp_backward(const float *prm, const float *X, const float *T, const int32_t *idx, int B, float inv_n,
               float *grad, float *sse) {
    extern __shared__ __align__(16) unsigned char smem[];
    BwdSmem &S = *reinterpret_cast<BwdSmem *>(smem);
    // gather this tile's rows into a dense staging copy of X (in z1 scratch)
    for (int row0 = blockIdx.x * ROWS; row0 < B; row0 += gridDim.x * ROWS) {
        // forward, reading X through idx
        for (int i = threadIdx.x; i < ROWS * IN; i += blockDim.x) {
            const int r = i / IN, row = row0 + r;
            float v = 0.f;
            if (row < B) {
                const int src = idx ? idx[row] : row;
                v = X[(size_t)src * IN + (i % IN)];
            }
            S.f.x[i] = __float2bfloat16_rn(v);
        }
        for (int i = threadIdx.x; i < IN * HID; i += blockDim.x) S.f.w1[i] = __float2bfloat16_rn(prm[OFF_W1 + i]);
        for (int i = threadIdx.x; i < HID * HID; i += blockDim.x) S.f.w2[i] = __float2bfloat16_rn(prm[OFF_W2 + i]);
        __syncthreads();
        cta_gemm(View{S.f.x, IN, 1}, View{S.f.w1, HID, 1}, S.f.z1, HID, ROWS, HID, IN, false);
        __syncthreads();
        for (int i = threadIdx.x; i < ROWS * HID; i += blockDim.x) {
            const float z = S.f.z1[i] + prm[OFF_B1 + (i % HID)];
            S.f.z1[i] = z;
            S.f.h1b[i] = __float2bfloat16_rn(z > 0.f ? z : 0.f);
        }
        __syncthreads();
        cta_gemm(View{S.f.h1b, HID, 1}, View{S.f.w2, HID, 1}, S.f.z2, HID, ROWS, HID, HID, false);
        __syncthreads();
        for (int i = threadIdx.x; i < ROWS * HID; i += blockDim.x) S.f.z2[i] += prm[OFF_B2 + (i % HID)];
        __syncthreads();
        // output layer and dL/dy
        for (int r = threadIdx.x; r < ROWS; r += blockDim.x) {
            const int row = row0 + r;
            float d = 0.f;
            if (row < B) {
                const float y = out_row(prm, S.f, r);
                const int src = idx ? idx[row] : row;
                const float e = y - T[src];
                atomicAdd(sse, e * e);
                d = e * inv_n;
            }
            S.dy[r] = d;
        }
        __syncthreads();
        // w3, b3 and dz2 = dy * w3 * relu'(z2)
        for (int j = threadIdx.x; j < HID; j += blockDim.x) {
            float gw3 = 0.f;
            for (int r = 0; r < ROWS; r++) {
                const float h = S.f.z2[r * HID + j];
                gw3 += S.dy[r] * (h > 0.f ? h : 0.f);
            }
            atomicAdd(&grad[OFF_W3 + j], gw3);
        }
        if (threadIdx.x == 0) {
            float gb3 = 0.f;
            for (int r = 0; r < ROWS; r++) gb3 += S.dy[r];
            atomicAdd(&grad[OFF_B3], gb3);
        }
        for (int i = threadIdx.x; i < ROWS * HID; i += blockDim.x) {
            const int r = i / HID, j = i % HID;
            const float d = S.f.z2[i] > 0.f ? S.dy[r] * prm[OFF_W3 + j] : 0.f;
            S.dz2[i] = d;
            S.dz2b[i] = __float2bfloat16_rn(d);
        }
        __syncthreads();
        // dW2 = h1^T dz2 (64 x 64, K = rows); dz1 = (dz2 W2^T) * relu'(z1)
        cta_gemm(View{S.f.h1b, 1, HID}, View{S.dz2b, HID, 1}, S.gw2, HID, HID, HID, ROWS, false);
        cta_gemm(View{S.dz2b, HID, 1}, View{S.f.w2, 1, HID}, S.dz1, HID, ROWS, HID, HID, false);
        __syncthreads();
        for (int i = threadIdx.x; i < HID * HID; i += blockDim.x) atomicAdd(&grad[OFF_W2 + i], S.gw2[i]);
        for (int j = threadIdx.x; j < HID; j += blockDim.x) {
            float gb2 = 0.f;
            for (int r = 0; r < ROWS; r++) gb2 += S.dz2[r * HID + j];
            atomicAdd(&grad[OFF_B2 + j], gb2);
        }
        for (int i = threadIdx.x; i < ROWS * HID; i += blockDim.x) {
            const float d = S.f.z1[i] > 0.f ? S.dz1[i] : 0.f;
            S.dz1[i] = d;
            S.dz1b[i] = __float2bfloat16_rn(d);
        }
        __syncthreads();
        // dW1 = x^T dz1 (16 x 64, K = rows)
        cta_gemm(View{S.f.x, 1, IN}, View{S.dz1b, HID, 1}, S.gw1, HID, IN, HID, ROWS, false);
        __syncthreads();
        for (int i = threadIdx.x; i < IN * HID; i += blockDim.x) atomicAdd(&grad[OFF_W1 + i], S.gw1[i]);
        for (int j = threadIdx.x; j < HID; j += blockDim.x) {
            float gb1 = 0.f;
            for (int r = 0; r < ROWS; r++) gb1 += S.dz1[r * HID + j];
            atomicAdd(&grad[OFF_B1 + j], gb1);
        }
        __syncthreads();
    }
}

// Adam step on FP32 master weights (bias-corrected), then clear the gradient.
__global__ void k_mlp_adam(float *prm, float *grad, float *m1, float *m2, int step, float lr) {
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    const float c1 = 1.f - powf(b1, (float)step), c2 = 1.f - powf(b2, (float)step);
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < NPARAM; i += gridDim.x * blockDim.x) {
        const float gi = grad[i];
        m1[i] = b1 * m1[i] + (1.f - b1) * gi;
        m2[i] = b2 * m2[i] + (1.f - b2) * gi * gi;
        prm[i] -= lr * (m1[i] / c1) / (sqrtf(m2[i] / c2) + eps);
        grad[i] = 0.f;
    }
}

// Minibatch row indices from a counter-based hash (SplitMix64 finaliser).
__device__ __forceinline__ int32_t sample_row(int batch, int n, uint64_t seed, int step, int i) {
    uint64_t z = seed + 0x9E3779B97F4A7C15ull * (uint64_t)((int64_t)step * batch + i + 1);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    z ^= z >> 31;
    return (int32_t)(z % (uint64_t)n);
}

__global__ void k_mlp_sample(int32_t *idx, int batch, int n, uint64_t seed, int step) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < batch; i += gridDim.x * blockDim.x)
        idx[i] = sample_row(batch, n, seed, step, i);
}

// ------------------------------------------------------------- training loop
//
// All Adam steps of a training call in one kernel, one thread-block cluster.
// A step is a chain of small products and reductions, so its time is latency:
// as three kernels and a memset (sampling, backward over 64-row blocks with
// atomics into one gradient, Adam) it took 37 us at 256 rows, 28 of them in the
// backward kernel with its scalar fragment loads.  Here a block holds the weights in
// shared memory (bf16, as the products want them) and 64 rows at a time; warp w
// owns columns 8w..8w+7 of both hidden layers, so its gradients of those columns
// stay in registers; fragments are loaded with ldmatrix.  The blocks' gradients
// are summed slice by slice through distributed shared memory, in rank order (so
// two runs give the same bits), the slice's owner does its Adam step on FP32
// masters and writes the new weights to all blocks: two cluster barriers a step,
// 8.2 us up to 512 rows.  Always eight blocks, since the Adam step is split over
// them too: with one block for 32 rows a step took 25 us.  16 warps a block, a
// half of the rows each, took 8.8.
//
// Sums run in the order of the kernels per step: 64-row tiles, rows and columns
// one after the other, the tiles' sums added up.  Training amplifies every other
// rounding (a hidden value that falls to the neighbouring bf16 changes all that
// follows), so another order, though no less exact, ends further away: 2e-5 of
// the scores after 63 steps with rows summed lane by lane.

namespace cg = cooperative_groups;

constexpr int TR = ROWS;           // rows per block and chunk
constexpr int TTHREADS = 256;      // 8 warps
constexpr int LDH = HID + 8, LDX = IN + 8;     // row strides: ldmatrix rows on distinct banks
constexpr int kTrainCluster = 8;   // blocks
constexpr int kTrainMaxBatch = 4096;   // rows up to which the fused loop is used

struct TrainSmem {
    alignas(16) __nv_bfloat16 w1[IN * LDH], w2[HID * LDH];
    alignas(16) __nv_bfloat16 x[TR * LDX], h1[TR * LDH], dz2[TR * LDH], dz1[TR * LDH];
    float b1[HID], b2[HID], w3[HID], b3;
    float t[TR], dy[TR];
    float h2[TR][HID + 1], dz2f[TR][HID + 1], dz1f[TR][HID + 1];
    float grad[NPARAM];
    float corr[2];                 // Adam's bias corrections of this step
    float sse[TR / 32];
};

struct TrainArgs {
    float *prm, *m1, *m2, *sse;
    const float *X, *T;
    int N, batch, rows;            // rows: per block
    int steps, step0, adam0;       // steps of this launch, sampling steps and Adam steps before it
    uint64_t seed;
    float lr;
};

__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

template <bool TRANS>
__device__ __forceinline__ void ldm4(uint32_t (&r)[4], const void *p) {
    if (TRANS)
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(smem_addr(p)) : "memory");
    else
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(smem_addr(p)) : "memory");
}
template <bool TRANS>
__device__ __forceinline__ void ldm2(uint32_t (&r)[2], const void *p) {
    if (TRANS)
        asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];"
                     : "=r"(r[0]), "=r"(r[1]) : "r"(smem_addr(p)) : "memory");
    else
        asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0,%1}, [%2];"
                     : "=r"(r[0]), "=r"(r[1]) : "r"(smem_addr(p)) : "memory");
}
__device__ __forceinline__ void mma16816(float (&c)[4], const uint32_t (&a)[4], const uint32_t (&b)[2]) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 "
        "{%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// Fragments of a 16 x 16 A tile / a 16 x 8 B tile.  M: row-major matrix with row
// stride ld holding A (rows m, columns k) or A^T; B (rows k, columns n) or B^T.
__device__ __forceinline__ void frag_a(uint32_t (&r)[4], const __nv_bfloat16 *M, int ld, int m0, int k0) {
    const int l = threadIdx.x & 31;
    ldm4<false>(r, M + (m0 + (l & 15)) * ld + k0 + 8 * (l >> 4));
}
__device__ __forceinline__ void frag_at(uint32_t (&r)[4], const __nv_bfloat16 *M, int ld, int m0, int k0) {
    const int l = threadIdx.x & 31;     // tiles in the order (m, k), (m + 8, k), (m, k + 8), (m + 8, k + 8)
    ldm4<true>(r, M + (k0 + (l & 7) + 8 * (l >> 4)) * ld + m0 + 8 * ((l >> 3) & 1));
}
__device__ __forceinline__ void frag_b(uint32_t (&r)[2], const __nv_bfloat16 *M, int ld, int k0, int n0) {
    const int l = threadIdx.x & 15;
    ldm2<true>(r, M + (k0 + l) * ld + n0);
}
__device__ __forceinline__ void frag_bt(uint32_t (&r)[2], const __nv_bfloat16 *M, int ld, int k0, int n0) {
    const int l = threadIdx.x & 15;
    ldm2<false>(r, M + (n0 + (l & 7)) * ld + k0 + 8 * (l >> 3));
}

// New value of parameter i in a block's working copy.
__device__ __forceinline__ void put_param(TrainSmem &S, int i, float v) {
    if (i < OFF_B1) S.w1[(i / HID) * LDH + i % HID] = __float2bfloat16_rn(v);
    else if (i < OFF_W2) S.b1[i - OFF_B1] = v;
    else if (i < OFF_B2) S.w2[((i - OFF_W2) / HID) * LDH + (i - OFF_W2) % HID] = __float2bfloat16_rn(v);
    else if (i < OFF_W3) S.b2[i - OFF_B2] = v;
    else if (i < OFF_B3) S.w3[i - OFF_W3] = v;
    else S.b3 = v;
}

__global__ void __launch_bounds__(TTHREADS) k_mlp_train(TrainArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    TrainSmem &S = *reinterpret_cast<TrainSmem *>(smem);
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank();
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, g = lane >> 2, tq = lane & 3;
    const int n0 = 8 * w, c0 = n0 + 2 * tq;              // the warp's columns, this lane's first one
    // this thread's share of the block's slice of the parameters
    constexpr int C = kTrainCluster, slice = (NPARAM + C - 1) / C, kOwn = (slice + TTHREADS - 1) / TTHREADS;
    const int own0 = rank * slice;
    float p[kOwn], m1[kOwn], m2[kOwn];
#pragma unroll
    for (int k = 0; k < kOwn; k++) {
        const int j = tid + k * TTHREADS, i = own0 + j;
        p[k] = m1[k] = m2[k] = 0.f;
        if (j < slice && i < NPARAM) { p[k] = a.prm[i]; m1[k] = a.m1[i]; m2[k] = a.m2[i]; }
    }
    for (int i = tid; i < NPARAM; i += TTHREADS) put_param(S, i, a.prm[i]);
    const int first = rank * a.rows, last = min(a.batch, first + a.rows);     // this block's rows
    const int chunks = (a.rows + TR - 1) / TR;
    const float inv_n = 1.f / (float)a.batch;
    // a chunk's inputs: four features per thread, and a target for the first 64,
    // fetched one chunk ahead
    float4 nx = make_float4(0.f, 0.f, 0.f, 0.f);
    float nt = 0.f;
    auto fetch = [&](int step, int chunk) {
        nx = make_float4(0.f, 0.f, 0.f, 0.f);
        nt = 0.f;
        if (step >= a.steps) return;
        const int row = first + chunk * TR + (tid >> 2);
        if (row < last) {
            const int src = sample_row(a.batch, a.N, a.seed, a.step0 + step, row);
            nx = *reinterpret_cast<const float4 *>(a.X + (size_t)src * IN + 4 * (tid & 3));
        }
        const int trow = first + chunk * TR + tid;
        if (tid < TR && trow < last) nt = a.T[sample_row(a.batch, a.N, a.seed, a.step0 + step, trow)];
    };
    constexpr int MT = TR / 16;                          // 16-row tiles
    fetch(0, 0);
    for (int step = 0; step < a.steps; step++) {
        float gw2[4][4] = {}, gw1[4] = {}, gcol = 0.f, sse = 0.f;
        for (int chunk = 0; chunk < chunks; chunk++) {
            {
                __nv_bfloat16 *d = S.x + (tid >> 2) * LDX + 4 * (tid & 3);
                d[0] = __float2bfloat16_rn(nx.x);
                d[1] = __float2bfloat16_rn(nx.y);
                d[2] = __float2bfloat16_rn(nx.z);
                d[3] = __float2bfloat16_rn(nx.w);
            }
            if (tid < TR) S.t[tid] = nt;
            else if (tid < TR + 2 && chunk == 0)
                S.corr[tid - TR] = 1.f - powf(tid == TR ? 0.9f : 0.999f, (float)(a.adam0 + step + 1));
            __syncthreads();
            if (chunk + 1 < chunks) fetch(step, chunk + 1);
            else fetch(step + 1, 0);
            // h1 = relu(X W1 + b1)
            uint32_t pos1 = 0;                           // z1 > 0, per fragment element
            {
                uint32_t b[2];
                frag_b(b, S.w1, LDH, 0, n0);
#pragma unroll
                for (int mt = 0; mt < MT; mt++) {
                    uint32_t f[4];
                    float z[4] = {};
                    frag_a(f, S.x, LDX, 16 * mt, 0);
                    mma16816(z, f, b);
#pragma unroll
                    for (int i = 0; i < 4; i++) {
                        z[i] += S.b1[c0 + (i & 1)];
                        if (z[i] > 0.f) pos1 |= 1u << (4 * mt + i);
                        else z[i] = 0.f;
                    }
                    __nv_bfloat16 *h = S.h1 + (16 * mt + g) * LDH + c0;
                    *reinterpret_cast<__nv_bfloat162 *>(h) = __floats2bfloat162_rn(z[0], z[1]);
                    *reinterpret_cast<__nv_bfloat162 *>(h + 8 * LDH) = __floats2bfloat162_rn(z[2], z[3]);
                }
            }
            __syncthreads();
            // h2 = relu(h1 W2 + b2)
            float z2[MT][4] = {};
#pragma unroll
            for (int k = 0; k < HID; k += 16) {
                uint32_t b[2];
                frag_b(b, S.w2, LDH, k, n0);
#pragma unroll
                for (int mt = 0; mt < MT; mt++) {
                    uint32_t f[4];
                    frag_a(f, S.h1, LDH, 16 * mt, k);
                    mma16816(z2[mt], f, b);
                }
            }
#pragma unroll
            for (int mt = 0; mt < MT; mt++)
#pragma unroll
                for (int i = 0; i < 4; i++) {
                    z2[mt][i] += S.b2[c0 + (i & 1)];
                    S.h2[16 * mt + 8 * (i >> 1) + g][c0 + (i & 1)] = z2[mt][i] > 0.f ? z2[mt][i] : 0.f;
                }
            __syncthreads();
            // y = h2 w3 + b3 and dL/dy
            if (tid < TR) {
                float y = S.b3, e = 0.f;
#pragma unroll
                for (int j = 0; j < HID; j++) y += S.h2[tid][j] * S.w3[j];
                if (first + chunk * TR + tid < last) e = y - S.t[tid];
                S.dy[tid] = e * inv_n;
                sse += e * e;
            }
            __syncthreads();
            // dz2 = dy w3 relu'(z2)
#pragma unroll
            for (int mt = 0; mt < MT; mt++) {
#pragma unroll
                for (int i = 0; i < 4; i++) {
                    const int r = 16 * mt + 8 * (i >> 1) + g;
                    z2[mt][i] = z2[mt][i] > 0.f ? S.dy[r] * S.w3[c0 + (i & 1)] : 0.f;
                    S.dz2f[r][c0 + (i & 1)] = z2[mt][i];
                }
                __nv_bfloat16 *d = S.dz2 + (16 * mt + g) * LDH + c0;
                *reinterpret_cast<__nv_bfloat162 *>(d) = __floats2bfloat162_rn(z2[mt][0], z2[mt][1]);
                *reinterpret_cast<__nv_bfloat162 *>(d + 8 * LDH) = __floats2bfloat162_rn(z2[mt][2], z2[mt][3]);
            }
            __syncthreads();
            // dz1 = (dz2 W2^T) relu'(z1)
            float d1[MT][4] = {};
#pragma unroll
            for (int k = 0; k < HID; k += 16) {
                uint32_t b[2];
                frag_bt(b, S.w2, LDH, k, n0);
#pragma unroll
                for (int mt = 0; mt < MT; mt++) {
                    uint32_t f[4];
                    frag_a(f, S.dz2, LDH, 16 * mt, k);
                    mma16816(d1[mt], f, b);
                }
            }
#pragma unroll
            for (int mt = 0; mt < MT; mt++) {
#pragma unroll
                for (int i = 0; i < 4; i++) {
                    if (!((pos1 >> (4 * mt + i)) & 1u)) d1[mt][i] = 0.f;
                    S.dz1f[16 * mt + 8 * (i >> 1) + g][c0 + (i & 1)] = d1[mt][i];
                }
                __nv_bfloat16 *d = S.dz1 + (16 * mt + g) * LDH + c0;
                *reinterpret_cast<__nv_bfloat162 *>(d) = __floats2bfloat162_rn(d1[mt][0], d1[mt][1]);
                *reinterpret_cast<__nv_bfloat162 *>(d + 8 * LDH) = __floats2bfloat162_rn(d1[mt][2], d1[mt][3]);
            }
            __syncthreads();
            // gradients of this chunk: w3 (threads 0..63), b2, b1 and b3 row by row,
            // dW2 = h1^T dz2 and dW1 = x^T dz1 for the warp's columns
            const int j = tid & 63;
            float s = 0.f;
            if (tid < 64) {
#pragma unroll 16
                for (int r = 0; r < TR; r++) s += S.dy[r] * S.h2[r][j];
            } else if (tid < 128) {
#pragma unroll 16
                for (int r = 0; r < TR; r++) s += S.dz2f[r][j];
            } else if (tid < 192) {
#pragma unroll 16
                for (int r = 0; r < TR; r++) s += S.dz1f[r][j];
            } else if (tid == 192) {
#pragma unroll 16
                for (int r = 0; r < TR; r++) s += S.dy[r];
            }
            gcol += s;
            __syncwarp();
            float c2[4][4] = {}, c1[4] = {};
#pragma unroll
            for (int k = 0; k < TR; k += 16) {
                uint32_t f[4], b[2];
                frag_b(b, S.dz2, LDH, k, n0);
#pragma unroll
                for (int mt = 0; mt < 4; mt++) {
                    frag_at(f, S.h1, LDH, 16 * mt, k);
                    mma16816(c2[mt], f, b);
                }
                frag_at(f, S.x, LDX, 0, k);
                frag_b(b, S.dz1, LDH, k, n0);
                mma16816(c1, f, b);
            }
#pragma unroll
            for (int i = 0; i < 4; i++) {
                gw1[i] += c1[i];
#pragma unroll
                for (int mt = 0; mt < 4; mt++) gw2[mt][i] += c2[mt][i];
            }
            __syncthreads();                             // all of it is rewritten by the next chunk
        }
        // the block's gradient
#pragma unroll
        for (int mt = 0; mt < 4; mt++)
#pragma unroll
            for (int i = 0; i < 4; i++)
                S.grad[OFF_W2 + (16 * mt + 8 * (i >> 1) + g) * HID + c0 + (i & 1)] = gw2[mt][i];
#pragma unroll
        for (int i = 0; i < 4; i++) S.grad[OFF_W1 + (8 * (i >> 1) + g) * HID + c0 + (i & 1)] = gw1[i];
        if (tid < 64) S.grad[OFF_W3 + tid] = gcol;
        else if (tid < 128) S.grad[OFF_B2 + tid - 64] = gcol;
        else if (tid < 192) S.grad[OFF_B1 + tid - 128] = gcol;
        else if (tid == 192) S.grad[OFF_B3] = gcol;
        if (tid < TR) {                                  // rows were taken by the first two warps
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) sse += __shfl_xor_sync(0xFFFFFFFFu, sse, o);
            if (lane == 0) S.sse[w] = sse;
        }
        cluster.sync();
        // sum the blocks' gradients of this block's slice, Adam step, new weights to all blocks
        const float corr1 = S.corr[0], corr2 = S.corr[1];
#pragma unroll
        for (int k = 0; k < kOwn; k++) {
            const int j = tid + k * TTHREADS, i = own0 + j;
            if (j >= slice || i >= NPARAM) break;
            float gi = 0.f;
#pragma unroll
            for (int r = 0; r < C; r++) gi += *cluster.map_shared_rank(&S.grad[i], r);
            m1[k] = 0.9f * m1[k] + (1.f - 0.9f) * gi;
            m2[k] = 0.999f * m2[k] + (1.f - 0.999f) * gi * gi;
            p[k] -= a.lr * (m1[k] / corr1) / (sqrtf(m2[k] / corr2) + 1e-8f);
#pragma unroll
            for (int r = 0; r < C; r++) put_param(*cluster.map_shared_rank(&S, r), i, p[k]);
        }
        if (step == a.steps - 1 && rank == 0 && tid == 0) {
            float sum = 0.f;
            for (int r = 0; r < C; r++) 
                for (int k = 0; k < TR / 32; k++) sum += *cluster.map_shared_rank(&S.sse[k], r);
            *a.sse = sum;
        }
        cluster.sync();
    }
#pragma unroll
    for (int k = 0; k < kOwn; k++) {
        const int j = tid + k * TTHREADS, i = own0 + j;
        if (j < slice && i < NPARAM) { a.prm[i] = p[k]; a.m1[i] = m1[k]; a.m2[i] = m2[k]; }
    }
}

}  // namespace ccpm

using namespace ccpm;

struct ccpm_mlp {
    int device = 0;
    cudaStream_t stream = nullptr;
    float *prm = nullptr, *grad = nullptr, *m1 = nullptr, *m2 = nullptr, *sse = nullptr;
    int adam_step = 0;
    // scratch of the public forward call (pipelines score with their context's own)
    ccpm::MlpScratch own;
    std::mutex mu;               // public forward calls may come from several threads
};

namespace {

size_t fwd_smem() { return sizeof(FwdSmem); }
size_t bwd_smem() { return sizeof(BwdSmem); }

// The fused loop's launch: one cluster.
struct TrainLaunch {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute cluster = {};
    explicit TrainLaunch(cudaStream_t s) {
        cluster.id = cudaLaunchAttributeClusterDimension;
        cluster.val.clusterDim.x = (unsigned)kTrainCluster;
        cluster.val.clusterDim.y = cluster.val.clusterDim.z = 1;
        cfg.gridDim = dim3((unsigned)kTrainCluster);
        cfg.blockDim = dim3(TTHREADS);
        cfg.dynamicSmemBytes = sizeof(TrainSmem);
        cfg.stream = s;
        cfg.attrs = &cluster;
        cfg.numAttrs = 1;
    }
    TrainLaunch(const TrainLaunch &) = delete;
    // Can the current device hold it?  Not where the process is given only some of
    // the SMs and no eight of them share a cluster's reach.
    bool fits() const {
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, k_mlp_train, &cfg) == cudaSuccess) return n > 0;
        cudaGetLastError();
        return false;
    }
};

int configure_kernels(bool *fused = nullptr) {
    // once per device, as settings belong to the current device's copy of a
    // kernel; under a lock, as batch workers reach this concurrently
    constexpr int kDevices = 64;     // those past it are configured by every call
    static std::mutex mu;
    static bool done[kDevices] = {}, fits[kDevices] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return CCPM_ECUDA;
    std::lock_guard<std::mutex> lock(mu);
    if (dev < kDevices && done[dev]) {
        if (fused) *fused = fits[dev];
        return CCPM_OK;
    }
    if (cudaFuncSetAttribute(k_mlp_forward, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)fwd_smem()) != cudaSuccess)
        return CCPM_ECUDA;
    if (cudaFuncSetAttribute(k_mlp_backward, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bwd_smem()) != cudaSuccess)
        return CCPM_ECUDA;
    if (cudaFuncSetAttribute(k_mlp_train, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(TrainSmem)) !=
        cudaSuccess)
        return CCPM_ECUDA;
    const bool takes_cluster = TrainLaunch(nullptr).fits();
    if (fused) *fused = takes_cluster;
    if (dev < kDevices) { done[dev] = true; fits[dev] = takes_cluster; }
    return CCPM_OK;
}

// A refused allocation: reported by its own call, and not once more by the
// check after the next launch.
int no_memory() {
    cudaGetLastError();
    return CCPM_ENOMEM;
}

// Device scratch for one call (X, targets, sampled rows).
struct Scratch {
    float *x = nullptr, *t = nullptr;
    int32_t *idx = nullptr;
    ~Scratch() { cudaFree(x); }  // the others lie behind x
    int alloc(size_t rows, size_t picks) {
        if (cudaMalloc(&x, sizeof(float) * rows * (IN + 1) + sizeof(int32_t) * picks) != cudaSuccess)
            return no_memory();
        t = x + rows * IN;
        idx = (int32_t *)(t + rows);
        return CCPM_OK;
    }
};

int tiles(int B) { return (B + ROWS - 1) / ROWS; }

}  // namespace

namespace ccpm {

void mlp_scratch_free(MlpScratch &sc) {
    cudaFree(sc.dx);             // dy and hy lie behind dx and hx
    if (sc.hx) cudaFreeHost(sc.hx);
    sc = MlpScratch{};
}

// Forward pass for the pruning pipeline's ordering decisions (host arrays),
// with the caller's scratch: no lock is held while the GPU works, so batch
// workers that score at the same time do not wait for one another.
int mlp_score(ccpm_mlp *m, int B, const float *host_x, float *host_y, void *stream, MlpScratch &sc, void *wait_ev) {
    cudaStream_t s = (cudaStream_t)stream;
    if (!m || B <= 0) return CCPM_EINVAL;
    if (configure_kernels()) return CCPM_ECUDA;
    if (B > sc.cap) {
        mlp_scratch_free(sc);
        const int cap = std::max(B, 256);
        if (cudaMalloc(&sc.dx, sizeof(float) * (size_t)cap * (IN + 1)) != cudaSuccess ||
            cudaMallocHost(&sc.hx, sizeof(float) * (size_t)cap * (IN + 1)) != cudaSuccess) {
            mlp_scratch_free(sc);
            return no_memory();
        }
        sc.dy = sc.dx + (size_t)cap * IN;
        sc.hy = sc.hx + (size_t)cap * IN;
        sc.cap = cap;
    }
    std::memcpy(sc.hx, host_x, sizeof(float) * (size_t)B * IN);
    cudaError_t e = cudaMemcpyAsync(sc.dx, sc.hx, sizeof(float) * (size_t)B * IN, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) {
        k_mlp_forward<<<tiles(B), THREADS, fwd_smem(), s>>>(m->prm, sc.dx, B, sc.dy);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(sc.hy, sc.dy, sizeof(float) * (size_t)B, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess && wait_ev) {
        cudaEvent_t ev = (cudaEvent_t)wait_ev;
        e = cudaEventRecord(ev, s);
        if (e == cudaSuccess)
            while ((e = cudaEventQuery(ev)) == cudaErrorNotReady) std::this_thread::yield();
    } else if (e == cudaSuccess) {
        e = cudaStreamSynchronize(s);
    }
    if (e == cudaSuccess) std::memcpy(host_y, sc.hy, sizeof(float) * (size_t)B);
    return e == cudaSuccess ? CCPM_OK : CCPM_ECUDA;
}

}  // namespace ccpm

extern "C" {

int ccpm_mlp_create(ccpm_ctx_t ctx, uint64_t seed, ccpm_mlp_t *out) {
    if (!ctx || !out) return CCPM_EINVAL;
    *out = nullptr;
    int dev = ctx_device(ctx);
    if (cudaSetDevice(dev) != cudaSuccess) return CCPM_ECUDA;
    ccpm_mlp *m = new (std::nothrow) ccpm_mlp();
    if (!m) return CCPM_ENOMEM;
    m->device = dev;
    m->stream = (cudaStream_t)ctx_stream_ptr(ctx);
    // one allocation: each allocation and release costs tens of microseconds,
    // as much as several training steps
    if (cudaMalloc(&m->prm, sizeof(float) * (4 * NPARAM + 1)) != cudaSuccess) {
        ccpm_mlp_destroy(m);
        return no_memory();
    }
    m->grad = m->prm + NPARAM;
    m->m1 = m->grad + NPARAM;
    m->m2 = m->m1 + NPARAM;
    m->sse = m->m2 + NPARAM;
    // He-uniform initial weights from a SplitMix64 stream, zero biases
    std::vector<float> p(NPARAM, 0.f);
    uint64_t st = seed;
    auto next = [&]() {
        uint64_t z = (st += 0x9E3779B97F4A7C15ull);
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
        z ^= z >> 31;
        return (double)(z >> 11) * (1.0 / 9007199254740992.0);
    };
    auto fill = [&](int off, int count, int fan_in) {
        const double a = std::sqrt(6.0 / fan_in);
        for (int i = 0; i < count; i++) p[(size_t)(off + i)] = (float)((2.0 * next() - 1.0) * a);
    };
    fill(OFF_W1, IN * HID, IN);
    fill(OFF_W2, HID * HID, HID);
    fill(OFF_W3, HID, HID);
    int rc = ccpm_mlp_set_params(m, p.data());
    if (rc) { ccpm_mlp_destroy(m); return rc; }
    *out = m;
    return CCPM_OK;
}

void ccpm_mlp_destroy(ccpm_mlp_t m) {
    if (!m) return;
    cudaSetDevice(m->device);
    cudaFree(m->prm);
    ccpm::mlp_scratch_free(m->own);
    delete m;
}

int ccpm_mlp_set_params(ccpm_mlp_t m, const float *host_params) {
    if (!m || !host_params) return CCPM_EINVAL;
    if (cudaSetDevice(m->device) != cudaSuccess) return CCPM_ECUDA;
    cudaError_t e = cudaMemcpyAsync(m->prm, host_params, sizeof(float) * NPARAM, cudaMemcpyHostToDevice, m->stream);
    if (e == cudaSuccess)        // gradient and both moments
        e = cudaMemsetAsync(m->grad, 0, sizeof(float) * 3 * NPARAM, m->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
    m->adam_step = 0;
    return e == cudaSuccess ? CCPM_OK : CCPM_ECUDA;
}

int ccpm_mlp_get_params(ccpm_mlp_t m, float *host_params) {
    if (!m || !host_params) return CCPM_EINVAL;
    if (cudaSetDevice(m->device) != cudaSuccess) return CCPM_ECUDA;
    cudaError_t e = cudaMemcpyAsync(host_params, m->prm, sizeof(float) * NPARAM, cudaMemcpyDeviceToHost, m->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
    return e == cudaSuccess ? CCPM_OK : CCPM_ECUDA;
}

int ccpm_mlp_forward(ccpm_mlp_t m, int B, const float *host_x, float *host_y) {
    if (!m || B <= 0 || !host_x || !host_y) return CCPM_EINVAL;
    if (cudaSetDevice(m->device) != cudaSuccess) return CCPM_ECUDA;
    std::lock_guard<std::mutex> lock(m->mu);
    return mlp_score(m, B, host_x, host_y, (void *)m->stream, m->own);
}

int ccpm_mlp_gradient(ccpm_mlp_t m, int B, const float *host_x, const float *host_t, float *host_grad,
                      float *loss) {
    if (!m || B <= 0 || !host_x || !host_t || !host_grad) return CCPM_EINVAL;
    if (cudaSetDevice(m->device) != cudaSuccess) return CCPM_ECUDA;
    if (configure_kernels()) return CCPM_ECUDA;
    Scratch sc;
    if (sc.alloc((size_t)B, 0)) return CCPM_ENOMEM;
    cudaStream_t s = m->stream;
    cudaError_t e = cudaMemcpyAsync(sc.x, host_x, sizeof(float) * (size_t)B * IN, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(sc.t, host_t, sizeof(float) * (size_t)B, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(m->grad, 0, sizeof(float) * NPARAM, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(m->sse, 0, sizeof(float), s);
    if (e == cudaSuccess) {
        k_mlp_backward<<<tiles(B), THREADS, bwd_smem(), s>>>(m->prm, sc.x, sc.t, nullptr, B, 1.f / (float)B, m->grad,
                                                              m->sse);
        e = cudaGetLastError();
    }
    float sse = 0.f;
    if (e == cudaSuccess) e = cudaMemcpyAsync(host_grad, m->grad, sizeof(float) * NPARAM, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&sse, m->sse, sizeof(float), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(m->grad, 0, sizeof(float) * NPARAM, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (loss) *loss = 0.5f * sse / (float)B;
    return e == cudaSuccess ? CCPM_OK : CCPM_ECUDA;
}

int ccpm_mlp_train(ccpm_mlp_t m, int N, const float *host_x, const float *host_t, int steps, int batch, float lr,
                   uint64_t seed, float *final_loss) {
    if (!m || N <= 0 || !host_x || !host_t || steps < 0 || batch <= 0) return CCPM_EINVAL;
    if (cudaSetDevice(m->device) != cudaSuccess) return CCPM_ECUDA;
    bool fused = false;
    if (configure_kernels(&fused)) return CCPM_ECUDA;
    Scratch sc;
    if (sc.alloc((size_t)N, (size_t)batch)) return CCPM_ENOMEM;
    cudaStream_t s = m->stream;
    cudaError_t e = cudaMemcpyAsync(sc.x, host_x, sizeof(float) * (size_t)N * IN, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(sc.t, host_t, sizeof(float) * (size_t)N, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(m->grad, 0, sizeof(float) * NPARAM, s);
    // Up to kTrainMaxBatch every step in one kernel, a few thousand steps a
    // launch: 8.2 us a step up to 512 rows, 12 at 1024, 35 at 4096, 45 at 8192 (a
    // block takes its rows 64 at a time).  The kernels per step, which spread
    // over the whole GPU, take 37 to 40 us up to 4096 rows and 41 at 8192.
    const TrainLaunch launch(s);
    fused = fused && batch <= kTrainMaxBatch;
    for (int it = 0; fused && it < steps && e == cudaSuccess;) {
        const int C = kTrainCluster;      // also where a block gets few rows: the Adam step is split, too
        TrainArgs a;
        a.prm = m->prm;
        a.m1 = m->m1;
        a.m2 = m->m2;
        a.sse = m->sse;
        a.X = sc.x;
        a.T = sc.t;
        a.N = N;
        a.batch = batch;
        a.rows = ((batch + C - 1) / C + TR - 1) / TR * TR;       // whole tiles
        a.steps = std::min(steps - it, 4096);
        a.step0 = it;
        a.adam0 = m->adam_step;
        a.seed = seed;
        a.lr = lr;
        e = cudaLaunchKernelEx(&launch.cfg, k_mlp_train, a);
        if (e == cudaSuccess) e = cudaGetLastError();
        it += a.steps;
        m->adam_step += a.steps;
    }
    for (int it = 0; !fused && it < steps && e == cudaSuccess; it++) {
        e = cudaMemsetAsync(m->sse, 0, sizeof(float), s);
        if (e != cudaSuccess) break;
        k_mlp_sample<<<(batch + 255) / 256, 256, 0, s>>>(sc.idx, batch, N, seed, it);
        k_mlp_backward<<<tiles(batch), THREADS, bwd_smem(), s>>>(m->prm, sc.x, sc.t, sc.idx, batch,
                                                                  1.f / (float)batch, m->grad, m->sse);
        m->adam_step++;
        k_mlp_adam<<<(NPARAM + 255) / 256, 256, 0, s>>>(m->prm, m->grad, m->m1, m->m2, m->adam_step, lr);
        e = cudaGetLastError();
    }
    float sse = 0.f;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&sse, m->sse, sizeof(float), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (final_loss) *final_loss = 0.5f * sse / (float)batch;
    return e == cudaSuccess ? CCPM_OK : CCPM_ECUDA;
}

}  // extern "C"
