// Warm-start network on the 5th-generation tensor cores (tcgen05, sm_103a).
//
// 16 inputs (9 features, zero padded) -> 4 hidden layers of 128 units (exact GELU) -> 16
// outputs (the first 3 used: n, u_y, T in normalised form).  Layer l: z_l = h_{l-1} W_l + b_l,
// W_l stored [inputs][outputs] in FP32 (master copy); BF16 operands, FP32 accumulation.
//
// Every GEMM is D[128 x N] (+)= A[128 x K] B[N x K]^T with A and B in shared memory in the
// K-major "core matrix" layout (8 rows x 16 bytes per 128-byte core matrix; neighbours along
// K 128 bytes apart, 8-row groups 16 K bytes apart), issued as tcgen05.mma kind::f16 (M = 128,
// K = 16 per instruction) by one thread, accumulated in tensor memory, completed through an
// mbarrier and read back with tcgen05.ld (thread t of the 128-thread block owns TMEM lane t).
//
// Forward: one block per 128-point tile, the weights' BF16 images copied into shared memory, the
// activation tile chained through one shared buffer.  Backward (training): per tile,
// dW_l = H_{l-1}^T dZ_l and dH_{l-1} = dZ_l W_l^T as tcgen05 GEMMs; each block writes its
// gradient to its own slot of a partial buffer, and the Adam kernel adds the slots in block
// order (deterministic) before the update and refreshes the BF16 images.  This network has no
// counterpart in the paper.
//
// What bounds a tile: the activation functions and the staging of operands between the GEMMs
// (the tensor pipe is busy for under 1 %).  So a block has 16 warps: tensor memory lane quarter
// w % 4 (a warp reaches no other) and column quarter w / 4, one point and 32 columns per thread;
// operands whose 8 consecutive columns belong to one thread are stored 16 bytes at a time; the
// pre-activations go to global memory with the point fastest, so that a warp writes and reads
// whole lines.
#include "../../include/fdlb.h"

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <cstring>
#include <string>
#include <vector>

namespace {

constexpr int NIN = 16, NH = 128, NOUT = 16, NUSED = 3;
// flat parameter offsets (W1, b1, ..., W5, b5)
constexpr int OW1 = 0, OB1 = OW1 + NIN * NH;
constexpr int OW2 = OB1 + NH, OB2 = OW2 + NH * NH;
constexpr int OW3 = OB2 + NH, OB3 = OW3 + NH * NH;
constexpr int OW4 = OB3 + NH, OB4 = OW4 + NH * NH;
constexpr int OW5 = OB4 + NH, OB5 = OW5 + NH * NOUT;
constexpr int NPARAM = OB5 + NOUT;                 // 53776
constexpr int TILE = 128;
constexpr int THREADS = 512;                       // 16 warps: 4 lane quarters x 4 column quarters
constexpr int WAIT_LIMIT = 4000000;                // bounded mbarrier wait

__host__ __device__ constexpr int woff(int l) { return l == 1 ? OW1 : l == 2 ? OW2 : l == 3 ? OW3 : l == 4 ? OW4 : OW5; }
__host__ __device__ constexpr int boff(int l) { return l == 1 ? OB1 : l == 2 ? OB2 : l == 3 ? OB3 : l == 4 ? OB4 : OB5; }

// byte offset of element (r, k) of an operand with K columns in the core-matrix layout
__device__ __forceinline__ int cm(int r, int k, int K) { return (r >> 3) * (16 * K) + (k >> 3) * 128 + (r & 7) * 16 + (k & 7) * 2; }

__device__ __forceinline__ uint64_t sdesc(uint32_t saddr, int K) {
    uint64_t d = (uint64_t)((saddr >> 4) & 0x3FFF);
    d |= (uint64_t)((128 >> 4) & 0x3FFF) << 16;          // leading byte offset: K-neighbour core matrices
    d |= (uint64_t)(((16 * K) >> 4) & 0x3FFF) << 32;     // stride byte offset: 8-row groups
    d |= (uint64_t)1 << 46;                               // descriptor version
    return d;                                             // no swizzle
}

__device__ __forceinline__ uint32_t idesc(int N) {
    // FP32 accumulate, BF16 A and B, both K-major, N >> 3, M = 128 >> 4
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(TILE >> 4) << 24);
}

__device__ __forceinline__ uint32_t saddr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// D(tmem) (+)= A(smem, 128 x K) B(smem, N x K)^T, issued by the calling thread.
__device__ __forceinline__ void mma(uint32_t tmem, const unsigned char* A, const unsigned char* B, int K, int N, bool acc) {
    const uint32_t a0 = saddr(A), b0 = saddr(B), id = idesc(N);
    for (int s = 0; s < K / 16; ++s) {
        const uint64_t ad = sdesc(a0 + s * 256, K), bd = sdesc(b0 + s * 256, K);
        const uint32_t en = (acc || s > 0) ? 1u : 0u;
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                     "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
                     :: "r"(tmem), "l"(ad), "l"(bd), "r"(id), "r"(en) : "memory");
    }
}

__device__ __forceinline__ void commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" :: "r"(saddr(bar)) : "memory");
}

// Wait for phase `parity` of the mbarrier, at most WAIT_LIMIT polls; false on timeout.
__device__ __forceinline__ bool wait_bar(uint64_t* bar, uint32_t parity) {
    uint32_t done = 0;
    for (int it = 0; it < WAIT_LIMIT && !done; ++it)
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(done) : "r"(saddr(bar)), "r"(parity) : "memory");
    return done != 0;
}

__device__ __forceinline__ void sync_for_mma() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// 32 consecutive FP32 columns of this thread's TMEM lane.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float* v) {
    uint32_t r[32];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
                 "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                   "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
                   "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
                   "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
                 : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(r[j]);
}

__device__ __forceinline__ void tmem_alloc(uint32_t* slot, int cols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" :: "r"(saddr(slot)), "r"(cols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_free(uint32_t tmem, int cols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem), "r"(cols) : "memory");
}

__device__ __forceinline__ float gelu(float z) { return 0.5f * z * (1.0f + erff(z * 0.70710678118654752f)); }
// GELU and its derivative from one error function.
__device__ __forceinline__ float gelu_both(float z, float& grad) {
    const float phi = 1.0f + erff(z * 0.70710678118654752f);
    grad = 0.5f * phi + z * expf(-0.5f * z * z) * 0.39894228040143268f;
    return 0.5f * z * phi;
}

__device__ __forceinline__ void put_bf16(unsigned char* base, int off, float v) {
    *reinterpret_cast<__nv_bfloat16*>(base + off) = __float2bfloat16_rn(v);
}
__device__ __forceinline__ uint32_t pack2(float a, float b) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t*>(&h);
}
// 8 consecutive columns of one row (one 16-byte line of a core matrix)
__device__ __forceinline__ void put8(unsigned char* base, int off, const float* v) {
    *reinterpret_cast<uint4*>(base + off) = make_uint4(pack2(v[0], v[1]), pack2(v[2], v[3]), pack2(v[4], v[5]), pack2(v[6], v[7]));
}

// ------------------------------------------------------------------------------ packed weights
// The BF16 core-matrix images of the weights that the forward and backward kernels use as
// GEMM operands.  They belong to the handle's state like the FP32 master copy: written whenever
// that is (initialisation, set_params, the Adam update), and copied into each block's shared
// memory with bulk asynchronous copies.
constexpr int PK_FWD = 106496;                 // W1t, W2t..W4t, W5t (the forward's first bytes)
constexpr int PK_BWD = 102400;                 // W2n..W4n, W5n (the backward's first bytes)
constexpr int PK_BYTES = PK_FWD + PK_BWD;

__device__ __forceinline__ void bulk_copy(unsigned char* dst, const unsigned char* src, uint32_t bytes, uint64_t* bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 :: "r"(saddr(dst)), "l"(src), "r"(bytes), "r"(saddr(bar)) : "memory");
}

// bytes (a multiple of 4096, 16-byte aligned at both ends) into shared memory by the block's
// threads, 4 KB per copy; false when the copies did not complete within the wait limit
__device__ bool load_packed(unsigned char* dst, const unsigned char* src, int bytes, uint64_t* cbar) {
    const int tid = threadIdx.x;
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(saddr(cbar)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" :: "r"(saddr(cbar)), "r"((uint32_t)bytes) : "memory");
    }
    __syncthreads();
    for (int c = tid; c < bytes / 4096; c += blockDim.x) bulk_copy(dst + c * 4096, src + c * 4096, 4096, cbar);
    return __syncthreads_and(wait_bar(cbar, 0) ? 1 : 0) != 0;
}

// BF16 images of parameter e (value v): forward operands B = W_l^T (rows: outputs, K = inputs);
// backward B = W_l (rows: inputs, K = outputs) for l >= 2; byte offsets as in the kernels'
// shared-memory layouts.  Biases have none.
__device__ __forceinline__ void pack_param(unsigned char* pk, int e, float v) {
    unsigned char* fw = pk;
    unsigned char* bw = pk + PK_FWD;
    if (e < OB1) {
        put_bf16(fw, cm(e % NH, e / NH, NIN), v);
    } else {
        for (int l = 2; l <= 4; ++l) {
            const int q = e - woff(l);
            if (q >= 0 && q < NH * NH) {
                const int a = q / NH, b = q % NH;
                put_bf16(fw + 4096 + (l - 2) * 32768, cm(b, a, NH), v);
                put_bf16(bw + (l - 2) * 32768, cm(a, b, NH), v);
            }
        }
        const int q = e - OW5;
        if (q >= 0 && q < NH * NOUT) {
            const int a = q / NOUT, b = q % NOUT;
            put_bf16(fw + 4096 + 3 * 32768, cm(b, a, NH), v);
            put_bf16(bw + 3 * 32768, cm(a, b, NOUT), v);
        }
    }
}

__global__ void k_mlp_pack(const float* __restrict__ prm, unsigned char* __restrict__ pk) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e < NPARAM) pack_param(pk, e, prm[e]);
}

// ------------------------------------------------------------------------------ forward
// Shared bytes: W1t 4096 | W2t..W4t 3 x 32768 | W5t 4096 | A 32768 | bias 2112
constexpr int F_W1 = 0, F_W2 = 4096, F_W3 = F_W2 + 32768, F_W4 = F_W3 + 32768, F_W5 = F_W4 + 32768;
constexpr int F_A = F_W5 + 4096, F_BIAS = F_A + 32768, F_BYTES = F_BIAS + 4 * 4 * NH + 4 * NOUT;

// Pre-activations kept for the backward pass, point fastest: Zs[tile][layer][column][point], the last
// tile with its own number of points.
__device__ __forceinline__ float* z_row(float* Zs, int row) { return Zs + (size_t)blockIdx.x * (4 * NH * TILE) + row; }
__device__ __forceinline__ int z_stride(int P) { return min(TILE, P - (int)blockIdx.x * TILE); }

__global__ void __launch_bounds__(THREADS) k_mlp_fwd(const float* __restrict__ prm, const unsigned char* __restrict__ pk,
                                                     const float* __restrict__ X, int P, float* __restrict__ pred,
                                                     float* __restrict__ Zs, int* err) {
    extern __shared__ __align__(1024) unsigned char sm[];
    __shared__ __align__(8) uint64_t bar, cbar;
    __shared__ uint32_t tslot;
    const int tid = threadIdx.x, wid = tid >> 5;
    const int row = (wid & 3) * 32 + (tid & 31), cg = (wid >> 2) * 32;   // this thread's point and columns
    const int p = blockIdx.x * TILE + row;
    const bool valid = p < P;
    float* z = z_row(Zs, row);
    const int zs = z_stride(P);
    if (tid < 32) tmem_alloc(&tslot, NH);
    // input tile (K = 16): four features per thread
    {
        const int r = tid >> 2, k = (tid & 3) * 4, q = blockIdx.x * TILE + r;
        float x[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        if (q < P)
            for (int j = 0; j < 4; ++j) x[j] = X[(size_t)q * NIN + k + j];
        *reinterpret_cast<uint2*>(sm + F_A + cm(r, k, NIN)) = make_uint2(pack2(x[0], x[1]), pack2(x[2], x[3]));
    }
    float* bias = reinterpret_cast<float*>(sm + F_BIAS);
    for (int e = tid; e < 4 * NH + NOUT; e += THREADS) bias[e] = e < 4 * NH ? prm[boff(e / NH + 1) + e % NH] : prm[OB5 + e - 4 * NH];
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(saddr(&bar)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // weights as B operands (N = outputs x K = inputs): the packed BF16 image, biases
    static_assert(F_A == PK_FWD, "packed forward image = the weight region of shared memory");
    bool ok = load_packed(sm, pk, PK_FWD, &cbar);
    sync_for_mma();
    const uint32_t tmem = tslot;
    const uint32_t lane_addr = tmem + ((uint32_t)((wid & 3) * 32) << 16);
    for (int l = 1; l <= 5 && ok; ++l) {
        const int K = l == 1 ? NIN : NH, N = l == 5 ? NOUT : NH;
        const unsigned char* W = sm + (l == 1 ? F_W1 : l == 2 ? F_W2 : l == 3 ? F_W3 : l == 4 ? F_W4 : F_W5);
        if (tid == 0) {
            mma(tmem, sm + F_A, W, K, N, false);
            commit(&bar);
        }
        ok = __syncthreads_and(wait_bar(&bar, (uint32_t)((l - 1) & 1)) ? 1 : 0) != 0;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (!ok) break;                      // uniform across the block
        const float* bl = bias + (l - 1) * NH;
        if (cg < N) {                        // layer 5: the first column quarter only
            float v[32];
            tmem_ld32(lane_addr + cg, v);    // 32 columns (all inside the 128 allocated)
            if (l < 5) {
#pragma unroll
                for (int c = 0; c < 32; c += 8) {
                    float h[8];
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const float x = v[c + j] + bl[cg + c + j];
                        if (Zs && valid) z[((l - 1) * NH + cg + c + j) * zs] = x;
                        h[j] = gelu(x);
                    }
                    put8(sm + F_A, cm(row, cg + c, NH), h);
                }
            } else if (valid) {
                for (int c = 0; c < NUSED; ++c) pred[(size_t)p * NUSED + c] = v[c] + bl[c];
            }
        }
        sync_for_mma();
    }
    if (!ok && tid == 0) atomicExch(err, 1);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (tid < 32) tmem_free(tmem, NH);
}

// ------------------------------------------------------------------------------ backward
// Shared bytes: W2n..W4n 3 x 32768 (natural: N = inputs x K = outputs) | W5n 4096 (N = 128 x K = 16)
//               | OpA 32768 | OpB 32768 | OpC 32768
constexpr int B_W2 = 0, B_W3 = 32768, B_W4 = 65536, B_W5 = 98304, B_A = B_W5 + 4096, B_B = B_A + 32768, B_C = B_B + 32768;
constexpr int B_BYTES = B_C + 32768;

__global__ void __launch_bounds__(THREADS) k_mlp_bwd(const unsigned char* __restrict__ pk, const float* __restrict__ X,
                                                     const float* __restrict__ Y, int P, const float* __restrict__ pred,
                                                     float* __restrict__ Zs, float* __restrict__ gpart,
                                                     float* __restrict__ lpart, int* err) {
    extern __shared__ __align__(1024) unsigned char sm[];
    __shared__ __align__(8) uint64_t bar, cbar;
    __shared__ uint32_t tslot;
    __shared__ float red[TILE / 32];
    const int tid = threadIdx.x, wid = tid >> 5, lane = tid & 31;
    const int row = (wid & 3) * 32 + lane, cg = (wid >> 2) * 32;         // this thread's point and columns
    const int p = blockIdx.x * TILE + row;
    const bool valid = p < P;
    float* g = gpart + (size_t)blockIdx.x * NPARAM;
    const float* z = z_row(Zs, row);
    const int zs = z_stride(P);
    if (tid < 32) tmem_alloc(&tslot, 2 * NH);
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(saddr(&bar)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // weights as B operands of the dH GEMMs (N = inputs x K = outputs): the packed BF16 image
    static_assert(B_A == PK_BWD, "packed backward image = the weight region of shared memory");
    bool ok = load_packed(sm, pk + PK_FWD, PK_BWD, &cbar);
    // dZ_5 = dL/dpred on the used outputs (columns 0..2 of the first column quarter); loss partial
    float d[32];
    float sq = 0.0f;
#pragma unroll
    for (int j = 0; j < 32; ++j) d[j] = 0.0f;
    if (valid && cg == 0)
#pragma unroll
        for (int j = 0; j < NUSED; ++j) {
            const float df = pred[(size_t)p * NUSED + j] - Y[(size_t)p * NUSED + j];
            sq += df * df;
            d[j] = 2.0f * df / (float)(NUSED * P);
        }
    for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
    if (cg == 0 && lane == 0) red[wid & 3] = sq;
    sync_for_mma();
    if (tid == 0) lpart[blockIdx.x] = red[0] + red[1] + red[2] + red[3];
    const uint32_t tmem = tslot;
    const uint32_t lane_addr = tmem + ((uint32_t)((wid & 3) * 32) << 16);
    uint32_t phase = 0;
    for (int l = 5; l >= 1 && ok; --l) {
        const int N = l == 5 ? NOUT : NH;          // outputs of layer l
        // operands: dW GEMM  A = H_{l-1}^T (rows: inputs), B = dZ^T (rows: outputs), K = points;
        //           layer 1: A = dZ_1^T (rows: outputs), B = X^T (rows: inputs).
        //           dH GEMM  A = dZ (rows: points, K = outputs), B = W_l natural (rows: inputs).
        float dg[32];                              // GELU'(Z_{l-1}) of this thread's columns
        if (l >= 2) {
#pragma unroll
            for (int c = 0; c < 32; ++c) {
                const float h = gelu_both(valid ? z[((l - 2) * NH + cg + c) * zs] : 0.0f, dg[c]);
                put_bf16(sm + B_A, cm(cg + c, row, TILE), valid ? h : 0.0f);
                if (!valid) dg[c] = 0.0f;
            }
            if (cg < N) {
                const int n = N < 32 ? N : 32;
#pragma unroll
                for (int j = 0; j < 32; ++j)
                    if (j < n) put_bf16(sm + B_B, cm(cg + j, row, TILE), d[j]);
#pragma unroll
                for (int j = 0; j < 32; j += 8)
                    if (j < n) put8(sm + B_C, cm(row, cg + j, N), d + j);
            }
        } else {
#pragma unroll
            for (int j = 0; j < 32; ++j) put_bf16(sm + B_A, cm(cg + j, row, TILE), d[j]);
            // X^T: four features per thread
            for (int k = (wid >> 2) * 4; k < (wid >> 2) * 4 + 4; ++k)
                put_bf16(sm + B_B, cm(k, row, TILE), valid ? X[(size_t)p * NIN + k] : 0.0f);
        }
        sync_for_mma();
        if (tid == 0) {
            mma(tmem, sm + B_A, sm + B_B, TILE, l >= 2 ? N : NIN, false);
            if (l >= 2) mma(tmem + NH, sm + B_C, sm + (l == 2 ? B_W2 : l == 3 ? B_W3 : l == 4 ? B_W4 : B_W5), N, NH, false);
            commit(&bar);
        }
        ok = __syncthreads_and(wait_bar(&bar, phase) ? 1 : 0) != 0;
        phase ^= 1;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (!ok) break;                      // uniform across the block
        // weight gradient: row `row`, columns from cg, of the dW accumulator
        const int NW = l >= 2 ? N : NIN;
        float v[32];
        if (cg < NW) {
            tmem_ld32(lane_addr + cg, v);        // 32 columns inside the dW accumulator's 128
            if (l == 1) {
#pragma unroll
                for (int j = 0; j < NIN; ++j) g[OW1 + j * NH + row] = v[j];            // dW_1[in = j][out = row]
            } else {
                // dW_l[in = row][out = cg + j], 16 bytes at a time (woff(l) and N are multiples of 4)
                float4* o = reinterpret_cast<float4*>(g + woff(l) + row * N + cg);
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    if (4 * j < NW) o[j] = make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
            }
        }
        // bias gradient: column sums of dZ_l over the tile's points, four threads per column
        {
            const unsigned char* src = sm + (l >= 2 ? B_B : B_A);
            const int col = tid >> 2, part = tid & 3;
            float s = 0.0f;
            if (col < N)
                for (int q = part * 32; q < part * 32 + 32; q += 8) {
                    const uint4 w = *reinterpret_cast<const uint4*>(src + cm(col, q, TILE));
                    const uint32_t x[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const float2 f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&x[j]));
                        s += f.x;
                        s += f.y;
                    }
                }
            s += __shfl_xor_sync(0xffffffffu, s, 1);
            s += __shfl_xor_sync(0xffffffffu, s, 2);
            if (part == 0 && col < N) g[boff(l) + col] = s;
        }
        if (l >= 2) {
            // dH_{l-1} (row = point), then dZ_{l-1} = dH * GELU'(Z_{l-1})
            tmem_ld32(lane_addr + NH + cg, v);
#pragma unroll
            for (int j = 0; j < 32; ++j) d[j] = v[j] * dg[j];
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    }
    if (!ok && tid == 0) atomicExch(err, 1);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (tid < 32) tmem_free(tmem, 2 * NH);
}

// ------------------------------------------------------------------------------ Adam
__global__ void k_mlp_adam(float* prm, float* m, float* v, const float* gpart, int nblk, float lr, float b1t, float b2t,
                           float* gout, unsigned char* pk) {
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= NPARAM) return;
    float gsum = 0.0f;
    // (in block order; the loads of a batch in flight together)
    constexpr int B = 16;
    for (int b = 0; b < nblk; b += B) {
        float x[B];
#pragma unroll
        for (int j = 0; j < B; ++j) x[j] = b + j < nblk ? gpart[(size_t)(b + j) * NPARAM + q] : 0.0f;
#pragma unroll
        for (int j = 0; j < B; ++j) gsum += x[j];
    }
    if (gout) gout[q] = gsum;
    if (lr == 0.0f) return;
    const float mq = 0.9f * m[q] + 0.1f * gsum;
    const float vq = 0.999f * v[q] + 0.001f * gsum * gsum;
    m[q] = mq;
    v[q] = vq;
    const float w = prm[q] - lr * (mq / (1.0f - b1t)) / (sqrtf(vq / (1.0f - b2t)) + 1e-8f);
    prm[q] = w;
    pack_param(pk, q, w);
}

// Glorot-uniform weights from a counter-based hash (splitmix64 of seed and index), zero biases;
// output columns beyond the 3 used are zero.
__global__ void k_mlp_init(float* prm, float* m, float* v, unsigned long long seed) {
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= NPARAM) return;
    m[q] = 0.0f;
    v[q] = 0.0f;
    int l = 5;
    for (int j = 1; j <= 5; ++j)
        if (q < boff(j) + (j == 5 ? NOUT : NH)) { l = j; break; }
    if (q >= boff(l)) { prm[q] = 0.0f; return; }
    const int fin = l == 1 ? NIN : NH, fout = l == 5 ? NOUT : NH;
    if (l == 5 && (q - OW5) % NOUT >= NUSED) { prm[q] = 0.0f; return; }
    unsigned long long z = seed + 0x9E3779B97F4A7C15ull * (unsigned long long)(q + 1);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    z ^= z >> 31;
    const float u = (float)((z >> 40) * (1.0 / 16777216.0)) * 2.0f - 1.0f;
    prm[q] = u * sqrtf(6.0f / (float)(fin + fout));
}

}  // namespace

// ------------------------------------------------------------------------------ C ABI
struct fdlb_mlp {
    float* prm = nullptr;
    float* m = nullptr;
    float* v = nullptr;
    float* gpart = nullptr;
    float* lpart = nullptr;
    float* Zs = nullptr;
    float* pred = nullptr;
    int* err = nullptr;
    unsigned char* pk = nullptr;      // packed BF16 weight images (k_mlp_pack)
    int max_points = 0;
    long long t = 0;
    cudaStream_t stream = nullptr;
    std::string msg;
};

static thread_local std::string g_mlp_err;

static size_t al256(size_t b) { return (b + 255) & ~size_t(255); }

static size_t mlp_layout(int max_points, size_t* off) {
    const size_t nblk = (size_t)(max_points + TILE - 1) / TILE;
    size_t o = 0;
    off[0] = o; o += al256(sizeof(float) * NPARAM);               // parameters
    off[1] = o; o += al256(sizeof(float) * NPARAM);               // Adam m
    off[2] = o; o += al256(sizeof(float) * NPARAM);               // Adam v
    off[3] = o; o += al256(sizeof(float) * NPARAM * nblk);        // per-block gradients
    off[4] = o; o += al256(sizeof(float) * nblk);                 // per-block loss
    off[5] = o; o += al256(sizeof(float) * 4 * NH * (size_t)max_points);   // pre-activations
    off[6] = o; o += al256(sizeof(float) * NUSED * (size_t)max_points);    // predictions
    off[7] = o; o += al256(sizeof(int));
    off[8] = o; o += al256(PK_BYTES);                            // packed BF16 weight images
    return o;
}

static int mlp_fail(fdlb_mlp* h, int code, const std::string& s) {
    if (h) h->msg = s;
    g_mlp_err = s;
    return code;
}

static int mlp_cuda(fdlb_mlp* h, cudaError_t e, const char* what) {
    if (e == cudaSuccess) return FDLB_OK;
    return mlp_fail(h, FDLB_ECUDA, std::string(what) + ": " + cudaGetErrorString(e));
}

extern "C" int32_t fdlb_mlp_param_count(void) { return NPARAM; }

extern "C" size_t fdlb_mlp_workspace_bytes(int32_t max_points) {
    if (max_points < 1) return 0;
    size_t off[9];
    return mlp_layout(max_points, off);
}

extern "C" const char* fdlb_mlp_last_error(const fdlb_mlp* h) { return h ? h->msg.c_str() : g_mlp_err.c_str(); }

extern "C" int fdlb_mlp_create(fdlb_mlp** out, void* dev_ws, size_t bytes, int32_t max_points, uint64_t seed, void* stream) {
    if (!out || !dev_ws || max_points < 1) return mlp_fail(nullptr, FDLB_EINVAL, "fdlb_mlp_create: bad arguments");
    size_t off[9];
    const size_t need = mlp_layout(max_points, off);
    if (bytes < need || (reinterpret_cast<uintptr_t>(dev_ws) & 255))
        return mlp_fail(nullptr, FDLB_ENOMEM, "fdlb_mlp_create: workspace smaller than fdlb_mlp_workspace_bytes or misaligned");
    fdlb_mlp* h = new fdlb_mlp();
    char* b = static_cast<char*>(dev_ws);
    h->prm = reinterpret_cast<float*>(b + off[0]);
    h->m = reinterpret_cast<float*>(b + off[1]);
    h->v = reinterpret_cast<float*>(b + off[2]);
    h->gpart = reinterpret_cast<float*>(b + off[3]);
    h->lpart = reinterpret_cast<float*>(b + off[4]);
    h->Zs = reinterpret_cast<float*>(b + off[5]);
    h->pred = reinterpret_cast<float*>(b + off[6]);
    h->err = reinterpret_cast<int*>(b + off[7]);
    h->pk = reinterpret_cast<unsigned char*>(b + off[8]);
    h->max_points = max_points;
    h->stream = reinterpret_cast<cudaStream_t>(stream);
    int rc = mlp_cuda(h, cudaFuncSetAttribute(k_mlp_fwd, cudaFuncAttributeMaxDynamicSharedMemorySize, F_BYTES), "attributes");
    if (!rc) rc = mlp_cuda(h, cudaFuncSetAttribute(k_mlp_bwd, cudaFuncAttributeMaxDynamicSharedMemorySize, B_BYTES), "attributes");
    if (!rc) {
        k_mlp_init<<<(NPARAM + 255) / 256, 256, 0, h->stream>>>(h->prm, h->m, h->v, (unsigned long long)seed);
        k_mlp_pack<<<(NPARAM + 255) / 256, 256, 0, h->stream>>>(h->prm, h->pk);
        rc = mlp_cuda(h, cudaGetLastError(), "init kernel");
    }
    if (!rc) rc = mlp_cuda(h, cudaMemsetAsync(h->err, 0, sizeof(int), h->stream), "clear");
    if (!rc) rc = mlp_cuda(h, cudaStreamSynchronize(h->stream), "synchronize");
    if (rc) { g_mlp_err = h->msg; delete h; return rc; }
    *out = h;
    return FDLB_OK;
}

extern "C" void fdlb_mlp_destroy(fdlb_mlp* h) { delete h; }

extern "C" int fdlb_mlp_get_params(fdlb_mlp* h, float* host) {
    if (!h || !host) return mlp_fail(h, FDLB_EINVAL, "fdlb_mlp_get_params: bad arguments");
    int rc = mlp_cuda(h, cudaMemcpyAsync(host, h->prm, sizeof(float) * NPARAM, cudaMemcpyDeviceToHost, h->stream), "copy");
    if (!rc) rc = mlp_cuda(h, cudaStreamSynchronize(h->stream), "synchronize");
    return rc;
}

extern "C" int fdlb_mlp_set_params(fdlb_mlp* h, const float* host) {
    if (!h || !host) return mlp_fail(h, FDLB_EINVAL, "fdlb_mlp_set_params: bad arguments");
    int rc = mlp_cuda(h, cudaMemcpyAsync(h->prm, host, sizeof(float) * NPARAM, cudaMemcpyHostToDevice, h->stream), "copy");
    if (!rc) rc = mlp_cuda(h, cudaMemsetAsync(h->m, 0, sizeof(float) * NPARAM, h->stream), "clear");
    if (!rc) rc = mlp_cuda(h, cudaMemsetAsync(h->v, 0, sizeof(float) * NPARAM, h->stream), "clear");
    if (!rc) {
        k_mlp_pack<<<(NPARAM + 255) / 256, 256, 0, h->stream>>>(h->prm, h->pk);
        rc = mlp_cuda(h, cudaGetLastError(), "pack kernel");
    }
    if (!rc) rc = mlp_cuda(h, cudaStreamSynchronize(h->stream), "synchronize");
    h->t = 0;
    return rc;
}

static int check_err(fdlb_mlp* h) {
    int e = 0;
    int rc = mlp_cuda(h, cudaMemcpyAsync(&e, h->err, sizeof(int), cudaMemcpyDeviceToHost, h->stream), "copy");
    if (!rc) rc = mlp_cuda(h, cudaStreamSynchronize(h->stream), "synchronize");
    if (!rc && e) rc = mlp_fail(h, FDLB_ETIMEOUT, "tensor-core completion wait timed out");
    return rc;
}

extern "C" int fdlb_mlp_predict(fdlb_mlp* h, const float* dev_x, int32_t points, float* dev_y) {
    if (!h || !dev_x || !dev_y || points < 1) return mlp_fail(h, FDLB_EINVAL, "fdlb_mlp_predict: bad arguments");
    const int nblk = (points + TILE - 1) / TILE;
    k_mlp_fwd<<<nblk, THREADS, F_BYTES, h->stream>>>(h->prm, h->pk, dev_x, points, dev_y, nullptr, h->err);
    int rc = mlp_cuda(h, cudaGetLastError(), "forward kernel");
    if (!rc) rc = check_err(h);
    return rc;
}

extern "C" int fdlb_mlp_train_step(fdlb_mlp* h, const float* dev_x, const float* dev_y, int32_t points, float lr,
                                   float* dev_grad, double* host_loss) {
    if (!h || !dev_x || !dev_y || points < 1 || points > h->max_points || !(lr >= 0.0f))
        return mlp_fail(h, FDLB_EINVAL, "fdlb_mlp_train_step: bad arguments (points must be <= max_points)");
    const int nblk = (points + TILE - 1) / TILE;
    k_mlp_fwd<<<nblk, THREADS, F_BYTES, h->stream>>>(h->prm, h->pk, dev_x, points, h->pred, h->Zs, h->err);
    k_mlp_bwd<<<nblk, THREADS, B_BYTES, h->stream>>>(h->pk, dev_x, dev_y, points, h->pred, h->Zs, h->gpart, h->lpart, h->err);
    if (lr > 0.0f) h->t += 1;
    const float b1t = lr > 0.0f ? (float)std::pow(0.9, (double)h->t) : 0.0f;
    const float b2t = lr > 0.0f ? (float)std::pow(0.999, (double)h->t) : 0.0f;
    k_mlp_adam<<<(NPARAM + 255) / 256, 256, 0, h->stream>>>(h->prm, h->m, h->v, h->gpart, nblk, lr, b1t, b2t, dev_grad, h->pk);
    int rc = mlp_cuda(h, cudaGetLastError(), "training kernels");
    if (!rc && host_loss) {
        std::vector<float> lp(nblk);
        rc = mlp_cuda(h, cudaMemcpyAsync(lp.data(), h->lpart, sizeof(float) * nblk, cudaMemcpyDeviceToHost, h->stream), "copy");
        if (!rc) rc = mlp_cuda(h, cudaStreamSynchronize(h->stream), "synchronize");
        double s = 0.0;
        for (float x : lp) s += x;
        if (!rc) *host_loss = s / (NUSED * (double)points);
    }
    if (!rc) rc = check_err(h);
    return rc;
}
