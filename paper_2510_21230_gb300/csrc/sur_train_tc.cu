// sur_train_tc.cu -- training of the surrogate MLP (32 -> 64 -> 64 -> 3, SiLU)
// on the fifth-generation tensor cores: forward and backward GEMMs as
// tcgen05.mma with bfloat16 operands in shared memory and FP32 accumulators
// in tensor memory (TMEM); FP32 master weights, FP32 gradients.
//
// One CTA of 512 threads per 128-sample tile (persistent over tiles); the four
// threads t, t + 128, .. share sample t and TMEM lane t, a quarter of the columns
// of every layer each.  A step of 8,192 samples has 64 tiles, fewer than SMs, so
// the tile's chain of latencies bounds it: 46 us a step with one thread per
// sample, 39 with four, 22 with rows, weights and gradients moved 16 bytes at a
// time and the vectors fetched beside the first layers (their rows are random
// lines of the data set).  What does not depend on the step before runs
// beside its Adam kernel: 50 steps 1,441 -> 1,210 us.  Per tile:
//   forward   Z1 = X W1, H1 = silu(Z1 + b1); Z2 = H1 W2, H2 = silu(Z2 + b2);
//             w = H2 W3 + b3 (the inference kernel's arithmetic: bfloat16
//             inputs, weights and hidden activations), F = sum_m w_m v_m
//   loss      L = norm sum |F - F_ref|^2, dL/dw_m = 2 norm (F - F_ref) . v_m
//   backward  dH2 = dY W3^T (CUDA cores, K = 3), dZ2 = dH2 silu'(Z2);
//             dH1 = dZ2 W2^T (tensor cores), dZ1 = dH1 silu'(Z1);
//             dW3 = H2^T dY, dW2 = H1^T dZ2, dW1 = X^T dZ1 (tensor cores,
//             contracting over the 128 samples), and the bias gradients
//             from the same GEMMs: the transposed left operands carry a row
//             of ones, whose output row is the column sum of the right one.
// silu'(z) (FP32) is kept in TMEM between the forward and the backward pass
// (tcgen05.st / tcgen05.ld).  The transposed operands (K = samples) are
// written element by element by the sample's thread.  Left operands of the
// weight gradients have M = 128 rows: rows beyond the weight rows and the
// ones row are zero.
//
// TMEM columns (256 per CTA, one CTA per SM by its shared memory):
//   [0, 64)    Z1 -> silu'(Z2) -> dH1
//   [64, 128)  Z2 -> dW2 (row 64: db2)
//   [128, 144) w
//   [144, 160) dW3 (row 64: db3)
//   [160, 224) silu'(Z1) -> dW1 (row 32: db1)
// Every wait on the MMA barrier is bounded; a wait that gives up stops the
// CTA (after freeing its TMEM) and sets ST_TIMEOUT.
#include <cuda_bf16.h>
#include <stdint.h>

#include "surrogate.cuh"
#include "tc_common.cuh"

namespace atm3 {

namespace {
using namespace tc;

constexpr int TR_M = 128;             // samples per tile = TMEM lanes
constexpr int TR_T = 512;             // threads: four per sample
constexpr int TR_VS = SUR_NV + 4;     // row stride of the staged vectors (16-byte reads without conflicts)
constexpr uint32_t TR_COLS = 256;     // TMEM columns per CTA
constexpr uint32_t SBO_K32 = 4 * 128, SBO_K64 = 8 * 128, SBO_K128 = 16 * 128;

struct TrSmem {
    alignas(128) unsigned char w1t[64 * 32 * 2];    // B, layer 1: N 64 x K 32 (W1^T)
    alignas(128) unsigned char w2t[64 * 64 * 2];    // B, layer 2: N 64 x K 64 (W2^T)
    alignas(128) unsigned char w3t[16 * 64 * 2];    // B, layer 3: N 16 x K 64 (W3^T)
    alignas(128) unsigned char w2[64 * 64 * 2];     // B of dH1 = dZ2 W2^T: N 64 (k) x K 64 (j)
    alignas(128) unsigned char x[TR_M * 32 * 2];    // A, layer 1: M 128 x K 32
    alignas(128) unsigned char h[TR_M * 64 * 2];    // A: H1 (layer 2), H2 (layer 3), dZ2 (dH1)
    alignas(128) unsigned char xt[128 * TR_M * 2];  // A of dW1: rows q < 32 X^T, row 32 ones
    alignas(128) unsigned char h1t[128 * TR_M * 2]; // A of dW2: rows k < 64 H1^T, row 64 ones
    alignas(128) unsigned char h2t[128 * TR_M * 2]; // A of dW3: rows k < 64 H2^T, row 64 ones
    alignas(128) unsigned char dyt[16 * TR_M * 2];  // B of dW3: N 16 (dL/dw_m) x K samples
    alignas(128) unsigned char dz2t[64 * TR_M * 2]; // B of dW2: N 64 x K samples
    alignas(128) unsigned char dz1t[64 * TR_M * 2]; // B of dW1: N 64 x K samples
    alignas(16) float v[TR_M * TR_VS];              // the samples' vectors
    float w3[SUR_NH * SUR_NO];                      // FP32 master W3
    float b1[64], b2[64], b3[SUR_NO];
    double lsum[TR_M / 32];
    alignas(8) unsigned long long mbar;
    uint32_t tmem_base;
};

static_assert(sizeof(TrSmem) <= 227 * 1024, "one CTA's shared memory");

// element (row, k) of a K-major operand with kchunks 8-element chunks per row
__device__ __forceinline__ void put_bf(unsigned char* base, int row, int k, int kchunks, float v)
{
    *reinterpret_cast<__nv_bfloat16*>(base + cm_off(row, k >> 3, kchunks) + 2 * (k & 7)) =
        __float2bfloat16_rn(v);
}

// 16 floats to a 16-byte aligned row
__device__ __forceinline__ void store16(float* to, const float (&o)[16])
{
#pragma unroll
    for (int i = 0; i < 4; i++)
        reinterpret_cast<float4*>(to)[i] = make_float4(o[4 * i], o[4 * i + 1], o[4 * i + 2], o[4 * i + 3]);
}
static_assert(SUR_OFF_W1 % 4 == 0 && SUR_OFF_W2 % 4 == 0 && SUR_OFF_W3 % 4 == 0 && SUR_NP % 4 == 0, "rows of store16");

// sigmoid and silu'(z) = s (1 + z (1 - s)); silu itself as the inference kernel forms it
__device__ __forceinline__ float sigm(float z) { return __fdividef(1.0f, 1.0f + __expf(-z)); }

}  // namespace

namespace {

__global__ void __launch_bounds__(TR_T) k_sur_grad_tc(const SurGradArgs A)
{
    extern __shared__ __align__(1024) unsigned char smraw[];
    TrSmem& S = *reinterpret_cast<TrSmem*>(smraw);
    const int tid = threadIdx.x, warp = tid >> 5;
    const int t = tid & (TR_M - 1), part = tid / TR_M;  // sample, quarter of the columns
    const SurPacked* model = A.packed;

    // ---- what does not depend on the step before, beside its Adam kernel: constant
    // rows of the padded operands, and the first tile's rows on their way to L2
    {
        // zero rows of the padded left operands: beyond the weight rows (a group of
        // 8 rows takes 2048 bytes)
        const uint4 z = make_uint4(0u, 0u, 0u, 0u);
        for (int e = tid; e < 12 * 128; e += TR_T) reinterpret_cast<uint4*>(S.xt + 4 * 2048)[e] = z;
        for (int e = tid; e < 8 * 128; e += TR_T) {
            reinterpret_cast<uint4*>(S.h1t + 8 * 2048)[e] = z;
            reinterpret_cast<uint4*>(S.h2t + 8 * 2048)[e] = z;
        }
    }
    {
        const long long row = blockIdx.x * (long long)TR_M + t;
        if (row < A.batch && (A.S > 0 || !A.idx)) {
            const long long smp = A.S > 0 ? sur_sample(A.seed, A.step, row, A.S) : row;
            const float* at = part == 0 ? A.D + smp * SUR_ND
                                        : (part == 3 ? A.T + 3 * smp : A.V + smp * SUR_NV + (part == 2 ? SUR_NV - 1 : 0));
            asm volatile("prefetch.global.L2 [%0];" ::"l"(at));
        }
    }
    after_previous();
    // ---- once per CTA: weights, barrier, TMEM
    for (int e = tid; e < 64 * 4; e += TR_T) {
        const int r = e >> 2, j = e & 3;
        put_chunk(S.w1t, r, j, 4, *reinterpret_cast<const uint4*>(model->w1t + r * SUR_XS + 8 * j));
    }
    for (int e = tid; e < 64 * 8; e += TR_T) {
        const int r = e >> 3, j = e & 7;
        put_chunk(S.w2t, r, j, 8, *reinterpret_cast<const uint4*>(model->w2t + r * SUR_HS + 8 * j));
    }
    for (int e = tid; e < 16 * 8; e += TR_T) {
        const int r = e >> 3, j = e & 7;
        const uint4 z = make_uint4(0u, 0u, 0u, 0u);
        put_chunk(S.w3t, r, j, 8, r < SUR_NO ? *reinterpret_cast<const uint4*>(model->w3t + r * SUR_HS + 8 * j) : z);
    }
    // W2 itself (row k holds W2[k][j], j contiguous) for dH1 = dZ2 W2^T
    for (int e = tid; e < 64 * 8; e += TR_T) {
        const float4* w = reinterpret_cast<const float4*>(A.P + SUR_OFF_W2 + 8 * e);
        const float4 a = w[0], b = w[1];
        put_chunk(S.w2, e >> 3, e & 7, 8, make_uint4(pack_bf2(a.x, a.y), pack_bf2(a.z, a.w),
                                                     pack_bf2(b.x, b.y), pack_bf2(b.z, b.w)));
    }
    for (int e = tid; e < SUR_NH * SUR_NO; e += TR_T) S.w3[e] = A.P[SUR_OFF_W3 + e];
    if (tid < 64) {
        S.b1[tid] = model->b1[tid];
        S.b2[tid] = model->b2[tid];
    }
    if (tid < SUR_NO) S.b3[tid] = model->b3[tid];
    __syncthreads();
    // the rows of ones: their output rows are the bias gradients
    if (part == 0) put_bf(S.xt, SUR_ND, t, 16, 1.0f);
    if (part == 1) put_bf(S.h1t, SUR_NH, t, 16, 1.0f);
    if (part == 2) put_bf(S.h2t, SUR_NH, t, 16, 1.0f);
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&S.mbar)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(&S.tmem_base)),
                     "r"(TR_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    fence_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = S.tmem_base;
    const uint32_t lane = tmem + ((uint32_t)((warp & 3) * 32) << 16);  // this warp's lane quarter
    const uint32_t id64 = idesc_bf16(TR_M, 64), id16 = idesc_bf16(TR_M, 16);

    uint32_t phase = 0u;
    bool ok = true;
    // every thread waits on the MMA barrier's phase; all agree on the outcome
    auto wait_mma = [&]() {
        bool done = false;
        for (long it = 0; it < TC_WAIT_TRIES && !done; it++) done = mbar_try_wait(&S.mbar, phase);
        phase ^= 1u;
        ok = __syncthreads_and(done) != 0;
        tc_fence_after();
    };
    // operands written by the threads become visible to the tensor cores
    auto publish = [&]() {
        fence_async_smem();
        tc_fence_before();
        __syncthreads();
    };
    // D (+)= A B over K / 16 instructions of K = 16
    auto mma = [&](uint32_t d, const unsigned char* a, const unsigned char* b, uint32_t sbo, int k,
                   uint32_t idesc) {
        for (int kk = 0; kk < k / 16; kk++)
            umma_bf16(d, sdesc(a + kk * 2 * TC_LBO, sbo), sdesc(b + kk * 2 * TC_LBO, sbo), idesc, kk > 0);
    };

    const long long ntiles = (A.batch + TR_M - 1) / TR_M;
    for (long long tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x) {
        const long long row = tile * TR_M + t;
        const bool active = row < A.batch;
        const long long smp = !active ? 0 : (A.S > 0 ? sur_sample(A.seed, A.step, row, A.S)
                                                     : (A.idx ? A.idx[row] : row));

        // ---- inputs: normalised descriptors (X and X^T), vectors, target
        {
            float xv[8];
            const int q0 = 8 * part;
            const float4* drow = reinterpret_cast<const float4*>(A.D + smp * SUR_ND + q0);
            const float4 d0 = drow[0], d1 = drow[1];
            const float dv[8] = {d0.x, d0.y, d0.z, d0.w, d1.x, d1.y, d1.z, d1.w};
#pragma unroll
            for (int q = 0; q < 8; q++)
                xv[q] = active ? (dv[q] - A.mean[q0 + q]) / A.scale[q0 + q] : 0.0f;
            put_chunk(S.x, t, part, 4, make_uint4(pack_bf2(xv[0], xv[1]), pack_bf2(xv[2], xv[3]),
                                                  pack_bf2(xv[4], xv[5]), pack_bf2(xv[6], xv[7])));
#pragma unroll
            for (int q = 0; q < 8; q++) put_bf(S.xt, q0 + q, t, 16, xv[q]);
        }
        float tg[3];
#pragma unroll
        for (int c = 0; c < 3; c++) tg[c] = active ? A.T[smp * 3 + c] : 0.0f;
        // the sample's 16 vectors to shared memory, 16 bytes at a time, beside the
        // first two layers (read row by row from global memory in the loss they took
        // 32 k of the tile's 66 k cycles)
        {
            const float* v = A.V + smp * SUR_NV + 12 * part;
#pragma unroll
            for (int q = 0; q < 3; q++)
                asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(smem_u32(S.v + t * TR_VS + 12 * part + 4 * q)),
                             "l"(v + 4 * q)
                             : "memory");
            asm volatile("cp.async.commit_group;" ::: "memory");
        }
        const float* vrow = S.v + t * TR_VS;
        publish();

        // ---- layer 1: TMEM [0, 64) = X W1
        if (tid == 0) {
            tc_fence_after();
            mma(tmem, S.x, S.w1t, SBO_K32, SUR_ND, id64);
            umma_commit(&S.mbar);
        }
        wait_mma();
        if (!ok) break;
        // H1 = silu(Z1 + b1) into the layer-2 operand and H1^T; silu'(Z1) to TMEM [160, 224)
        {
            const int q = part;
            float z[16], d[16];
            tmem_ld16(lane + 16 * q, z);
            uint32_t p[8];
#pragma unroll
            for (int i = 0; i < 16; i++) {
                const int k = 16 * q + i;
                const float zb = z[i] + S.b1[k], s = sigm(zb);
                d[i] = s * (1.0f + zb * (1.0f - s));
                z[i] = silu(zb);
                put_bf(S.h1t, k, t, 16, z[i]);
            }
#pragma unroll
            for (int i = 0; i < 8; i++) p[i] = pack_bf2(z[2 * i], z[2 * i + 1]);
            put_chunk(S.h, t, 2 * q, 8, make_uint4(p[0], p[1], p[2], p[3]));
            put_chunk(S.h, t, 2 * q + 1, 8, make_uint4(p[4], p[5], p[6], p[7]));
            tmem_st16(lane + 160 + 16 * q, d);
        }
        publish();

        // ---- layer 2: TMEM [64, 128) = H1 W2
        if (tid == 0) {
            tc_fence_after();
            mma(tmem + 64, S.h, S.w2t, SBO_K64, SUR_NH, id64);
            umma_commit(&S.mbar);
        }
        wait_mma();
        if (!ok) break;
        // H2 (over H1: layer 2 has read it), H2^T; silu'(Z2) to TMEM [0, 64)
        {
            const int q = part;
            float z[16], d[16];
            tmem_ld16(lane + 64 + 16 * q, z);
            uint32_t p[8];
#pragma unroll
            for (int i = 0; i < 16; i++) {
                const int k = 16 * q + i;
                const float zb = z[i] + S.b2[k], s = sigm(zb);
                d[i] = s * (1.0f + zb * (1.0f - s));
                z[i] = silu(zb);
                put_bf(S.h2t, k, t, 16, z[i]);
            }
#pragma unroll
            for (int i = 0; i < 8; i++) p[i] = pack_bf2(z[2 * i], z[2 * i + 1]);
            put_chunk(S.h, t, 2 * q, 8, make_uint4(p[0], p[1], p[2], p[3]));
            put_chunk(S.h, t, 2 * q + 1, 8, make_uint4(p[4], p[5], p[6], p[7]));
            tmem_st16(lane + 16 * q, d);
        }
        publish();

        asm volatile("cp.async.wait_group 0;" ::: "memory");  // (ordered by wait_mma's barrier)

        // ---- layer 3: TMEM [128, 144) = H2 W3
        if (tid == 0) {
            tc_fence_after();
            mma(tmem + 128, S.h, S.w3t, SBO_K64, SUR_NH, id16);
            umma_commit(&S.mbar);
        }
        wait_mma();
        if (!ok) break;
        double loss = 0.0;
        float dy[SUR_NO];
        {
            float o[16];
            tmem_ld16(lane + 128, o);
            float r[3];
#pragma unroll
            for (int c = 0; c < 3; c++) {
                float fc = 0.0f;
                if (active) {
#pragma unroll
                    for (int m = 0; m < SUR_NO; m++) fc = fmaf(o[m] + S.b3[m], vrow[3 * m + c], fc);
                }
                r[c] = fc - tg[c];
                if (part == 0) loss += (double)r[c] * (double)r[c];
            }
            loss *= (double)A.norm;
            const float two_norm = 2.0f * A.norm;
#pragma unroll
            for (int m = 0; m < SUR_NO; m++) {
                dy[m] = active ? two_norm * (r[0] * vrow[3 * m] + r[1] * vrow[3 * m + 1] +
                                             r[2] * vrow[3 * m + 2])
                               : 0.0f;
                if ((m >> 2) == part) put_bf(S.dyt, m, t, 16, dy[m]);
            }
        }
        // dZ2 = (dY W3^T) silu'(Z2) over H2 (layer 3 has read it) and into dZ2^T
        {
            const int q = part;
            float s2[16], dz[16];
            tmem_ld16(lane + 16 * q, s2);
            uint32_t p[8];
#pragma unroll
            for (int i = 0; i < 16; i++) {
                const int k = 16 * q + i;
                float dh = 0.0f;
#pragma unroll
                for (int m = 0; m < SUR_NO; m++) dh = fmaf(dy[m], S.w3[SUR_NO * k + m], dh);
                dz[i] = dh * s2[i];
                put_bf(S.dz2t, k, t, 16, dz[i]);
            }
#pragma unroll
            for (int i = 0; i < 8; i++) p[i] = pack_bf2(dz[2 * i], dz[2 * i + 1]);
            put_chunk(S.h, t, 2 * q, 8, make_uint4(p[0], p[1], p[2], p[3]));
            put_chunk(S.h, t, 2 * q + 1, 8, make_uint4(p[4], p[5], p[6], p[7]));
        }
        publish();

        // ---- dW3 (TMEM [144, 160)), dH1 (TMEM [0, 64)), dW2 (TMEM [64, 128))
        if (tid == 0) {
            tc_fence_after();
            mma(tmem + 144, S.h2t, S.dyt, SBO_K128, TR_M, id16);
            mma(tmem, S.h, S.w2, SBO_K64, SUR_NH, id64);
            mma(tmem + 64, S.h1t, S.dz2t, SBO_K128, TR_M, id64);
            umma_commit(&S.mbar);
        }
        wait_mma();
        if (!ok) break;
        // dZ1 = dH1 silu'(Z1) into dZ1^T
        {
            const int q = part;
            float dh[16], s1[16];
            tmem_ld16(lane + 16 * q, dh);
            tmem_ld16(lane + 160 + 16 * q, s1);
#pragma unroll
            for (int i = 0; i < 16; i++) put_bf(S.dz1t, 16 * q + i, t, 16, dh[i] * s1[i]);
        }
        // gradient rows of layers 3 and 2 (TMEM lane = output row)
        float* G = A.part + tile * SUR_NP;
        if (part == 0) {
            float o[16];
            tmem_ld16(lane + 144, o);
            if (t < SUR_NH)
                store16(G + SUR_OFF_W3 + t * SUR_NO, o);
            else if (t == SUR_NH)
                for (int m = 0; m < SUR_NO; m++) G[SUR_OFF_B3 + m] = o[m];
        }
        {
            const int q = part;
            float o[16];
            tmem_ld16(lane + 64 + 16 * q, o);
            if (t < SUR_NH)
                store16(G + SUR_OFF_W2 + t * SUR_NH + 16 * q, o);
            else if (t == SUR_NH)
                for (int i = 0; i < 16; i++) G[SUR_OFF_B2 + 16 * q + i] = o[i];
        }
        publish();

        // ---- dW1 (TMEM [160, 224): silu'(Z1) has been read)
        if (tid == 0) {
            tc_fence_after();
            mma(tmem + 160, S.xt, S.dz1t, SBO_K128, TR_M, id64);
            umma_commit(&S.mbar);
        }
        wait_mma();
        if (!ok) break;
        {
            const int q = part;
            float o[16];
            tmem_ld16(lane + 160 + 16 * q, o);
            if (t < SUR_ND)
                store16(G + SUR_OFF_W1 + t * SUR_NH + 16 * q, o);
            else if (t == SUR_ND)
                for (int i = 0; i < 16; i++) G[SUR_OFF_B1 + 16 * q + i] = o[i];
        }
        // the tile's loss, in thread order
        if (part == 0) {
            for (int o = 16; o > 0; o >>= 1) loss += __shfl_down_sync(0xffffffffu, loss, o);
            if ((tid & 31) == 0) S.lsum[warp] = loss;
        }
        tc_fence_before();
        __syncthreads();  // TMEM reads and operand reads done before the next tile
        tc_fence_after();
        if (tid == 0) A.part_loss[tile] = ((S.lsum[0] + S.lsum[1]) + S.lsum[2]) + S.lsum[3];
    }
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TR_COLS)
                     : "memory");
    if (!ok && tid == 0) atomicOr(A.status, ST_TIMEOUT);
}

}  // namespace

int sur_grad_tc_tiles(long long batch) { return (int)((batch + TR_M - 1) / TR_M); }

cudaError_t launch_sur_grad_tc(const SurGradArgs& a, int sms, cudaStream_t st)
{
    const long long ntiles = (a.batch + TR_M - 1) / TR_M;
    if (ntiles <= 0) return cudaSuccess;
    const size_t smem = sizeof(TrSmem);
    cudaError_t e = cudaFuncSetAttribute(k_sur_grad_tc, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem);
    if (e != cudaSuccess) return e;
    const long long grid = ntiles < (long long)sms ? ntiles : (long long)sms;
    if (a.chained) return launch_after(k_sur_grad_tc, grid, TR_T, smem, st, a);
    k_sur_grad_tc<<<(unsigned)grid, TR_T, smem, st>>>(a);
    return cudaGetLastError();
}

}  // namespace atm3
