// rt_mlp.cu -- learned path-gain surrogate (not in the paper; it cites
// neural path-loss prediction as related work, Sec. I): Fourier features of
// (tx, rx) -> n_hidden ReLU layers -> (path logit, path gain in dB).
//
// Dense layers are tcgen05 GEMMs: BF16 operands staged in shared memory by
// TMA (128-byte swizzle, 4-stage mbarrier pipeline), FP32 accumulators in
// TMEM, one thread issuing MMAs, the four warps reading TMEM in the
// epilogue (bias, ReLU, BF16 or FP32 store). Inference and training run all
// layers of a tile in one kernel each; the weight gradients of all layers are
// one more, Adam another. Shapes those do not take go layer by layer.
#include <cuda.h>
#include <cuda_bf16.h>

#include <cmath>
#include <cstring>
#include <random>
#include <string>
#include <vector>

#include "rt_internal.h"
#include "rt_tc.cuh"

namespace {

constexpr int GM = 128, GK = 64, GSTAGES = 4;

// sin and cos of 2 pi a for a in [-0.5, 0.5] (the reduced Fourier phase):
// the hardware approximation, absolute error about 4e-7 on [-pi, pi], far
// below the BF16 rounding the features then get.
__device__ __forceinline__ void feature_sincos(float a, float* s, float* c) {
    __sincosf(6.283185307179586f * a, s, c);
}

__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
    __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<uint32_t*>(&v);
}

// C[M x N] = act(A[M x K] B[N x K]^T + bias), A and B BF16 row-major (K
// contiguous), C FP32 or BF16 row-major with leading dimension ldc. MASK: C is
// zero where mask (BF16 [M x N], same leading dimension) is not positive, the
// derivative of the ReLU that produced it (a variant of its own: as a test of
// the pointer it cost every layer of a forward pass 2 to 4 us).
template <int BN, bool MASK>
__global__ void __launch_bounds__(128, 1) k_gemm(const __grid_constant__ CUtensorMap ta,
                                                  const __grid_constant__ CUtensorMap tb, int M, int N, int K,
                                                  const float* __restrict__ bias, int relu, int out_bf16,
                                                  void* __restrict__ C, int ldc,
                                                  const __nv_bfloat16* __restrict__ mask, unsigned* err) {
    extern __shared__ uint8_t dyn[];
    __shared__ __align__(8) uint64_t bar_full[GSTAGES], bar_empty[GSTAGES], bar_done;
    __shared__ uint32_t tmem_slot;
    constexpr uint32_t A_BYTES = GM * GK * 2, B_BYTES = BN * GK * 2, ST_BYTES = A_BYTES + B_BYTES;
    constexpr uint32_t TCOLS = BN;  // 64, 128 or 256 FP32 columns
    uint8_t* base = (uint8_t*)(((uintptr_t)dyn + 1023) & ~(uintptr_t)1023);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int m0 = blockIdx.x * GM, n0 = blockIdx.y * BN;
    const int nk = (K + GK - 1) / GK;
    if (warp == 0) {
        tmem_alloc(su32(&tmem_slot), TCOLS);
        tmem_relinquish();
    }
    if (threadIdx.x == 32) {
        for (int s = 0; s < GSTAGES; s++) {
            mbar_init(su32(&bar_full[s]), 1);
            mbar_init(su32(&bar_empty[s]), 1);
        }
        mbar_init(su32(&bar_done), 1);
        mbar_fence_init();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;
    if (warp == 0 && lane == 0) {
        // TMA producer
        for (int kb = 0; kb < nk; kb++) {
            const int s = kb % GSTAGES;
            if (kb >= GSTAGES && !mbar_wait(su32(&bar_empty[s]), ((kb / GSTAGES) - 1) & 1, err)) break;
            const uint32_t sa = su32(base + s * ST_BYTES), sb = sa + A_BYTES;
            mbar_expect_tx(su32(&bar_full[s]), ST_BYTES);
            tma_load_2d(sa, &ta, kb * GK, m0, su32(&bar_full[s]));
            tma_load_2d(sb, &tb, kb * GK, n0, su32(&bar_full[s]));
        }
    } else if (warp == 1 && lane == 0) {
        // MMA issuer
        constexpr uint32_t idesc = idesc_bf16(GM, BN);
        for (int kb = 0; kb < nk; kb++) {
            const int s = kb % GSTAGES;
            if (!mbar_wait(su32(&bar_full[s]), (kb / GSTAGES) & 1, err)) break;
            tc_fence_after();
            const uint32_t sa = su32(base + s * ST_BYTES), sb = sa + A_BYTES;
#pragma unroll
            for (int k = 0; k < GK / 16; k++)
                mma_bf16(tmem, desc_sw128(sa + k * 32), desc_sw128(sb + k * 32), idesc, (kb | k) != 0 ? 1u : 0u);
            mma_commit(su32(&bar_empty[s]));
        }
        mma_commit(su32(&bar_done));
    }
    __syncwarp();
    const bool done = mbar_wait(su32(&bar_done), 0, err);
    tc_fence_after();
    const int row = m0 + warp * 32 + lane;
    if (done) {
        for (int c0 = 0; c0 < BN; c0 += 32) {
            uint32_t r[32];
            tmem_ld32(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c0, r);
            tmem_wait_ld();
            const int col = n0 + c0;
            if (row >= M || col >= N) continue;
            float v[32];
#pragma unroll
            for (int j = 0; j < 32; j++) {
                float x = __uint_as_float(r[j]);
                if (bias && col + j < N) x += bias[col + j];
                if (relu) x = fmaxf(x, 0.0f);
                v[j] = x;
            }
            if (MASK) {
                const __nv_bfloat16* mp = mask + (size_t)row * ldc + col;
                if (col + 32 <= N) {
#pragma unroll
                    for (int q = 0; q < 4; q++) {
                        const uint4 h = *reinterpret_cast<const uint4*>(mp + 8 * q);
                        const uint32_t hw[4] = {h.x, h.y, h.z, h.w};
#pragma unroll
                        for (int u = 0; u < 4; u++) {
                            const __nv_bfloat162 b2 = *reinterpret_cast<const __nv_bfloat162*>(&hw[u]);
                            if (!(__low2float(b2) > 0.0f)) v[8 * q + 2 * u] = 0.0f;
                            if (!(__high2float(b2) > 0.0f)) v[8 * q + 2 * u + 1] = 0.0f;
                        }
                    }
                } else {
#pragma unroll
                    for (int j = 0; j < 32; j++)
                        if (col + j < N && !(__bfloat162float(mp[j]) > 0.0f)) v[j] = 0.0f;
                }
            }
            if (col + 32 <= N) {
                if (out_bf16) {
                    uint4* p = reinterpret_cast<uint4*>((__nv_bfloat16*)C + (size_t)row * ldc + col);
#pragma unroll
                    for (int q = 0; q < 4; q++)
                        p[q] = make_uint4(pack_bf16(v[8 * q], v[8 * q + 1]), pack_bf16(v[8 * q + 2], v[8 * q + 3]),
                                          pack_bf16(v[8 * q + 4], v[8 * q + 5]), pack_bf16(v[8 * q + 6], v[8 * q + 7]));
                } else {
                    float4* p = reinterpret_cast<float4*>((float*)C + (size_t)row * ldc + col);
#pragma unroll
                    for (int q = 0; q < 8; q++) p[q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
                }
            } else {
                for (int j = 0; j < 32 && col + j < N; j++) {
                    if (out_bf16)
                        ((__nv_bfloat16*)C)[(size_t)row * ldc + col + j] = __float2bfloat16_rn(v[j]);
                    else
                        ((float*)C)[(size_t)row * ldc + col + j] = v[j];
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, TCOLS);
}

// ------------------------------------------------------------ CUDA-core parts
// features: x [B x 6] (tx xyz, rx xyz) -> [sin(2 pi Bx'), cos(2 pi Bx')] (BF16 [B x 2F]),
// x' = 2 (x - lo) / (hi - lo) - 1 per coordinate.
__global__ void k_features(const float* __restrict__ x, int64_t n, const float* __restrict__ Bf, int F,
                           const float* __restrict__ lo, const float* __restrict__ hi,
                           __nv_bfloat16* __restrict__ out) {
    int64_t i = (int64_t)blockIdx.x * blockDim.y + threadIdx.y;
    if (i >= n) return;
    float xn[6];
    for (int k = 0; k < 6; k++) xn[k] = 2.0f * (x[6 * i + k] - lo[k]) / (hi[k] - lo[k]) - 1.0f;
    for (int j = threadIdx.x; j < F; j += blockDim.x) {
        float a = 0.0f;
        for (int k = 0; k < 6; k++) a = fmaf(Bf[6 * j + k], xn[k], a);
        a -= rintf(a);  // integer periods drop out of sin/cos(2 pi a)
        float s, c;
        feature_sincos(a, &s, &c);
        out[(size_t)i * 2 * F + j] = __float2bfloat16_rn(s);
        out[(size_t)i * 2 * F + F + j] = __float2bfloat16_rn(c);
    }
}

// head: y[b][o] = sum_j H[b][j] W[o][j] + bias[o], o in {0, 1}; one warp per row
__global__ void k_head(const __nv_bfloat16* __restrict__ H, int64_t n, int W, const float* __restrict__ Wh,
                       const float* __restrict__ bh, float* __restrict__ y) {
    int64_t i = (int64_t)blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32;
    int lane = threadIdx.x & 31;
    if (i >= n) return;
    float a0 = 0.0f, a1 = 0.0f;
    for (int j = lane; j < W; j += 32) {
        float h = __bfloat162float(H[(size_t)i * W + j]);
        a0 = fmaf(h, Wh[j], a0);
        a1 = fmaf(h, Wh[W + j], a1);
    }
    for (int o = 16; o > 0; o >>= 1) {
        a0 += __shfl_xor_sync(0xffffffffu, a0, o);
        a1 += __shfl_xor_sync(0xffffffffu, a1, o);
    }
    if (lane == 0) {
        y[2 * i] = a0 + bh[0];
        y[2 * i + 1] = a1 + bh[1];
    }
}

// Free-space gain 20 log10(lambda / (4 pi d)) in dB of the query x [6]
// (d = |rx - tx|, at least 1 m); 0 when lam == 0 (no baseline).
__device__ __forceinline__ float fspl_db(const float* __restrict__ x, float lam) {
    if (lam <= 0.0f) return 0.0f;
    float dx = x[3] - x[0], dy = x[4] - x[1], dz = x[5] - x[2];
    float d = fmaxf(sqrtf(dx * dx + dy * dy + dz * dz), 1.0f);
    return 20.0f * log10f(lam / (4.0f * RT_PI_F * d));
}

// outputs in user units: (path logit, gain dB = y1 * scale + offset + baseline)
__global__ void k_head_out(const float* __restrict__ y, const float* __restrict__ x, int64_t n, float scale,
                           float offset, float lam, float* __restrict__ out) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    out[2 * i] = y[2 * i];
    out[2 * i + 1] = y[2 * i + 1] * scale + offset + fspl_db(x + 6 * i, lam);
}

// loss = mean_b [BCE(logit, has) + has * (y1 - t)^2], t = (gain_db - offset) / scale;
// dy = d loss / d y. Returns one row's term (not yet divided by n).
__device__ __forceinline__ float loss_row(float z, float y1, const float* __restrict__ tgt, const float* __restrict__ x,
                                          int n, float scale, float offset, float lam, float& d0, float& d1) {
    float has = tgt[0], t = (tgt[1] - offset - fspl_db(x, lam)) / scale;
    float p = 1.0f / (1.0f + __expf(-z));
    // BCE with logits, stable form: max(z,0) - z has + log(1 + e^-|z|)
    float l = fmaxf(z, 0.0f) - z * has + log1pf(__expf(-fabsf(z)));
    float e = y1 - t;
    l += has * e * e;
    d0 = (p - has) / n;
    d1 = 2.0f * has * e / n;
    return l;
}

__global__ void k_loss(const float* __restrict__ y, const float* __restrict__ tgt, const float* __restrict__ x, int n,
                       float scale, float offset, float lam, float* __restrict__ dy, float* __restrict__ loss) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    float l = 0.0f;
    if (i < n)
        l = loss_row(y[2 * i], y[2 * i + 1], tgt + 2 * i, x + 6 * i, n, scale, offset, lam, dy[2 * i], dy[2 * i + 1]);
    for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
    if ((threadIdx.x & 31) == 0) atomicAdd(loss, l / n);
}

// Backward of the head over HB_ROWS rows per block, a thread per pair of
// columns: dZ[b][j] = (dy[b][0] Wh[0][j] + dy[b][1] Wh[1][j]) * (H[b][j] > 0)
// in BF16, and this block's part of the head's gradients
// part[block] = (sum_b dy[b][o] H[b][j] [2 x W], sum_b dy[b][o] [2]), summed in
// block order by k_adam. One read of H and one write of dZ, spread over
// B / 64 blocks: 5 us at B = 16384, W = 256 (the same sums over 8 blocks of
// all rows each took 845 us, dZ in a pass of its own 15 us).
constexpr int HB_ROWS = 64;
__global__ void k_head_bwd(const __nv_bfloat16* __restrict__ H, const float* __restrict__ dy, int W,
                           const float* __restrict__ Wh, __nv_bfloat16* __restrict__ dZ, float* __restrict__ part) {
    __shared__ float2 sd[HB_ROWS];
    const int b0 = blockIdx.x * HB_ROWS, c = threadIdx.x;   // blockDim = W / 2
    for (int r = threadIdx.x; r < HB_ROWS; r += blockDim.x) sd[r] = reinterpret_cast<const float2*>(dy)[b0 + r];
    __syncthreads();
    const float2 w0 = make_float2(Wh[2 * c], Wh[2 * c + 1]), w1 = make_float2(Wh[W + 2 * c], Wh[W + 2 * c + 1]);
    const uint32_t* Hp = reinterpret_cast<const uint32_t*>(H + (size_t)b0 * W) + c;
    uint32_t* Zp = reinterpret_cast<uint32_t*>(dZ + (size_t)b0 * W) + c;
    float a[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    float c0 = 0.0f, c1 = 0.0f;
#pragma unroll 8
    for (int r = 0; r < HB_ROWS; r++) {
        const uint32_t hw = Hp[(size_t)r * (W / 2)];
        const __nv_bfloat162 h2 = *reinterpret_cast<const __nv_bfloat162*>(&hw);
        const float hx = __low2float(h2), hy = __high2float(h2);
        const float2 d = sd[r];
        a[0] = fmaf(d.x, hx, a[0]);
        a[1] = fmaf(d.x, hy, a[1]);
        a[2] = fmaf(d.y, hx, a[2]);
        a[3] = fmaf(d.y, hy, a[3]);
        c0 += d.x;
        c1 += d.y;
        const float gx = d.x * w0.x + d.y * w1.x;
        const float gy = d.x * w0.y + d.y * w1.y;
        Zp[(size_t)r * (W / 2)] = pack_bf16(hx > 0.0f ? gx : 0.0f, hy > 0.0f ? gy : 0.0f);
    }
    float* o = part + (size_t)blockIdx.x * (2 * W + 2);
    o[2 * c] = a[0];
    o[2 * c + 1] = a[1];
    o[W + 2 * c] = a[2];
    o[W + 2 * c + 1] = a[3];
    if (c == 0) {
        o[2 * W] = c0;
        o[2 * W + 1] = c1;
    }
}

// Weight gradients dW_l[o][i] = sum_b dZ_l[b][o] H_l[b][i] and bias gradients
// sum_b dZ_l[b][o] of every hidden layer in one launch. Both operands of the
// contraction over the batch lie with the batch outermost in memory, so they
// go to the tensor cores as they are, as MN-major operands (TMA boxes of 64
// rows by 64 or 32 columns, 128- and 64-byte swizzle), with no transposed
// copies. A CTA takes 128 outputs o by 32 inputs i of one layer over the whole
// batch: the sum runs through one accumulator in batch order, as the GEMM over
// transposed copies ran it (the tensor cores round their FP32 accumulators
// towards zero, so splitting the batch would change the sums by 3e-5). 16 CTAs
// per 256 x 256 layer, 116 at L = 8, 2F = 64. Warps 2 and 3 add up 16 columns
// of the staged dZ for the bias, in 8 interleaved sums (all 128 columns in one
// CTA of a layer held the others up: 126 us).
// Bound by what an SM takes in (20 KB per 64 rows: 5.2 MB per CTA at B =
// 16384); eight stages cover the L2 latency. B = 16384, W = 256, L = 8: 97 us,
// where transposed copies, a GEMM per layer and a column sum per layer took
// 1.3 ms.
constexpr int WG_ROWS = 64, WG_ST = 8, WG_N = 32;
constexpr uint32_t WG_CHUNK = WG_ROWS * 128;            // 64 rows x 64 columns of dZ
constexpr uint32_t WG_STAGE = 2 * WG_CHUNK + WG_ROWS * WG_N * 2;
struct WgradArgs {
    int W, K0, L, B;
    int64_t cap;   // rows between consecutive layers of dZ (and of H)
    int layer;     // the only layer of this launch, or -1: all
    int64_t z0;    // first row of its dZ
    float* g;      // gradient vector
    unsigned* err;
};

// K-step of 16 rows of an MN-major operand in 128-byte rows (64-column chunks
// WG_CHUNK apart, groups of 8 rows 1024 B apart), or in 64-byte rows (one
// chunk of 32 columns, groups of 8 rows 512 B apart).
__device__ __forceinline__ uint64_t desc_mn_sw128(uint32_t saddr) {
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)(WG_CHUNK >> 4) << 16) | ((uint64_t)(1024 >> 4) << 32) |
           ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}
__device__ __forceinline__ uint64_t desc_mn_sw64(uint32_t saddr) {
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)(512 >> 4) << 16) | ((uint64_t)(512 >> 4) << 32) |
           ((uint64_t)1 << 46) | ((uint64_t)4 << 61);
}

__global__ void __launch_bounds__(128, 1) k_wgrad(const __grid_constant__ CUtensorMap tz,
                                                  const __grid_constant__ CUtensorMap th0,
                                                  const __grid_constant__ CUtensorMap th, WgradArgs a) {
    extern __shared__ uint8_t dyn[];
    __shared__ __align__(8) uint64_t bar_full[WG_ST], bar_empty[WG_ST], bar_done;
    __shared__ uint32_t tmem_slot;
    __shared__ float s_bias[8][16];
    uint8_t* base = (uint8_t*)(((uintptr_t)dyn + 1023) & ~(uintptr_t)1023);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // layer, 128-output tile and 32-input tile of this CTA
    const int mt = (a.W + 127) / 128, nt0 = (a.K0 + WG_N - 1) / WG_N, nt1 = a.W / WG_N;
    int l, t = blockIdx.x;
    if (a.layer >= 0) {
        l = a.layer;
    } else if (t < mt * nt0) {
        l = 0;
    } else {
        t -= mt * nt0;
        l = 1 + t / (mt * nt1);
        t -= (l - 1) * mt * nt1;
    }
    const int nt = t / mt, m = t - nt * mt;
    const int K = l == 0 ? a.K0 : a.W;   // inputs of the layer
    const int nkb = a.B / WG_ROWS;
    // the layer's tiles share the bias sums of these 128 outputs: groups of 16
    // columns nt, nt + ntl, ...
    const int ntl = l == 0 ? nt0 : nt1, ngr = min(8, (a.W - 128 * m) / 16);
    const bool do_bias = nt < ngr;
    if (warp == 0) {
        tmem_alloc(su32(&tmem_slot), 32);
        tmem_relinquish();
    }
    if (threadIdx.x == 32) {
        for (int s = 0; s < WG_ST; s++) {
            mbar_init(su32(&bar_full[s]), 1);
            mbar_init(su32(&bar_empty[s]), do_bias ? 3 : 1);   // the MMA commit and the bias warps
        }
        mbar_init(su32(&bar_done), 1);
        mbar_fence_init();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;
    // the layer's place in the gradient vector (W then b of every layer)
    float* out = a.g + (l == 0 ? 0 : (int64_t)a.W * a.K0 + a.W + (int64_t)(l - 1) * (a.W * a.W + a.W));
    if (warp == 0 && lane == 0) {
        const int zr = (int)(a.layer >= 0 ? a.z0 : l * a.cap), hr = l == 0 ? 0 : (int)((l - 1) * a.cap);
        const CUtensorMap* mh = l == 0 ? &th0 : &th;
        int issued = 0;
        for (int kb = 0; kb < nkb; kb++, issued++) {
            const int s = kb % WG_ST;
            if (kb >= WG_ST && !mbar_wait(su32(&bar_empty[s]), ((kb / WG_ST) - 1) & 1, a.err)) break;
            const uint32_t sa = su32(base) + (uint32_t)s * WG_STAGE;
            mbar_expect_tx(su32(&bar_full[s]), WG_STAGE);
            // columns past the layer's width or inputs read as zero
            tma_load_2d(sa, &tz, 128 * m, zr + kb * WG_ROWS, su32(&bar_full[s]));
            tma_load_2d(sa + WG_CHUNK, &tz, 128 * m + 64, zr + kb * WG_ROWS, su32(&bar_full[s]));
            tma_load_2d(sa + 2 * WG_CHUNK, mh, WG_N * nt, hr + kb * WG_ROWS, su32(&bar_full[s]));
        }
        // the last loads have landed before the CTA ends
        for (int j = issued > WG_ST ? issued - WG_ST : 0; j < issued; j++)
            mbar_wait(su32(&bar_full[j % WG_ST]), (j / WG_ST) & 1, a.err);
    } else if (warp == 1 && lane == 0) {
        // BF16 A and B, both MN-major (bits 15, 16), FP32 accumulators
        constexpr uint32_t idesc = idesc_bf16(128, WG_N) | (1u << 15) | (1u << 16);
        for (int kb = 0; kb < nkb; kb++) {
            const int s = kb % WG_ST;
            if (!mbar_wait(su32(&bar_full[s]), (kb / WG_ST) & 1, a.err)) break;
            tc_fence_after();
            const uint32_t sa = su32(base) + (uint32_t)s * WG_STAGE;
#pragma unroll
            for (int k = 0; k < WG_ROWS / 16; k++)
                mma_bf16(tmem, desc_mn_sw128(sa + k * 2048u), desc_mn_sw64(sa + 2 * WG_CHUNK + k * 1024u), idesc,
                         (kb | k) != 0 ? 1u : 0u);
            mma_commit(su32(&bar_empty[s]));
        }
        mma_commit(su32(&bar_done));
    } else if (warp >= 2 && do_bias) {
        // column sums of the staged dZ: thread (pair of columns, row phase of 8)
        const int cp = threadIdx.x & 7, ph = (threadIdx.x - 64) >> 3;
        float bx[8], by[8];
#pragma unroll
        for (int i = 0; i < 8; i++) bx[i] = by[i] = 0.0f;
        for (int kb = 0; kb < nkb; kb++) {
            const int s = kb % WG_ST;
            if (!__all_sync(0xffffffffu, mbar_wait(su32(&bar_full[s]), (kb / WG_ST) & 1, a.err))) break;
            const uint8_t* q = base + (uint32_t)s * WG_STAGE + ph * 128;
#pragma unroll
            for (int i = 0; i < 8; i++) {
                const int gr = nt + i * ntl;   // group of 16 columns (warp-uniform)
                if (gr >= ngr) break;
                const uint8_t* qc = q + (uint32_t)(gr >> 2) * WG_CHUNK + (((2 * (gr & 3) + (cp >> 2)) ^ ph) << 4) + 4 * (cp & 3);
#pragma unroll
                for (int r8 = 0; r8 < WG_ROWS; r8 += 8) {
                    const __nv_bfloat162 z = *reinterpret_cast<const __nv_bfloat162*>(qc + r8 * 128);
                    bx[i] += __low2float(z);
                    by[i] += __high2float(z);
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(su32(&bar_empty[s]));
        }
        // the 8 phases of a column, in order
#pragma unroll
        for (int i = 0; i < 8; i++) {
            const int gr = nt + i * ntl;
            if (gr >= ngr) break;
            s_bias[ph][2 * cp] = bx[i];
            s_bias[ph][2 * cp + 1] = by[i];
            asm volatile("bar.sync 1, 64;" ::: "memory");
            if (threadIdx.x < 64 + 16) {
                float t8 = 0.0f;
                for (int r = 0; r < 8; r++) t8 += s_bias[r][threadIdx.x - 64];
                out[(int64_t)a.W * K + 128 * m + 16 * gr + threadIdx.x - 64] = t8;
            }
            asm volatile("bar.sync 1, 64;" ::: "memory");
        }
    }
    __syncwarp();
    const bool done = mbar_wait(su32(&bar_done), 0, a.err);
    tc_fence_after();
    const int row = 128 * m + warp * 32 + lane;
    if (done) {
        uint32_t r[32];
        tmem_ld32(tmem + ((uint32_t)(warp * 32) << 16), r);
        tmem_wait_ld();
        if (row < a.W) {
            float* o = out + (int64_t)row * K + WG_N * nt;
            if (WG_N * (nt + 1) <= K) {
#pragma unroll
                for (int q = 0; q < 8; q++)
                    reinterpret_cast<float4*>(o)[q] = make_float4(__uint_as_float(r[4 * q]), __uint_as_float(r[4 * q + 1]),
                                                                  __uint_as_float(r[4 * q + 2]), __uint_as_float(r[4 * q + 3]));
            } else {
#pragma unroll
                for (int j = 0; j < 32; j++)
                    if (WG_N * nt + j < K) o[j] = __uint_as_float(r[j]);
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, 32);
}

// All parameters in one pass: Adam (Kingma & Ba 2015) on the gradients of the
// hidden layers (k_wgrad) and of the head (the blocks' partial sums of
// k_head_bwd, a warp per value), then the BF16 copies W [out x in] and W^T
// [in x out] of the hidden layers. One launch over the parameter vector where
// every tensor had its own (18 launches of 3 to 5 us each at L = 8).
struct AdamArgs {
    int W, K0, L, hblocks;
    float *w, *m, *v, *g;     // parameter vector layout (rt_mlp_get_params)
    const float* hpart;       // [hblocks][2W + 2]
    __nv_bfloat16 *wb, *wtb;  // hidden layers one after another
    float lr, b1, b2, eps, c1, c2;
};

__device__ __forceinline__ float adam_update(const AdamArgs& a, int64_t k, float gk) {
    const float mk_ = a.b1 * a.m[k] + (1.0f - a.b1) * gk;
    const float vk = a.b2 * a.v[k] + (1.0f - a.b2) * gk * gk;
    a.m[k] = mk_;
    a.v[k] = vk;
    const float x = a.w[k] - a.lr * (mk_ / a.c1) / (sqrtf(vk / a.c2) + a.eps);
    a.w[k] = x;
    return x;
}

__global__ void __launch_bounds__(256) k_adam(AdamArgs a, int hidden_blocks) {
    const int64_t n0 = (int64_t)a.W * a.K0 + a.W, n1 = (int64_t)a.W * a.W + a.W;
    const int64_t nh = n0 + (a.L - 1) * n1;
    if ((int)blockIdx.x < hidden_blocks) {
        const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
        if (k >= nh) return;
        const float x = adam_update(a, k, a.g[k]);
        const int l = k < n0 ? 0 : 1 + (int)((k - n0) / n1);
        const int64_t off = l == 0 ? 0 : n0 + (l - 1) * n1, j = k - off;
        const int in = l == 0 ? a.K0 : a.W;
        if (j < (int64_t)a.W * in) {
            const int64_t wo = off - (int64_t)l * a.W;   // weights before this layer (no biases)
            const int o = (int)j / in, i = (int)j - o * in;
            const __nv_bfloat16 xb = __float2bfloat16_rn(x);
            a.wb[wo + j] = xb;
            a.wtb[wo + (int64_t)i * a.W + o] = xb;
        }
        return;
    }
    const int q = ((int)blockIdx.x - hidden_blocks) * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    const int hn = 2 * a.W + 2;
    if (q >= hn) return;
    float gk = 0.0f;
    for (int s = lane; s < a.hblocks; s += 32) gk += a.hpart[(size_t)s * hn + q];
    for (int o = 16; o > 0; o >>= 1) gk += __shfl_xor_sync(0xffffffffu, gk, o);
    if (lane == 0) {
        a.g[nh + q] = gk;
        adam_update(a, nh + q, gk);
    }
}

// BF16 copies of the hidden layers' weights (see k_adam)
__global__ void k_to_bf16(const float* __restrict__ w, int W, int K0, int L, __nv_bfloat16* __restrict__ wb,
                          __nv_bfloat16* __restrict__ wtb) {
    const int64_t n0 = (int64_t)W * K0 + W, n1 = (int64_t)W * W + W;
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n0 + (L - 1) * n1) return;
    const int l = k < n0 ? 0 : 1 + (int)((k - n0) / n1);
    const int64_t off = l == 0 ? 0 : n0 + (l - 1) * n1, j = k - off;
    const int in = l == 0 ? K0 : W;
    if (j >= (int64_t)W * in) return;
    const int64_t wo = off - (int64_t)l * W;
    const int o = (int)j / in, i = (int)j - o * in;
    const __nv_bfloat16 xb = __float2bfloat16_rn(w[k]);
    wb[wo + j] = xb;
    wtb[wo + (int64_t)i * W + o] = xb;
}

// ------------------------------------------------------ fused inference
// All layers for a pair of 128-query tiles (A, B; one query per row) in a
// persistent CTA, with warp roles and mbarrier handshakes:
//   warp 8 (one lane)  streams each layer's weights by TMA in K-chunks
//                      (W output rows x 64 inputs) through a ring of NS
//                      slots; every chunk serves both tiles, so weight
//                      traffic per query is half of a one-tile design;
//   warp 9 (one lane)  issues tcgen05.mma (M = 128, N = W, K = 16) per chunk,
//                      first for tile A then for tile B, into TMEM columns
//                      [0, W) and [W, 2W); commits each slot back to the
//                      producer and each tile's last chunk to its epilogue;
//   warps 0-3 / 4-7    tile A / tile B: the Fourier features, then per layer
//                      the epilogue: read the accumulator (one TMEM lane
//                      quarter per warp), add the bias, apply ReLU, round to
//                      BF16 and write the next layer's input in place
//                      (128-byte-swizzled K-major, the layout TMA produces);
//                      after the last layer the 2-wide head.
// Tile A's epilogue overlaps tile B's last chunk, tile B's epilogue overlaps
// tile A's next layer. Every wait is bounded; after a timeout all roles
// skip their remaining work.
constexpr int FM_MAX_L = 16;
constexpr int FM_NS = 2;          // weight ring slots (W x 64 BF16 each)
constexpr int FM_THREADS = 320;   // 8 epilogue warps + producer + MMA issuer
struct alignas(64) FusedMaps {
    CUtensorMap w[FM_MAX_L];  // BF16 weights [W x K_l], box 64 x W
};

struct FusedArgs {
    const float* x;      // [n x 6]
    float* out;          // [n x 2]
    int64_t n;
    int F, W, L;
    const float* Bf;     // [F x 6]
    const float* lo;
    const float* hi;
    const float* params;       // parameter vector (W then b of every layer)
    const float* head_w;       // [2 x W]
    const float* head_b;       // [2]
    float db_scale, db_offset;
    float lam;           // free-space baseline wavelength (0 = none)
    unsigned* err;
};

__device__ __forceinline__ uint32_t sw128_off(int r, int c) {
    // byte offset of element (r, c) inside a 64-column K-chunk (128 B rows)
    return (uint32_t)r * 128u + ((((uint32_t)c >> 3) ^ ((uint32_t)r & 7u)) << 4) + (((uint32_t)c & 7u) << 1);
}

// Shared-memory layout (offsets from a 1024-aligned base).
struct FusedLayout {
    uint32_t act_bytes, act0, act1, ring, bias, head, bf, bars;
    __host__ __device__ FusedLayout(int F, int W, int L) {
        const int kmax = (2 * F > W ? 2 * F : W) / 64;
        act_bytes = (uint32_t)kmax * 16384u;
        act0 = 0;
        act1 = act_bytes;
        ring = 2 * act_bytes;
        bias = ring + FM_NS * (uint32_t)W * 128u;
        head = bias + 4u * (uint32_t)(L * W);
        bf = head + 4u * (uint32_t)(2 * W + 2);
        bars = (bf + 4u * (uint32_t)(6 * F + 12) + 7u) & ~7u;
    }
    // ring full/empty, per tile: MMA done, input ready; MMA drain
    __host__ __device__ uint32_t bytes() const { return bars + 8u * (2 * FM_NS + 5); }
};

__global__ void __launch_bounds__(FM_THREADS, 1) k_mlp_fused(const __grid_constant__ FusedMaps maps, FusedArgs a) {
    extern __shared__ uint8_t dyn[];
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int abort_flag;
    uint8_t* base = (uint8_t*)(((uintptr_t)dyn + 1023) & ~(uintptr_t)1023);
    const int W = a.W, L = a.L, F = a.F;
    const FusedLayout lay(F, W, L);
    uint8_t* act[2] = {base + lay.act0, base + lay.act1};   // tile A, tile B
    uint8_t* ring = base + lay.ring;
    float* s_bias = (float*)(base + lay.bias);
    float* s_head = (float*)(base + lay.head);
    float* s_bf = (float*)(base + lay.bf);
    uint64_t* bars = (uint64_t*)(base + lay.bars);
    const uint32_t full0 = su32(bars), empty0 = su32(bars + FM_NS);
    const uint32_t mma_done0 = su32(bars + 2 * FM_NS), in_ready0 = su32(bars + 2 * FM_NS + 2);
    const uint32_t drain = su32(bars + 2 * FM_NS + 4);
    const uint32_t slot_bytes = (uint32_t)W * 128u;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    for (int i = tid; i < L * W; i += FM_THREADS) {
        const int l = i / W;   // biases of layer l follow its weights
        s_bias[i] = a.params[2 * F * W + l * (W * W + W) + i % W];
    }
    for (int i = tid; i < 2 * W; i += FM_THREADS) s_head[i] = a.head_w[i];
    if (tid < 2) s_head[2 * W + tid] = a.head_b[tid];
    for (int i = tid; i < 6 * F; i += FM_THREADS) s_bf[i] = a.Bf[i];
    if (tid < 6) {
        s_bf[6 * F + tid] = a.lo[tid];
        s_bf[6 * F + 6 + tid] = a.hi[tid];
    }
    const uint32_t tcols = 2u * (uint32_t)W <= 256u ? 256u : 512u;
    if (warp == 0) {
        tmem_alloc(su32(&tmem_slot), tcols);
        tmem_relinquish();
    }
    if (tid == 32) {
        for (int s = 0; s < FM_NS; s++) {
            mbar_init(full0 + 8 * s, 1);
            mbar_init(empty0 + 8 * s, 1);
        }
        for (int t = 0; t < 2; t++) {
            mbar_init(mma_done0 + 8 * t, 1);
            mbar_init(in_ready0 + 8 * t, 128);
        }
        mbar_init(drain, 1);
        mbar_fence_init();
        abort_flag = 0;
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;
    const int64_t ntiles = (a.n + 127) / 128;
    const int64_t npairs = (ntiles + 1) / 2;
    auto fail = [&]() { abort_flag = 1; };

    if (warp == 8) {
        // ---------------------------------------------------------- producer
        if (lane == 0) {
            uint32_t it = 0;
            for (int64_t pr = blockIdx.x; pr < npairs && !abort_flag; pr += gridDim.x) {
                for (int l = 0; l < L && !abort_flag; l++) {
                    const int nkc = (l == 0 ? 2 * F : W) / 64;
                    for (int kc = 0; kc < nkc; kc++, it++) {
                        const uint32_t s = it % FM_NS, ph = (it / FM_NS) & 1u;
                        if (it >= FM_NS && !mbar_wait(empty0 + 8 * s, ph ^ 1u, a.err)) {
                            fail();
                            break;
                        }
                        mbar_expect_tx(full0 + 8 * s, slot_bytes);
                        tma_load_2d(su32(ring + s * slot_bytes), &maps.w[l], kc * 64, 0, full0 + 8 * s);
                    }
                }
            }
            // drain: the last loads issued have landed before the CTA ends
            for (uint32_t j = it > FM_NS ? it - FM_NS : 0; j < it; j++)
                mbar_wait(full0 + 8 * (j % FM_NS), (j / FM_NS) & 1u, a.err);
        }
    } else if (warp == 9) {
        // -------------------------------------------------------- MMA issuer
        if (lane == 0) {
            const uint32_t idesc = idesc_bf16(128, W);
            uint32_t it = 0, in_ph[2] = {0, 0};
            for (int64_t pr = blockIdx.x; pr < npairs && !abort_flag; pr += gridDim.x) {
                for (int l = 0; l < L && !abort_flag; l++) {
                    const int nkc = (l == 0 ? 2 * F : W) / 64;
                    for (int kc = 0; kc < nkc; kc++, it++) {
                        const uint32_t s = it % FM_NS, ph = (it / FM_NS) & 1u;
                        if (!mbar_wait(full0 + 8 * s, ph, a.err)) { fail(); break; }
                        bool okk = true;
                        for (int t = 0; t < 2; t++) {
                            // a layer's input (features for layer 0) and free TMEM columns
                            if (kc == 0) {
                                if (!mbar_wait(in_ready0 + 8 * t, in_ph[t], a.err)) { okk = false; break; }
                                in_ph[t] ^= 1u;
                            }
                            tc_fence_after();
#pragma unroll
                            for (int k = 0; k < 4; k++)
                                mma_bf16(tmem + (uint32_t)(t * W), desc_sw128(su32(act[t] + kc * 16384) + k * 32),
                                         desc_sw128(su32(ring + s * slot_bytes) + k * 32), idesc,
                                         (kc | k) != 0 ? 1u : 0u);
                            if (kc == nkc - 1) mma_commit(mma_done0 + 8 * t);
                        }
                        mma_commit(empty0 + 8 * s);
                        if (!okk) { fail(); break; }
                    }
                }
            }
            // drain: every MMA issued has completed before TMEM is released
            mma_commit(drain);
            mbar_wait(drain, 0, a.err);
        }
    } else {
        // ---------------------------------------- features + epilogue, per tile
        const int t = warp >> 2;                       // 0: tile A, 1: tile B
        const int row = (warp & 3) * 32 + lane;        // query row = TMEM lane
        const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
        const uint32_t col0 = (uint32_t)(t * W);
        uint8_t* buf = act[t];
        uint32_t done_ph = 0;
        for (int64_t pr = blockIdx.x; pr < npairs; pr += gridDim.x) {
            const int64_t q = (2 * pr + t) * 128 + row;
            {
                float xn[6];
                for (int k = 0; k < 6; k++) {
                    float xv = q < a.n ? a.x[6 * q + k] : 0.0f;
                    xn[k] = 2.0f * (xv - s_bf[6 * F + k]) / (s_bf[6 * F + 6 + k] - s_bf[6 * F + k]) - 1.0f;
                }
                for (int j = 0; j < F; j += 2) {
                    float s2[2], c2[2];
                    for (int hh = 0; hh < 2; hh++) {
                        float v = 0.0f;
                        for (int k = 0; k < 6; k++) v = fmaf(s_bf[6 * (j + hh) + k], xn[k], v);
                        v -= rintf(v);
                        feature_sincos(v, &s2[hh], &c2[hh]);
                    }
                    *(uint32_t*)(buf + (j / 64) * 16384 + sw128_off(row, j % 64)) = pack_bf16(s2[0], s2[1]);
                    *(uint32_t*)(buf + ((F + j) / 64) * 16384 + sw128_off(row, (F + j) % 64)) =
                        pack_bf16(c2[0], c2[1]);
                }
            }
            fence_async_smem();
            tc_fence_before();
            mbar_arrive(in_ready0 + 8 * t);
            float h0 = 0.0f, h1 = 0.0f;
            bool ok = true;
            for (int l = 0; l < L; l++) {
                bool got = !abort_flag && mbar_wait(mma_done0 + 8 * t, done_ph, a.err);
                done_ph ^= 1u;
                got = __all_sync(0xffffffffu, got);
                if (!got) { fail(); ok = false; break; }
                tc_fence_after();
                for (int cc = 0; cc < W; cc += 64) {
                    // two 32-column loads in flight per wait
                    uint32_t r2[2][32];
                    tmem_ld32(tmem + lane_base + col0 + (uint32_t)cc, r2[0]);
                    tmem_ld32(tmem + lane_base + col0 + (uint32_t)cc + 32u, r2[1]);
                    tmem_wait_ld();
#pragma unroll
                    for (int hh = 0; hh < 2; hh++) {
                    const int c0 = cc + 32 * hh;
                    const uint32_t* r = r2[hh];
                    uint32_t packed[16];
                    const float4* bv = reinterpret_cast<const float4*>(s_bias + l * W + c0);
#pragma unroll
                    for (int j4 = 0; j4 < 8; j4++) {
                        const float4 b = bv[j4];
                        const int j = 4 * j4;
                        packed[2 * j4] = add2_relu_bf16x2(__uint_as_float(r[j]), b.x, __uint_as_float(r[j + 1]), b.y);
                        packed[2 * j4 + 1] =
                            add2_relu_bf16x2(__uint_as_float(r[j + 2]), b.z, __uint_as_float(r[j + 3]), b.w);
                    }
                    if (l == L - 1) {
#pragma unroll
                        for (int j = 0; j < 32; j += 2) {
                            __nv_bfloat162 b2 = *reinterpret_cast<__nv_bfloat162*>(&packed[j / 2]);
                            float r0 = __low2float(b2), r1 = __high2float(b2);
                            h0 = fmaf(r0, s_head[c0 + j], fmaf(r1, s_head[c0 + j + 1], h0));
                            h1 = fmaf(r0, s_head[W + c0 + j], fmaf(r1, s_head[W + c0 + j + 1], h1));
                        }
                    }
                    if (l < L - 1) {
#pragma unroll
                        for (int u = 0; u < 4; u++) {
                            const int c = c0 + 8 * u;
                            *(uint4*)(buf + (c / 64) * 16384 + sw128_off(row, c % 64)) =
                                make_uint4(packed[4 * u], packed[4 * u + 1], packed[4 * u + 2], packed[4 * u + 3]);
                        }
                    }
                    }
                }
                if (l < L - 1) {
                    // the next layer's input is in place and this tile's TMEM columns are free
                    fence_async_smem();
                    tc_fence_before();
                    mbar_arrive(in_ready0 + 8 * t);
                }
            }
            if (!ok) break;
            if (q < a.n) {
                a.out[2 * q] = h0 + s_head[2 * W];
                a.out[2 * q + 1] = (h1 + s_head[2 * W + 1]) * a.db_scale + a.db_offset + fspl_db(a.x + 6 * q, a.lam);
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, tcols);
}

// ------------------------------------------------------ fused training chain
// Forward, loss and the backward chain of a 128-row tile in one CTA: the
// activations stay in shared memory (one buffer, 64-column chunks, updated in
// place) and the accumulators in TMEM (two buffers, alternating by pass), and
// what the weight gradients need (features, hidden outputs H_l and the
// gradients dZ_l) leaves by TMA stores from that buffer. L forward passes
// (H_l = ReLU(H_{l-1} W_l^T + b_l)), the head, the loss and its gradient, then
// L - 1 backward passes (dZ_{l-1} = (dZ_l W_l) * (H_l > 0), the signs kept as
// bits). Roles:
//   warps 0-7   features, then every pass's epilogue: chunk c by warps
//               4 (c & 1) .. + 3, so that the next pass starts on chunk 0 while
//               chunks 2 and 3 are still in TMEM (W = 64: each four warps take
//               half of the columns of the one chunk);
//   warp 8      streams the weights by TMA, W and later W^T, in 64-column chunks;
//   warp 9      issues tcgen05.mma (M 128, N W, K 16) chunk by chunk;
//   warp 10     stores every finished chunk.
// Values are those of the layer-by-layer kernels bit for bit (same MMA shapes
// and order, same sums in the head and the loss). A wait by parity tells a phase
// from the one after it, not from the next but one, so no barrier completes a
// second phase before every waiter has seen the first: warps 0-7 all arrive in
// each pass after their own waits, and the chunks that are only stored (H_L and
// dZ_0) have barriers that warp 10 alone waits on, since warp 9 holds up nothing
// between them and the chunks after them. Every wait is bounded; after
// a timeout the roles run on without waiting, on the same control flow.
// One tile per CTA: 128 CTAs at B = 16384, and the per-pass latency (first
// chunk's epilogue + four chunks of MMA) bounds it: 67 us for B = 16384,
// W = 256, L = 8, where a kernel per layer and step took 1.0 ms.
constexpr int TC_THREADS = 352;
struct TrainArgs {
    const float* x;        // [B x 6]
    const float* target;   // [B x 2]
    int B, F, W, L, NS;    // NS: weight ring slots
    const float *Bf, *lo, *hi;
    const float* params;
    float scale, offset, lam;
    float* loss;
    float* hpart;          // [B / HB_ROWS][2W + 2]
    int64_t cap;
    unsigned* err;
};
struct TrainMaps {
    CUtensorMap w0, wx, wt;   // W_0; W_1.. and W_1^T.. one below another
    CUtensorMap h0, h, z;     // features, [L * cap] hidden outputs, [L * cap] gradients
};

struct TrainLayout {
    uint32_t act, ring, mask, bias, head, bf, dy, bars;
    __host__ __device__ TrainLayout(int F, int W, int L, int NS) {
        const int kmax = (2 * F > W ? 2 * F : W) / 64;
        act = 0;
        ring = (uint32_t)kmax * 16384u;
        mask = ring + (uint32_t)NS * (uint32_t)W * 128u;
        bias = mask + (uint32_t)L * (uint32_t)(W / 32) * 512u;
        head = bias + 4u * (uint32_t)(L * W);
        bf = head + 4u * (uint32_t)(2 * W + 2);
        dy = (bf + 4u * (uint32_t)(6 * F + 12) + 7u) & ~7u;
        bars = dy + 128u * 8u;
    }
    // ring full / empty, chunks ready, chunks ready to be stored only, features ready, MMA done, stored, drain
    __host__ __device__ uint32_t bytes(int NS) const { return bars + 8u * (2 * NS + 4 + 4 + 4); }
};

__global__ void __launch_bounds__(TC_THREADS, 1) k_train_chain(const __grid_constant__ TrainMaps maps, TrainArgs a) {
    extern __shared__ uint8_t dyn[];
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int abort_flag;
    uint8_t* base = (uint8_t*)(((uintptr_t)dyn + 1023) & ~(uintptr_t)1023);
    const int W = a.W, L = a.L, F = a.F, NS = a.NS, nc = W / 64, nc0 = 2 * F / 64;
    const TrainLayout lay(F, W, L, NS);
    uint8_t* act = base + lay.act;
    uint32_t* s_mask = (uint32_t*)(base + lay.mask);   // [L][W / 32][128]
    float* s_bias = (float*)(base + lay.bias);
    float* s_head = (float*)(base + lay.head);
    float* s_bf = (float*)(base + lay.bf);
    float2* s_dy = (float2*)(base + lay.dy);
    uint64_t* bars = (uint64_t*)(base + lay.bars);
    const uint32_t full0 = su32(bars), empty0 = su32(bars + NS), chunk0 = su32(bars + 2 * NS);
    const uint32_t only0 = su32(bars + 2 * NS + 4);
    const uint32_t feat = su32(bars + 2 * NS + 8), done = su32(bars + 2 * NS + 9), stored = su32(bars + 2 * NS + 10);
    const uint32_t drain = su32(bars + 2 * NS + 11);
    const uint32_t slot_bytes = (uint32_t)W * 128u;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    for (int i = tid; i < L * W; i += TC_THREADS) {
        const int l = i / W;   // biases of layer l follow its weights
        s_bias[i] = a.params[2 * F * W + l * (W * W + W) + i % W];
    }
    const float* head = a.params + (size_t)2 * F * W + W + (size_t)(L - 1) * (W * W + W);
    for (int i = tid; i < 2 * W + 2; i += TC_THREADS) s_head[i] = head[i];
    for (int i = tid; i < 6 * F; i += TC_THREADS) s_bf[i] = a.Bf[i];
    if (tid < 6) {
        s_bf[6 * F + tid] = a.lo[tid];
        s_bf[6 * F + 6 + tid] = a.hi[tid];
    }
    const uint32_t tcols = 2u * (uint32_t)W <= 128u ? 128u : 2u * (uint32_t)W <= 256u ? 256u : 512u;
    if (warp == 0) {
        tmem_alloc(su32(&tmem_slot), tcols);
        tmem_relinquish();
    }
    if (tid == 32) {
        for (int s = 0; s < NS; s++) {
            mbar_init(full0 + 8 * s, 1);
            mbar_init(empty0 + 8 * s, 1);
        }
        for (int c = 0; c < 4; c++) {
            mbar_init(chunk0 + 8 * c, nc == 1 ? 256 : 128);
            mbar_init(only0 + 8 * c, nc == 1 ? 256 : 128);
        }
        mbar_init(feat, 256);
        mbar_init(done, 1);
        mbar_init(stored, 1);
        mbar_init(drain, 1);
        mbar_fence_init();
        abort_flag = 0;
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;
    const int tiles = a.B / 128, passes = 2 * L - 1;
    auto wait = [&](uint32_t bar, uint32_t parity) {
        if (!abort_flag && !mbar_wait(bar, parity & 1u, a.err)) abort_flag = 1;
    };

    if (warp == 8) {
        if (lane == 0) {
            uint32_t it = 0;
            for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x)
                for (int p = 0; p < passes; p++) {
                    const bool fwd = p < L;
                    const int l = fwd ? p : 2 * L - 1 - p;   // the pass's layer
                    const CUtensorMap* mp = l == 0 ? &maps.w0 : fwd ? &maps.wx : &maps.wt;
                    const int y = l == 0 ? 0 : (l - 1) * W, nk = l == 0 ? nc0 : nc;
                    for (int kc = 0; kc < nk && !abort_flag; kc++, it++) {
                        const uint32_t s = it % NS;
                        if (it >= (uint32_t)NS) wait(empty0 + 8 * s, it / NS + 1);
                        if (abort_flag) break;
                        mbar_expect_tx(full0 + 8 * s, slot_bytes);
                        tma_load_2d(su32(base + lay.ring + s * slot_bytes), mp, kc * 64, y, full0 + 8 * s);
                    }
                }
            // the last loads issued have landed before the CTA ends
            for (uint32_t j = it > (uint32_t)NS ? it - NS : 0; j < it; j++)
                mbar_wait(full0 + 8 * (j % NS), (j / NS) & 1u, a.err);
        }
    } else if (warp == 9) {
        if (lane == 0) {
            const uint32_t idesc = idesc_bf16(128, W);
            uint32_t it = 0, stage = 0, pass = 0, ft = 0;   // chunk phases seen, passes issued, tiles started
            for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x, ft++)
                for (int p = 0; p < passes; p++, pass++) {
                    const int nk = p == 0 ? nc0 : nc;
                    if (p == 0) wait(feat, ft);
                    for (int kc = 0; kc < nk; kc++, it++) {
                        const uint32_t s = it % NS;
                        if (p > 0) wait(chunk0 + 8 * kc, stage);
                        wait(full0 + 8 * s, it / NS);
                        if (abort_flag) break;
                        tc_fence_after();
#pragma unroll
                        for (int k = 0; k < 4; k++)
                            mma_bf16(tmem + (pass & 1u) * (uint32_t)W, desc_sw128(su32(act + kc * 16384) + k * 32),
                                     desc_sw128(su32(base + lay.ring + s * slot_bytes) + k * 32), idesc,
                                     (kc | k) != 0 ? 1u : 0u);
                        mma_commit(empty0 + 8 * s);
                    }
                    mma_commit(done);
                    if (p > 0) stage++;
                }
            // every MMA issued has completed before TMEM is released
            mma_commit(drain);
            mbar_wait(drain, 0, a.err);
        }
    } else if (warp == 10) {
        if (lane == 0) {
            uint32_t ft = 0, stage = 0, only = 0;   // tiles, phases of the two kinds of chunk barriers
            for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x, ft++)
                for (int q = 0; q <= 2 * L; q++) {   // features, H_1 .. H_L, dZ_{L-1} .. dZ_0
                    const CUtensorMap* mp = q == 0 ? &maps.h0 : q <= L ? &maps.h : &maps.z;
                    const int64_t r0 = q == 0 ? 0 : q <= L ? (int64_t)(q - 1) * a.cap : (int64_t)(2 * L - q) * a.cap;
                    const int nk = q == 0 ? nc0 : nc;
                    const bool last = q == L || q == 2 * L;   // H_L, dZ_0: no MMA's input
                    if (q == 0) wait(feat, ft);
                    for (int c = 0; c < nk; c++) {
                        if (q > 0) wait((last ? only0 : chunk0) + 8 * c, last ? only : stage);
                        if (!abort_flag)
                            tma_store_2d(mp, su32(act + c * 16384), c * 64, (int)(r0 + (int64_t)tile * 128));
                    }
                    if (last) only++;
                    else if (q > 0) stage++;
                    bulk_commit();
                    bulk_wait_read0();
                    mbar_arrive(stored);
                }
            bulk_wait0();
        }
    } else {
        const int g = warp >> 2, row = (warp & 3) * 32 + lane;
        const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
        const int c_first = nc == 1 ? 0 : g;
        uint32_t nst = 0, pass = 0;   // store phases and passes so far
        for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
            const int64_t q = (int64_t)tile * 128 + row;
            if (nst > 0) wait(stored, nst - 1);   // the buffer's last contents have been read
            {
                float xn[6];
                for (int k = 0; k < 6; k++)
                    xn[k] = 2.0f * (a.x[6 * q + k] - s_bf[6 * F + k]) / (s_bf[6 * F + 6 + k] - s_bf[6 * F + k]) - 1.0f;
                for (int j = g * (F / 2); j < (g + 1) * (F / 2); j += 2) {
                    float s2[2], c2[2];
                    for (int hh = 0; hh < 2; hh++) {
                        float v = 0.0f;
                        for (int k = 0; k < 6; k++) v = fmaf(s_bf[6 * (j + hh) + k], xn[k], v);
                        v -= rintf(v);
                        feature_sincos(v, &s2[hh], &c2[hh]);
                    }
                    *(uint32_t*)(act + (j / 64) * 16384 + sw128_off(row, j % 64)) = pack_bf16(s2[0], s2[1]);
                    *(uint32_t*)(act + ((F + j) / 64) * 16384 + sw128_off(row, (F + j) % 64)) = pack_bf16(c2[0], c2[1]);
                }
            }
            fence_async_smem();
            tc_fence_before();
            mbar_arrive(feat);
            nst++;
            for (int p = 0; p < passes; p++, pass++) {
                const bool fwd = p < L;
                const int l = fwd ? p : 2 * L - 1 - p;
                const uint32_t acc = tmem + lane_base + (pass & 1u) * (uint32_t)W;
                wait(done, pass);
                __syncwarp();
                tc_fence_after();
                wait(stored, nst - 1);
                nst++;
                // bits of H_{l+1} > 0 written forward; those of H_l applied backward
                uint32_t* mk = s_mask + (size_t)(fwd ? l : l - 1) * (W / 32) * 128 + row;
                const uint32_t ready = p == L - 1 || p == passes - 1 ? only0 : chunk0;
                for (int c = c_first; c < nc; c += 2) {
                    uint32_t r2[2][32];
                    tmem_ld32(acc + (uint32_t)c * 64u, r2[0]);
                    tmem_ld32(acc + (uint32_t)c * 64u + 32u, r2[1]);
                    tmem_wait_ld();
#pragma unroll
                    for (int hh = 0; hh < 2; hh++) {
                        if (nc == 1 && hh != g) continue;
                        uint32_t packed[16];
                        const int c0 = 64 * c + 32 * hh;
                        if (fwd) {
                            const float4* bv = reinterpret_cast<const float4*>(s_bias + l * W + c0);
                            uint32_t bits = 0;
#pragma unroll
                            for (int j4 = 0; j4 < 8; j4++) {
                                const float4 b = bv[j4];
                                const float v0 = fmaxf(__uint_as_float(r2[hh][4 * j4]) + b.x, 0.0f);
                                const float v1 = fmaxf(__uint_as_float(r2[hh][4 * j4 + 1]) + b.y, 0.0f);
                                const float v2 = fmaxf(__uint_as_float(r2[hh][4 * j4 + 2]) + b.z, 0.0f);
                                const float v3 = fmaxf(__uint_as_float(r2[hh][4 * j4 + 3]) + b.w, 0.0f);
                                // what rounds to a BF16 above zero (2^-134 is the tie with zero)
                                const float tie = __uint_as_float(0x00008000u);
                                if (v0 > tie) bits |= 1u << (4 * j4);
                                if (v1 > tie) bits |= 2u << (4 * j4);
                                if (v2 > tie) bits |= 4u << (4 * j4);
                                if (v3 > tie) bits |= 8u << (4 * j4);
                                packed[2 * j4] = pack_bf16(v0, v1);
                                packed[2 * j4 + 1] = pack_bf16(v2, v3);
                            }
                            mk[(2 * c + hh) * 128] = bits;
                        } else {
                            const uint32_t bits = mk[(2 * c + hh) * 128];
#pragma unroll
                            for (int j = 0; j < 32; j += 2)
                                packed[j / 2] = pack_bf16(bits & (1u << j) ? __uint_as_float(r2[hh][j]) : 0.0f,
                                                          bits & (2u << j) ? __uint_as_float(r2[hh][j + 1]) : 0.0f);
                        }
#pragma unroll
                        for (int u = 0; u < 4; u++)
                            *(uint4*)(act + c * 16384 + sw128_off(row, 32 * hh + 8 * u)) =
                                make_uint4(packed[4 * u], packed[4 * u + 1], packed[4 * u + 2], packed[4 * u + 3]);
                    }
                    fence_async_smem();
                    tc_fence_before();
                    mbar_arrive(ready + 8 * c);
                }
                if (p != L - 1) continue;
                // the head, the loss and their gradients
                if (g == 0) {
                    // y_o = sum_j H[j] Wh[o][j] in 32 interleaved sums and a tree over them
                    float a0[32], a1[32];
#pragma unroll
                    for (int j = 0; j < 32; j++) a0[j] = a1[j] = 0.0f;
                    for (int c0 = 0; c0 < W; c0 += 32) {
                        uint32_t r[32];
                        tmem_ld32(acc + (uint32_t)c0, r);
                        tmem_wait_ld();
#pragma unroll
                        for (int j = 0; j < 32; j++) {
                            const float v = fmaxf(__uint_as_float(r[j]) + s_bias[l * W + c0 + j], 0.0f);
                            const float h = __bfloat162float(__float2bfloat16_rn(v));
                            a0[j] = fmaf(h, s_head[c0 + j], a0[j]);
                            a1[j] = fmaf(h, s_head[W + c0 + j], a1[j]);
                        }
                    }
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
                        for (int j = 0; j < o; j++) {
                            a0[j] += a0[j + o];
                            a1[j] += a1[j + o];
                        }
                    float d0, d1;
                    float ls = loss_row(a0[0] + s_head[2 * W], a1[0] + s_head[2 * W + 1], a.target + 2 * q, a.x + 6 * q,
                                        a.B, a.scale, a.offset, a.lam, d0, d1);
                    s_dy[row] = make_float2(d0, d1);
                    for (int o = 16; o > 0; o >>= 1) ls += __shfl_xor_sync(0xffffffffu, ls, o);
                    if (lane == 0) atomicAdd(a.loss, ls / a.B);
                }
                asm volatile("bar.sync 1, 256;" ::: "memory");
                {
                    // this tile's part of the head's gradients, 64 rows at a time (see k_head_bwd)
                    const int half = tid >> 7, cc = 2 * (tid & 127);
                    if (cc < W) {
                        float s0 = 0.0f, s1 = 0.0f, s2 = 0.0f, s3 = 0.0f, e0 = 0.0f, e1 = 0.0f;
                        const uint8_t* col = act + (cc / 64) * 16384;
#pragma unroll 8
                        for (int r = 64 * half; r < 64 * half + 64; r++) {
                            const __nv_bfloat162 h2 = *(const __nv_bfloat162*)(col + sw128_off(r, cc % 64));
                            const float2 d = s_dy[r];
                            s0 = fmaf(d.x, __low2float(h2), s0);
                            s1 = fmaf(d.x, __high2float(h2), s1);
                            s2 = fmaf(d.y, __low2float(h2), s2);
                            s3 = fmaf(d.y, __high2float(h2), s3);
                            e0 += d.x;
                            e1 += d.y;
                        }
                        float* o = a.hpart + ((size_t)tile * 2 + half) * (2 * W + 2);
                        o[cc] = s0;
                        o[cc + 1] = s1;
                        o[W + cc] = s2;
                        o[W + cc + 1] = s3;
                        if (cc == 0) {
                            o[2 * W] = e0;
                            o[2 * W + 1] = e1;
                        }
                    }
                }
                asm volatile("bar.sync 1, 256;" ::: "memory");
                wait(stored, nst - 1);
                nst++;
                const float2 d = s_dy[row];
                for (int c = c_first; c < nc; c += 2) {
#pragma unroll
                    for (int hh = 0; hh < 2; hh++) {
                        if (nc == 1 && hh != g) continue;
                        const int c0 = 64 * c + 32 * hh;
                        const uint32_t bits = mk[(2 * c + hh) * 128];
#pragma unroll
                        for (int u = 0; u < 4; u++) {
                            uint32_t pk[4];
#pragma unroll
                            for (int v = 0; v < 4; v++) {
                                const int j = 8 * u + 2 * v;
                                const float gx = d.x * s_head[c0 + j] + d.y * s_head[W + c0 + j];
                                const float gy = d.x * s_head[c0 + j + 1] + d.y * s_head[W + c0 + j + 1];
                                pk[v] = pack_bf16(bits & (1u << j) ? gx : 0.0f, bits & (2u << j) ? gy : 0.0f);
                            }
                            *(uint4*)(act + c * 16384 + sw128_off(row, 32 * hh + 8 * u)) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
                        }
                    }
                    fence_async_smem();
                    tc_fence_before();
                    mbar_arrive((L == 1 ? only0 : chunk0) + 8 * c);
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, tcols);
}

// ------------------------------------------------------------- tensor maps
typedef CUresult (*EncodeTiled)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiled g_encode = nullptr;

bool load_encoder() {
    if (g_encode) return true;
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess || !fn) {
        cudaGetLastError();
        return false;
    }
    g_encode = (EncodeTiled)fn;
    return true;
}

// BF16 row-major [rows x cols] (cols % 8 == 0), box = 64 columns x box_rows
// rows with 128-byte swizzle, or 32 columns with 64-byte swizzle
bool make_map(CUtensorMap* m, const void* ptr, uint64_t rows, uint64_t cols, uint32_t box_rows, uint32_t box_cols = 64) {
    if (!load_encoder()) return false;
    cuuint64_t dims[2] = {cols, rows};
    cuuint64_t strides[1] = {cols * 2};
    cuuint32_t box[2] = {box_cols, box_rows};
    cuuint32_t es[2] = {1, 1};
    CUresult r = g_encode(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(ptr), dims, strides, box, es,
                          CU_TENSOR_MAP_INTERLEAVE_NONE,
                          box_cols == 32 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B,
                          CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

int pick_bn(int N) { return N <= 64 ? 64 : (N <= 128 ? 128 : 256); }

template <int BN>
size_t gemm_smem() {
    return (size_t)GSTAGES * (GM * GK * 2 + BN * GK * 2) + 1024;
}

template <int BN, bool MASK>
cudaError_t launch_gemm_m(cudaStream_t st, const CUtensorMap& ta, const CUtensorMap& tb, int M, int N, int K,
                          const float* bias, int relu, int out_bf16, void* C, int ldc, const void* mask,
                          unsigned* err) {
    size_t smem = gemm_smem<BN>();
    cudaError_t e = ensure_smem_attr((const void*)k_gemm<BN, MASK>, smem);
    if (e != cudaSuccess) return e;
    dim3 grid((unsigned)((M + GM - 1) / GM), (unsigned)((N + BN - 1) / BN));
    k_gemm<BN, MASK><<<grid, 128, smem, st>>>(ta, tb, M, N, K, bias, relu, out_bf16, C, ldc, (const __nv_bfloat16*)mask, err);
    return cudaGetLastError();
}
template <int BN>
cudaError_t launch_gemm_t(cudaStream_t st, const CUtensorMap& ta, const CUtensorMap& tb, int M, int N, int K,
                          const float* bias, int relu, int out_bf16, void* C, int ldc, const void* mask,
                          unsigned* err) {
    return (mask ? launch_gemm_m<BN, true> : launch_gemm_m<BN, false>)(st, ta, tb, M, N, K, bias, relu, out_bf16, C, ldc,
                                                                       mask, err);
}

}  // namespace

// C = act(A B^T + bias): A [M x K], B [N x K] BF16 row-major (device), M, N,
// K with K % 8 == 0 and N % 8 == 0 (TMA strides); C FP32 or BF16 [M x N].
cudaError_t gemm_bf16(cudaStream_t st, const void* A, const void* B, int M, int N, int K, const float* bias, int relu,
                      int out_bf16, void* C, int ldc, unsigned* err, const void* mask = nullptr) {
    const int BN = pick_bn(N);
    alignas(64) CUtensorMap ta, tb;
    if (!make_map(&ta, A, M, K, GM) || !make_map(&tb, B, N, K, BN)) return cudaErrorInvalidValue;
    if (BN == 64) return launch_gemm_t<64>(st, ta, tb, M, N, K, bias, relu, out_bf16, C, ldc, mask, err);
    if (BN == 128) return launch_gemm_t<128>(st, ta, tb, M, N, K, bias, relu, out_bf16, C, ldc, mask, err);
    return launch_gemm_t<256>(st, ta, tb, M, N, K, bias, relu, out_bf16, C, ldc, mask, err);
}

// ------------------------------------------------------------- MLP object
struct rt_mlp {
    int device = 0;
    cudaStream_t stream = nullptr;
    int F = 32, W = 256, L = 8;  // Fourier frequencies, width, hidden layers
    float db_scale = 20.0f, db_offset = -100.0f;
    float lam = 0.0f;            // free-space baseline wavelength (0 = none)
    std::string err;
    DevBuf Bf, lo, hi, errw, loss;
    // parameters, Adam moments and gradients, each one vector in the layout
    // of rt_mlp_get_params (without the Fourier matrix); BF16 copies W and
    // W^T of the hidden layers one after another
    DevBuf w, mom, var, g, wbf, wtbf;
    DevBuf H0, H;         // features [B x 2F]; hidden outputs [L][cap x W]
    DevBuf y, dy, dZ;     // dZ: [L][cap x W], gradients of the layers' inputs to the ReLU
    DevBuf hpart;         // partial sums of the head's gradients (k_head_bwd)
    int64_t cap = 0;      // rows of the activation buffers
    int64_t tcap = 0;     // rows of the training buffers
    int zl = 0;           // layers that dZ holds: L, or 2 in turn where memory has no room for all
    int step = 0;
    int in_dim(int l) const { return l == 0 ? 2 * F : W; }
    int out_dim(int l) const { return l == L ? 2 : W; }
    int64_t off(int l) const { return l == 0 ? 0 : (int64_t)W * 2 * F + W + (int64_t)(l - 1) * (W * W + W); }
    int64_t woff(int l) const { return off(l) - (int64_t)l * W; }   // weights alone
    int64_t n_w() const { return off(L) + 2 * W + 2; }
    float* wp(int l) { return bp<float>(w) + off(l); }
    float* bias(int l) { return wp(l) + (int64_t)in_dim(l) * out_dim(l); }
    __nv_bfloat16* hid(int l) { return l == 0 ? bp<__nv_bfloat16>(H0) : bp<__nv_bfloat16>(H) + (size_t)(l - 1) * cap * W; }
    __nv_bfloat16* wb(int l) { return bp<__nv_bfloat16>(wbf) + woff(l); }
    __nv_bfloat16* wtb(int l) { return bp<__nv_bfloat16>(wtbf) + woff(l); }
};

static int mlp_err(rt_mlp* m, int code, const std::string& s) {
    m->err = s;
    return code;
}
#define MT(expr)                                                                                  \
    do {                                                                                          \
        cudaError_t e_ = (expr);                                                                  \
        if (e_ != cudaSuccess) return mlp_err(m, e_ == cudaErrorMemoryAllocation ? RT_ERR_OOM : RT_ERR_CUDA, \
                                              std::string(#expr) + ": " + cudaGetErrorString(e_)); \
    } while (0)

static int mlp_reserve(rt_mlp* m, int64_t B) {
    if (B <= m->cap) return RT_OK;
    m->cap = 0;   // a failed reservation leaves nothing to use
    MT(buf_reserve(m->H0, sizeof(__nv_bfloat16) * B * 2 * m->F));
    MT(buf_reserve(m->H, sizeof(__nv_bfloat16) * B * m->W * m->L));
    MT(buf_reserve(m->y, sizeof(float) * 2 * B));
    m->cap = B;
    return RT_OK;
}

static int mlp_reserve_train(rt_mlp* m, int64_t B) {
    int rc = mlp_reserve(m, B);
    if (rc) return rc;
    if (m->cap <= m->tcap) return RT_OK;
    m->tcap = 0;
    MT(buf_reserve(m->dy, sizeof(float) * 2 * m->cap));
    MT(buf_reserve(m->hpart, sizeof(float) * (size_t)(m->cap / HB_ROWS + 1) * (2 * m->W + 2)));
    const size_t layer = sizeof(__nv_bfloat16) * (size_t)m->cap * m->W;
    m->zl = m->L;
    cudaError_t e = buf_reserve(m->dZ, layer * m->L);
    if (e == cudaErrorMemoryAllocation && m->L > 2) {
        m->zl = 2;
        e = buf_reserve(m->dZ, layer * 2);
    }
    MT(e);
    m->tcap = m->cap;
    return RT_OK;
}

static int mlp_forward(rt_mlp* m, const float* x, int64_t B) {
    cudaStream_t st = m->stream;
    unsigned* err = bp<unsigned>(m->errw);
    dim3 fb(32, 8);
    k_features<<<(unsigned)((B + 7) / 8), fb, 0, st>>>(x, B, bp<float>(m->Bf), m->F, bp<float>(m->lo),
                                                       bp<float>(m->hi), m->hid(0));
    MT(cudaGetLastError());
    for (int l = 0; l < m->L; l++)
        MT(gemm_bf16(st, m->hid(l), m->wb(l), (int)B, m->W, m->in_dim(l), m->bias(l), 1, 1, m->hid(l + 1), m->W,
                     err));
    k_head<<<(unsigned)((B + 7) / 8), 256, 0, st>>>(m->hid(m->L), B, m->W, m->wp(m->L), m->bias(m->L),
                                                    bp<float>(m->y));
    MT(cudaGetLastError());
    return RT_OK;
}

// BF16 copies of the FP32 weights
static void mlp_to_bf16(rt_mlp* m, cudaStream_t st) {
    k_to_bf16<<<(unsigned)((m->off(m->L) + 255) / 256), 256, 0, st>>>(bp<float>(m->w), m->W, 2 * m->F, m->L,
                                                                     bp<__nv_bfloat16>(m->wbf),
                                                                     bp<__nv_bfloat16>(m->wtbf));
}

// k_train_chain on a batch: hidden outputs, gradients of the layers, loss and
// the head's partial sums
static int launch_train_chain(rt_mlp* m, const float* x, const float* target, int B, float* loss, int NS) {
    const int W = m->W, L = m->L, K0 = 2 * m->F;
    alignas(64) TrainMaps t;
    bool ok = make_map(&t.w0, m->wb(0), W, K0, W) && make_map(&t.h0, m->H0.p, m->cap, K0, 128) &&
              make_map(&t.h, m->H.p, (uint64_t)L * m->cap, W, 128) && make_map(&t.z, m->dZ.p, (uint64_t)L * m->cap, W, 128);
    if (L > 1)
        ok = ok && make_map(&t.wx, m->wb(1), (uint64_t)(L - 1) * W, W, W) &&
             make_map(&t.wt, m->wtb(1), (uint64_t)(L - 1) * W, W, W);
    else
        t.wx = t.wt = t.w0;
    if (!ok) return mlp_err(m, RT_ERR_CUDA, "tensor map of the training buffers");
    TrainArgs a;
    a.x = x;
    a.target = target;
    a.B = B;
    a.F = m->F;
    a.W = W;
    a.L = L;
    a.NS = NS;
    a.Bf = bp<float>(m->Bf);
    a.lo = bp<float>(m->lo);
    a.hi = bp<float>(m->hi);
    a.params = bp<float>(m->w);
    a.scale = m->db_scale;
    a.offset = m->db_offset;
    a.lam = m->lam;
    a.loss = loss;
    a.hpart = bp<float>(m->hpart);
    a.cap = m->cap;
    a.err = bp<unsigned>(m->errw);
    const size_t smem = 1024 + TrainLayout(m->F, W, L, NS).bytes(NS);
    MT(ensure_smem_attr((const void*)k_train_chain, smem));
    int sms = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, m->device);
    k_train_chain<<<std::min(B / 128, sms), TC_THREADS, smem, m->stream>>>(t, a);
    MT(cudaGetLastError());
    return RT_OK;
}

extern "C" {

int rt_mlp_create(rt_mlp** out, int device, void* stream, int32_t n_freq, int32_t width, int32_t n_hidden,
                  float sigma, uint64_t seed, const float* lo_host, const float* hi_host) {
    if (!out || n_freq < 4 || n_freq % 4 || width < 64 || width > 256 || width % 64 || n_hidden < 1 ||
        n_hidden > 16 || !lo_host || !hi_host)
        return RT_ERR_INVALID_ARG;
    *out = nullptr;
    if (cudaSetDevice(device) != cudaSuccess) return RT_ERR_INVALID_ARG;
    rt_mlp* m = new rt_mlp();
    m->device = device;
    m->stream = (cudaStream_t)stream;
    m->F = n_freq;
    m->W = width;
    m->L = n_hidden;
    if (!load_encoder()) {
        delete m;
        return RT_ERR_CUDA;
    }
    std::mt19937_64 rng(seed);
    std::normal_distribution<float> nd(0.0f, sigma);
    std::vector<float> Bf(6 * n_freq);
    for (auto& v : Bf) v = nd(rng);
    int n = m->L + 1;
    int rc = RT_OK;
    auto up = [&](DevBuf& d, const std::vector<float>& h) -> int {
        if (buf_reserve(d, sizeof(float) * h.size()) != cudaSuccess) return RT_ERR_OOM;
        return cudaMemcpy(d.p, h.data(), sizeof(float) * h.size(), cudaMemcpyHostToDevice) == cudaSuccess ? RT_OK
                                                                                                          : RT_ERR_CUDA;
    };
    rc |= up(m->Bf, Bf);
    rc |= up(m->lo, std::vector<float>(lo_host, lo_host + 6));
    rc |= up(m->hi, std::vector<float>(hi_host, hi_host + 6));
    std::vector<float> wv(m->n_w(), 0.0f), zero(m->n_w(), 0.0f);
    for (int l = 0; l < n; l++) {
        int fi = m->in_dim(l), fo = m->out_dim(l);
        float bound = std::sqrt(6.0f / fi) * (l == m->L ? 0.1f : 1.0f);  // He-uniform; small head
        std::uniform_real_distribution<float> ud(-bound, bound);
        for (int64_t k = 0; k < (int64_t)fi * fo; k++) wv[m->off(l) + k] = ud(rng);
    }
    if (!rc) rc |= up(m->w, wv);
    if (!rc) rc |= up(m->mom, zero);
    if (!rc) rc |= up(m->var, zero);
    if (!rc) rc |= up(m->g, zero);
    const size_t nb = sizeof(__nv_bfloat16) * (size_t)m->woff(m->L);
    if (!rc && (buf_reserve(m->wbf, nb) != cudaSuccess || buf_reserve(m->wtbf, nb) != cudaSuccess)) rc = RT_ERR_OOM;
    if (!rc) mlp_to_bf16(m, nullptr);
    if (!rc && (buf_reserve(m->errw, 64) != cudaSuccess || buf_reserve(m->loss, 64) != cudaSuccess)) rc = RT_ERR_OOM;
    if (!rc) {
        cudaMemset(m->errw.p, 0, 64);
        if (cudaDeviceSynchronize() != cudaSuccess) rc = RT_ERR_CUDA;
    }
    if (rc) {
        rt_mlp_destroy(m);
        return rc < 0 ? rc : RT_ERR_CUDA;
    }
    *out = m;
    return RT_OK;
}

int rt_mlp_destroy(rt_mlp* m) {
    if (!m) return RT_OK;
    cudaSetDevice(m->device);
    if (m->stream) cudaStreamSynchronize(m->stream);
    for (DevBuf* d : {&m->Bf, &m->lo, &m->hi, &m->errw, &m->loss, &m->w, &m->mom, &m->var, &m->g, &m->wbf, &m->wtbf,
                      &m->H0, &m->H, &m->y, &m->dy, &m->dZ, &m->hpart})
        buf_free(*d);
    delete m;
    return RT_OK;
}

int rt_mlp_set_stream(rt_mlp* m, void* stream) {
    if (!m) return RT_ERR_INVALID_ARG;
    m->stream = (cudaStream_t)stream;
    return RT_OK;
}

int rt_mlp_last_error(const rt_mlp* m, char* buf, size_t len) {
    if (!m || !buf || !len) return RT_ERR_INVALID_ARG;
    size_t n = std::min(len - 1, m->err.size());
    memcpy(buf, m->err.data(), n);
    buf[n] = 0;
    return RT_OK;
}

int rt_mlp_infer(rt_mlp* m, const float* x, int64_t n, float* out) {
    if (!m || (n > 0 && (!x || !out))) return RT_ERR_INVALID_ARG;
    if (cudaSetDevice(m->device) != cudaSuccess) return RT_ERR_CUDA;
    if ((2 * m->F) % 64 || m->W % 64 || m->L > FM_MAX_L) return rt_mlp_infer_layers(m, x, n, out);
    if (n == 0) return RT_OK;
    alignas(64) FusedMaps maps;
    for (int l = 0; l < m->L; l++)
        if (!make_map(&maps.w[l], m->wb(l), m->W, m->in_dim(l), m->W))
            return mlp_err(m, RT_ERR_CUDA, "tensor map of a weight matrix");
    FusedArgs a;
    a.x = x;
    a.out = out;
    a.n = n;
    a.F = m->F;
    a.W = m->W;
    a.L = m->L;
    a.Bf = bp<float>(m->Bf);
    a.lo = bp<float>(m->lo);
    a.hi = bp<float>(m->hi);
    a.params = bp<float>(m->w);
    a.head_w = m->wp(m->L);
    a.head_b = m->bias(m->L);
    a.db_scale = m->db_scale;
    a.db_offset = m->db_offset;
    a.lam = m->lam;
    a.err = bp<unsigned>(m->errw);
    const size_t smem = 1024 + FusedLayout(m->F, m->W, m->L).bytes();
    if (smem > 227 * 1024) return rt_mlp_infer_layers(m, x, n, out);
    MT(ensure_smem_attr((const void*)k_mlp_fused, smem));
    int sms = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, m->device);
    int64_t npairs = ((n + 127) / 128 + 1) / 2;
    int grid = (int)std::min<int64_t>(npairs, sms);
    k_mlp_fused<<<grid, FM_THREADS, smem, m->stream>>>(maps, a);
    MT(cudaGetLastError());
    return RT_OK;
}

// Layer-by-layer inference through the generic GEMM (activations in HBM):
// the reference path the fused kernel is checked against.
int rt_mlp_infer_layers(rt_mlp* m, const float* x, int64_t n, float* out) {
    if (!m || (n > 0 && (!x || !out))) return RT_ERR_INVALID_ARG;
    if (cudaSetDevice(m->device) != cudaSuccess) return RT_ERR_CUDA;
    const int64_t chunk = 1 << 18;
    int rc = mlp_reserve(m, std::min<int64_t>(std::max<int64_t>(n, 128), chunk));
    if (rc) return rc;
    for (int64_t s = 0; s < n; s += chunk) {
        int64_t c = std::min(chunk, n - s);
        rc = mlp_forward(m, x + 6 * s, c);
        if (rc) return rc;
        k_head_out<<<(unsigned)((c + 255) / 256), 256, 0, m->stream>>>(bp<float>(m->y), x + 6 * s, c, m->db_scale,
                                                                       m->db_offset, m->lam, out + 2 * s);
        MT(cudaGetLastError());
    }
    return RT_OK;
}

int rt_mlp_set_baseline(rt_mlp* m, float wavelength) {
    if (!m || !(wavelength >= 0.0f)) return RT_ERR_INVALID_ARG;
    m->lam = wavelength;
    return RT_OK;
}

int rt_mlp_train_step(rt_mlp* m, const float* x, const float* target, int32_t B, float lr, float* loss_out) {
    if (!m || !x || !target || B < 128 || B % 128) return RT_ERR_INVALID_ARG;
    if (cudaSetDevice(m->device) != cudaSuccess) return RT_ERR_CUDA;
    const int W = m->W, L = m->L, K0 = 2 * m->F;
    int rc = mlp_reserve_train(m, B);
    if (rc) return rc;
    cudaStream_t st = m->stream;
    unsigned* err = bp<unsigned>(m->errw);
    float* loss = loss_out ? loss_out : bp<float>(m->loss);
    // one launch for forward, loss and backward chain where the features come
    // in whole 64-column chunks and the activations, the signs and two weight
    // slots fit in shared memory; else layer by layer
    int NS = 0;
    for (int n = 4; n >= 2 && !NS; n--)
        if (1024 + TrainLayout(m->F, W, L, n).bytes(n) <= 227 * 1024) NS = n;
    const bool all_dz = m->zl == L;
    // dW_l = dZ_l^T H_l and the bias gradients of all hidden layers, or of one
    WgradArgs wa;
    wa.W = W;
    wa.K0 = K0;
    wa.L = L;
    wa.B = B;
    wa.cap = m->cap;
    wa.g = bp<float>(m->g);
    wa.err = err;
    alignas(64) CUtensorMap tz, th0, th;
    if (!make_map(&tz, m->dZ.p, (uint64_t)m->zl * m->cap, W, WG_ROWS) ||
        !make_map(&th0, m->H0.p, m->cap, K0, WG_ROWS, WG_N) ||
        !make_map(&th, m->H.p, (uint64_t)L * m->cap, W, WG_ROWS, WG_N))
        return mlp_err(m, RT_ERR_CUDA, "tensor map of the training buffers");
    const size_t smem = 1024 + (size_t)WG_ST * WG_STAGE;
    MT(ensure_smem_attr((const void*)k_wgrad, smem));
    const int mt = (W + 127) / 128, nt0 = (K0 + WG_N - 1) / WG_N, nt1 = W / WG_N;
    auto wgrad = [&](int layer, int slot) -> cudaError_t {
        wa.layer = layer;
        wa.z0 = (int64_t)slot * m->cap;
        const int tiles = mt * (layer < 0 ? nt0 + (L - 1) * nt1 : layer == 0 ? nt0 : nt1);
        k_wgrad<<<(unsigned)tiles, 128, smem, st>>>(tz, th0, th, wa);
        return cudaGetLastError();
    };
    if (K0 % 64 == 0 && NS && all_dz) {
        rc = launch_train_chain(m, x, target, B, loss, NS);
        if (rc) return rc;
    } else {
        rc = mlp_forward(m, x, B);
        if (rc) return rc;
        k_loss<<<(B + 255) / 256, 256, 0, st>>>(bp<float>(m->y), target, x, B, m->db_scale, m->db_offset, m->lam,
                                               bp<float>(m->dy), loss);
        // where a layer's gradient lies
        auto slot = [&](int l) { return all_dz ? l : l & 1; };
        auto dz = [&](int l) { return bp<__nv_bfloat16>(m->dZ) + (size_t)slot(l) * m->cap * W; };
        k_head_bwd<<<B / HB_ROWS, W / 2, 0, st>>>(m->hid(L), bp<float>(m->dy), W, m->wp(L), dz(L - 1),
                                                  bp<float>(m->hpart));
        MT(cudaGetLastError());
        // dH_l = dZ_l W_l, then through the ReLU of layer l's input
        for (int l = L - 1; l >= 0; l--) {
            if (!all_dz) MT(wgrad(l, slot(l)));   // before the layer below the next takes its place
            if (l > 0) MT(gemm_bf16(st, dz(l), m->wtb(l), B, W, W, nullptr, 0, 1, dz(l - 1), W, err, m->hid(l)));
        }
    }
    if (all_dz) MT(wgrad(-1, 0));
    m->step++;
    AdamArgs aa;
    aa.W = W;
    aa.K0 = K0;
    aa.L = L;
    aa.hblocks = B / HB_ROWS;
    aa.w = bp<float>(m->w);
    aa.m = bp<float>(m->mom);
    aa.v = bp<float>(m->var);
    aa.g = bp<float>(m->g);
    aa.hpart = bp<float>(m->hpart);
    aa.wb = bp<__nv_bfloat16>(m->wbf);
    aa.wtb = bp<__nv_bfloat16>(m->wtbf);
    aa.lr = lr;
    aa.b1 = 0.9f;
    aa.b2 = 0.999f;
    aa.eps = 1e-8f;
    aa.c1 = 1.0f - std::pow(aa.b1, (float)m->step);
    aa.c2 = 1.0f - std::pow(aa.b2, (float)m->step);
    const int hb = (int)((m->off(L) + 255) / 256);
    k_adam<<<hb + (2 * W + 2 + 7) / 8, 256, 0, st>>>(aa, hb);
    MT(cudaGetLastError());
    return RT_OK;
}

int rt_mlp_num_params(const rt_mlp* m, int64_t* n) {
    if (!m || !n) return RT_ERR_INVALID_ARG;
    *n = m->n_w() + 6 * m->F;
    return RT_OK;
}

// Parameters as one FP32 vector: per layer W [out x in] then b [out], then
// the Fourier matrix [F x 6]. dir 0: model -> dst, 1: src -> model.
static int mlp_params(rt_mlp* m, float* p, int dir) {
    if (!m || !p) return RT_ERR_INVALID_ARG;
    if (cudaSetDevice(m->device) != cudaSuccess) return RT_ERR_CUDA;
    cudaStream_t st = m->stream;
    const size_t nw = (size_t)m->n_w();
    if (dir == 0) {
        MT(cudaMemcpyAsync(p, m->w.p, 4 * nw, cudaMemcpyDeviceToDevice, st));
        MT(cudaMemcpyAsync(p + nw, m->Bf.p, 4 * 6 * m->F, cudaMemcpyDeviceToDevice, st));
    } else {
        MT(cudaMemcpyAsync(m->w.p, p, 4 * nw, cudaMemcpyDeviceToDevice, st));
        MT(cudaMemcpyAsync(m->Bf.p, p + nw, 4 * 6 * m->F, cudaMemcpyDeviceToDevice, st));
        mlp_to_bf16(m, st);
    }
    MT(cudaGetLastError());
    return RT_OK;
}

int rt_mlp_get_params(rt_mlp* m, float* dst) { return mlp_params(m, dst, 0); }
int rt_mlp_set_params(rt_mlp* m, const float* src) { return mlp_params(m, const_cast<float*>(src), 1); }

// Serialised model (rt_mlp_save / rt_mlp_load), little-endian host bytes:
//   "RTMLP001" | int32 F, W, L, 0 | float lo[6], hi[6], lam, db_scale,
//   db_offset, 0 | int64 n_params | float params[n_params] (the
//   rt_mlp_get_params layout) | uint64 FNV-1a hash of everything before it.
namespace {
constexpr char MLP_MAGIC[8] = {'R', 'T', 'M', 'L', 'P', '0', '0', '1'};
constexpr size_t MLP_HDR = 8 + 4 * 4 + 16 * 4 + 8;

uint64_t fnv1a(const unsigned char* p, size_t n) {
    uint64_t h = 1469598103934665603ull;
    for (size_t i = 0; i < n; i++) {
        h ^= p[i];
        h *= 1099511628211ull;
    }
    return h;
}
}  // namespace

int rt_mlp_save(rt_mlp* m, void* buf, int64_t cap, int64_t* size_out) {
    if (!m || !size_out) return RT_ERR_INVALID_ARG;
    int64_t np = 0;
    rt_mlp_num_params(m, &np);
    const size_t need = MLP_HDR + 4 * (size_t)np + 8;
    *size_out = (int64_t)need;
    if (!buf) return RT_OK;
    if (cap < (int64_t)need) return mlp_err(m, RT_ERR_CAPACITY, "mlp_save: buffer smaller than the size query");
    if (cudaSetDevice(m->device) != cudaSuccess) return RT_ERR_CUDA;
    unsigned char* out = (unsigned char*)buf;
    std::memcpy(out, MLP_MAGIC, 8);
    const int32_t dims[4] = {m->F, m->W, m->L, 0};
    std::memcpy(out + 8, dims, sizeof(dims));
    float box[16] = {0};
    MT(cudaMemcpyAsync(box, m->lo.p, 24, cudaMemcpyDeviceToHost, m->stream));
    MT(cudaMemcpyAsync(box + 6, m->hi.p, 24, cudaMemcpyDeviceToHost, m->stream));
    float* params = (float*)(out + MLP_HDR);
    const int64_t nw = m->n_w();
    MT(cudaMemcpyAsync(params, m->w.p, 4 * (size_t)nw, cudaMemcpyDeviceToHost, m->stream));
    MT(cudaMemcpyAsync(params + nw, m->Bf.p, 4 * 6 * m->F, cudaMemcpyDeviceToHost, m->stream));
    MT(cudaStreamSynchronize(m->stream));
    box[12] = m->lam;
    box[13] = m->db_scale;
    box[14] = m->db_offset;
    std::memcpy(out + 8 + 16, box, sizeof(box));
    std::memcpy(out + 8 + 16 + 64, &np, 8);
    const uint64_t h = fnv1a(out, need - 8);
    std::memcpy(out + need - 8, &h, 8);
    return RT_OK;
}

int rt_mlp_load(rt_mlp** out, int device, void* cuda_stream, const void* buf, int64_t size) {
    if (!out || !buf || size < (int64_t)(MLP_HDR + 8)) return RT_ERR_INVALID_ARG;
    *out = nullptr;
    const unsigned char* in = (const unsigned char*)buf;
    if (std::memcmp(in, MLP_MAGIC, 8) != 0) return RT_ERR_INVALID_ARG;
    int32_t dims[4];
    float box[16];
    int64_t np = 0;
    std::memcpy(dims, in + 8, sizeof(dims));
    std::memcpy(box, in + 8 + 16, sizeof(box));
    std::memcpy(&np, in + 8 + 16 + 64, 8);
    if (np < 0 || size != (int64_t)(MLP_HDR + 4 * (size_t)np + 8)) return RT_ERR_INVALID_ARG;
    uint64_t h = 0;
    std::memcpy(&h, in + size - 8, 8);
    if (h != fnv1a(in, (size_t)size - 8)) return RT_ERR_INVALID_ARG;
    rt_mlp* m = nullptr;
    int rc = rt_mlp_create(&m, device, cuda_stream, dims[0], dims[1], dims[2], 1.0f, 0, box, box + 6);
    if (rc) return rc;
    int64_t want = 0;
    rt_mlp_num_params(m, &want);
    if (want != np) {
        rt_mlp_destroy(m);
        return RT_ERR_INVALID_ARG;
    }
    DevBuf tmp;
    if (buf_reserve(tmp, 4 * (size_t)np) != cudaSuccess) {
        rt_mlp_destroy(m);
        return RT_ERR_OOM;
    }
    cudaError_t e = cudaMemcpy(tmp.p, in + MLP_HDR, 4 * (size_t)np, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) rc = mlp_params(m, bp<float>(tmp), 1);
    if (e == cudaSuccess && !rc) e = cudaStreamSynchronize(m->stream);
    buf_free(tmp);
    if (e != cudaSuccess || rc) {
        rt_mlp_destroy(m);
        return rc ? rc : RT_ERR_CUDA;
    }
    m->lam = box[12];
    m->db_scale = box[13];
    m->db_offset = box[14];
    *out = m;
    return RT_OK;
}

// Gradients of the last rt_mlp_train_step (before its Adam update), same
// layout as the parameters (Fourier matrix entries are 0: not trained).
int rt_mlp_get_grads(rt_mlp* m, float* dst) {
    if (!m || !dst) return RT_ERR_INVALID_ARG;
    if (cudaSetDevice(m->device) != cudaSuccess) return RT_ERR_CUDA;
    MT(cudaMemcpyAsync(dst, m->g.p, 4 * (size_t)m->n_w(), cudaMemcpyDeviceToDevice, m->stream));
    MT(cudaMemsetAsync(dst + m->n_w(), 0, 4 * 6 * m->F, m->stream));
    return RT_OK;
}

int rt_mlp_status(rt_mlp* m, uint32_t* status) {
    if (!m || !status) return RT_ERR_INVALID_ARG;
    MT(cudaMemcpy(status, m->errw.p, 4, cudaMemcpyDeviceToHost));
    return RT_OK;
}

int rt_gemm_bf16(void* stream, const void* A, const void* B, int32_t M, int32_t N, int32_t K, const float* bias,
                 int32_t relu, int32_t out_bf16, void* C, uint32_t* status) {
    if (!A || !B || !C || M < 1 || N < 8 || K < 8 || N % 8 || K % 8) return RT_ERR_INVALID_ARG;
    cudaError_t e = gemm_bf16((cudaStream_t)stream, A, B, M, N, K, bias, relu, out_bf16, C, N, status);
    return e == cudaSuccess ? RT_OK : RT_ERR_CUDA;
}

}  // extern "C"
