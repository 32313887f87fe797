// sph_mlp.cu -- the boid-force surrogate: a 272 -> 256 -> 256 -> 256 -> 16
// MLP (exact-erf GELU) whose inference (k_mlp_fused; small batches
// k_train_rows) and training (k_train_*) run on the tensor cores
// (tcgen05.mma kind::f16: BF16 operands staged by TMA, FP32 accumulators in
// tensor memory), with Adam on FP32 master weights.
//
// The surrogate is not in the paper; it predicts the fluid force the SPH
// coupling of section "Boid Motion and Agent Fluid Interaction" puts on a
// boid (F_b in v_b += sph_factor dt F_b) from the flow around the boid.
//
// Layout: a layer's weight W is [out][in] (K-major for the B operand of the
// forward products) with a transposed BF16 copy W^T [in][out] for the
// backward ones; activations are [batch][features] with transposed copies
// [features][batch] for the weight gradients (which contract over the
// batch).  Every product is C[M][N] = A[M][K] . B[N][K]^T with both operands
// K-major.
#include <cudaTypedefs.h>
#include <math.h>
#include <stdarg.h>
#include <stdio.h>
#include <string.h>

#include <mutex>
#include <new>

#include "sph_umma.cuh"

namespace sphk {

constexpr int BM = 128;  // rows per tile (UMMA M)
constexpr int BK = 64;   // K elements per pipeline stage (one 128-byte row)
constexpr int UK = 16;   // K per tcgen05.mma of kind::f16

struct GemmEpi {
    int M, N;                 // valid rows / columns of C
    int kb_total;             // K blocks of BK
    int kb_per_split;         // K blocks per blockIdx.z
    float* out_f32;           // [M][ld_f32] + blockIdx.z * split_stride
    int ld_f32;
    long long split_stride;
    unsigned* err;
};

// Phi(-|z|) = erfc(|z| / sqrt 2) / 2, the standard normal lower tail, by
// formula 7.1.26 of Abramowitz and Stegun, "Handbook of Mathematical
// Functions": erfc x = t (a1 + t (a2 + t (a3 + t (a4 + t a5)))) exp(-x^2),
// t = 1 / (1 + p x), x >= 0, absolute error <= 1.5e-7 (here with x =
// |z| / sqrt 2: p / sqrt 2 and a_k / 2 folded into the constants).
// Evaluated in float32 with the hardware reciprocal and exponential
// approximations, which add a few 1e-7: far below the BF16 rounding of the
// activations (2^-9 relative).  The GELU epilogue bounds the fused forward
// pass; this form takes about half the instructions of the library erff.
// Also returns exp(-z^2 / 2) for the derivative.
__device__ __forceinline__ float phi_lower(float z, float* gauss)
{
    const float az = fabsf(z);
    const float t = __fdividef(1.0f, fmaf(0.23164190f, az, 1.0f));  // p / sqrt 2 = 0.3275911 / 1.41421356
    float poly = fmaf(t, 0.5307027145f, -0.7265760135f);            // a_k / 2
    poly = fmaf(t, poly, 0.7107068705f);
    poly = fmaf(t, poly, -0.142248368f);
    poly = fmaf(t, poly, 0.127414796f);
    poly *= t;
    const float e = __expf(-0.5f * z * z);
    *gauss = e;
    return poly * e;
}

// GELU(z) = z Phi(z) and its derivative Phi(z) + z phi(z), phi the standard
// normal density, with Phi(z) = 1 - Phi(-z) for z >= 0.
__device__ __forceinline__ float gelu_f(float z)
{
    float e;
    const float lt = phi_lower(z, &e);
    return z * (z >= 0.0f ? 1.0f - lt : lt);
}

__device__ __forceinline__ float gelu_grad_f(float z)
{
    float e;
    const float lt = phi_lower(z, &e);
    return (z >= 0.0f ? 1.0f - lt : lt) + z * e * 0.39894228040143268f;
}

// GELU of two values with the packed FP32x2 instructions (the fused
// forward's epilogue): the same formula as gelu_f, with
// exp(-z^2 / 2) = 2^(-z^2 log2(e) / 2) on the hardware base-2 exponential
// and Phi(z) = 1/2 + sign(z) (1/2 - Phi(-|z|)), the sign bit of z moved onto
// the bracket, so that each step but the reciprocal and the exponential
// works on both values at once.
__device__ __forceinline__ float ex2_approx(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ float2 gelu2_f(float2 z)
{
    const float2 az = make_float2(fabsf(z.x), fabsf(z.y));
    const float2 d = __ffma2_rn(make_float2(0.23164190f, 0.23164190f), az, make_float2(1.0f, 1.0f));
    const float2 t = make_float2(__fdividef(1.0f, d.x), __fdividef(1.0f, d.y));
    float2 poly = __ffma2_rn(t, make_float2(0.5307027145f, 0.5307027145f), make_float2(-0.7265760135f, -0.7265760135f));
    poly = __ffma2_rn(t, poly, make_float2(0.7107068705f, 0.7107068705f));
    poly = __ffma2_rn(t, poly, make_float2(-0.142248368f, -0.142248368f));
    poly = __ffma2_rn(t, poly, make_float2(0.127414796f, 0.127414796f));
    poly = __fmul2_rn(poly, t);
    // -z^2 log2(e) / 2
    const float2 a = __fmul2_rn(__fmul2_rn(z, make_float2(-0.72134752f, -0.72134752f)), z);
    const float2 e = make_float2(ex2_approx(a.x), ex2_approx(a.y));
    const float2 lt = __fmul2_rn(poly, e);                                              // Phi(-|z|)
    const float2 hb = __ffma2_rn(lt, make_float2(-1.0f, -1.0f), make_float2(0.5f, 0.5f));  // 1/2 - Phi(-|z|)
    const float2 sh = make_float2(__uint_as_float(__float_as_uint(hb.x) ^ (__float_as_uint(z.x) & 0x80000000u)),
                                  __uint_as_float(__float_as_uint(hb.y) ^ (__float_as_uint(z.y) & 0x80000000u)));
    return __fmul2_rn(z, __fadd2_rn(sh, make_float2(0.5f, 0.5f)));
}

__global__ void k_debug_gelu(const float* __restrict__ z, int n, int grad, float* __restrict__ out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    if (grad == 2) {
        out[i] = gelu2_f(make_float2(z[i], 0.0f)).x;
        return;
    }
    out[i] = grad ? gelu_grad_f(z[i]) : gelu_f(z[i]);
}

// Epilogue, in column chunks of EC (32, or NT when NT < 32), through shared
// memory so that every global store is a coalesced row segment: each thread
// (one accumulator row) writes EC columns from TMEM to the FP32 staging tile
// F[128][EC + 4], then the CTA walks F with 4 consecutive columns per thread.
template <int NT>
struct EpiShape {
    static constexpr int EC = NT < 32 ? NT : 32;   // columns per chunk
    static constexpr int FLD = EC + 4;               // F row stride (floats)
    static constexpr uint32_t BYTES = BM * FLD * 4;
};

template <int NT>
__device__ __forceinline__ void gemm_epilogue(const GemmEpi& e, uint32_t tmem, int m0, int n0, uint8_t* stage)
{
    using S = EpiShape<NT>;
    constexpr int EC = S::EC, FLD = S::FLD;
    float* F = reinterpret_cast<float*>(stage);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int r_own = warp * 32 + lane;
    constexpr int TPR = EC / 4;          // threads per row
    constexpr int RPP = 128 / TPR;       // rows per pass of the CTA
#pragma unroll 1
    for (int c0 = 0; c0 < NT; c0 += EC) {
#pragma unroll
        for (int h = 0; h < EC; h += 16) {
            float v[16];
            tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(c0 + h), v);
            // float4 stores: the 8 lanes of one store phase hit 32 distinct banks
#pragma unroll
            for (int j = 0; j < 16; j += 4)
                *reinterpret_cast<float4*>(F + r_own * FLD + h + j) = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
        }
        __syncthreads();
        const int cq = (threadIdx.x % TPR) * 4;
        const int n = n0 + c0 + cq;
#pragma unroll 1
        for (int r = threadIdx.x / TPR; r < BM; r += RPP) {
            const int row = m0 + r;
            const float4 x = *reinterpret_cast<const float4*>(F + r * FLD + cq);
            if (row < e.M && n < e.N)
                *reinterpret_cast<float4*>(e.out_f32 + (size_t)blockIdx.z * e.split_stride + (size_t)row * e.ld_f32 + n) = x;
        }
        __syncthreads();
    }
}

template <int NT, int STAGES>
struct GemmSmem {
    static constexpr uint32_t A_BYTES = BM * BK * 2;
    static constexpr uint32_t B_BYTES = NT * BK * 2;
    static constexpr uint32_t STAGE = A_BYTES + B_BYTES;
    static constexpr uint32_t TILES = STAGES * STAGE > EpiShape<NT>::BYTES ? STAGES * STAGE : EpiShape<NT>::BYTES;
    static constexpr uint32_t TOTAL = 1024 + TILES + 8 * (2 * STAGES + 1) + 16;
    static constexpr uint32_t TMEM_COLS = NT < 32 ? 32 : NT;
};

// For the consumer of a ring of stages that gave up at copy `first` of `total`:
// let the copies that may be in flight by then land, within the waits' limit.
// The loader may have issued its last ones and be done, and the block must not
// go away under them; a loader that gives up waits for its own.
// (Out of line, so that the kernels' loops are compiled as without it.)
__device__ __noinline__ void drain_ring(int stages, int first, int total, uint32_t full0, unsigned* err)
{
    for (int i = first; i < min(total, first + stages); ++i)
        mbar_wait(full0 + 8u * (uint32_t)(i % stages), (uint32_t)(i / stages) & 1u, err);
}

// A product by itself, C = A B^T: only sph_debug_gemm launches it (the network
// runs in k_mlp_fused and k_train_*).
// One CTA of 128 threads per (M tile, N tile, K split).  Warp 0 lane 0
// streams the A and B tiles through a STAGES-deep TMA ring, warp 1 lane 0
// issues the tcgen05.mma and frees each stage with tcgen05.commit, and all
// four warps read the 128 x NT FP32 accumulator out of tensor memory (warp
// w owns rows 32w .. 32w+31) for the epilogue.  Every wait is bounded; on a
// timeout the kernel records SPH_DEV_TIMEOUT, lets its own copies land,
// frees its tensor memory and returns.
template <int NT, int STAGES>
__global__ void __launch_bounds__(128, 2)
k_gemm(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB, GemmEpi e)
{
    using L = GemmSmem<NT, STAGES>;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t tiles = (raw + 1023u) & ~1023u;
    const uint32_t bars = tiles + L::TILES;
    auto full = [&](int s) { return bars + 8u * (uint32_t)s; };
    auto empty = [&](int s) { return bars + 8u * (uint32_t)(STAGES + s); };
    const uint32_t done = bars + 8u * (uint32_t)(2 * STAGES);
    const uint32_t tmem_slot = done + 8u;
    uint32_t* tmem_slot_ptr = reinterpret_cast<uint32_t*>(smem_raw + (tmem_slot - raw));

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int m0 = blockIdx.x * BM, n0 = blockIdx.y * NT;
    const int kb0 = blockIdx.z * e.kb_per_split;
    const int nk = min(e.kb_per_split, e.kb_total - kb0);

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(full(s), 1);
            mbar_init(empty(s), 1);
        }
        mbar_init(done, 1);
        mbar_fence_init();
    }
    if (warp == 0) tmem_alloc(tmem_slot, L::TMEM_COLS);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot_ptr;

    if (warp == 0 && lane == 0) {
        // ---- TMA producer
        int issued = 0;
        bool ok = true;
        for (int i = 0; i < nk; ++i) {
            const int s = i % STAGES;
            if (i >= STAGES && !mbar_wait(empty(s), (uint32_t)((i / STAGES) - 1) & 1u, e.err)) {
                ok = false;
                break;
            }
            const uint32_t a = tiles + (uint32_t)s * L::STAGE;
            mbar_expect_tx(full(s), L::STAGE);
            tma_load_2d(&mapA, full(s), a, (kb0 + i) * BK, m0);
            tma_load_2d(&mapB, full(s), a + L::A_BYTES, (kb0 + i) * BK, n0);
            ++issued;
        }
        if (!ok) {
            // let the copies still in flight land before the CTA goes away
            for (int i = max(0, issued - STAGES); i < issued; ++i)
                mbar_wait(full(i % STAGES), (uint32_t)(i / STAGES) & 1u, e.err);
        }
    } else if (warp == 1 && lane == 0) {
        // ---- MMA issuer
        constexpr uint32_t idesc = umma_idesc_bf16(BM, NT);
        for (int i = 0; i < nk; ++i) {
            const int s = i % STAGES;
            if (!mbar_wait(full(s), (uint32_t)(i / STAGES) & 1u, e.err)) {
                drain_ring(STAGES, i, nk, full(0), e.err);
                break;
            }
            tc_fence_after();
            const uint32_t a = tiles + (uint32_t)s * L::STAGE;
            const uint32_t b = a + L::A_BYTES;
#pragma unroll
            for (int k = 0; k < BK / UK; ++k)
                umma_bf16(tmem, sw128_desc(a + k * UK * 2), sw128_desc(b + k * UK * 2), idesc,
                          (uint32_t)((i | k) != 0));
            umma_commit(empty(s));
        }
        umma_commit(done);
    }
    __syncwarp();

    // ---- epilogue (the stage buffers are idle once every MMA completed)
    const bool ok = mbar_wait(done, 0, e.err);
    tc_fence_after();
    // the CTA agrees on ok, so that the barriers inside are reached by all
    if (__syncthreads_and(ok ? 1 : 0))
        gemm_epilogue<NT>(e, tmem, m0, n0, smem_raw + (tiles - raw));
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, L::TMEM_COLS);
}

// ------------------------------------------------------------ host side

static PFN_cuTensorMapEncodeTiled_v12000 g_encode = nullptr;
static std::mutex g_encode_mutex;

static cudaError_t get_encoder()
{
    std::lock_guard<std::mutex> lock(g_encode_mutex);
    if (g_encode) return cudaSuccess;
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult q;
    cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q);
    if (e != cudaSuccess) return e;
    if (q != cudaDriverEntryPointSuccess || !fn) return cudaErrorNotSupported;
    g_encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
    return cudaSuccess;
}

// Tensor map of a row-major BF16 matrix [rows][cols] (row stride ld
// elements), boxes of 64 columns x box_rows rows, 128-byte swizzle,
// out-of-range elements read as zero.
static cudaError_t make_map(CUtensorMap* map, const void* ptr, int rows, int cols, int ld, int box_rows)
{
    cudaError_t e = get_encoder();
    if (e != cudaSuccess) return e;
    cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
    cuuint32_t box[2] = {(cuuint32_t)BK, (cuuint32_t)box_rows};
    cuuint32_t elem[2] = {1, 1};
    auto encode = [&] {
        return g_encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(ptr), dims, strides, box, elem,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                        CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    };
    CUresult r = encode();
    if (r != CUDA_SUCCESS) {
        // the encoder needs a current context, which a host thread without a
        // launch or a copy so far has not: bind its device's
        int dev = 0;
        if ((e = cudaGetDevice(&dev)) != cudaSuccess || (e = cudaSetDevice(dev)) != cudaSuccess) return e;
        r = encode();
    }
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

template <int NT>
static cudaError_t launch_gemm_t(const CUtensorMap& ma, const CUtensorMap& mb, const GemmEpi& e, int splits,
                                 cudaStream_t s)
{
    constexpr int STAGES = NT >= 256 ? 4 : 6;
    using L = GemmSmem<NT, STAGES>;
    static bool attr = false;
    if (!attr) {
        cudaError_t r = cudaFuncSetAttribute(k_gemm<NT, STAGES>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)L::TOTAL);
        if (r != cudaSuccess) return r;
        attr = true;
    }
    dim3 grid((e.M + BM - 1) / BM, (e.N + NT - 1) / NT, splits);
    k_gemm<NT, STAGES><<<grid, 128, L::TOTAL, s>>>(ma, mb, e);
    return cudaGetLastError();
}

// C[M][N] = A[M][K] . B[N][K]^T; A, B row-major BF16 with leading
// dimensions lda, ldb (elements, multiples of 8).  NT chooses the N tile.
static cudaError_t gemm(int NT, const __nv_bfloat16* A, int lda, const __nv_bfloat16* B, int ldb, int M,
                        int N, int K, int splits, GemmEpi e, cudaStream_t s, long long* launches)
{
    CUtensorMap ma, mb;
    cudaError_t r = make_map(&ma, A, M, K, lda, BM);
    if (r != cudaSuccess) return r;
    r = make_map(&mb, B, N, K, ldb, NT);
    if (r != cudaSuccess) return r;
    e.M = M;
    e.N = N;
    e.kb_total = (K + BK - 1) / BK;
    splits = splits < 1 ? 1 : (splits > e.kb_total ? e.kb_total : splits);
    e.kb_per_split = (e.kb_total + splits - 1) / splits;
    splits = (e.kb_total + e.kb_per_split - 1) / e.kb_per_split;
    ++*launches;
    if (NT == 16) return launch_gemm_t<16>(ma, mb, e, splits, s);
    if (NT == 128) return launch_gemm_t<128>(ma, mb, e, splits, s);
    if (NT == 256) return launch_gemm_t<256>(ma, mb, e, splits, s);
    return cudaErrorInvalidValue;
}

// ---------------------------------------------------------- MLP kernels

constexpr int MLP_IN = SPH_MLP_IN, MLP_H = SPH_MLP_HIDDEN, MLP_OUT = SPH_MLP_OUT;

// Offsets of the packed parameter vector: W1 b1 W2 b2 W3 b3 W4 b4.
struct ParamLayout {
    int w[4], b[4], wn[4], in[4], out[4];
    __host__ __device__ ParamLayout()
    {
        const int ins[4] = {MLP_IN, MLP_H, MLP_H, MLP_H}, outs[4] = {MLP_H, MLP_H, MLP_H, MLP_OUT};
        int o = 0;
        for (int l = 0; l < 4; ++l) {
            in[l] = ins[l];
            out[l] = outs[l];
            w[l] = o;
            wn[l] = ins[l] * outs[l];
            o += wn[l];
            b[l] = o;
            o += outs[l];
        }
    }
};

// fp32 master -> BF16 W [out][in] and W^T [in][out] for every layer.
__global__ void k_cast_weights(const float* __restrict__ P, __nv_bfloat16* __restrict__ W,
                               __nv_bfloat16* __restrict__ WT)
{
    const ParamLayout L;
    const int total = L.b[3] + MLP_OUT;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < total; t += gridDim.x * blockDim.x) {
        for (int l = 0; l < 4; ++l) {
            if (t >= L.w[l] && t < L.w[l] + L.wn[l]) {
                const int r = (t - L.w[l]) / L.in[l], c = (t - L.w[l]) % L.in[l];
                const __nv_bfloat16 v = __float2bfloat16_rn(P[t]);
                W[t] = v;
                WT[L.w[l] + c * L.out[l] + r] = v;
            }
        }
    }
}

// ------------------------------------------------------------- fused forward

// The forward pass of 128-row tiles (inference), one persistent CTA per SM
// with two tiles in flight (slots 0 and 1), so that the tensor cores work
// on one tile while the epilogue works on the other.  Per slot the input
// tile and then each hidden layer's output stay in one shared-memory buffer
// in the layout the tensor cores read (K-major, 64-column tiles of 128-byte
// rows with the 128-byte swizzle that TMA writes): a layer's epilogue
// starts once that layer's MMAs have completed, so it writes its output
// over its input.  Each slot has a 128 x 256 FP32 accumulator in tensor
// memory (columns 256 j ..).  The 17 weight tiles of the four layers stream
// through a two-stage TMA ring, once per tile and layer.  Warp 16 loads,
// warp 17 issues the MMAs, warps 0 .. 15 are the epilogue (warp w reads
// tensor-memory lanes 32 (w % 4) .. and, in each 64-column K tile, the 16
// columns 16 (w / 4) ..): bias, GELU, BF16, written straight into the next
// layer's operand tile; the last layer's 16 columns go to y with their
// bias.  All three take the work items (tile pair, layer, slot) in the
// same order: for each pair of tiles, layer by layer, slot 0 then slot 1,
// so the MMAs of one slot's next layer run during the epilogue of the
// other slot's current layer.  The K order and the epilogue arithmetic are
// those of per-layer GEMMs.  Every wait is bounded.
namespace fused {
constexpr int KB_IN = (MLP_IN + BK - 1) / BK;   // 5 K tiles of the input
constexpr int KB_H = MLP_H / BK;                // 4 K tiles of a hidden layer
constexpr uint32_t A_TILE = BM * BK * 2;        // 16 KB: 128 rows x 64 BF16
constexpr uint32_t W_TILE = MLP_H * BK * 2;     // 32 KB: 256 rows x 64 BF16
constexpr uint32_t BUF = KB_IN * A_TILE;        // 80 KB per slot: the input, then each layer's output
constexpr uint32_t RING = 2 * BUF;
constexpr int STAGES = 2;
constexpr uint32_t BARS = RING + STAGES * W_TILE;
// barriers: full[2], empty[2], then per slot x_full, buf_free, acc_full,
// epi_done; then the TMEM slot
constexpr uint32_t TOTAL = 1024 + BARS + 8 * 12 + 16;
constexpr int EPI_WARPS = 16;
constexpr int LOAD_WARP = EPI_WARPS, MMA_WARP = EPI_WARPS + 1;
constexpr int THREADS = 32 * (EPI_WARPS + 2);
constexpr int EPI_THREADS = 32 * EPI_WARPS;
}  // namespace fused

// byte offset of element (r, c) in a K-major 64-column tile with 128-byte swizzle
__device__ __forceinline__ uint32_t sw128_offset(int r, int c)
{
    return (uint32_t)(r * 128 + ((((c * 2) >> 4) ^ (r & 7)) << 4) + ((c * 2) & 15));
}

__global__ void __launch_bounds__(fused::THREADS, 1)
k_mlp_fused(const __grid_constant__ CUtensorMap mapX, const __grid_constant__ CUtensorMap mapW0,
            const __grid_constant__ CUtensorMap mapW1, const __grid_constant__ CUtensorMap mapW2,
            const __grid_constant__ CUtensorMap mapW3, const float* __restrict__ P, int B, float* __restrict__ y,
            unsigned* __restrict__ err)
{
    using namespace fused;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    uint8_t* gbase = smem_raw + (base - raw);
    const uint32_t bars = base + BARS;
    auto full = [&](int s) { return bars + 8u * (uint32_t)s; };
    auto empty = [&](int s) { return bars + 16u + 8u * (uint32_t)s; };
    // slot j: its input tile landed; its buffer read by its last layer's
    // MMAs; its accumulator complete; its epilogue done (every epilogue
    // thread arrives: the layer's output written, the accumulator read)
    auto x_full = [&](int j) { return bars + 32u + 32u * (uint32_t)j; };
    auto buf_free = [&](int j) { return bars + 40u + 32u * (uint32_t)j; };
    auto acc_full = [&](int j) { return bars + 48u + 32u * (uint32_t)j; };
    auto epi_done = [&](int j) { return bars + 56u + 32u * (uint32_t)j; };
    const uint32_t tmem_slot = bars + 96;
    uint32_t* tmem_slot_ptr = reinterpret_cast<uint32_t*>(gbase + BARS + 96);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const ParamLayout L;

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(full(s), 1);
            mbar_init(empty(s), 1);
        }
        for (int j = 0; j < 2; ++j) {
            mbar_init(x_full(j), 1);
            mbar_init(buf_free(j), 1);
            mbar_init(acc_full(j), 1);
            mbar_init(epi_done(j), EPI_THREADS);
        }
        mbar_fence_init();
    }
    if (warp == LOAD_WARP) tmem_alloc(tmem_slot, 2 * MLP_H);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot_ptr;

    // tiles of this CTA: t = blockIdx.x + i gridDim.x, i = 0 .. ntl - 1; tile
    // i sits in slot i & 1 as that slot's (i >> 1)-th tile.  Work item it =
    // 8 p + 2 l + j: pair p, layer l, slot j (tile 2 p + j, skipped past
    // ntl).  Per slot, its barriers complete one phase per tile (x_full,
    // buf_free) or per tile and layer (acc_full, epi_done: parity l & 1),
    // and none can run two phases ahead of its waiter: each next phase
    // needs an action that follows the wait on the current one.
    const int ntiles = (B + BM - 1) / BM;
    const int ntl = blockIdx.x < ntiles ? (ntiles - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
    const int items = 8 * ((ntl + 1) / 2);
    auto tile_row = [&](int i) { return ((int)blockIdx.x + i * (int)gridDim.x) * BM; };

    if (warp == LOAD_WARP) {
        if (lane == 0) {
            // ---- loads, in work-item order: a slot's input tile before its
            // layer 0 (once the slot's previous tile has left the buffer),
            // then the item's weight tiles
            int g = 0, nx[2] = {0, 0};  // weight tiles, input tiles per slot issued
            bool ok = true;
            for (int it = 0; it < items && ok; ++it) {
                const int p = it >> 3, l = (it >> 1) & 3, j = it & 1, i = 2 * p + j;
                if (i >= ntl) continue;
                if (l == 0) {
                    if (p > 0 && !mbar_wait(buf_free(j), (uint32_t)(p - 1) & 1u, err)) {
                        ok = false;
                        break;
                    }
                    mbar_expect_tx(x_full(j), KB_IN * A_TILE);
                    for (int kb = 0; kb < KB_IN; ++kb)
                        tma_load_2d(&mapX, x_full(j), base + j * BUF + kb * A_TILE, kb * BK, tile_row(i));
                    ++nx[j];
                }
                const CUtensorMap* map = l == 0 ? &mapW0 : l == 1 ? &mapW1 : l == 2 ? &mapW2 : &mapW3;
                const uint32_t bytes = l == 3 ? MLP_OUT * BK * 2 : W_TILE;
                const int nkb = l == 0 ? KB_IN : KB_H;
                for (int kb = 0; kb < nkb; ++kb, ++g) {
                    const int s = g % STAGES;
                    if (g >= STAGES && !mbar_wait(empty(s), (uint32_t)((g / STAGES) - 1) & 1u, err)) {
                        ok = false;
                        break;
                    }
                    mbar_expect_tx(full(s), bytes);
                    tma_load_2d(map, full(s), base + RING + s * W_TILE, kb * BK, 0);
                }
            }
            if (!ok) {  // let the copies in flight land before the CTA goes away
                for (int h = (g > STAGES ? g - STAGES : 0); h < g; ++h)
                    mbar_wait(full(h % STAGES), (uint32_t)(h / STAGES) & 1u, err);
                for (int j = 0; j < 2; ++j)
                    if (nx[j] > 0) mbar_wait(x_full(j), (uint32_t)(nx[j] - 1) & 1u, err);
            }
        }
    } else if (warp == MMA_WARP) {
        if (lane == 0) {
            // ---- MMA issue, in work-item order: layer l of a slot once the
            // slot's input tile has landed (l = 0) or once its epilogue of
            // layer l - 1 (of the previous tile for l = 0) is done
            bool ok = true;
            int g = 0;
            for (int it = 0; it < items && ok; ++it) {
                const int p = it >> 3, l = (it >> 1) & 3, j = it & 1, i = 2 * p + j;
                if (i >= ntl) continue;
                if (l == 0) {
                    ok = mbar_wait(x_full(j), (uint32_t)p & 1u, err);
                    if (ok && p > 0) ok = mbar_wait(epi_done(j), 1u, err);  // layer 3 of the slot's previous tile
                } else {
                    ok = mbar_wait(epi_done(j), (uint32_t)(l - 1) & 1u, err);
                }
                if (!ok) break;
                tc_fence_after();
                const uint32_t a_buf = base + j * BUF;
                const uint32_t d_tmem = tmem + (uint32_t)(j * MLP_H);
                const int nkb = l == 0 ? KB_IN : KB_H;
                const uint32_t idesc = umma_idesc_bf16(BM, l == 3 ? MLP_OUT : MLP_H);
                for (int kb = 0; kb < nkb; ++kb, ++g) {
                    const int s = g % STAGES;
                    if (!mbar_wait(full(s), (uint32_t)(g / STAGES) & 1u, err)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t a = a_buf + kb * A_TILE;
                    const uint32_t b = base + RING + s * W_TILE;
#pragma unroll
                    for (int k = 0; k < BK / UK; ++k)
                        umma_bf16(d_tmem, sw128_desc(a + k * UK * 2), sw128_desc(b + k * UK * 2), idesc,
                                  (uint32_t)((kb | k) != 0));
                    umma_commit(empty(s));
                }
                if (!ok) break;
                if (l == 3) umma_commit(buf_free(j));  // the slot's buffer is free once these MMAs are done
                umma_commit(acc_full(j));
            }
            if (!ok) {  // so that the epilogue does not wait for nothing
                umma_commit(acc_full(0));
                umma_commit(acc_full(1));
                drain_ring(STAGES, g, ntl * (KB_IN + 3 * KB_H), full(0), err);
            }
        }
    } else {
        // ---- epilogue warps, in work-item order
        const int q = warp & 3, part = warp >> 2;
        const int r = q * 32 + lane;  // tile row of this thread
        for (int it = 0; it < items; ++it) {
            const int p = it >> 3, l = (it >> 1) & 3, j = it & 1, i = 2 * p + j;
            if (i >= ntl) continue;
            const bool ok = mbar_wait(acc_full(j), (uint32_t)l & 1u, err);
            tc_fence_after();
            if (!ok) break;
            const float* bias = P + L.b[l];
            const uint32_t tb = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(j * MLP_H);
            if (l < 3) {
                uint8_t* out = gbase + j * BUF;
                // columns c0 .. c0+15 from the registers of their load: bias
                // (four 16-byte loads), GELU, BF16, then K tile c0 / 64 as two
                // 16-byte chunks
                auto emit = [&](const uint32_t (&rv)[16], int c0) {
                    const float4* b4 = reinterpret_cast<const float4*>(bias + c0);
                    float bb[16];
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const float4 t = __ldg(b4 + e);
                        bb[4 * e] = t.x;
                        bb[4 * e + 1] = t.y;
                        bb[4 * e + 2] = t.z;
                        bb[4 * e + 3] = t.w;
                    }
                    uint32_t pk[8];
#pragma unroll
                    for (int e = 0; e < 16; e += 2) {
                        const float2 gv = gelu2_f(__fadd2_rn(make_float2(__uint_as_float(rv[e]), __uint_as_float(rv[e + 1])),
                                                             make_float2(bb[e], bb[e + 1])));
                        const __nv_bfloat162 h2 = __floats2bfloat162_rn(gv.x, gv.y);
                        pk[e >> 1] = *reinterpret_cast<const uint32_t*>(&h2);
                    }
                    uint8_t* tile = out + (c0 / BK) * A_TILE;
                    const int cc = c0 % BK;
                    *reinterpret_cast<uint4*>(tile + sw128_offset(r, cc)) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
                    *reinterpret_cast<uint4*>(tile + sw128_offset(r, cc + 8)) = make_uint4(pk[4], pk[5], pk[6], pk[7]);
                };
                // warp part p takes columns 64 kt + 16 p .. + 15 of each K
                // tile kt; the next chunk's accumulator load runs while this
                // chunk is worked on
                auto col = [&](int kt) { return kt * BK + part * 16; };
                uint32_t ra[16], rb[16];
                tmem_ld16_async(tb + (uint32_t)col(0), ra);
                tmem_wait16(ra);
#pragma unroll
                for (int kt = 0; kt < KB_H; kt += 2) {
                    tmem_ld16_async(tb + (uint32_t)col(kt + 1), rb);
                    emit(ra, col(kt));
                    tmem_wait16(rb);
                    if (kt + 2 < KB_H) tmem_ld16_async(tb + (uint32_t)col(kt + 2), ra);
                    emit(rb, col(kt + 1));
                    if (kt + 2 < KB_H) tmem_wait16(ra);
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            } else if (part == 0) {
                float v[16];
                tmem_ld16(tb, v);
                const int row = tile_row(i) + r;
                if (row < B) {
                    float4* o = reinterpret_cast<float4*>(y + (size_t)row * MLP_OUT);
#pragma unroll
                    for (int e = 0; e < 16; e += 4)
                        o[e / 4] = make_float4(v[e] + __ldg(bias + e), v[e + 1] + __ldg(bias + e + 1),
                                               v[e + 2] + __ldg(bias + e + 2), v[e + 3] + __ldg(bias + e + 3));
                }
            }
            tc_fence_before();
            asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(epi_done(j)) : "memory");
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == LOAD_WARP) tmem_dealloc(tmem, 2 * MLP_H);
}

// ------------------------------------------------------------------ training

// A training step is three launches: k_train_rows (forward and backward
// through all layers for a few batch rows per CTA), k_train_dw (every
// layer's weight and bias gradient, split over the batch) and k_train_update
// (the splits' sum, Adam, the BF16 copies).
//
// k_train_rows: one CTA per NB batch rows.  The products run transposed,
// out^T[feature][row] = W[feature][k] . act[row][k]^T, with the weights as
// the 128-row A operand (two halves of 256 features) and the CTA's rows as
// the N dimension, because a training batch is small: 2,048 rows make
// 128 CTAs of 16 rows where 128-row tiles make 16.  Seven steps: layers 0 .. 3,
// then the backward products through W4, W3, W2.  The rows' activations stay
// in one shared-memory buffer (K-major 64-column tiles, 128-byte swizzle),
// each step's epilogue writing its output over its input once the step's
// MMAs are done; the three layers' pre-activations stay in tensor memory in
// FP32 (2 NB columns each) until the backward pass takes their GELU', and
// the other steps share a fourth region.  An epilogue thread owns a feature
// and a half of the rows, so what the weight gradients contract over the
// batch ([feature][batch], BF16) is written straight from its registers.
// The 26 weight tiles (32 KB) stream through a TMA ring ahead of the steps.
// Every wait is bounded.
//
// What bounds it: the chain of seven dependent steps (MMA, epilogue and
// barrier each), not bandwidth: 0.68 MB of weights per CTA from L2.  A
// training step of 2,048 rows took 432 us as 26 launches (four 110 us
// column sums of one thread per column among them); now 21 us here, 10 in
// k_train_dw, 6 in k_train_update, with the host's part 50.
namespace train {
constexpr int STEPS = 7, STAGES = 5, KB_IN = (MLP_IN + BK - 1) / BK, KB_H = MLP_H / BK;
constexpr uint32_t W_TILE = MLP_H * BK * 2;  // 32 KB: 256 features x 64 BF16
constexpr int EPI_WARPS = 16, LOAD_WARP = EPI_WARPS, MMA_WARP = EPI_WARPS + 1;
constexpr int THREADS = 32 * (EPI_WARPS + 2), EPI_THREADS = 32 * EPI_WARPS;
// K tiles of a step, bytes of one of its weight tiles
__host__ __device__ constexpr int kblocks(int s) { return s == 0 ? KB_IN : (s == 4 ? 1 : KB_H); }
__host__ __device__ constexpr uint32_t tile_bytes(int s) { return s == 3 ? MLP_OUT * BK * 2 : W_TILE; }

template <int NB>
struct Smem {
    static constexpr uint32_t ACT_TILE = NB * BK * 2;  // NB rows x 64 BF16
    static constexpr uint32_t RING = KB_IN * ACT_TILE;
    static constexpr uint32_t BARS = RING + STAGES * W_TILE;
    // full[STAGES], empty[STAGES], x_full, acc_full, epi_done, then the TMEM slot
    static constexpr uint32_t TOTAL = 1024 + BARS + 8 * (2 * STAGES + 3) + 16;
    static constexpr uint32_t TMEM_COLS = 8 * NB;
};
}  // namespace train

struct TrainMaps {
    CUtensorMap w[4];       // W of layers 0 .. 3
    CUtensorMap wt[3];      // W^T of layers 3, 2, 1 (steps 4, 5, 6)
};

struct TrainArgs {
    const float* P;
    const float* target;    // [B][4], or NULL: the output gradient is given
    const float* dy;        // [B][16]
    int B, phase;
    int trunk;              // 0: stop after the output gradient
    int ld_t;               // row length of the transposed arrays
    __nv_bfloat16 *xt, *ht[3], *dt[3], *dyt;
    float* loss_part;       // two partial losses per CTA
    float* y;               // [B][16] (the forward pass alone)
    unsigned* err;
};

// FWD: the forward pass alone (inference of few rows): y [B][16] and nothing
// else, with the fused forward's GELU form, so that both give the same bits.
template <int NB, bool FWD>
__global__ void __launch_bounds__(train::THREADS, 1)
k_train_rows(const __grid_constant__ CUtensorMap mapX, const __grid_constant__ TrainMaps maps, TrainArgs a)
{
    using namespace train;
    using S = Smem<NB>;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    uint8_t* gbase = smem_raw + (base - raw);
    const uint32_t bars = base + S::BARS;
    auto full = [&](int s) { return bars + 8u * (uint32_t)s; };
    auto empty = [&](int s) { return bars + 8u * (uint32_t)(STAGES + s); };
    const uint32_t x_full = bars + 8u * (2 * STAGES), acc_full = x_full + 8u, epi_done = x_full + 16u;
    const uint32_t tmem_slot = x_full + 24u;
    uint32_t* tmem_slot_ptr = reinterpret_cast<uint32_t*>(gbase + S::BARS + 8 * (2 * STAGES + 3));
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int row0 = blockIdx.x * NB;
    const int nsteps = !FWD && a.trunk ? STEPS : 4;
    const ParamLayout L;

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(full(s), 1);
            mbar_init(empty(s), 1);
        }
        mbar_init(x_full, 1);
        mbar_init(acc_full, 1);
        mbar_init(epi_done, EPI_THREADS);
        mbar_fence_init();
    }
    if (warp == LOAD_WARP) tmem_alloc(tmem_slot, S::TMEM_COLS);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot_ptr;
    // accumulator of a step: layers 0 .. 2 keep theirs, the others share one
    auto acc_cols = [&](int s) { return tmem + (uint32_t)((s < 3 ? s : 3) * 2 * NB); };

    if (warp == LOAD_WARP) {
        if (lane == 0) {
            mbar_expect_tx(x_full, KB_IN * S::ACT_TILE);
            for (int kb = 0; kb < KB_IN; ++kb) tma_load_2d(&mapX, x_full, base + kb * S::ACT_TILE, kb * BK, row0);
            int g = 0;
            bool ok = true;
            for (int s = 0; s < nsteps && ok; ++s) {
                const CUtensorMap* map = s < 4 ? &maps.w[s] : &maps.wt[s - 4];
                for (int kb = 0; kb < kblocks(s); ++kb, ++g) {
                    const int st = g % STAGES;
                    if (g >= STAGES && !mbar_wait(empty(st), (uint32_t)((g / STAGES) - 1) & 1u, a.err)) {
                        ok = false;
                        break;
                    }
                    mbar_expect_tx(full(st), tile_bytes(s));
                    tma_load_2d(map, full(st), base + S::RING + st * W_TILE, kb * BK, 0);
                }
            }
            if (!ok) {  // let the copies in flight land before the CTA goes away
                for (int h = (g > STAGES ? g - STAGES : 0); h < g; ++h)
                    mbar_wait(full(h % STAGES), (uint32_t)(h / STAGES) & 1u, a.err);
                mbar_wait(x_full, 0, a.err);
            }
        }
    } else if (warp == MMA_WARP) {
        if (lane == 0) {
            constexpr uint32_t idesc = umma_idesc_bf16(BM, NB);
            bool ok = true;
            int g = 0;
            for (int s = 0; s < nsteps && ok; ++s) {
                // step s reads the input tile, or what the epilogue of step s - 1 wrote
                ok = s == 0 ? mbar_wait(x_full, 0, a.err) : mbar_wait(epi_done, (uint32_t)(s - 1) & 1u, a.err);
                if (!ok) break;
                tc_fence_after();
                for (int kb = 0; kb < kblocks(s); ++kb, ++g) {
                    const int st = g % STAGES;
                    if (!mbar_wait(full(st), (uint32_t)(g / STAGES) & 1u, a.err)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t w = base + S::RING + st * W_TILE, act = base + kb * S::ACT_TILE;
                    // the output layer has 16 features: the other rows of its A
                    // tile are leftovers of the ring, their lanes never read
                    const uint64_t wd = sw128_desc(w), ad = sw128_desc(act);
                    // a K step of 16 is 32 bytes, 2 in the descriptor's address
                    // field; the second half of the features 16 KB, 1024 there
                    auto issue = [&](int hf, int k) {
                        umma_bf16(acc_cols(s) + (uint32_t)(hf * NB), wd + (uint64_t)(hf * (int)(W_TILE / 32) + 2 * k),
                                  ad + (uint64_t)(2 * k), idesc, (uint32_t)((kb | k) != 0));
                    };
                    if (s == 4) {  // 16 columns
                        issue(0, 0);
                        issue(1, 0);
                    } else {
#pragma unroll
                        for (int k = 0; k < BK / UK; ++k) {
                            issue(0, k);
                            if (s != 3) issue(1, k);
                        }
                    }
                    umma_commit(empty(st));
                }
                if (!ok) break;
                umma_commit(acc_full);
            }
            if (!ok) {
                umma_commit(acc_full);  // so that the epilogue does not wait for nothing
                int total = 0;
                for (int s = 0; s < nsteps; ++s) total += kblocks(s);
                drain_ring(STAGES, g, total, full(0), a.err);
            }
        }
    } else {
        // warp w reads tensor-memory lanes 32 (w % 4) ..; part w / 4 picks the
        // feature half and the half of the rows
        constexpr int CH = NB >= 32 ? 16 : 8;  // rows (accumulator columns) per chunk
        auto tmem_ld = [](uint32_t addr, float (&v)[CH]) {
            if constexpr (CH == 16) tmem_ld16(addr, v);
            else tmem_ld8(addr, v);
        };
        const int q = warp & 3, part = warp >> 2, hf = part >> 1, f = hf * 128 + q * 32 + lane;
        const int n0 = (part & 1) * (NB / 2);
        const uint32_t lanes = (uint32_t)(q * 32) << 16;
        bool ok = mbar_wait(x_full, 0, a.err);
        if (!FWD && a.trunk && ok) {  // x^T for the first layer's weight gradient
            for (int e = threadIdx.x; e < MLP_IN * (NB / 8); e += EPI_THREADS) {
                const int c = e % MLP_IN, r8 = (e / MLP_IN) * 8;
                const uint8_t* tile = gbase + (c / BK) * S::ACT_TILE;
                uint32_t pk[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const uint32_t lo = *reinterpret_cast<const uint16_t*>(tile + sw128_offset(r8 + 2 * k, c % BK));
                    const uint32_t hi = *reinterpret_cast<const uint16_t*>(tile + sw128_offset(r8 + 2 * k + 1, c % BK));
                    pk[k] = lo | (hi << 16);
                }
                *reinterpret_cast<uint4*>(a.xt + (size_t)c * a.ld_t + row0 + r8) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
            }
        }
        if (!FWD) asm volatile("bar.sync 1, %0;" ::"n"(EPI_THREADS) : "memory");  // x read before any epilogue overwrites it
        // this thread's biases, before the steps' critical path
        const float bias[3] = {__ldg(a.P + L.b[0] + f), __ldg(a.P + L.b[1] + f), __ldg(a.P + L.b[2] + f)};
#pragma unroll
        for (int s = 0; s < (FWD ? 4 : STEPS); ++s) {
            if (s >= nsteps) break;
            ok = mbar_wait(acc_full, (uint32_t)s & 1u, a.err);
            tc_fence_after();
            if (!ok) break;
            uint32_t pk[NB / 2 / CH][CH / 2];
            if (s == 3) {
                // the output layer: 16 features in the first lanes
                if (hf == 0 && q == 0) {
                    float loss = 0.0f;
#pragma unroll
                    for (int c = 0; c < NB / 2; c += CH) {
                        float v[CH];
                        tmem_ld(acc_cols(3) + lanes + (uint32_t)(n0 + c), v);
                        if (lane < MLP_OUT) {
                            const float b = __ldg(a.P + L.b[3] + lane);
                            if constexpr (FWD) {
#pragma unroll
                                for (int e = 0; e < CH; ++e)
                                    if (row0 + n0 + c + e < a.B)
                                        a.y[(size_t)(row0 + n0 + c + e) * MLP_OUT + lane] = v[e] + b;
                                continue;
                            }
                            uint32_t(&p)[CH / 2] = pk[c / CH];
#pragma unroll
                            for (int e = 0; e < CH; ++e) {
                                const int row = row0 + n0 + c + e;
                                float g = 0.0f;
                                if (a.dy) {
                                    g = __ldg(a.dy + (size_t)row * MLP_OUT + lane);
                                } else if (a.phase == 0 ? lane < 3 : lane == 3) {
                                    const float d = v[e] + b - __ldg(a.target + (size_t)row * 4 + lane);
                                    loss += 0.5f * d * d;
                                    g = d / (float)a.B;
                                }
                                const __nv_bfloat16 gb = __float2bfloat16_rn(g);
                                const uint16_t u = *reinterpret_cast<const uint16_t*>(&gb);
                                if (e & 1) p[e >> 1] |= (uint32_t)u << 16;
                                else p[e >> 1] = u;
                                if (a.trunk)
                                    *reinterpret_cast<uint16_t*>(gbase + sw128_offset(n0 + c + e, lane)) = u;
                            }
                        }
                    }
                    if constexpr (!FWD) {
#pragma unroll
                        for (int o = 16; o > 0; o >>= 1) loss += __shfl_xor_sync(FULL, loss, o);
                        if (lane == 0) a.loss_part[2 * blockIdx.x + part] = loss;
                    }
                }
            } else {
                const int l = s < 3 ? s : 6 - s;  // layer whose pre-activation the step meets
                const float b = bias[l];
#pragma unroll
                for (int c = 0; c < NB / 2; c += CH) {
                    const uint32_t cols = lanes + (uint32_t)(hf * NB + n0 + c);
                    float z[CH], v[CH];
                    tmem_ld(acc_cols(l) + cols, z);
                    if (s > 3) tmem_ld(acc_cols(s) + cols, v);
                    uint32_t(&p)[CH / 2] = pk[c / CH];
#pragma unroll
                    for (int e = 0; e < CH; e += 2) {
                        const float z0 = z[e] + b, z1 = z[e + 1] + b;
                        const float2 g2 = FWD ? gelu2_f(make_float2(z0, z1)) : make_float2(0.f, 0.f);
                        const __nv_bfloat162 h2 =
                            FWD ? __floats2bfloat162_rn(g2.x, g2.y) : s < 3 ? __floats2bfloat162_rn(gelu_f(z0), gelu_f(z1))
                                  : __floats2bfloat162_rn(v[e] * gelu_grad_f(z0), v[e + 1] * gelu_grad_f(z1));
                        p[e >> 1] = *reinterpret_cast<const uint32_t*>(&h2);
                    }
                    if (s < 6) {  // the next step's operand: (row n0 + c + e, feature f)
                        uint8_t* tile = gbase + (f / BK) * S::ACT_TILE;
#pragma unroll
                        for (int e = 0; e < CH; ++e)
                            *reinterpret_cast<uint16_t*>(tile + sw128_offset(n0 + c + e, f % BK)) =
                                (uint16_t)(p[e >> 1] >> (16 * (e & 1)));
                    }
                }
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            tc_fence_before();
            asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(epi_done) : "memory");
            // the transposed copy, off the next step's path (a warp's stores go
            // to 32 rows and would hold up the operand's)
            __nv_bfloat16* out = s == 3 ? a.dyt : (s < 3 ? a.ht[s < 3 ? s : 0] : a.dt[s < 4 ? 0 : 6 - s]);
            const bool mine = s == 3 ? hf == 0 && q == 0 && lane < MLP_OUT : a.trunk || s == 2;
            if (!FWD && mine)
#pragma unroll
                for (int c = 0; c < NB / 2; c += CH) {
                    uint4* o = reinterpret_cast<uint4*>(out + (size_t)f * a.ld_t + row0 + n0 + c);
                    const uint32_t(&p)[CH / 2] = pk[c / CH];
#pragma unroll
                    for (int k = 0; k < CH / 8; ++k)
                        o[k] = make_uint4(p[4 * k], p[4 * k + 1], p[4 * k + 2], p[4 * k + 3]);
                }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == LOAD_WARP) tmem_dealloc(tmem, S::TMEM_COLS);
}

// Weight and bias gradients of every layer: dW[out][in] = dT[out][B] .
// inT[in][B]^T over a slice of the batch.  blockIdx.x: a tile of 128 outputs
// x 144 inputs of a layer (two N tiles cover 256 or 272 inputs: 14 tiles in
// all), blockIdx.y: the slice.  Partials go to part[slice] in the packed
// parameter layout.  One kernel for all layers: a product alone would use
// 16 SMs.  The last blocks of the first slice sum dT over the batch, the
// bias gradients: a thread per output adds its row in batch order, one
// float32 sum (its last bit reaches the next step's activations, so the
// order is part of the result).  That chain of additions bounds the kernel
// (the weight tiles alone take 6.6 us for 2,048 rows), so its warp does
// nothing else: the rows come by TMA from a warp of the copies' own, two
// blocks of 64 a wait, and the BF16 value is an operand of the addition.  A
// warp of 32 outputs a block, mixed additions and one wait for two blocks:
// 13.9 -> 10.2 us (with conversions and a wait a block 14.1, with the mixed
// additions alone 12.8; read straight from memory, a warp's loads of 32 rows
// were 32 wavefronts each: 21).
namespace dw {
constexpr int NT = 144, STAGES = 4, TILES = 14;  // weight tiles
constexpr int BR = 32, BIAS = 25, BIAS_STAGES = 8;  // bias blocks of 32 outputs: 8 a hidden layer, then the output layer's
constexpr uint32_t A_BYTES = BM * BK * 2, B_BYTES = NT * BK * 2, STAGE = A_BYTES + B_BYTES;
constexpr uint32_t BARS = STAGES * STAGE;
constexpr uint32_t BIAS_BYTES = 2 * BR * BK * 2;  // a stage: two blocks of the batch
constexpr uint32_t TOTAL = 1024 + BARS + 8 * (2 * BIAS_STAGES + 2) + 16;
constexpr uint32_t TMEM_COLS = 256;
static_assert(STAGE % 1024 == 0 && BIAS_BYTES % 1024 == 0, "operand tiles start on 1024-byte boundaries");
static_assert(BIAS_STAGES >= STAGES && BIAS_STAGES * BIAS_BYTES <= BARS, "the biases' ring fits the operands'");
}  // namespace dw

struct DwMaps {
    CUtensorMap d[4];   // dT of layers 0 .. 3, boxes of 128 rows
    CUtensorMap in[4];  // inT of layers 0 .. 3, boxes of 144 rows
    CUtensorMap b[4];   // dT of layers 0 .. 3, boxes of 32 rows
};

__global__ void __launch_bounds__(160)
k_train_dw(const __grid_constant__ DwMaps maps, int first_tile, int kb_total, int kb_per_split,
           float* __restrict__ part, unsigned* __restrict__ err)
{
    using namespace dw;
    const int tile = first_tile + (int)blockIdx.x;
    const bool bias = tile >= TILES;
    if (bias && blockIdx.y) return;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    uint8_t* gbase = smem_raw + (base - raw);
    const uint32_t bars = base + BARS;
    auto full = [&](int s) { return bars + 8u * (uint32_t)s; };
    auto empty = [&](int s) { return bars + 8u * (uint32_t)(BIAS_STAGES + s); };
    const uint32_t done = bars + 8u * (2 * BIAS_STAGES), tmem_slot = done + 8u;
    uint32_t* tmem_slot_ptr = reinterpret_cast<uint32_t*>(gbase + BARS + 8 * (2 * BIAS_STAGES + 1));
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const ParamLayout L;
    if (threadIdx.x == 0) {
        for (int s = 0; s < (bias ? BIAS_STAGES : STAGES); ++s) {
            mbar_init(full(s), 1);
            mbar_init(empty(s), bias ? BR : 1);
        }
        mbar_init(done, 1);
        mbar_fence_init();
    }
    if (bias) {
        // blocks 0 .. 23: the hidden layers, 24: the output layer (the last
        // block, also where it is the only one)
        const int blk = BIAS - ((int)gridDim.x - (int)blockIdx.x), l = blk >> 3, m0 = (blk & 7) * BR;
        const int n = kb_total / 2;  // the batch is a multiple of two blocks
        __syncthreads();
        if (warp == 4) {  // the copies' own warp: in a summing warp they would hold up its chain
            if (lane == 0) {
                int i = 0;
                for (; i < n; ++i) {
                    const int st = i % BIAS_STAGES;
                    if (i >= BIAS_STAGES && !mbar_wait(empty(st), (uint32_t)((i / BIAS_STAGES) - 1) & 1u, err)) break;
                    mbar_expect_tx(full(st), BIAS_BYTES);
                    for (int h = 0; h < 2; ++h)
                        tma_load_2d(&maps.b[l], full(st), base + st * BIAS_BYTES + h * (BIAS_BYTES / 2), (2 * i + h) * BK, m0);
                }
                if (i < n)  // let the copies in flight land before the CTA goes away
                    for (int q = max(0, i - BIAS_STAGES); q < i; ++q)
                        mbar_wait(full(q % BIAS_STAGES), (uint32_t)(q / BIAS_STAGES) & 1u, err);
            }
            return;
        }
        if (warp) return;
        // a row's 64 values of a block are loaded while the block before is added
        uint4 v[2][BK / 8];
        float s = 0.f;
        auto wait = [&](int i) { return mbar_wait(full(i % BIAS_STAGES), (uint32_t)(i / BIAS_STAGES) & 1u, err); };
        auto fetch = [&](int i, int h) {
            const uint8_t* row = gbase + (i % BIAS_STAGES) * BIAS_BYTES + h * (BIAS_BYTES / 2);
#pragma unroll
            for (int c = 0; c < BK / 8; ++c) v[h][c] = *reinterpret_cast<const uint4*>(row + sw128_offset(lane, 8 * c));
        };
        auto sum = [&](const uint4 (&from)[BK / 8]) {
#pragma unroll
            for (int c = 0; c < BK / 8; ++c) {
                const uint32_t w[4] = {from[c].x, from[c].y, from[c].z, from[c].w};
#pragma unroll
                for (int j = 0; j < 4; ++j)  // float32 + BF16, rounded once
                    asm("{.reg .b16 l, h;\n\tmov.b32 {l, h}, %1;\n\tadd.rn.f32.bf16 %0, l, %0;\n\tadd.rn.f32.bf16 %0, h, %0;}"
                        : "+f"(s)
                        : "r"(w[j]));
            }
        };
        bool ok = wait(0);
        if (ok) fetch(0, 0);
        int i = 0;
        for (; ok && i < n; ++i) {
            fetch(i, 1);
            asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(empty(i % BIAS_STAGES)) : "memory");
            sum(v[0]);
            if (i + 1 < n && (ok = wait(i + 1))) fetch(i + 1, 0);
            sum(v[1]);
        }
        if (!ok) drain_ring(BIAS_STAGES, i, n, full(0), err);
        const int f = m0 + lane;
        if (ok && f < L.out[l])  // the other slices hold zeros
            for (int k = 0; k < (int)gridDim.y; ++k) part[(size_t)k * SPH_MLP_PARAMS + L.b[l] + f] = k ? 0.0f : s;
        return;
    }
    const int l = tile < 12 ? tile >> 2 : 3, mt = tile < 12 ? (tile >> 1) & 1 : 0, nt = tile & 1;
    const int m0 = mt * BM, n0 = nt * NT;
    const int kb0 = blockIdx.y * kb_per_split, nk = min(kb_per_split, kb_total - kb0);

    if (warp == 0) tmem_alloc(tmem_slot, TMEM_COLS);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot_ptr;

    if (warp == 0 && lane == 0) {
        int issued = 0;
        bool ok = true;
        for (int i = 0; i < nk; ++i) {
            const int s = i % STAGES;
            if (i >= STAGES && !mbar_wait(empty(s), (uint32_t)((i / STAGES) - 1) & 1u, err)) {
                ok = false;
                break;
            }
            mbar_expect_tx(full(s), STAGE);
            tma_load_2d(&maps.d[l], full(s), base + s * STAGE, (kb0 + i) * BK, m0);
            tma_load_2d(&maps.in[l], full(s), base + s * STAGE + A_BYTES, (kb0 + i) * BK, n0);
            ++issued;
        }
        if (!ok)
            for (int i = max(0, issued - STAGES); i < issued; ++i)
                mbar_wait(full(i % STAGES), (uint32_t)(i / STAGES) & 1u, err);
    } else if (warp == 1 && lane == 0) {
        constexpr uint32_t idesc = umma_idesc_bf16(BM, NT);
        for (int i = 0; i < nk; ++i) {
            const int s = i % STAGES;
            if (!mbar_wait(full(s), (uint32_t)(i / STAGES) & 1u, err)) {
                drain_ring(STAGES, i, nk, full(0), err);
                break;
            }
            tc_fence_after();
            const uint32_t a = base + s * STAGE, b = a + A_BYTES;
#pragma unroll
            for (int k = 0; k < BK / UK; ++k)
                umma_bf16(tmem, sw128_desc(a + k * UK * 2), sw128_desc(b + k * UK * 2), idesc, (uint32_t)((i | k) != 0));
            umma_commit(empty(s));
        }
        umma_commit(done);
    }
    __syncwarp();

    // warps 0 .. 3 each read their tensor-memory lanes
    const bool ok = warp < 4 && mbar_wait(done, 0, err);
    tc_fence_after();
    if (ok) {
        const int m = m0 + warp * 32 + lane, nin = L.in[l];
        const uint32_t row = tmem + ((uint32_t)(warp * 32) << 16);
        float* out = part + (size_t)blockIdx.y * SPH_MLP_PARAMS;
        // a thread's row goes through shared memory (the idle ring; the odd
        // number of 16-byte chunks per row spreads a warp's over the banks)
        // and out as one bulk copy: stored by the warp, 32 rows an instruction
        constexpr int LD = NT + 4;
        static_assert(128 * LD * 4 <= STAGES * STAGE, "the rows fit the ring");
        float* stage = reinterpret_cast<float*>(gbase) + threadIdx.x * LD;
        const int w = min(NT, nin - n0);  // 16-column chunks end with the layer's inputs
        for (int c = 0; c < w; c += 16) {
            float v[16];
            tmem_ld16(row + (uint32_t)c, v);
#pragma unroll
            for (int e = 0; e < 16; e += 4)
                *reinterpret_cast<float4*>(stage + c + e) = make_float4(v[e], v[e + 1], v[e + 2], v[e + 3]);
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        if (m < L.out[l]) {
            asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(out + L.w[l] + m * nin + n0),
                         "r"(smem_u32(stage)), "r"(w * 4)
                         : "memory");
            asm volatile("cp.async.bulk.commit_group;" ::: "memory");
        }
        asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, TMEM_COLS);
}

// G = the slices' sum, in order; then (adam) the Adam update (Kingma & Ba)
// of the FP32 master parameters a phase trains, with their BF16 copies W
// [out][in] and W^T [in][out].  [lo, SPH_MLP_PARAMS): the parameters with
// partials.  The first thread adds the partial losses.
struct AdamArgs {
    float lr, b1, b2, eps, c1, c2;
    int phase;
};

__global__ void __launch_bounds__(128)
k_train_update(const float* __restrict__ part, int splits, int lo, float* __restrict__ G, float* __restrict__ grads,
               int adam, AdamArgs o, float* __restrict__ P, float* __restrict__ Mo, float* __restrict__ Vo,
               __nv_bfloat16* __restrict__ W, __nv_bfloat16* __restrict__ WT, const float* __restrict__ loss_part,
               int nloss, int B, float* __restrict__ loss)
{
    const ParamLayout L;
    const int t = lo + 4 * (int)(blockIdx.x * 128 + threadIdx.x);
    if (loss && blockIdx.x == gridDim.x - 1) {  // the last block: few parameters, and the loss
        __shared__ float red[4];
        float s = 0.0f;
        for (int k = threadIdx.x; k < nloss; k += 128) s += loss_part[k];
#pragma unroll
        for (int q = 16; q > 0; q >>= 1) s += __shfl_xor_sync(FULL, s, q);
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
        __syncthreads();
        if (threadIdx.x == 0) {
            float tot = 0.0f;
            for (int w = 0; w < 4; ++w) tot += red[w];
            *loss = tot / (float)B;
        }
    }
    if (t >= SPH_MLP_PARAMS) return;
    // four parameters a thread: every weight row, bias vector and layer starts
    // at a multiple of four
    static_assert(SPH_MLP_PARAMS % 4 == 0 && MLP_IN % 4 == 0, "whole quads");
    auto at4 = [&](const float* p) { return *reinterpret_cast<const float4*>(p + t); };
    float g[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    for (int k = 0; k < splits; ++k) {
        const float4 p = at4(part + (size_t)k * SPH_MLP_PARAMS);
        g[0] += p.x;
        g[1] += p.y;
        g[2] += p.z;
        g[3] += p.w;
    }
    *reinterpret_cast<float4*>(G + t) = make_float4(g[0], g[1], g[2], g[3]);
    if (grads)
        for (int e = 0; e < 4; ++e) grads[t + e] = g[e];  // the caller's array, aligned as floats
    if (!adam) return;
    const int l = t >= L.w[3] ? 3 : (t >= L.w[2] ? 2 : (t >= L.w[1] ? 1 : 0));
    const int e0 = t - L.w[l], nin = l == 0 ? MLP_IN : MLP_H, nout = l == 3 ? MLP_OUT : MLP_H;
    const float4 P4 = at4(P), M4 = at4(Mo), V4 = at4(Vo);
    float p[4] = {P4.x, P4.y, P4.z, P4.w}, m[4] = {M4.x, M4.y, M4.z, M4.w}, v[4] = {V4.x, V4.y, V4.z, V4.w};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        // phase 0 leaves the error head (row 3 of W4, b4[3]), phase 1 trains it alone
        const bool head = (t >= L.w[3] + 3 * MLP_H && t < L.w[3] + 4 * MLP_H) || t + e == L.b[3] + 3;
        if (head != (o.phase == 1)) continue;
        // contracted in one fixed way: a last bit here decides now and then how
        // a weight rounds to BF16
        m[e] = __fmaf_rn(1.f - o.b1, g[e], __fmul_rn(o.b1, m[e]));
        v[e] = __fmaf_rn(__fmul_rn(1.f - o.b2, g[e]), g[e], __fmul_rn(o.b2, v[e]));
        p[e] -= o.lr * (m[e] / o.c1) / (sqrtf(v[e] / o.c2) + o.eps);
    }
    *reinterpret_cast<float4*>(Mo + t) = make_float4(m[0], m[1], m[2], m[3]);
    *reinterpret_cast<float4*>(Vo + t) = make_float4(v[0], v[1], v[2], v[3]);
    *reinterpret_cast<float4*>(P + t) = make_float4(p[0], p[1], p[2], p[3]);
    if (e0 < nin * nout) {
        const int r = e0 / nin, c = e0 % nin;
        const __nv_bfloat162 lo2 = __floats2bfloat162_rn(p[0], p[1]), hi2 = __floats2bfloat162_rn(p[2], p[3]);
        *reinterpret_cast<__nv_bfloat162*>(W + t) = lo2;
        *reinterpret_cast<__nv_bfloat162*>(W + t + 2) = hi2;
        __nv_bfloat16* wt = WT + L.w[l] + c * nout + r;
        wt[0] = lo2.x;
        wt[nout] = lo2.y;
        wt[2 * nout] = hi2.x;
        wt[3 * nout] = hi2.y;
    }
}

}  // namespace sphk

// ------------------------------------------------------------------ API

using namespace sphk;

struct sph_mlp {
    int max_batch;
    float *P, *G, *Mo, *Vo;            // packed parameters, gradients, Adam moments
    __nv_bfloat16 *W, *WT;             // BF16 weights and transposes (packed like P)
    __nv_bfloat16 *XT, *HT[3];         // transposed input and hidden activations [features][Bmax]
    __nv_bfloat16 *DT[3], *DYT;        // transposed gradients of the pre-activations and of the output
    float* part;                       // split-K partials: `splits` packed parameter vectors
    int splits;
    float* loss_part;                  // two partial losses per CTA of 16 rows or more
    float* loss;
    unsigned* err;
    long long step;
    long long launches;
    // tensor maps of the handle's own arrays (built with it: its calls, from
    // whatever thread, only read them)
    TrainMaps tmaps;
    DwMaps dmaps;
    char msg[512];
};

// Slices of the batch in the weight gradients: up to eight (14 tiles x 8 =
// 112 CTAs), fewer for small handles so that the partials do not outgrow
// the activations.
static int max_splits(int max_batch) { return max_batch >= 1152 ? 8 : 2 + max_batch / 192; }

static int mfail(sph_mlp* m, int code, const char* fmt, ...)
{
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof(buf), fmt, ap);
    va_end(ap);
    if (m) snprintf(m->msg, sizeof(m->msg), "%s", buf);
    sphk::set_handleless_error(buf);
    return code;
}

#define MLP_TRY(m, expr)                                                                           \
    do {                                                                                           \
        cudaError_t e_ = (expr);                                                                   \
        if (e_ != cudaSuccess)                                                                     \
            return mfail((m), SPH_ERR_CUDA, "%s: %s (%s:%d)", #expr, cudaGetErrorString(e_), __FILE__, \
                         __LINE__);                                                                \
    } while (0)

struct MCarver {
    uintptr_t base, off;
    template <class T>
    T* take(size_t count)
    {
        off = (off + 255) & ~(uintptr_t)255;
        T* p = reinterpret_cast<T*>(base + off);
        off += count * sizeof(T);
        return p;
    }
};

static size_t mlp_carve(sph_mlp* m, uintptr_t base)
{
    MCarver c{base, 0};
    const size_t P = SPH_MLP_PARAMS, B = (size_t)m->max_batch;
    m->P = c.take<float>(P);
    m->G = c.take<float>(P);
    m->Mo = c.take<float>(P);
    m->Vo = c.take<float>(P);
    m->W = c.take<__nv_bfloat16>(P);
    m->WT = c.take<__nv_bfloat16>(P);
    m->XT = c.take<__nv_bfloat16>((size_t)MLP_IN * B);
    for (int l = 0; l < 3; ++l) {
        m->HT[l] = c.take<__nv_bfloat16>((size_t)MLP_H * B);
        m->DT[l] = c.take<__nv_bfloat16>((size_t)MLP_H * B);
    }
    m->DYT = c.take<__nv_bfloat16>((size_t)MLP_OUT * B);
    m->splits = max_splits(m->max_batch);
    m->part = c.take<float>((size_t)m->splits * P);
    m->loss_part = c.take<float>(2 * (B / 16));
    m->loss = c.take<float>(4);
    m->err = c.take<unsigned>(4);
    return (c.off + 255) & ~(uintptr_t)255;
}

static int sms_of_device(sph_mlp* m, int* sms)
{
    int dev = 0;
    MLP_TRY(m, cudaGetDevice(&dev));
    MLP_TRY(m, cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, dev));
    return SPH_OK;
}

static int build_maps(sph_mlp* m)
{
    const ParamLayout L;
    for (int l = 0; l < 4; ++l)
        MLP_TRY(m, make_map(&m->tmaps.w[l], m->W + L.w[l], L.out[l], L.in[l], L.in[l], L.out[l]));
    for (int l = 3; l > 0; --l)
        MLP_TRY(m, make_map(&m->tmaps.wt[3 - l], m->WT + L.w[l], L.in[l], L.out[l], L.out[l], L.in[l]));
    for (int l = 0; l < 4; ++l) {
        MLP_TRY(m, make_map(&m->dmaps.d[l], l < 3 ? m->DT[l] : m->DYT, L.out[l], m->max_batch, m->max_batch, BM));
        MLP_TRY(m, make_map(&m->dmaps.in[l], l ? m->HT[l - 1] : m->XT, L.in[l], m->max_batch, m->max_batch, dw::NT));
        MLP_TRY(m, make_map(&m->dmaps.b[l], l < 3 ? m->DT[l] : m->DYT, L.out[l], m->max_batch, m->max_batch, dw::BR));
    }
    return SPH_OK;
}

template <int NB, bool FWD>
static int launch_rows(sph_mlp* m, const CUtensorMap& mx, const TrainArgs& a, cudaStream_t s)
{
    static bool attr = false;
    if (!attr) {
        MLP_TRY(m, cudaFuncSetAttribute(k_train_rows<NB, FWD>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        (int)train::Smem<NB>::TOTAL));
        attr = true;
    }
    k_train_rows<NB, FWD><<<a.B / NB, train::THREADS, train::Smem<NB>::TOTAL, s>>>(mx, m->tmaps, a);
    ++m->launches;
    MLP_TRY(m, cudaGetLastError());
    return SPH_OK;
}

// Inference: the four layers in one launch (k_mlp_fused), 128-row tiles.
static int mlp_forward_fused(sph_mlp* m, const __nv_bfloat16* x, int B, float* y, cudaStream_t s)
{
    CUtensorMap mx;
    int sms = 0, rc = sms_of_device(m, &sms);
    if (rc != SPH_OK) return rc;
    // Few rows: 16 or 32 a CTA instead of 128, so that more of the chip works
    // on them: 128 to 2,432 rows take 14 us instead of 22, up to 4,864 rows
    // 15 instead of 22.6; at 4,992 rows (64 a CTA) nothing would be gained.
    if (B <= 32 * sms) {
        const int NB = B <= 16 * sms ? 16 : 32;
        MLP_TRY(m, make_map(&mx, x, B, MLP_IN, MLP_IN, NB));
        TrainArgs a;
        memset(&a, 0, sizeof(a));
        a.P = m->P;
        a.B = B;
        a.y = y;
        a.err = m->err;
        return NB == 16 ? launch_rows<16, true>(m, mx, a, s) : launch_rows<32, true>(m, mx, a, s);
    }
    MLP_TRY(m, make_map(&mx, x, B, MLP_IN, MLP_IN, BM));
    static bool attr = false;
    if (!attr) {
        MLP_TRY(m, cudaFuncSetAttribute(k_mlp_fused, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)fused::TOTAL));
        attr = true;
    }
    const CUtensorMap* mw = m->tmaps.w;
    // persistent: one CTA per SM (the kernel takes one), each looping over
    // the 128-row tiles blockIdx.x, blockIdx.x + gridDim.x, ...
    const int tiles = (B + BM - 1) / BM;
    const int grid = tiles < sms ? tiles : sms;
    k_mlp_fused<<<grid, fused::THREADS, fused::TOTAL, s>>>(mx, mw[0], mw[1], mw[2], mw[3], m->P, B, y, m->err);
    ++m->launches;
    MLP_TRY(m, cudaGetLastError());
    return SPH_OK;
}

// Gradients of one batch (targets t: the phase's loss; else the output
// gradient dy), and with adam the update.
static int train_pass(sph_mlp* m, const __nv_bfloat16* x, const float* t, const float* dy, int B, int phase,
                      float* grads, const AdamArgs* adam, float* loss, cudaStream_t s)
{
    const ParamLayout L;
    int sms = 0, rc = sms_of_device(m, &sms);
    if (rc != SPH_OK) return rc;
    TrainArgs a;
    memset(&a, 0, sizeof(a));
    a.P = m->P;
    a.target = t;
    a.dy = dy;
    a.B = B;
    a.phase = phase;
    a.trunk = phase == 0;
    a.ld_t = m->max_batch;
    a.xt = m->XT;
    for (int l = 0; l < 3; ++l) {
        a.ht[l] = m->HT[l];
        a.dt[l] = m->DT[l];
    }
    a.dyt = m->DYT;
    a.loss_part = m->loss_part;
    a.err = m->err;
    // as few rows a CTA as one wave of CTAs allows: the epilogues (1.85 us a
    // step per 32 rows, bound by the GELU's reciprocals and exponentials) are
    // most of the chain
    const int NB = B <= 16 * sms ? 16 : (B <= 32 * sms ? 32 : 64);
    CUtensorMap mx;
    MLP_TRY(m, make_map(&mx, x, B, MLP_IN, MLP_IN, NB));
    rc = NB == 16   ? launch_rows<16, false>(m, mx, a, s)
         : NB == 32 ? launch_rows<32, false>(m, mx, a, s)
                    : launch_rows<64, false>(m, mx, a, s);
    if (rc != SPH_OK) return rc;
    static bool attr = false;
    if (!attr) {
        MLP_TRY(m, cudaFuncSetAttribute(k_train_dw, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dw::TOTAL));
        attr = true;
    }
    const int kb = B / BK;
    int splits = m->splits < kb ? m->splits : kb;
    const int per = (kb + splits - 1) / splits;
    splits = (kb + per - 1) / per;
    const int first = phase == 0 ? 0 : 12, lo = phase == 0 ? 0 : L.w[3];
    const int nbias = phase == 0 ? dw::BIAS : 1;
    k_train_dw<<<dim3(dw::TILES - first + nbias, splits), 160, dw::TOTAL, s>>>(m->dmaps, first, kb, per, m->part, m->err);
    AdamArgs none;
    memset(&none, 0, sizeof(none));
    // the kernel writes the caller's floats itself where they are aligned as
    // floats; elsewhere they are copied from the handle's
    auto aligned = [](float* p) { return ((uintptr_t)p & 3) == 0; };
    k_train_update<<<(SPH_MLP_PARAMS - lo + 511) / 512, 128, 0, s>>>(
        m->part, splits, lo, m->G, aligned(grads) ? grads : nullptr, adam != nullptr, adam ? *adam : none, m->P, m->Mo,
        m->Vo, m->W, m->WT, m->loss_part, 2 * (B / NB), B, aligned(loss) ? loss : m->loss);
    m->launches += 2;
    MLP_TRY(m, cudaGetLastError());
    if (!aligned(grads))
        MLP_TRY(m, cudaMemcpyAsync(grads, m->G, sizeof(float) * SPH_MLP_PARAMS, cudaMemcpyDeviceToDevice, s));
    if (!aligned(loss)) MLP_TRY(m, cudaMemcpyAsync(loss, m->loss, sizeof(float), cudaMemcpyDeviceToDevice, s));
    return SPH_OK;
}

static int check_batch(sph_mlp* m, int B)
{
    if (!m) return mfail(nullptr, SPH_ERR_ARG, "mlp is NULL");
    if (B <= 0 || B > m->max_batch || (B & 127))
        return mfail(m, SPH_ERR_ARG, "batch %d must be a positive multiple of 128 <= %d", B, m->max_batch);
    return SPH_OK;
}

extern "C" {

int sph_mlp_workspace_size(int max_batch, size_t* bytes)
{
    if (!bytes || max_batch <= 0 || (max_batch & 127))
        return mfail(nullptr, SPH_ERR_ARG, "max_batch must be a positive multiple of 128");
    sph_mlp t;
    memset(&t, 0, sizeof(t));
    t.max_batch = max_batch;
    *bytes = mlp_carve(&t, 0);
    return SPH_OK;
}

int sph_mlp_create(int max_batch, void* workspace, size_t ws_bytes, sph_mlp** out)
{
    size_t need = 0;
    int rc = sph_mlp_workspace_size(max_batch, &need);
    if (rc != SPH_OK) return rc;
    if (!out || !workspace || ((uintptr_t)workspace & 255) || ws_bytes < need)
        return mfail(nullptr, SPH_ERR_ARG, "workspace must be 256-byte aligned and >= %zu bytes", need);
    sph_mlp* m = new (std::nothrow) sph_mlp;
    if (!m) return mfail(nullptr, SPH_ERR_ARG, "out of host memory");
    memset(m, 0, sizeof(*m));
    m->max_batch = max_batch;
    mlp_carve(m, (uintptr_t)workspace);
    cudaError_t e = cudaMemset(workspace, 0, need);
    if (e != cudaSuccess) {
        delete m;
        return mfail(nullptr, SPH_ERR_CUDA, "cudaMemset: %s", cudaGetErrorString(e));
    }
    rc = build_maps(m);
    if (rc != SPH_OK) {
        delete m;
        return rc;
    }
    *out = m;
    return SPH_OK;
}

void sph_mlp_destroy(sph_mlp* m) { delete m; }

int sph_mlp_set_params(sph_mlp* m, const float* params, void* stream)
{
    if (!m || !params) return mfail(m, SPH_ERR_ARG, "NULL argument");
    cudaStream_t s = (cudaStream_t)stream;
    MLP_TRY(m, cudaMemcpyAsync(m->P, params, sizeof(float) * SPH_MLP_PARAMS, cudaMemcpyDeviceToDevice, s));
    MLP_TRY(m, cudaMemsetAsync(m->Mo, 0, sizeof(float) * SPH_MLP_PARAMS, s));
    MLP_TRY(m, cudaMemsetAsync(m->Vo, 0, sizeof(float) * SPH_MLP_PARAMS, s));
    k_cast_weights<<<256, 256, 0, s>>>(m->P, m->W, m->WT);
    ++m->launches;
    MLP_TRY(m, cudaGetLastError());
    m->step = 0;
    return SPH_OK;
}

int sph_mlp_get_optimizer_state(sph_mlp* m, float* grads, float* m1, float* m2, long long* step, void* stream)
{
    if (!m || !grads || !m1 || !m2 || !step) return mfail(m, SPH_ERR_ARG, "NULL argument");
    cudaStream_t s = (cudaStream_t)stream;
    const size_t bytes = sizeof(float) * SPH_MLP_PARAMS;
    MLP_TRY(m, cudaMemcpyAsync(grads, m->G, bytes, cudaMemcpyDeviceToDevice, s));
    MLP_TRY(m, cudaMemcpyAsync(m1, m->Mo, bytes, cudaMemcpyDeviceToDevice, s));
    MLP_TRY(m, cudaMemcpyAsync(m2, m->Vo, bytes, cudaMemcpyDeviceToDevice, s));
    *step = m->step;
    return SPH_OK;
}

int sph_mlp_set_optimizer_state(sph_mlp* m, const float* m1, const float* m2, long long step, void* stream)
{
    if (!m || !m1 || !m2) return mfail(m, SPH_ERR_ARG, "NULL argument");
    if (step < 0) return mfail(m, SPH_ERR_ARG, "step must be >= 0");
    cudaStream_t s = (cudaStream_t)stream;
    const size_t bytes = sizeof(float) * SPH_MLP_PARAMS;
    MLP_TRY(m, cudaMemcpyAsync(m->Mo, m1, bytes, cudaMemcpyDeviceToDevice, s));
    MLP_TRY(m, cudaMemcpyAsync(m->Vo, m2, bytes, cudaMemcpyDeviceToDevice, s));
    m->step = step;
    return SPH_OK;
}

int sph_mlp_get_params(sph_mlp* m, float* params, void* stream)
{
    if (!m || !params) return mfail(m, SPH_ERR_ARG, "NULL argument");
    MLP_TRY(m, cudaMemcpyAsync(params, m->P, sizeof(float) * SPH_MLP_PARAMS, cudaMemcpyDeviceToDevice,
                               (cudaStream_t)stream));
    return SPH_OK;
}

int sph_mlp_forward(sph_mlp* m, const void* x, int B, float* y, void* stream)
{
    int rc = check_batch(m, B);
    if (rc != SPH_OK) return rc;
    if (!x || !y || ((uintptr_t)x & 15) || ((uintptr_t)y & 15))
        return mfail(m, SPH_ERR_ARG, "x and y must be 16-byte aligned");
    return mlp_forward_fused(m, (const __nv_bfloat16*)x, B, y, (cudaStream_t)stream);
}

int sph_mlp_gradients(sph_mlp* m, const void* x, const float* dy, int B, float* grads, void* stream)
{
    int rc = check_batch(m, B);
    if (rc != SPH_OK) return rc;
    if (!x || !dy || !grads || ((uintptr_t)x & 15)) return mfail(m, SPH_ERR_ARG, "bad pointers");
    return train_pass(m, (const __nv_bfloat16*)x, nullptr, dy, B, 0, grads, nullptr, nullptr, (cudaStream_t)stream);
}

int sph_mlp_train_step(sph_mlp* m, const void* x, const float* target, int B, int phase, float lr,
                       float* loss_out, void* stream)
{
    int rc = check_batch(m, B);
    if (rc != SPH_OK) return rc;
    if (!x || !target || ((uintptr_t)x & 15)) return mfail(m, SPH_ERR_ARG, "bad pointers");
    if (phase != 0 && phase != 1) return mfail(m, SPH_ERR_ARG, "phase must be 0 or 1");
    const float b1 = 0.9f, b2 = 0.999f;
    // bias corrections 1 - beta^t in double (in float32 the difference
    // cancels: 1 - 0.999^t loses most of its digits for small t)
    const double k = (double)(m->step + 1);
    const AdamArgs adam{lr, b1, b2, 1e-8f, (float)(1.0 - pow((double)b1, k)), (float)(1.0 - pow((double)b2, k)), phase};
    rc = train_pass(m, (const __nv_bfloat16*)x, target, nullptr, B, phase, nullptr, &adam,
                    loss_out ? loss_out : m->loss, (cudaStream_t)stream);
    if (rc == SPH_OK) ++m->step;
    return rc;
}

int sph_mlp_status(sph_mlp* m, unsigned* bits, void* stream)
{
    if (!m || !bits) return mfail(m, SPH_ERR_ARG, "NULL argument");
    unsigned v = 0;
    MLP_TRY(m, cudaMemcpyAsync(&v, m->err, sizeof(unsigned), cudaMemcpyDeviceToHost, (cudaStream_t)stream));
    MLP_TRY(m, cudaStreamSynchronize((cudaStream_t)stream));
    *bits = v;
    return SPH_OK;
}

long long sph_mlp_launch_count(sph_mlp* m) { return m ? m->launches : 0; }

int sph_debug_gelu(const float* z, int n, int grad, float* out, void* stream)
{
    if (!z || !out || n < 0 || grad < 0 || grad > 2) return mfail(nullptr, SPH_ERR_ARG, "bad GELU arguments");
    if (n == 0) return SPH_OK;
    k_debug_gelu<<<(n + 255) / 256, 256, 0, (cudaStream_t)stream>>>(z, n, grad, out);
    MLP_TRY(nullptr, cudaGetLastError());
    return SPH_OK;
}

int sph_debug_gemm(const void* A, int lda, const void* B, int ldb, int M, int N, int K, int splits, float* C,
                   unsigned* err, void* stream)
{
    if (!A || !B || !C || !err || M <= 0 || N <= 0 || K <= 0 || (lda & 7) || (ldb & 7) || (N & 3) || splits < 1)
        return mfail(nullptr, SPH_ERR_ARG, "bad GEMM arguments");
    if (((uintptr_t)A & 15) || ((uintptr_t)B & 15) || ((uintptr_t)C & 15))
        return mfail(nullptr, SPH_ERR_ARG, "A, B, C must be 16-byte aligned");
    GemmEpi e;
    memset(&e, 0, sizeof(e));
    e.err = err;
    e.out_f32 = C;
    e.ld_f32 = N;
    e.split_stride = (long long)M * N;
    long long launches = 0;
    const int NT = N <= 16 ? 16 : (N <= 128 ? 128 : 256);
    cudaError_t r = gemm(NT, (const __nv_bfloat16*)A, lda, (const __nv_bfloat16*)B, ldb, M, N, K, splits,
                         e, (cudaStream_t)stream, &launches);
    if (r != cudaSuccess) return mfail(nullptr, SPH_ERR_CUDA, "GEMM: %s", cudaGetErrorString(r));
    return SPH_OK;
}

}  // extern "C"
