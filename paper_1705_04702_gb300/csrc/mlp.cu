// MLP surrogate of the dust-emission step: 32 band features -> 128 -> 128 ->
// 100 emission-shape logits (SiLU, SiLU, softmax).
//
// Inference (mlp_infer_kernel): one warp per 32 rows, the three layers as
// BF16 tensor-core products with FP32 accumulation (mma.sync m16n8k16 in
// inline PTX); weights staged once per block in shared memory, each fragment of
// them used for the warp's two 16-row tiles; activations go through the warp's
// own shared memory, so that the layers are loops over pairs of n-tiles that
// stay in the instruction cache.  Softmax over the 100 outputs is reduced across
// the four lanes that hold a row; the result times the cell's absorbed power
// is written as FP64 emission.  The same pass flags rows whose raw features
// leave the training hull (lane = row).  What bounds it are the tile's chains of
// dependent products and exponentials at 12 warps per SM (issue 47%, tensor pipe
// 25%): 4e6 dense rows 1.34 ms (42% of the copy rate), 8e6 torus rows 1.84 ms.
// With 16-row tiles, every layer unrolled and activations in registers the code
// outgrew the instruction cache (2.9 fetch stalls per issue): 1.57 and 2.45 ms,
// the same rows bit for bit; 10 or 8 warps of this form take 1.57 and 1.68 ms.
//
// Training (skirt_mlp_train): FP32 master weights; every step is one fused
// tensor-core kernel per 32 rows (forward, softmax cross-entropy, backward,
// weight-gradient products; mlp_train.cu) and one kernel that sums the
// partial gradients in order, takes the Adam step (cosine step decay) and
// refreshes the BF16 weights.  The standardisation, the hull and the guard come
// from two passes over the features and a radix selection on the device (0.9 ms
// for 3e5 rows; 2.5 with one block per feature and the selection on the host).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <mutex>
#include <vector>

#include "async_copy.cuh"
#include "skirt_internal.cuh"

namespace skirt {
namespace {

constexpr int NIN = SKIRT_NBANDS;      // 32
constexpr int NH = SKIRT_MLP_HIDDEN;   // 128
constexpr int NO = SKIRT_NEMIT;        // 100
constexpr int NO_PAD = 104;            // 13 n-tiles of 8
constexpr int NPARAM = SKIRT_MLP_NPARAM;
constexpr int OFF_W1 = 0, OFF_B1 = OFF_W1 + NH * NIN, OFF_W2 = OFF_B1 + NH, OFF_B2 = OFF_W2 + NH * NH,
              OFF_W3 = OFF_B2 + NH, OFF_B3 = OFF_W3 + NO * NH;
static_assert(OFF_B3 + NO == NPARAM, "packed parameter layout");

#define MCK(call)                                                                                       \
    do {                                                                                                \
        cudaError_t e_ = (call);                                                                        \
        if (e_ != cudaSuccess)                                                                          \
            return set_error(e_ == cudaErrorMemoryAllocation ? SKIRT_ERR_OOM : SKIRT_ERR_CUDA,          \
                             "%s failed: %s (%s:%d)", #call, cudaGetErrorString(e_), __FILE__, __LINE__); \
    } while (0)

// --------------------------------------------------------------------------
// inference
// --------------------------------------------------------------------------
constexpr int INF_WARPS = 12;
constexpr int INF_TILE = 32;                    // rows of a warp's tile
constexpr int INF_ROWS = INF_TILE * INF_WARPS;
// shared memory: W1 [128][32], W2 [128][128], W3 [104][128] (bf16) with
// every row padded by 8 elements, so that the eight rows one matrix load
// touches start 4 banks apart (conflict-free); biases [128 + 128 + 104]
// (fp32); mean / inv_std / lo / hi [32] each; per warp the feature tile that the
// bulk copy engine fills, the activations and an mbarrier
constexpr int KP1 = NIN + 8, KP2 = NH + 8;
constexpr size_t SM_W1 = 0;
constexpr size_t SM_W2 = SM_W1 + sizeof(uint16_t) * NH * KP1;
constexpr size_t SM_W3 = SM_W2 + sizeof(uint16_t) * NH * KP2;
constexpr size_t SM_B = SM_W3 + sizeof(uint16_t) * NO_PAD * KP2;
constexpr size_t SM_ST = SM_B + sizeof(float) * (NH + NH + NO_PAD);
constexpr size_t SM_X = (SM_ST + sizeof(float) * 4 * NIN + 127) & ~(size_t)127;  // [warp][32][32] fp32
constexpr size_t SM_A = SM_X + sizeof(float) * INF_WARPS * INF_TILE * NIN;         // [warp][32][KP2] bf16
constexpr size_t SM_BAR = SM_A + sizeof(uint16_t) * INF_WARPS * INF_TILE * KP2;
constexpr size_t SM_TOTAL = SM_BAR + sizeof(unsigned long long) * INF_WARPS;
static_assert(SM_TOTAL <= 227 * 1024, "shared memory of one block");
static_assert((KP1 * 2) % 16 == 0 && (KP2 * 2) % 16 == 0 && SM_ST % 16 == 0 && SM_A % 16 == 0 && SM_BAR % 8 == 0,
              "padded rows and parts keep 16-byte alignment");

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi)
{
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&v);
}

__device__ __forceinline__ void mma_bf16(float* c, uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                         uint32_t b1)
{
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

__device__ __forceinline__ float silu_f(float z) { return __fdividef(z, 1.f + __expf(-z)); }

// FP32 -> FP64 for a non-negative float by IEEE-754 field manipulation on the
// integer pipe (exact for normal floats; zero and subnormals map to zero), so
// that the epilogue issues no FP64-pipe instruction; infinities, NaN and
// negative values take the ordinary conversion
__device__ __forceinline__ double widen_pos(float f)
{
    const unsigned u = __float_as_uint(f);
    const unsigned e = u >> 23;
    if (e >= 255u) return (double)f;
    return e ? __hiloint2double((int)((u >> 3) + 0x38000000u), (int)(u << 29)) : 0.0;
}

__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], const void* p)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(smem_u32(p)));
}

// A fragments (16 x 16 KT) of the rows from r0 of the activations
template <int KT>
__device__ __forceinline__ void load_afrag(uint32_t (&a)[KT][4], const uint16_t* act, int r0, int lane)
{
    const int q = lane >> 3, j = lane & 7;
#pragma unroll
    for (int kk = 0; kk < KT; ++kk) ldsm4(a[kk], act + (r0 + (q & 1) * 8 + j) * KP2 + 16 * kk + (q >> 1) * 8);
}

// B fragments of the n-tiles at row n0 and n0 + 8 of W (row stride KP) for k-tile
// kk: b[0], b[1] and b[2], b[3]
template <int KP>
__device__ __forceinline__ void load_bfrag2(uint32_t (&b)[4], const uint16_t* W, int n0, int kk, int lane)
{
    const int q = lane >> 3, j = lane & 7;
    ldsm4(b, W + (n0 + (q >> 1) * 8 + j) * KP + 16 * kk + (q & 1) * 8);
}

// One hidden layer: act[32][8 NT] = SiLU(act[32][16 KT] W^T + bias) in place (the
// inputs are in registers before the first output is written)
template <int NT, int KT, int KP>
__device__ __forceinline__ void hidden_layer(uint16_t* act, const uint16_t* W, const float* bias, int lane)
{
    const int g = lane >> 2, t = lane & 3;
    uint32_t a0[KT][4], a1[KT][4];
    load_afrag<KT>(a0, act, 0, lane);
    load_afrag<KT>(a1, act, 16, lane);
    __syncwarp();
#pragma unroll 1
    for (int n0 = 0; n0 < 8 * NT; n0 += 16) {
        float c[2][2][4];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const float2 bb = *reinterpret_cast<const float2*>(bias + n0 + 8 * u + 2 * t);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                c[h][u][0] = c[h][u][2] = bb.x;
                c[h][u][1] = c[h][u][3] = bb.y;
            }
        }
#pragma unroll
        for (int kk = 0; kk < KT; ++kk) {
            uint32_t b[4];
            load_bfrag2<KP>(b, W, n0, kk, lane);
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                mma_bf16(c[0][u], a0[kk][0], a0[kk][1], a0[kk][2], a0[kk][3], b[2 * u], b[2 * u + 1]);
                mma_bf16(c[1][u], a1[kk][0], a1[kk][1], a1[kk][2], a1[kk][3], b[2 * u], b[2 * u + 1]);
            }
        }
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                uint16_t* o = act + (16 * h + g) * KP2 + n0 + 8 * u + 2 * t;
                *reinterpret_cast<uint32_t*>(o) = pack_bf16(silu_f(c[h][u][0]), silu_f(c[h][u][1]));
                *reinterpret_cast<uint32_t*>(o + 8 * KP2) = pack_bf16(silu_f(c[h][u][2]), silu_f(c[h][u][3]));
            }
    }
    __syncwarp();
}

// zeros into `count` emission rows from row r
__device__ __forceinline__ void zero_rows(double* emission, long long r, int count, int lane)
{
    double2* o = reinterpret_cast<double2*>(emission + r * NO);
    for (int k = lane; k < count * (NO / 2); k += 32) __stcs(o + k, make_double2(0.0, 0.0));
}

__global__ void __launch_bounds__(32 * INF_WARPS, 1) mlp_infer_kernel(
    const uint16_t* __restrict__ Wg, const float* __restrict__ Bg, const float* __restrict__ stats,
    const float* __restrict__ features, const double* __restrict__ total, long long n,
    double* __restrict__ emission, unsigned char* __restrict__ flags, float inv_share_max, int* timeout)
{
    extern __shared__ __align__(128) unsigned char sm[];
    // stage the weights (bf16, contiguous W1 W2 W3) and biases / statistics
    {
        // 16-byte chunks of the contiguous global rows into the padded rows
        const uint4* src = reinterpret_cast<const uint4*>(Wg);
        constexpr int c1 = NIN / 8, c2 = NH / 8;  // chunks per row
        for (int i = threadIdx.x; i < NH * c1; i += blockDim.x)
            *reinterpret_cast<uint4*>(sm + SM_W1 + sizeof(uint16_t) * ((i / c1) * KP1 + 8 * (i % c1))) = src[i];
        src += NH * c1;
        for (int i = threadIdx.x; i < NH * c2; i += blockDim.x)
            *reinterpret_cast<uint4*>(sm + SM_W2 + sizeof(uint16_t) * ((i / c2) * KP2 + 8 * (i % c2))) = src[i];
        src += NH * c2;
        for (int i = threadIdx.x; i < NO_PAD * c2; i += blockDim.x)
            *reinterpret_cast<uint4*>(sm + SM_W3 + sizeof(uint16_t) * ((i / c2) * KP2 + 8 * (i % c2))) = src[i];
        float* sb = reinterpret_cast<float*>(sm + SM_B);
        for (int i = threadIdx.x; i < NH + NH + NO_PAD; i += blockDim.x) sb[i] = Bg[i];
        float* ss = reinterpret_cast<float*>(sm + SM_ST);
        for (int i = threadIdx.x; i < 4 * NIN; i += blockDim.x) ss[i] = stats[i];
    }
    __syncthreads();
    const uint16_t* W1 = reinterpret_cast<const uint16_t*>(sm + SM_W1);
    const uint16_t* W2 = reinterpret_cast<const uint16_t*>(sm + SM_W2);
    const uint16_t* W3 = reinterpret_cast<const uint16_t*>(sm + SM_W3);
    const float* B1 = reinterpret_cast<const float*>(sm + SM_B);
    const float* B2 = B1 + NH;
    const float* B3 = B2 + NH;
    const float4* mean4 = reinterpret_cast<const float4*>(sm + SM_ST);
    const float4* istd4 = mean4 + NIN / 4;
    const float4* lo4 = istd4 + NIN / 4;
    const float4* hi4 = lo4 + NIN / 4;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = lane >> 2, t = lane & 3;
    float* xbuf = reinterpret_cast<float*>(sm + SM_X) + warp * INF_TILE * NIN;
    uint16_t* act = reinterpret_cast<uint16_t*>(sm + SM_A) + warp * INF_TILE * KP2;
    unsigned long long* bar = reinterpret_cast<unsigned long long*>(sm + SM_BAR) + warp;
    if (lane == 0) {
        mbar_init(bar, 1);
        fence_barrier_init();
    }
    __syncwarp();
    const long long stride = (long long)gridDim.x * INF_ROWS;
    // the feature rows of the tile at row b (fewer at the end), 128 bytes each
    auto fetch = [&](long long b) {
        const long long rows = n - b < INF_TILE ? n - b : INF_TILE;
        fence_proxy_async();
        bulk_load(xbuf, features + b * NIN, (unsigned)(rows * NIN * sizeof(float)), bar);
    };
    long long base = (long long)blockIdx.x * INF_ROWS + warp * INF_TILE;
    if (lane == 0 && base < n) fetch(base);
    unsigned parity = 0;
    for (; base < n; base += stride, parity ^= 1u) {
        const int rows = n - base < INF_TILE ? (int)(n - base) : INF_TILE;
        const double tot = lane < rows ? __ldcs(total + base + lane) : 0.0;  // of row `lane`
        if (!__all_sync(0xffffffffu, mbar_wait(bar, parity))) {
            atomicOr(timeout, 1);
            mbar_wait(bar, parity);  // the copy lands in this block's memory: give it its time
            break;
        }
        // ---- lane = row: the row's features in 8 groups of four, in an order rotated
        // by the lane (the rows lie 32 banks apart), standardised into act, and the
        // guard.  A row leaves the training hull when a feature leaves its range, or
        // when its dominant band holds a larger share of the cell's absorbed power
        // than the guard allows: sum_b 10^(f_b - f_max) is the inverse of that share.
        // The sum joins groups 4, 2, 1 apart and then the four places, an order that
        // the rotation leaves alone.
        {
            float4 v[8];
            float mx = -INFINITY;
            bool in = true;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const int c = (k + lane) & 7;
                v[k] = reinterpret_cast<const float4*>(xbuf + lane * NIN)[c];
                const float4 mu = mean4[c], is = istd4[c];
                *reinterpret_cast<uint2*>(act + lane * KP2 + 4 * c) =
                    make_uint2(pack_bf16((v[k].x - mu.x) * is.x, (v[k].y - mu.y) * is.y),
                               pack_bf16((v[k].z - mu.z) * is.z, (v[k].w - mu.w) * is.w));
                if (flags) {
                    const float4 l = lo4[c], h = hi4[c];
                    in = in && v[k].x >= l.x && v[k].x <= h.x && v[k].y >= l.y && v[k].y <= h.y && v[k].z >= l.z &&
                         v[k].z <= h.z && v[k].w >= l.w && v[k].w <= h.w;
                    mx = fmaxf(mx, fmaxf(fmaxf(v[k].x, v[k].y), fmaxf(v[k].z, v[k].w)));
                }
            }
            if (flags) {
                const auto ex = [&](float f) { return exp2f((f - mx) * 3.32192809f); };
                float4 e[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) e[k] = make_float4(ex(v[k].x), ex(v[k].y), ex(v[k].z), ex(v[k].w));
                const auto add = [](float4 p, float4 q) {
                    return make_float4(p.x + q.x, p.y + q.y, p.z + q.z, p.w + q.w);
                };
#pragma unroll
                for (int k = 0; k < 4; ++k) e[k] = add(e[k], e[k + 4]);
                e[0] = add(e[0], e[2]);
                e[1] = add(e[1], e[3]);
                e[0] = add(e[0], e[1]);
                const float sum = (e[0].x + e[0].z) + (e[0].y + e[0].w);
                // a cell without absorbed power emits nothing: no fallback needed
                if (lane < rows) flags[base + lane] = (!in || sum < inv_share_max) && tot > 0.0 ? 1 : 0;
            }
        }
        __syncwarp();  // every lane is done with the feature tile
        if (lane == 0 && base + stride < n) fetch(base + stride);
        // a tile none of whose 32 rows absorbs power (empty space): its emission rows
        // are zeros (the epilogue scales every row by its FP32 total), so its products
        // are skipped; so is the last layer of a half of the tile
        const float ftot = (float)tot;
        const unsigned live = __ballot_sync(0xffffffffu, ftot != 0.f);
        if (live == 0u) {
            zero_rows(emission, base, rows, lane);
            continue;
        }
        // ---- layers
        hidden_layer<NH / 8, 2, KP1>(act, W1, B1, lane);
        hidden_layer<NH / 8, NH / 16, KP2>(act, W2, B2, lane);
#pragma unroll 1
        for (int h = 0; h < 2; ++h) {
            const long long r0 = base + 16 * h + g, r1 = r0 + 8;
            if (((live >> (16 * h)) & 0xFFFFu) == 0u) {
                if (rows > 16 * h) zero_rows(emission, base + 16 * h, rows - 16 * h < 16 ? rows - 16 * h : 16, lane);
                continue;
            }
            uint32_t a[NH / 16][4];
            load_afrag<NH / 16>(a, act, 16 * h, lane);
            float z[NO_PAD / 8][4];
#pragma unroll
            for (int j = 0; j < NO_PAD / 8; ++j) {
                const float2 bb = *reinterpret_cast<const float2*>(B3 + 8 * j + 2 * t);
                z[j][0] = z[j][2] = bb.x;
                z[j][1] = z[j][3] = bb.y;
            }
            // n-tiles in pairs (the last alone), two k-tiles per matrix load for it
#pragma unroll
            for (int j = 0; j + 1 < NO_PAD / 8; j += 2)
#pragma unroll
                for (int kk = 0; kk < NH / 16; ++kk) {
                    uint32_t b[4];
                    load_bfrag2<KP2>(b, W3, 8 * j, kk, lane);
                    mma_bf16(z[j], a[kk][0], a[kk][1], a[kk][2], a[kk][3], b[0], b[1]);
                    mma_bf16(z[j + 1], a[kk][0], a[kk][1], a[kk][2], a[kk][3], b[2], b[3]);
                }
            {
                constexpr int j = NO_PAD / 8 - 1;
                const int q = lane >> 3, r = lane & 7;
#pragma unroll
                for (int kk = 0; kk < NH / 16; kk += 2) {
                    uint32_t b[4];
                    ldsm4(b, W3 + (8 * j + r) * KP2 + 16 * kk + q * 8);
                    mma_bf16(z[j], a[kk][0], a[kk][1], a[kk][2], a[kk][3], b[0], b[1]);
                    mma_bf16(z[j], a[kk + 1][0], a[kk + 1][1], a[kk + 1][2], a[kk + 1][3], b[2], b[3]);
                }
            }
            // ---- softmax over the 100 outputs of rows g and g+8 (4 lanes per row)
            float m0 = -3.0e38f, m1 = -3.0e38f;
#pragma unroll
            for (int j = 0; j < NO_PAD / 8; ++j) {
                if (8 * j + 2 * t < NO) { m0 = fmaxf(m0, fmaxf(z[j][0], z[j][1])); m1 = fmaxf(m1, fmaxf(z[j][2], z[j][3])); }
            }
            m0 = fmaxf(m0, __shfl_xor_sync(0xffffffffu, m0, 1));
            m0 = fmaxf(m0, __shfl_xor_sync(0xffffffffu, m0, 2));
            m1 = fmaxf(m1, __shfl_xor_sync(0xffffffffu, m1, 1));
            m1 = fmaxf(m1, __shfl_xor_sync(0xffffffffu, m1, 2));
            float s0 = 0.f, s1 = 0.f;
#pragma unroll
            for (int j = 0; j < NO_PAD / 8; ++j) {
                const bool ok = 8 * j + 2 * t < NO;
                z[j][0] = ok ? __expf(z[j][0] - m0) : 0.f;
                z[j][1] = ok ? __expf(z[j][1] - m0) : 0.f;
                z[j][2] = ok ? __expf(z[j][2] - m1) : 0.f;
                z[j][3] = ok ? __expf(z[j][3] - m1) : 0.f;
                s0 += z[j][0] + z[j][1];
                s1 += z[j][2] + z[j][3];
            }
            s0 += __shfl_xor_sync(0xffffffffu, s0, 1);
            s0 += __shfl_xor_sync(0xffffffffu, s0, 2);
            s1 += __shfl_xor_sync(0xffffffffu, s1, 1);
            s1 += __shfl_xor_sync(0xffffffffu, s1, 2);
            // emission = shape x absorbed power, formed in FP32 (the shape is an FP32
            // softmax) and widened exactly to FP64
            const float f0 = __shfl_sync(0xffffffffu, ftot, 16 * h + g) / s0;
            const float f1 = __shfl_sync(0xffffffffu, ftot, 16 * h + g + 8) / s1;
#pragma unroll
            for (int j = 0; j < NO_PAD / 8; ++j) {
                const int c = 8 * j + 2 * t;
                if (c < NO) {
                    if (r0 < n)
                        __stcs(reinterpret_cast<double2*>(emission + r0 * NO + c),
                               make_double2(widen_pos(f0 * z[j][0]), widen_pos(f0 * z[j][1])));
                    if (r1 < n)
                        __stcs(reinterpret_cast<double2*>(emission + r1 * NO + c),
                               make_double2(widen_pos(f1 * z[j][2]), widen_pos(f1 * z[j][3])));
                }
            }
        }
        __syncwarp();  // every lane is done with the activations
    }
}

// --------------------------------------------------------------------------
// training helpers (the step itself is in mlp_train.cu)
// --------------------------------------------------------------------------
// out[r][c] = in[r][c] / sum_c in[r][c] in FP32 (one warp per row; zero rows stay zero)
__global__ void normalize_rows_kernel(const double* __restrict__ in, float* __restrict__ out, long long rows)
{
    const long long r = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (r >= rows) return;
    double s = 0.0;
    for (int c = lane; c < NO; c += 32) s += in[r * NO + c];
    for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    const double inv = s > 0.0 ? 1.0 / s : 0.0;
    for (int c = lane; c < NO; c += 32) out[r * NO + c] = (float)(in[r * NO + c] * inv);
}

// share of a row's absorbed power in its dominant band, from its 32 band
// features (log10 of the band powers per unit mass): 1 / sum_b 10^(f_b - f_max)
__global__ void dominant_share_kernel(const float* __restrict__ feat, long long n, float* __restrict__ share)
{
    for (long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x; r < n; r += (long long)gridDim.x * blockDim.x) {
        const float* f = feat + r * NIN;
        float m = f[0];
        for (int b = 1; b < NIN; ++b) m = fmaxf(m, f[b]);
        float e = 0.f;
        for (int b = 0; b < NIN; ++b) e += exp2f((f[b] - m) * 3.32192809f);
        share[r] = 1.f / e;
    }
}

// Per-feature sums over n samples (sum, sum of squares, min, max): lane = feature, a
// warp per row, so that a row is one 128-byte read and its FP64 additions serve 32
// features; the blocks' partial results [block][32][4] are joined in block order
// by the second kernel.
constexpr int STAT_BLOCKS = 152, STAT_WARPS = 8;

__global__ void __launch_bounds__(32 * STAT_WARPS) feature_stats_kernel(const float* __restrict__ feat, long long n,
                                                                        double* __restrict__ part)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double s = 0.0, s2 = 0.0;
    float lo = 3.0e38f, hi = -3.0e38f;
    for (long long r = (long long)blockIdx.x * STAT_WARPS + warp; r < n; r += (long long)gridDim.x * STAT_WARPS) {
        const float v = feat[r * NIN + lane];
        s += v;
        s2 += (double)v * v;
        lo = fminf(lo, v);
        hi = fmaxf(hi, v);
    }
    __shared__ double rs[STAT_WARPS][32], rs2[STAT_WARPS][32];
    __shared__ float rl[STAT_WARPS][32], rh[STAT_WARPS][32];
    rs[warp][lane] = s; rs2[warp][lane] = s2; rl[warp][lane] = lo; rh[warp][lane] = hi;
    __syncthreads();
    if (warp > 0) return;
    for (int w = 1; w < STAT_WARPS; ++w) {
        s += rs[w][lane];
        s2 += rs2[w][lane];
        lo = fminf(lo, rl[w][lane]);
        hi = fmaxf(hi, rh[w][lane]);
    }
    double* o = part + ((size_t)blockIdx.x * 32 + lane) * 4;
    o[0] = s; o[1] = s2; o[2] = lo; o[3] = hi;
}

__global__ void feature_stats_join_kernel(const double* __restrict__ part, int nblocks, double* __restrict__ out)
{
    const int c = threadIdx.x;  // one warp
    double s = 0.0, s2 = 0.0, lo = 3.0e38, hi = -3.0e38;
    for (int b = 0; b < nblocks; ++b) {
        const double* p = part + ((size_t)b * 32 + c) * 4;
        s += p[0];
        s2 += p[1];
        lo = p[2] < lo ? p[2] : lo;
        hi = p[3] > hi ? p[3] : hi;
    }
    out[4 * c + 0] = s;
    out[4 * c + 1] = s2;
    out[4 * c + 2] = lo;
    out[4 * c + 3] = hi;
}

// The k-th smallest of n non-negative floats by their bits, 11 + 11 + 10 of them at a
// time: a histogram of the next bits of the values that agree so far, then the
// bin that holds rank k.  state: [0] the bits found, [1] the rank left.
constexpr int SEL_BINS = 2048;

__global__ void select_hist_kernel(const float* __restrict__ v, long long n, const unsigned long long* state, int shift,
                                   int bits, unsigned* __restrict__ hist)
{
    __shared__ unsigned h[SEL_BINS];
    for (int i = threadIdx.x; i < SEL_BINS; i += blockDim.x) h[i] = 0u;
    __syncthreads();
    const unsigned found = (unsigned)state[0];
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const unsigned u = __float_as_uint(v[i]);
        if (shift + bits >= 32 || (u >> (shift + bits)) == found) atomicAdd(&h[(u >> shift) & ((1u << bits) - 1u)], 1u);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < SEL_BINS; i += blockDim.x)
        if (h[i]) atomicAdd(&hist[i], h[i]);
}

__global__ void select_bin_kernel(unsigned* __restrict__ hist, unsigned long long* state, int bits)
{
    // one warp: lane l sums its 64 bins, then the lane holding the rank walks them
    constexpr int PER = SEL_BINS / 32;
    const int lane = threadIdx.x;
    unsigned long long sum = 0;
    for (int i = 0; i < PER; ++i) sum += hist[lane * PER + i];
    unsigned long long inc = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    const unsigned long long k = state[1], before = inc - sum;
    __syncwarp();
    if (k >= before && k < inc) {
        unsigned long long left = k - before;
        int b = lane * PER;
        while (left >= hist[b]) left -= hist[b++];
        state[0] = (state[0] << bits) | (unsigned)b;
        state[1] = left;
    }
    __syncwarp();
    for (int i = 0; i < PER; ++i) hist[lane * PER + i] = 0u;
}

// bf16 copies of the weights (W3 padded to 104 rows with zeros) and the fp32
// biases (b3 padded with -inf-like values so that padded logits vanish)
__global__ void pack_inference_kernel(const float* __restrict__ P, uint16_t* __restrict__ W, float* __restrict__ B)
{
    const int nW = NH * NIN + NH * NH + NO_PAD * NH;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < nW; i += gridDim.x * blockDim.x) {
        float v;
        if (i < NH * NIN) v = P[OFF_W1 + i];
        else if (i < NH * NIN + NH * NH) v = P[OFF_W2 + (i - NH * NIN)];
        else {
            const int k = i - NH * NIN - NH * NH;
            v = k < NO * NH ? P[OFF_W3 + k] : 0.f;
        }
        __nv_bfloat16 b = __float2bfloat16_rn(v);
        W[i] = *reinterpret_cast<uint16_t*>(&b);
    }
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < NH + NH + NO_PAD; i += gridDim.x * blockDim.x) {
        if (i < NH) B[i] = P[OFF_B1 + i];
        else if (i < 2 * NH) B[i] = P[OFF_B2 + i - NH];
        else B[i] = (i - 2 * NH) < NO ? P[OFF_B3 + i - 2 * NH] : -1.0e30f;
    }
}

int blocks_for(long long n, int block)
{
    long long b = (n + block - 1) / block;
    if (b > 4096) b = 4096;
    return (int)(b < 1 ? 1 : b);
}

// splitmix64: the library's host-side generator for the initial weights
uint64_t splitmix64(uint64_t& s)
{
    uint64_t z = (s += 0x9E3779B97F4A7C15ull);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

}  // namespace
}  // namespace skirt

using namespace skirt;

struct skirt_mlp_s {
    float* P = nullptr;        // FP32 master parameters [NPARAM]
    float* G = nullptr;        // gradient [NPARAM]
    float* Mo = nullptr;       // Adam first moment
    float* Vo = nullptr;       // Adam second moment
    uint16_t* Wb = nullptr;    // bf16 weights for inference
    float* Bb = nullptr;       // fp32 biases for inference (b3 padded)
    float* stats = nullptr;    // device: mean[32], 1/std[32], lo[32], hi[32]
    float host_stats[4 * NIN]; // mean, std, lo, hi
    float share_max = 1.f;     // guard: rows whose dominant band holds more of the power go to the exact solver
    bool packed = false;
    // working tables of skirt_dust_emission's surrogate mode (features, totals,
    // flags, fallback rows), grown on demand and kept until the network is
    // destroyed; ws_mu serialises the calls that use them
    std::mutex ws_mu;
    void* ws = nullptr;
    size_t ws_bytes = 0;
};

namespace skirt {

static int upload_stats(skirt_mlp_s* net)
{
    float d[4 * NIN];
    for (int k = 0; k < NIN; ++k) {
        d[k] = net->host_stats[k];
        d[NIN + k] = 1.f / net->host_stats[NIN + k];
        d[2 * NIN + k] = net->host_stats[2 * NIN + k];
        d[3 * NIN + k] = net->host_stats[3 * NIN + k];
    }
    MCK(cudaMemcpy(net->stats, d, sizeof d, cudaMemcpyHostToDevice));
    return SKIRT_OK;
}

static int repack(skirt_mlp_s* net, cudaStream_t s)
{
    pack_inference_kernel<<<64, 256, 0, s>>>(net->P, net->Wb, net->Bb);
    MCK(cudaGetLastError());
    net->packed = true;
    return SKIRT_OK;
}

std::mutex& mlp_workspace_mutex(skirt_mlp_s* net) { return net->ws_mu; }

int mlp_workspace(skirt_mlp_s* net, size_t bytes, void** p)
{
    if (bytes > net->ws_bytes) {
        // the previous calls have synchronised their streams: the old tables are idle
        cudaFree(net->ws);
        net->ws = nullptr;
        net->ws_bytes = 0;
        MCK(cudaMalloc(&net->ws, bytes));
        net->ws_bytes = bytes;
    }
    *p = net->ws;
    return SKIRT_OK;
}

// timeout: a zero in device memory that belongs to the call (concurrent calls must
// not clear or see each other's); a wait for a bulk copy that runs out sets it, and
// mlp_check_timeout reports what the call read back from it
int mlp_forward_internal(skirt_mlp_s* net, const float* features, const double* total, long long n, double* emission,
                         unsigned char* flags, int* timeout, cudaStream_t s)
{
    if ((reinterpret_cast<uintptr_t>(features) & 15) != 0)
        return set_error(SKIRT_ERR_INVALID_ARG, "features must be 16-byte aligned");
    if (!net->packed) {
        int r = repack(net, s);
        if (r) return r;
    }
    MCK(cudaFuncSetAttribute(mlp_infer_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SM_TOTAL));
    int sms = 0, dev = 0, per_sm = 0;
    MCK(cudaGetDevice(&dev));
    MCK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    MCK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, mlp_infer_kernel, 32 * INF_WARPS, SM_TOTAL));
    long long tiles = (n + INF_ROWS - 1) / INF_ROWS;
    long long grid = (long long)sms * (per_sm > 0 ? per_sm : 1);
    if (grid > tiles) grid = tiles;
    if (grid < 1) grid = 1;
    const float inv_share_max = net->share_max > 0.f ? 1.f / net->share_max : 3.0e38f;
    mlp_infer_kernel<<<(int)grid, 32 * INF_WARPS, SM_TOTAL, s>>>(net->Wb, net->Bb, net->stats, features, total, n,
                                                                  emission, flags, inv_share_max, timeout);
    MCK(cudaGetLastError());
    return SKIRT_OK;
}

int mlp_check_timeout(int v)
{
    return v ? set_error(SKIRT_ERR_CUDA, "surrogate inference: a feature copy did not complete in time") : SKIRT_OK;
}

}  // namespace skirt

// ---------------------------------------------------------------- C ABI
extern "C" int skirt_mlp_create(skirt_mlp_t* out, uint64_t seed)
{
    if (!out) return set_error(SKIRT_ERR_INVALID_ARG, "out is NULL");
    *out = nullptr;
    skirt_mlp_s* net = new skirt_mlp_s;
    auto bail = [&](int code) {
        skirt_mlp_destroy(net);
        return code;
    };
    cudaError_t e;
    if ((e = cudaMalloc(&net->P, sizeof(float) * NPARAM)) || (e = cudaMalloc(&net->G, sizeof(float) * NPARAM)) ||
        (e = cudaMalloc(&net->Mo, sizeof(float) * NPARAM)) || (e = cudaMalloc(&net->Vo, sizeof(float) * NPARAM)) ||
        (e = cudaMalloc(&net->Wb, sizeof(uint16_t) * (NH * NIN + NH * NH + NO_PAD * NH))) ||
        (e = cudaMalloc(&net->Bb, sizeof(float) * (NH + NH + NO_PAD))) ||
        (e = cudaMalloc(&net->stats, sizeof(float) * 4 * NIN)))
        return bail(set_error(SKIRT_ERR_OOM, "mlp buffers: %s", cudaGetErrorString(e)));
    // Kaiming-uniform weights U(-sqrt(6 / fan_in), +sqrt(6 / fan_in)), zero biases
    std::vector<float> h(NPARAM, 0.f);
    uint64_t st = seed;
    auto fill = [&](int off, int rows, int cols) {
        const double b = std::sqrt(6.0 / cols);
        for (int i = 0; i < rows * cols; ++i) {
            const double u = (double)(splitmix64(st) >> 11) * (1.0 / 9007199254740992.0);
            h[off + i] = (float)((2.0 * u - 1.0) * b);
        }
    };
    fill(OFF_W1, NH, NIN);
    fill(OFF_W2, NH, NH);
    fill(OFF_W3, NO, NH);
    if ((e = cudaMemcpy(net->P, h.data(), sizeof(float) * NPARAM, cudaMemcpyHostToDevice)))
        return bail(set_error(SKIRT_ERR_CUDA, "mlp init: %s", cudaGetErrorString(e)));
    for (int k = 0; k < NIN; ++k) {
        net->host_stats[k] = 0.f;
        net->host_stats[NIN + k] = 1.f;
        net->host_stats[2 * NIN + k] = -3.0e38f;
        net->host_stats[3 * NIN + k] = 3.0e38f;
    }
    if (int r = upload_stats(net)) return bail(r);
    *out = net;
    return SKIRT_OK;
}

extern "C" int skirt_mlp_destroy(skirt_mlp_t net)
{
    if (!net) return SKIRT_OK;
    cudaFree(net->P);
    cudaFree(net->G);
    cudaFree(net->Mo);
    cudaFree(net->Vo);
    cudaFree(net->Wb);
    cudaFree(net->Bb);
    cudaFree(net->stats);
    cudaFree(net->ws);
    delete net;
    return SKIRT_OK;
}

extern "C" int skirt_mlp_set_params(skirt_mlp_t net, const float* params, const float* x_mean, const float* x_std,
                                    const float* hull_lo, const float* hull_hi)
{
    if (!net) return set_error(SKIRT_ERR_INVALID_ARG, "net is NULL");
    if (params) {
        for (int i = 0; i < NPARAM; ++i)
            if (!std::isfinite(params[i])) return set_error(SKIRT_ERR_INVALID_ARG, "params[%d] is not finite", i);
        MCK(cudaMemcpy(net->P, params, sizeof(float) * NPARAM, cudaMemcpyHostToDevice));
        net->packed = false;
    }
    if (x_std)
        for (int k = 0; k < NIN; ++k)
            if (!(x_std[k] > 0)) return set_error(SKIRT_ERR_INVALID_ARG, "x_std[%d] must be > 0", k);
    if (x_mean) std::memcpy(net->host_stats, x_mean, sizeof(float) * NIN);
    if (x_std) std::memcpy(net->host_stats + NIN, x_std, sizeof(float) * NIN);
    if (hull_lo) std::memcpy(net->host_stats + 2 * NIN, hull_lo, sizeof(float) * NIN);
    if (hull_hi) std::memcpy(net->host_stats + 3 * NIN, hull_hi, sizeof(float) * NIN);
    return upload_stats(net);
}

extern "C" int skirt_mlp_set_guard(skirt_mlp_t net, float share_max)
{
    if (!net) return set_error(SKIRT_ERR_INVALID_ARG, "net is NULL");
    if (!(share_max > 0.f)) return set_error(SKIRT_ERR_INVALID_ARG, "share_max must be > 0");
    net->share_max = share_max;
    return SKIRT_OK;
}

extern "C" int skirt_mlp_get_guard(skirt_mlp_t net, float* share_max)
{
    if (!net || !share_max) return set_error(SKIRT_ERR_INVALID_ARG, "net / share_max is NULL");
    *share_max = net->share_max;
    return SKIRT_OK;
}

extern "C" int skirt_mlp_get_params(skirt_mlp_t net, float* params, float* x_mean, float* x_std, float* hull_lo,
                                    float* hull_hi)
{
    if (!net) return set_error(SKIRT_ERR_INVALID_ARG, "net is NULL");
    if (params) MCK(cudaMemcpy(params, net->P, sizeof(float) * NPARAM, cudaMemcpyDeviceToHost));
    if (x_mean) std::memcpy(x_mean, net->host_stats, sizeof(float) * NIN);
    if (x_std) std::memcpy(x_std, net->host_stats + NIN, sizeof(float) * NIN);
    if (hull_lo) std::memcpy(hull_lo, net->host_stats + 2 * NIN, sizeof(float) * NIN);
    if (hull_hi) std::memcpy(hull_hi, net->host_stats + 3 * NIN, sizeof(float) * NIN);
    return SKIRT_OK;
}

extern "C" int skirt_mlp_train_opts_default(skirt_mlp_train_opts* o)
{
    if (!o) return set_error(SKIRT_ERR_INVALID_ARG, "opts is NULL");
    o->epochs = 200;
    o->batch = 2048;
    o->lr = 2e-3f;
    o->beta1 = 0.9f;
    o->beta2 = 0.999f;
    o->eps = 1e-8f;
    o->seed = 1;
    o->guard_quantile = 0.99f;
    return SKIRT_OK;
}

namespace {

// Per-call scratch of a training step: the per-CTA partial gradients and
// losses, and the loss accumulator.
struct Work {
    float* part = nullptr;
    float* part_loss = nullptr;
    float* loss = nullptr;
    cudaError_t alloc(int rows, cudaStream_t s)
    {
        const int ncta = (rows + train_rows_per_cta() - 1) / train_rows_per_cta();
        cudaError_t e;
        if ((e = cudaMallocAsync((void**)&part, sizeof(float) * (size_t)ncta * NPARAM, s))) return e;
        if ((e = cudaMallocAsync((void**)&part_loss, sizeof(float) * (size_t)ncta, s))) return e;
        if ((e = cudaMallocAsync((void**)&loss, sizeof(float), s))) return e;
        return cudaMemsetAsync(loss, 0, sizeof(float), s);
    }
    void release(cudaStream_t s)
    {
        for (float** p : {&part, &part_loss, &loss}) {
            if (*p) cudaFreeAsync(*p, s);
            *p = nullptr;
        }
    }
};

// steps per replayed graph
constexpr int TRAIN_UNROLL = 8;

// Everything a training call acquires, released on every return path (the
// stream-ordered frees go on the caller's stream, after the private stream's
// work has been joined to it).
struct TrainScope {
    cudaStream_t s = nullptr;
    Work w;
    float* target = nullptr;
    float* x_in = nullptr;    // the gradient call's copies of its rows
    float* t_in = nullptr;
    double* d_st = nullptr;
    unsigned long long* d_ab = nullptr;
    float* d_sched = nullptr;
    long long* d_t = nullptr;
    cudaStream_t cs = nullptr;
    cudaEvent_t ready = nullptr;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t gexec = nullptr;   // TRAIN_UNROLL steps
    cudaGraphExec_t gexec1 = nullptr;  // one step
    explicit TrainScope(cudaStream_t st) : s(st) {}
    ~TrainScope()
    {
        if (cs) {
            if (ready && cudaEventRecord(ready, cs) == cudaSuccess) cudaStreamWaitEvent(s, ready, 0);
            cudaStreamSynchronize(cs);
        }
        if (gexec) cudaGraphExecDestroy(gexec);
        if (gexec1) cudaGraphExecDestroy(gexec1);
        if (graph) cudaGraphDestroy(graph);
        if (cs) cudaStreamDestroy(cs);
        if (ready) cudaEventDestroy(ready);
        w.release(s);
        if (target) cudaFreeAsync(target, s);
        if (x_in) cudaFreeAsync(x_in, s);
        if (t_in) cudaFreeAsync(t_in, s);
        if (d_st) cudaFreeAsync(d_st, s);
        if (d_ab) cudaFreeAsync(d_ab, s);
        if (d_sched) cudaFreeAsync(d_sched, s);
        if (d_t) cudaFreeAsync(d_t, s);
        cudaGetLastError();
    }
};

}  // namespace

extern "C" int skirt_mlp_grad(skirt_mlp_t net, const float* x_std, const float* target, int n, float* grad,
                              float* loss, void* stream)
{
    if (!net || !x_std || !target || n < 1) return set_error(SKIRT_ERR_INVALID_ARG, "net / x_std / target / n");
    cudaStream_t s = (cudaStream_t)stream;
    TrainScope sc(s);
    Work& w = sc.w;
    MCK(w.alloc(n, s));
    float*& d_x = sc.x_in;
    float*& d_t = sc.t_in;
    MCK(cudaMallocAsync((void**)&d_x, sizeof(float) * (size_t)n * NIN, s));
    MCK(cudaMallocAsync((void**)&d_t, sizeof(float) * (size_t)n * NO, s));
    MCK(cudaMemcpyAsync(d_x, x_std, sizeof(float) * (size_t)n * NIN, cudaMemcpyDefault, s));
    MCK(cudaMemcpyAsync(d_t, target, sizeof(float) * (size_t)n * NO, cudaMemcpyDefault, s));
    if (int r = repack(net, s)) return r;
    MCK(launch_train_step(net->Wb, net->P, nullptr, d_t, nullptr, nullptr, nullptr, 0, n, d_x, n, w.part, w.part_loss,
                          net->G, 0, nullptr, nullptr, nullptr, nullptr, 0.f, 0.f, 0.f, nullptr, w.loss, 0, 0, s));
    if (grad) MCK(cudaMemcpyAsync(grad, net->G, sizeof(float) * NPARAM, cudaMemcpyDeviceToHost, s));
    float l = 0.f;
    MCK(cudaMemcpyAsync(&l, w.loss, sizeof(float), cudaMemcpyDeviceToHost, s));
    MCK(cudaStreamSynchronize(s));
    if (loss) *loss = l;
    return SKIRT_OK;
}

extern "C" int skirt_mlp_train(skirt_mlp_t net, const float* features, const double* emission, long long n,
                               const skirt_mlp_train_opts* opts, float* loss_history, void* stream)
{
    if (!net || !features || !emission || !opts) return set_error(SKIRT_ERR_INVALID_ARG, "net / data / opts is NULL");
    const int B = opts->batch;
    if (B < 32 || B > (1 << 16) || n < B) return set_error(SKIRT_ERR_INVALID_ARG, "batch must be in [32, 65536] and <= n");
    if (opts->epochs < 1 || !(opts->lr > 0)) return set_error(SKIRT_ERR_INVALID_ARG, "epochs / lr invalid");
    if (!(opts->guard_quantile > 0.f)) return set_error(SKIRT_ERR_INVALID_ARG, "guard_quantile must be > 0");
    cudaStream_t s = (cudaStream_t)stream;
    TrainScope sc(s);
    // target shapes: every emission row normalised to sum 1
    float*& target = sc.target;
    MCK(cudaMallocAsync((void**)&target, sizeof(float) * NO * (size_t)n, s));
    normalize_rows_kernel<<<(unsigned)((n * 32 + 255) / 256), 256, 0, s>>>(emission, target, n);
    MCK(cudaGetLastError());
    // standardisation and hull from the training features
    double*& d_st = sc.d_st;
    MCK(cudaMallocAsync((void**)&d_st, sizeof(double) * 4 * NIN * (STAT_BLOCKS + 1), s));
    const int stat_blocks = (int)std::min<long long>(STAT_BLOCKS, (n + STAT_WARPS - 1) / STAT_WARPS);
    feature_stats_kernel<<<stat_blocks, 32 * STAT_WARPS, 0, s>>>(features, n, d_st + 4 * NIN);
    feature_stats_join_kernel<<<1, NIN, 0, s>>>(d_st + 4 * NIN, stat_blocks, d_st);
    MCK(cudaGetLastError());
    double st[4 * NIN];
    MCK(cudaMemcpyAsync(st, d_st, sizeof st, cudaMemcpyDeviceToHost, s));
    MCK(cudaStreamSynchronize(s));
    for (int k = 0; k < NIN; ++k) {
        const double mean = st[4 * k] / (double)n;
        const double var = st[4 * k + 1] / (double)n - mean * mean;
        net->host_stats[k] = (float)mean;
        net->host_stats[NIN + k] = (float)std::sqrt(var > 1e-12 ? var : 1e-12);
        net->host_stats[2 * NIN + k] = (float)st[4 * k + 2];
        net->host_stats[3 * NIN + k] = (float)st[4 * k + 3];
    }
    if (int r = upload_stats(net)) return r;
    // the guard: the guard_quantile quantile of the training rows' dominant-band share
    if (opts->guard_quantile >= 1.f) {
        net->share_max = 1.f;
    } else {
        float*& d_share = sc.x_in;
        MCK(cudaMallocAsync((void**)&d_share, sizeof(float) * (size_t)n, s));
        dominant_share_kernel<<<blocks_for(n, 256), 256, 0, s>>>(features, n, d_share);
        MCK(cudaGetLastError());
        // its rank among the rows, by radix selection on the device
        unsigned long long*& d_sel = sc.d_ab;  // state, then the histogram
        MCK(cudaMallocAsync((void**)&d_sel, 2 * sizeof(unsigned long long) + SEL_BINS * sizeof(unsigned), s));
        unsigned* hist = reinterpret_cast<unsigned*>(d_sel + 2);
        const unsigned long long init[2] = {0ull, (unsigned long long)((double)opts->guard_quantile * (double)(n - 1))};
        MCK(cudaMemsetAsync(hist, 0, SEL_BINS * sizeof(unsigned), s));
        MCK(cudaMemcpyAsync(d_sel, init, sizeof init, cudaMemcpyHostToDevice, s));
        const int sel[3][2] = {{21, 11}, {10, 11}, {0, 10}};  // shift and width of the bits
        for (const auto& b : sel) {
            select_hist_kernel<<<(int)std::min<long long>(blocks_for(n, 256), 304), 256, 0, s>>>(d_share, n, d_sel, b[0], b[1],
                                                                                               hist);
            select_bin_kernel<<<1, 32, 0, s>>>(hist, d_sel, b[1]);
        }
        MCK(cudaGetLastError());
        unsigned long long found = 0;
        MCK(cudaMemcpyAsync(&found, d_sel, sizeof found, cudaMemcpyDeviceToHost, s));
        MCK(cudaStreamSynchronize(s));
        MCK(cudaFreeAsync(d_sel, s));
        d_sel = nullptr;
        const unsigned bits = (unsigned)found;
        std::memcpy(&net->share_max, &bits, sizeof bits);
    }
    MCK(cudaMemsetAsync(net->Mo, 0, sizeof(float) * NPARAM, s));
    MCK(cudaMemsetAsync(net->Vo, 0, sizeof(float) * NPARAM, s));
    Work& w = sc.w;
    MCK(w.alloc(B, s));
    const long long steps = n / B;
    const long long total_steps = steps * opts->epochs;
    // per-epoch permutations (affine i -> (a i + b) mod n with a coprime to n)
    // and the per-step schedule (cosine learning rate, Adam bias corrections),
    // computed on the host and read on the device at the step counter
    std::vector<unsigned long long> ab(2 * (size_t)opts->epochs);
    std::vector<float> sched(3 * (size_t)total_steps);
    uint64_t rs = opts->seed ^ 0x5DEECE66Dull;
    auto gcd = [](unsigned long long x, unsigned long long y) {
        while (y) { unsigned long long r = x % y; x = y; y = r; }
        return x;
    };
    for (int ep = 0; ep < opts->epochs; ++ep) {
        unsigned long long a = (splitmix64(rs) % (unsigned long long)n) | 1ull;
        while (gcd(a, (unsigned long long)n) != 1) a += 2;
        ab[2 * ep] = a;
        ab[2 * ep + 1] = splitmix64(rs) % (unsigned long long)n;
    }
    for (long long t = 0; t < total_steps; ++t) {
        const double frac = (double)t / (double)(total_steps > 1 ? total_steps - 1 : 1);
        sched[3 * t] = (float)(opts->lr * (0.05 + 0.95 * 0.5 * (1.0 + std::cos(M_PI * frac))));
        sched[3 * t + 1] = 1.f - std::pow(opts->beta1, (float)(t + 1));
        sched[3 * t + 2] = 1.f - std::pow(opts->beta2, (float)(t + 1));
    }
    unsigned long long*& d_ab = sc.d_ab;
    float*& d_sched = sc.d_sched;
    long long*& d_t = sc.d_t;
    MCK(cudaMallocAsync((void**)&d_ab, sizeof(unsigned long long) * ab.size(), s));
    MCK(cudaMallocAsync((void**)&d_sched, sizeof(float) * sched.size(), s));
    MCK(cudaMallocAsync((void**)&d_t, sizeof(long long), s));
    MCK(cudaMemcpyAsync(d_ab, ab.data(), sizeof(unsigned long long) * ab.size(), cudaMemcpyHostToDevice, s));
    MCK(cudaMemcpyAsync(d_sched, sched.data(), sizeof(float) * sched.size(), cudaMemcpyHostToDevice, s));
    MCK(cudaMemsetAsync(d_t, 0, sizeof(long long), s));

    // the BF16 weights the first step reads
    if (int r = repack(net, s)) return r;
    // training steps (the fused tensor-core tile kernel, then the ordered gradient
    // sum with the Adam step and the step counter) as CUDA graphs of TRAIN_UNROLL
    // steps and of one, captured on a private stream and replayed: the device
    // counter tells a step which rows it takes.  Within a graph a kernel starts
    // while its predecessor ends (programmatic dependent launch).
    cudaStream_t& cs = sc.cs;
    MCK(cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking));
    cudaEvent_t& ready = sc.ready;
    MCK(cudaEventCreateWithFlags(&ready, cudaEventDisableTiming));
    MCK(cudaEventRecord(ready, s));
    MCK(cudaStreamWaitEvent(cs, ready, 0));
    const auto capture = [&](int count, cudaGraphExec_t& gexec) -> int {
        cudaError_t e = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
        if (e != cudaSuccess) return set_error(SKIRT_ERR_CUDA, "training graph: %s", cudaGetErrorString(e));
        for (int k = 0; k < count && e == cudaSuccess; ++k)
            e = launch_train_step(net->Wb, net->P, features, target, net->stats, d_ab, d_t, steps, n, nullptr, B,
                                  w.part, w.part_loss, net->G, 1, net->P, net->Mo, net->Vo, d_sched, opts->beta1,
                                  opts->beta2, opts->eps, net->Wb, w.loss, k, k == count - 1 ? count : 0, cs);
        const cudaError_t ec = cudaStreamEndCapture(cs, &sc.graph);
        if (e == cudaSuccess) e = ec;
        if (e == cudaSuccess) e = cudaGraphInstantiate(&gexec, sc.graph, 0);
        if (sc.graph) cudaGraphDestroy(sc.graph);
        sc.graph = nullptr;
        return e == cudaSuccess ? SKIRT_OK : set_error(SKIRT_ERR_CUDA, "training graph: %s", cudaGetErrorString(e));
    };
    const long long unrolled = steps / TRAIN_UNROLL * TRAIN_UNROLL;
    if (unrolled > 0)
        if (int r = capture(TRAIN_UNROLL, sc.gexec)) return r;
    if (unrolled < steps)
        if (int r = capture(1, sc.gexec1)) return r;
    int rc = SKIRT_OK;
    for (int ep = 0; ep < opts->epochs && rc == SKIRT_OK; ++ep) {
        cudaError_t e = cudaMemsetAsync(w.loss, 0, sizeof(float), cs);
        for (long long k = 0; k < unrolled && e == cudaSuccess; k += TRAIN_UNROLL) e = cudaGraphLaunch(sc.gexec, cs);
        for (long long k = unrolled; k < steps && e == cudaSuccess; ++k) e = cudaGraphLaunch(sc.gexec1, cs);
        if (e == cudaSuccess && loss_history) {
            float l = 0.f;
            e = cudaMemcpyAsync(&l, w.loss, sizeof(float), cudaMemcpyDeviceToHost, cs);
            if (e == cudaSuccess) e = cudaStreamSynchronize(cs);
            loss_history[ep] = l / (float)steps;
        }
        if (e != cudaSuccess) rc = set_error(SKIRT_ERR_CUDA, "training step: %s", cudaGetErrorString(e));
    }
    if (rc) return rc;  // the scope joins the private stream and frees everything
    // join the private stream before the repack on the caller's stream
    MCK(cudaEventRecord(ready, cs));
    MCK(cudaStreamWaitEvent(s, ready, 0));
    if (int r = repack(net, s)) return r;
    MCK(cudaStreamSynchronize(s));
    return SKIRT_OK;
}

extern "C" int skirt_mlp_forward(skirt_mlp_t net, const float* features, const double* total, long long n,
                                 double* emission, unsigned char* flags, void* stream)
{
    if (!net || !features || !total || !emission || n < 0) return set_error(SKIRT_ERR_INVALID_ARG, "mlp forward args");
    if (n == 0) return SKIRT_OK;
    cudaStream_t s = (cudaStream_t)stream;
    int* d_timeout = nullptr;
    int timeout = 0;
    MCK(cudaMallocAsync((void**)&d_timeout, sizeof(int), s));
    cudaError_t e = cudaMemsetAsync(d_timeout, 0, sizeof(int), s);
    const int r = e == cudaSuccess ? mlp_forward_internal(net, features, total, n, emission, flags, d_timeout, s) : SKIRT_OK;
    if (e == cudaSuccess && r == SKIRT_OK)
        e = cudaMemcpyAsync(&timeout, d_timeout, sizeof(int), cudaMemcpyDeviceToHost, s);
    cudaFreeAsync(d_timeout, s);
    if (r) return r;
    MCK(e);
    MCK(cudaStreamSynchronize(s));
    return mlp_check_timeout(timeout);
}
