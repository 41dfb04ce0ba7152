// Training step of the MLP surrogate on the tensor cores (BF16 products,
// FP32 accumulation, FP32 master weights).
//
// train_tile_kernel: one CTA per 32 rows of the batch, 16 warps.  The CTA
// gathers and standardises its rows and fetches their targets while the
// previous step still runs, then takes the BF16 weights into shared memory by
// asynchronous copies, a group per layer, and runs the whole step for its rows
// with mma.sync m16n8k16 in inline PTX:
//   forward   Z1 = X W1^T + b1, A1 = SiLU(Z1), Z2, A2, Z3 (logits);
//   softmax and cross-entropy, dZ3 = (p - t) / n;
//   backward  dZ2 = (dZ3 W3) * SiLU'(Z2), dZ1 = (dZ2 W2) * SiLU'(Z1)
//             (the products with W^T read W, stored [out][in], through
//             ldmatrix.trans);
//   weights   dW3 = dZ3^T A2, dW2 = dZ2^T A1, dW1 = dZ1^T X, biases = column
//             sums (the row dimension is the contraction; both operands come
//             from the row-major activation tiles through ldmatrix.trans).
// Every operand of a product is rounded to BF16 once: the standardised
// inputs, the weights, the activations and the dZ tiles; the SiLU
// derivatives, the softmax, the bias sums and the accumulators stay FP32.
// Each CTA writes its partial gradient (packed parameter layout) and its
// partial loss.
//
// train_reduce_kernel: the partial gradients summed over the CTAs in CTA
// order (deterministic), then (training) the Adam step at the learning rate
// and bias corrections of the step, the refreshed BF16 weights for the next
// step, and the loss.
//
// A step is a chain of latencies on less than half of the SMs (a batch of 2048
// rows has 64 tiles): 16.8 us, of which the weights' copy takes 1.0, the layers
// and the softmax 4.6, the way back 2.1, the weight gradients and their stores
// about 2.5, the hand-over to the sum 2.2 and the sum 1.5 (35 us with 8 warps
// that staged the weights and divided 64-bit row numbers in every thread, and
// with the kernels strictly one after the other).  Tiles of 16 rows would fill
// the chip but sum the gradients in another order, and the trained parameters
// are the same bit for bit as before.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "skirt_internal.cuh"

namespace skirt {
namespace {

constexpr int NIN = SKIRT_NBANDS;      // 32
constexpr int NH = SKIRT_MLP_HIDDEN;   // 128
constexpr int NO = SKIRT_NEMIT;        // 100
constexpr int NOP = 104;               // 13 n-tiles of 8 (forward output of layer 3)
constexpr int NOK = 112;               // 7 k-tiles of 16 (dZ3 as a contraction operand)
constexpr int NPARAM = SKIRT_MLP_NPARAM;
constexpr int OFF_W1 = 0, OFF_B1 = OFF_W1 + NH * NIN, OFF_W2 = OFF_B1 + NH, OFF_B2 = OFF_W2 + NH * NH,
              OFF_W3 = OFF_B2 + NH, OFF_B3 = OFF_W3 + NO * NH;

constexpr int TR = 32;      // rows per CTA
constexpr int TWARPS = 16;  // warps per CTA
// shared-memory row strides (elements), each row padded by 8 BF16 (16 bytes)
// so that the eight rows an ldmatrix touches start in different bank groups
constexpr int P1 = NIN + 8;   // 40
constexpr int P2 = NH + 8;    // 136
constexpr int P3 = NOK + 8;   // 120
constexpr size_t S_W1 = 0;                                            // [128][P1]
constexpr size_t S_W2 = S_W1 + 2 * NH * P1;                           // [128][P2]
constexpr size_t S_W3 = S_W2 + 2 * NH * P2;                           // [112][P2], rows >= 100 zero
constexpr size_t S_X = S_W3 + 2 * NOK * P2;                           // [32][P1]
constexpr size_t S_A1 = S_X + 2 * TR * P1;                            // [32][P2]
constexpr size_t S_A2 = S_A1 + 2 * TR * P2;
constexpr size_t S_D3 = S_A2 + 2 * TR * P2;                           // [32][P3], cols >= 100 zero
constexpr size_t S_D2 = S_D3 + 2 * TR * P3;                           // [32][P2]
constexpr size_t S_D1 = S_D2 + 2 * TR * P2;
constexpr size_t S_G1 = S_D1 + 2 * TR * P2;                           // fp32 [32][128]: SiLU'(Z1), then dZ1
constexpr size_t S_G2 = S_G1 + 4 * TR * NH;                           // fp32 [32][128]: SiLU'(Z2), then dZ2
constexpr size_t S_Z3 = S_G2 + 4 * TR * NH;                           // fp32 [32][104]: logits, then dZ3
constexpr size_t S_LOSS = S_Z3 + 4 * TR * NOP;                        // fp32 [32]
constexpr size_t S_T = S_LOSS + 4 * TR;                               // fp32 [32][100]: targets
constexpr size_t S_B = S_T + 4 * TR * NO;                             // fp32 b1 [128], b2 [128], b3 [100]
constexpr size_t S_IDX = S_B + 4 * (NH + NH + NO);                    // int64 [32]: the rows in the data
constexpr size_t S_TOTAL = S_IDX + 8 * TR;
static_assert(S_TOTAL <= 227 * 1024, "shared memory of one CTA");
static_assert(S_X % 16 == 0 && S_A1 % 16 == 0 && S_D3 % 16 == 0 && S_G1 % 16 == 0 && S_T % 16 == 0 && S_IDX % 8 == 0,
              "16-byte aligned tiles");

constexpr int STAGE = 16 * (8 * (NH / 16) + 4);  // floats of one warp's staging area
static_assert(4 * TWARPS * STAGE <= S_X, "the staging areas fit the weights' memory");

__device__ __forceinline__ unsigned su32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void cp_async16(void* dst, const void* src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(su32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait()
{
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Programmatic dependent launch: a kernel may start once every block of its
// predecessor has called launch_dependents, and waits for its results in
// wait_predecessor.
__device__ __forceinline__ void launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_predecessor() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], const void* p)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(su32(p)));
}

__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], const void* p)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(su32(p)));
}

__device__ __forceinline__ void mma16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

__device__ __forceinline__ uint16_t bf16_bits(float v)
{
    __nv_bfloat16 b = __float2bfloat16_rn(v);
    return *reinterpret_cast<uint16_t*>(&b);
}

__device__ __forceinline__ uint32_t pack2(float lo, float hi)
{
    return (uint32_t)bf16_bits(lo) | ((uint32_t)bf16_bits(hi) << 16);
}

__device__ __forceinline__ float sigmoid_f(float z) { return 1.f / (1.f + expf(-z)); }

// A fragment (16 x 16) of the row-major tile S [rows][stride] at (r0, c0)
template <int STRIDE>
__device__ __forceinline__ void frag_a(uint32_t (&a)[4], const uint16_t* S, int r0, int c0, int lane)
{
    const int m = lane >> 3, j = lane & 7;
    ldsm4(a, S + (size_t)(r0 + (m & 1) * 8 + j) * STRIDE + c0 + (m >> 1) * 8);
}

// A fragment (16 x 16) of S^T at (m0, k0), S row-major [k][m]
template <int STRIDE>
__device__ __forceinline__ void frag_at(uint32_t (&a)[4], const uint16_t* S, int m0, int k0, int lane)
{
    const int m = lane >> 3, j = lane & 7;
    ldsm4t(a, S + (size_t)(k0 + (m >> 1) * 8 + j) * STRIDE + m0 + (m & 1) * 8);
}

// B fragments of two n-tiles (n0, n0 + 8) for the k-tile at k0, where
// B[k][n] = S[k][n] with S row-major: b[0], b[1] for n-tile n0; b[2], b[3] for n0 + 8
template <int STRIDE>
__device__ __forceinline__ void frag_b2t(uint32_t (&b)[4], const uint16_t* S, int k0, int n0, int lane)
{
    const int m = lane >> 3, j = lane & 7;
    ldsm4t(b, S + (size_t)(k0 + (m & 1) * 8 + j) * STRIDE + n0 + (m >> 1) * 8);
}

// forward layer tile: C (16 x 8 per n-tile) = A (16 x 16*KT) x W^T for the
// n-tiles nts[] (W row-major [out][in] in shared memory)
template <int KT, int STRIDE_A, int STRIDE_W>
__device__ __forceinline__ void fwd_tile(float (&c)[4], const uint32_t (&a)[KT][4], const uint16_t* W, int nt, int g,
                                         int t)
{
    const uint16_t* wr = W + (size_t)(8 * nt + g) * STRIDE_W + 2 * t;
#pragma unroll
    for (int kk = 0; kk < KT; ++kk) {
        const uint32_t b0 = *reinterpret_cast<const uint32_t*>(wr + 16 * kk);
        const uint32_t b1 = *reinterpret_cast<const uint32_t*>(wr + 16 * kk + 8);
        mma16816(c, a[kk], b0, b1);
    }
}

// dst[o][i] (o < mrows, row stride outK) = sum over the 32 rows r of D[r][o] Act[r][i]
// for the output rows of m-tile mt and the NT n-tiles from nt0 of i: A = D^T,
// B = Act, both through ldmatrix.trans of the row-major tiles.  The 16 x 8 NT
// results go through the warp's staging area (rows padded by 4 floats) so that
// they leave in 16-byte stores along the rows: straight from the fragments, each
// store met 8 rows with 32 bytes and the stores took most of this phase.
template <int SD, int SA, int NT>
__device__ __forceinline__ void wgrad(const uint16_t* D, const uint16_t* Act, int nt0, int mt, int outK, int mrows,
                                      float* dst, float* stage, int lane)
{
    constexpr int PS = 8 * NT + 4;
    const int g = lane >> 2, t = lane & 3;
    uint32_t a0[4], a1[4];
    frag_at<SD>(a0, D, 16 * mt, 0, lane);
    frag_at<SD>(a1, D, 16 * mt, 16, lane);
    __syncwarp();  // the staging area is free
#pragma unroll
    for (int np = 0; np < NT; np += 2) {
        float acc0[4] = {0.f, 0.f, 0.f, 0.f}, acc1[4] = {0.f, 0.f, 0.f, 0.f};
        uint32_t b[4];
        frag_b2t<SA>(b, Act, 0, 8 * (nt0 + np), lane);
        mma16816(acc0, a0, b[0], b[1]);
        mma16816(acc1, a0, b[2], b[3]);
        frag_b2t<SA>(b, Act, 16, 8 * (nt0 + np), lane);
        mma16816(acc0, a1, b[0], b[1]);
        mma16816(acc1, a1, b[2], b[3]);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float* row = stage + (g + 8 * h) * PS + 8 * np + 2 * t;
            *reinterpret_cast<float2*>(row) = make_float2(acc0[2 * h], acc0[2 * h + 1]);
            *reinterpret_cast<float2*>(row + 8) = make_float2(acc1[2 * h], acc1[2 * h + 1]);
        }
    }
    __syncwarp();
    constexpr int C4 = 2 * NT;  // 16-byte pieces per row
#pragma unroll
    for (int k = lane; k < 16 * C4; k += 32) {
        const int o = 16 * mt + k / C4;
        if (o < mrows)
            *reinterpret_cast<float4*>(dst + (size_t)o * outK + 8 * nt0 + 4 * (k % C4)) =
                *reinterpret_cast<const float4*>(stage + (k / C4) * PS + 4 * (k % C4));
    }
}

struct TileArgs {
    const uint16_t* Wb;       // bf16 W1 [128][32], W2 [128][128], W3 [104][128] (rows >= 100 zero)
    const float* P;           // fp32 parameters (biases read from here)
    // rows: either gathered (feat != nullptr: row r of step t is (a (k B + r) + b) mod n_data of the
    // epoch's permutation, features standardised with stats) or direct (x_std, target)
    const float* feat;
    const float* target;      // [n_data][100] row shapes
    const float* stats;       // mean[32], 1/std[32]
    const unsigned long long* ab;
    const long long* t_dev;   // the step of the first launch of this graph
    int ahead;                // this launch's steps after it
    long long steps, n_data;
    const float* x_std;       // direct rows [nrows][32]
    int nrows;                // rows in this batch
    float inv_n;              // 1 / nrows
    float* part;              // [ncta][NPARAM] partial gradients
    float* part_loss;         // [ncta]
};

__global__ void __launch_bounds__(32 * TWARPS, 1) train_tile_kernel(const TileArgs A)
{
    extern __shared__ __align__(16) unsigned char sm[];
    uint16_t* W1 = reinterpret_cast<uint16_t*>(sm + S_W1);
    uint16_t* W2 = reinterpret_cast<uint16_t*>(sm + S_W2);
    uint16_t* W3 = reinterpret_cast<uint16_t*>(sm + S_W3);
    uint16_t* X = reinterpret_cast<uint16_t*>(sm + S_X);
    uint16_t* A1 = reinterpret_cast<uint16_t*>(sm + S_A1);
    uint16_t* A2 = reinterpret_cast<uint16_t*>(sm + S_A2);
    uint16_t* D3 = reinterpret_cast<uint16_t*>(sm + S_D3);
    uint16_t* D2 = reinterpret_cast<uint16_t*>(sm + S_D2);
    uint16_t* D1 = reinterpret_cast<uint16_t*>(sm + S_D1);
    float* G1 = reinterpret_cast<float*>(sm + S_G1);
    float* G2 = reinterpret_cast<float*>(sm + S_G2);
    float* Z3 = reinterpret_cast<float*>(sm + S_Z3);
    float* LS = reinterpret_cast<float*>(sm + S_LOSS);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int g = lane >> 2, t = lane & 3;
    const int row0 = blockIdx.x * TR;
    const int nvalid = min(TR, A.nrows - row0);

    float* T = reinterpret_cast<float*>(sm + S_T);
    float* SB = reinterpret_cast<float*>(sm + S_B);
    long long* idx = reinterpret_cast<long long*>(sm + S_IDX);
    // ---- what does not depend on the previous step, done while it ends: the rows'
    // places in the data (32 threads: the permutation's 64-bit modulus is slow)
    if (tid < TR) {
        long long at = -1;
        if (tid < nvalid) {
            at = row0 + tid;
            if (A.feat) {
                const long long st = *A.t_dev + A.ahead;
                const unsigned long long pa = A.ab[2 * (st / A.steps)], pb = A.ab[2 * (st / A.steps) + 1];
                const unsigned long long q = (unsigned long long)((st % A.steps) * (long long)A.nrows + at);
                at = (long long)((pa * q + pb) % (unsigned long long)A.n_data);
            }
        }
        idx[tid] = at;
    }
    // zero what no copy fills: W3's rows 104 .. 111, and dZ3's columns 100 .. 111,
    // which take part in the W3 products
    for (int i = tid; i < (NOK - NOP) * (NH / 8); i += blockDim.x)
        *reinterpret_cast<uint4*>(W3 + (NOP + i / (NH / 8)) * P2 + 8 * (i % (NH / 8))) = make_uint4(0u, 0u, 0u, 0u);
    for (int i = tid; i < TR * (NOK - NO); i += blockDim.x) D3[(i / (NOK - NO)) * P3 + NO + i % (NOK - NO)] = 0;
    __syncthreads();
    // the target shapes in T, the standardised features (bf16) in X
    for (int i = tid; i < TR * (NO / 4); i += blockDim.x) {
        const int r = i / (NO / 4), c = i % (NO / 4);
        if (idx[r] >= 0) cp_async16(T + r * NO + 4 * c, A.target + idx[r] * NO + 4 * c);
    }
    cp_commit();
    for (int i = tid; i < TR * NIN; i += blockDim.x) {
        const int r = i / NIN, c = i % NIN;
        const long long s = idx[r];
        float v = 0.f;
        if (s >= 0) v = A.feat ? (A.feat[s * NIN + c] - A.stats[c]) * A.stats[NIN + c] : A.x_std[s * NIN + c];
        X[r * P1 + c] = bf16_bits(v);
    }
    // the dependents are let go only now: they wait for this kernel, and so for the
    // previous step's results as well
    wait_predecessor();
    launch_dependents();
    // ---- the weights by asynchronous copies of 16 bytes into padded rows, each
    // layer's in a group of its own, so that a layer starts when its weights are in
    {
        const uint4* src = reinterpret_cast<const uint4*>(A.Wb);
        for (int i = tid; i < NH * (NIN / 8); i += blockDim.x)
            cp_async16(W1 + (i / (NIN / 8)) * P1 + 8 * (i % (NIN / 8)), src + i);
        cp_commit();
        src += NH * (NIN / 8);
        for (int i = tid; i < NH * (NH / 8); i += blockDim.x)
            cp_async16(W2 + (i / (NH / 8)) * P2 + 8 * (i % (NH / 8)), src + i);
        cp_commit();
        src += NH * (NH / 8);
        for (int i = tid; i < NOP * (NH / 8); i += blockDim.x)
            cp_async16(W3 + (i / (NH / 8)) * P2 + 8 * (i % (NH / 8)), src + i);
        cp_commit();
        for (int i = tid; i < NH + NH + NO; i += blockDim.x)
            SB[i] = i < NH ? A.P[OFF_B1 + i] : (i < 2 * NH ? A.P[OFF_B2 + i - NH] : A.P[OFF_B3 + i - 2 * NH]);
    }
    cp_wait<2>();
    __syncthreads();

    const int rt = warp & 1;          // row tile of this warp in the forward and backward products
    const int q8 = warp >> 1;         // its pair of n-tiles
    const float* b1v = SB;
    const float* b2v = SB + NH;
    const float* b3v = SB + 2 * NH;

    // ---- layer 1: Z1 = X W1^T + b1; A1 = SiLU(Z1) (bf16), G1 = SiLU'(Z1)
    {
        uint32_t a[2][4];
        frag_a<P1>(a[0], X, 16 * rt, 0, lane);
        frag_a<P1>(a[1], X, 16 * rt, 16, lane);
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int nt = 2 * q8 + j;
            const int c = 8 * nt + 2 * t;
            float acc[4] = {b1v[c], b1v[c + 1], b1v[c], b1v[c + 1]};
            fwd_tile<2, P1, P1>(acc, a, W1, nt, g, t);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int r = 16 * rt + g + 8 * h;
                const float z0 = acc[2 * h], z1 = acc[2 * h + 1];
                const float s0 = sigmoid_f(z0), s1 = sigmoid_f(z1);
                *reinterpret_cast<uint32_t*>(A1 + r * P2 + c) = pack2(z0 * s0, z1 * s1);
                *reinterpret_cast<float2*>(G1 + r * NH + c) =
                    make_float2(s0 * (1.f + z0 * (1.f - s0)), s1 * (1.f + z1 * (1.f - s1)));
            }
        }
    }
    cp_wait<1>();
    __syncthreads();
    // ---- layer 2
    {
        uint32_t a[8][4];
#pragma unroll
        for (int kk = 0; kk < 8; ++kk) frag_a<P2>(a[kk], A1, 16 * rt, 16 * kk, lane);
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int nt = 2 * q8 + j;
            const int c = 8 * nt + 2 * t;
            float acc[4] = {b2v[c], b2v[c + 1], b2v[c], b2v[c + 1]};
            fwd_tile<8, P2, P2>(acc, a, W2, nt, g, t);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int r = 16 * rt + g + 8 * h;
                const float z0 = acc[2 * h], z1 = acc[2 * h + 1];
                const float s0 = sigmoid_f(z0), s1 = sigmoid_f(z1);
                *reinterpret_cast<uint32_t*>(A2 + r * P2 + c) = pack2(z0 * s0, z1 * s1);
                *reinterpret_cast<float2*>(G2 + r * NH + c) =
                    make_float2(s0 * (1.f + z0 * (1.f - s0)), s1 * (1.f + z1 * (1.f - s1)));
            }
        }
    }
    cp_wait<0>();
    __syncthreads();
    // ---- layer 3: logits Z3 (n-tiles q8, q8 + 8 < 13)
    {
        uint32_t a[8][4];
#pragma unroll
        for (int kk = 0; kk < 8; ++kk) frag_a<P2>(a[kk], A2, 16 * rt, 16 * kk, lane);
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int nt = q8 + 8 * j;
            if (nt < NOP / 8) {
                const int c = 8 * nt + 2 * t;
                const float bb0 = c < NO ? b3v[c] : 0.f, bb1 = c + 1 < NO ? b3v[c + 1] : 0.f;
                float acc[4] = {bb0, bb1, bb0, bb1};
                fwd_tile<8, P2, P2>(acc, a, W3, nt, g, t);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int r = 16 * rt + g + 8 * h;
                    *reinterpret_cast<float2*>(Z3 + r * NOP + c) = make_float2(acc[2 * h], acc[2 * h + 1]);
                }
            }
        }
    }
    __syncthreads();
    // ---- softmax and cross-entropy, one warp per row: dZ3 = (p - t) / n
#pragma unroll
    for (int h = 0; h < TR / TWARPS; ++h) {
        const int r = warp + h * TWARPS;
        float v[4], m = -3.0e38f;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int c = lane + 32 * k;
            v[k] = c < NO ? Z3[r * NOP + c] : -3.0e38f;
            m = fmaxf(m, v[k]);
        }
        for (int o = 16; o; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
        float s = 0.f;
#pragma unroll
        for (int k = 0; k < 4; ++k) s += (lane + 32 * k < NO) ? expf(v[k] - m) : 0.f;
        for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        const float ls = logf(s);
        const bool live = r < nvalid;
        const float* tr = T + r * NO;
        float l = 0.f;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int c = lane + 32 * k;
            if (c < NO) {
                float d = 0.f;
                if (live) {
                    const float tv = tr[c];
                    const float logp = v[k] - m - ls;
                    l -= tv * logp;
                    d = (expf(logp) - tv) * A.inv_n;
                }
                Z3[r * NOP + c] = d;  // the FP32 dZ3, for the bias sums
                D3[r * P3 + c] = bf16_bits(d);
            }
        }
        for (int o = 16; o; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
        if (lane == 0) LS[r] = l * A.inv_n;
    }
    __syncthreads();
    // ---- dZ2 = (dZ3 W3) * SiLU'(Z2): K = 112 (7 k-tiles), W3^T through ldmatrix.trans
    {
        uint32_t a[7][4];
#pragma unroll
        for (int kk = 0; kk < 7; ++kk) frag_a<P3>(a[kk], D3, 16 * rt, 16 * kk, lane);
        {
            const int nt = 2 * q8;  // n-tiles nt, nt + 1
            float acc0[4] = {0.f, 0.f, 0.f, 0.f}, acc1[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int kk = 0; kk < 7; ++kk) {
                uint32_t b[4];
                frag_b2t<P2>(b, W3, 16 * kk, 8 * nt, lane);
                mma16816(acc0, a[kk], b[0], b[1]);
                mma16816(acc1, a[kk], b[2], b[3]);
            }
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const float* acc = u ? acc1 : acc0;
                const int c = 8 * (nt + u) + 2 * t;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int r = 16 * rt + g + 8 * h;
                    float2 gs = *reinterpret_cast<const float2*>(G2 + r * NH + c);
                    const float d0 = acc[2 * h] * gs.x, d1 = acc[2 * h + 1] * gs.y;
                    *reinterpret_cast<float2*>(G2 + r * NH + c) = make_float2(d0, d1);
                    *reinterpret_cast<uint32_t*>(D2 + r * P2 + c) = pack2(d0, d1);
                }
            }
        }
    }
    __syncthreads();
    // ---- dZ1 = (dZ2 W2) * SiLU'(Z1)
    {
        uint32_t a[8][4];
#pragma unroll
        for (int kk = 0; kk < 8; ++kk) frag_a<P2>(a[kk], D2, 16 * rt, 16 * kk, lane);
        {
            const int nt = 2 * q8;
            float acc0[4] = {0.f, 0.f, 0.f, 0.f}, acc1[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int kk = 0; kk < 8; ++kk) {
                uint32_t b[4];
                frag_b2t<P2>(b, W2, 16 * kk, 8 * nt, lane);
                mma16816(acc0, a[kk], b[0], b[1]);
                mma16816(acc1, a[kk], b[2], b[3]);
            }
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const float* acc = u ? acc1 : acc0;
                const int c = 8 * (nt + u) + 2 * t;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int r = 16 * rt + g + 8 * h;
                    float2 gs = *reinterpret_cast<const float2*>(G1 + r * NH + c);
                    const float d0 = acc[2 * h] * gs.x, d1 = acc[2 * h + 1] * gs.y;
                    *reinterpret_cast<float2*>(G1 + r * NH + c) = make_float2(d0, d1);
                    *reinterpret_cast<uint32_t*>(D1 + r * P2 + c) = pack2(d0, d1);
                }
            }
        }
    }
    __syncthreads();
    float* part = A.part + (size_t)blockIdx.x * NPARAM;
    // ---- bias gradients: column sums of the FP32 dZ tiles over the 32 rows, in row order
    for (int c = tid; c < NH + NH + NO; c += blockDim.x) {
        float s = 0.f;
        if (c < NH) {
            for (int r = 0; r < TR; ++r) s += G1[r * NH + c];
            part[OFF_B1 + c] = s;
        } else if (c < 2 * NH) {
            for (int r = 0; r < TR; ++r) s += G2[r * NH + c - NH];
            part[OFF_B2 + c - NH] = s;
        } else {
            for (int r = 0; r < TR; ++r) s += Z3[r * NOP + c - 2 * NH];
            part[OFF_B3 + c - 2 * NH] = s;
        }
    }
    if (tid == 32 * TWARPS - 1) {
        float l = 0.f;
        for (int r = 0; r < TR; ++r) l += r < nvalid ? LS[r] : 0.f;
        A.part_loss[blockIdx.x] = l;
    }
    // ---- weight gradients dW = dZ^T Act over the 32 rows (2 k-tiles): warp w takes
    // half of the n-tiles of m-tile w mod 8 of dW2 and dW1 and, below 7, of dW3;
    // the weights' shared memory, no longer needed, is the staging area
    const int mt = warp & 7, hf = warp >> 3;
    float* stage = reinterpret_cast<float*>(sm + S_W1) + warp * STAGE;
    wgrad<P2, P2, NH / 16>(D2, A1, hf * (NH / 16), mt, NH, NH, part + OFF_W2, stage, lane);
    if (mt < 7) wgrad<P3, P2, NH / 16>(D3, A2, hf * (NH / 16), mt, NH, NO, part + OFF_W3, stage, lane);
    wgrad<P2, P1, NIN / 16>(D1, X, hf * (NIN / 16), mt, NIN, NH, part + OFF_W1, stage, lane);
}

// g = sum over the CTAs of their partial gradients (in CTA order); with
// adam: the Adam step of the FP32 parameters and their BF16 copies for the
// next step.  The last block instead sums the loss (partials in CTA order).
// Nothing of the previous step is read before wait_predecessor: what a kernel
// wrote is promised only to kernels that wait for it, and the chain of waits
// leads from a sum through the next tile kernel to the next sum.  The step
// counter and the schedule do not change within a graph.
constexpr int RED_T = 128;   // threads per block
constexpr int RED_C = 64;    // partials per chunk
__global__ void __launch_bounds__(RED_T) train_reduce_kernel(
    const float* __restrict__ part, const float* __restrict__ part_loss, int ncta, float* __restrict__ G, int adam,
    float* __restrict__ P, float* __restrict__ Mo, float* __restrict__ Vo, const float* __restrict__ sched,
    const long long* t_dev, int ahead, float b1, float b2, float eps, uint16_t* __restrict__ Wb, float* loss_acc)
{
    launch_dependents();
    if (blockIdx.x == gridDim.x - 1) {
        __shared__ float sl[RED_T];
        float l = 0.f;
        wait_predecessor();
        for (int c0 = 0; c0 < ncta; c0 += RED_T) {
            const int n = min(RED_T, ncta - c0);
            if (threadIdx.x < n) sl[threadIdx.x] = part_loss[c0 + threadIdx.x];
            __syncthreads();
            if (threadIdx.x == 0)
                for (int c = 0; c < n; ++c) l += sl[c];
            __syncthreads();
        }
        if (threadIdx.x == 0) *loss_acc += l;
        return;
    }
    const int i = blockIdx.x * RED_T + threadIdx.x;
    const bool mine = i < NPARAM;
    float mi = 0.f, vi = 0.f, p = 0.f, lr = 0.f, c1 = 1.f, c2 = 1.f;
    if (adam && mine) {
        const long long st = *t_dev + ahead;
        lr = sched[3 * st];
        c1 = sched[3 * st + 1];
        c2 = sched[3 * st + 2];
    }
    wait_predecessor();
    if (adam && mine) {
        mi = Mo[i];
        vi = Vo[i];
        p = P[i];
    }
    float gi = 0.f;
    // a chunk of partials of the block's 128 parameters by asynchronous copies, all
    // in flight at once, then added in order
    __shared__ __align__(16) float sp[RED_C][RED_T];
    const int n4 = min(RED_T, NPARAM - (int)blockIdx.x * RED_T) / 4;  // NPARAM is a multiple of 4
    for (int c0 = 0; c0 < ncta; c0 += RED_C) {
        const int n = min(RED_C, ncta - c0);
        const float* src = part + (size_t)c0 * NPARAM + (size_t)blockIdx.x * RED_T;
        for (int k = threadIdx.x; k < n * (RED_T / 4); k += RED_T) {
            const int c = k / (RED_T / 4), q = k % (RED_T / 4);
            if (q < n4) cp_async16(&sp[c][4 * q], src + (size_t)c * NPARAM + 4 * q);
        }
        cp_commit();
        cp_wait<0>();
        __syncthreads();
#pragma unroll 16
        for (int c = 0; c < n; ++c) gi += sp[c][threadIdx.x];
        __syncthreads();
    }
    if (!mine) return;
    G[i] = gi;
    if (adam) {
        mi = fmaf(1.f - b1, gi, b1 * mi);
        vi = fmaf((1.f - b2) * gi, gi, b2 * vi);
        Mo[i] = mi;
        Vo[i] = vi;
        p = p - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
        P[i] = p;
        // the bf16 copy of a weight (biases stay fp32): W1, W2, W3 contiguous
        int w = -1;
        if (i < OFF_B1) w = i;
        else if (i >= OFF_W2 && i < OFF_B2) w = NH * NIN + (i - OFF_W2);
        else if (i >= OFF_W3 && i < OFF_B3) w = NH * NIN + NH * NH + (i - OFF_W3);
        if (w >= 0) Wb[w] = bf16_bits(p);
    }
}

// Moves the step counter on at the end of a graph: a kernel of its own, launched
// without the early start, so that every block that reads the counter has ended.
__global__ void advance_step_kernel(long long* t_dev, int steps) { *t_dev += steps; }

}  // namespace

size_t train_tile_smem_bytes() { return S_TOTAL; }
int train_rows_per_cta() { return TR; }

// One step (or one gradient): nrows rows, either gathered from feat/target
// with the permutation schedule (feat != nullptr) or taken from x_std/target.
// ahead: this step's place in the captured graph; advance: the graph's steps on
// its last one (0 elsewhere).
cudaError_t launch_train_step(const uint16_t* Wb, const float* P, const float* feat, const float* target,
                              const float* stats, const unsigned long long* ab, long long* t_dev,
                              long long steps, long long n_data, const float* x_std, int nrows, float* part,
                              float* part_loss, float* G, int adam, float* Pw, float* Mo, float* Vo,
                              const float* sched, float b1, float b2, float eps, uint16_t* Wb_out, float* loss_acc,
                              int ahead, int advance, cudaStream_t s)
{
    cudaError_t se = cudaFuncSetAttribute(train_tile_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S_TOTAL);
    if (se != cudaSuccess) return se;
    TileArgs A;
    A.Wb = Wb;
    A.P = P;
    A.feat = feat;
    A.target = target;
    A.stats = stats;
    A.ab = ab;
    A.t_dev = t_dev;
    A.ahead = ahead;
    A.steps = steps;
    A.n_data = n_data;
    A.x_std = x_std;
    A.nrows = nrows;
    A.inv_n = 1.f / (float)nrows;
    A.part = part;
    A.part_loss = part_loss;
    const int ncta = (nrows + TR - 1) / TR;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(ncta);
    cfg.blockDim = dim3(32 * TWARPS);
    cfg.dynamicSmemBytes = S_TOTAL;
    cfg.stream = s;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    cudaError_t e = cudaLaunchKernelEx(&cfg, train_tile_kernel, A);
    if (e != cudaSuccess) return e;
    cfg.gridDim = dim3((NPARAM + RED_T - 1) / RED_T + 1);
    cfg.blockDim = dim3(RED_T);
    cfg.dynamicSmemBytes = 0;
    e = cudaLaunchKernelEx(&cfg, train_reduce_kernel, (const float*)part, (const float*)part_loss, ncta, G, adam, Pw, Mo,
                           Vo, sched, (const long long*)t_dev, ahead, b1, b2, eps, Wb_out, loss_acc);
    if (e != cudaSuccess || advance == 0) return e;
    advance_step_kernel<<<1, 1, 0, s>>>(t_dev, advance);
    return cudaGetLastError();
}

}  // namespace skirt
