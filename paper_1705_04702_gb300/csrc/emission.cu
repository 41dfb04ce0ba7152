// Dust emission step (Sect. 3.2, dust emission phases; Sect. 1, instantaneous
// dust emission): per-cell emission spectra from the absorbed spectra.
//
//  * dust_mass_kernel      M = kappa*rho * cell volume
//  * band_features_kernel  32 log-spaced band sums per unit mass (log10) and
//                          the total absorbed power, one cell per lane
//  * exact_kernel          equilibrium temperatures of three grain
//                          populations by bracketed Newton on ln T (powers
//                          in 64-bit integers, FP64 per population, Planck
//                          terms in double-float), then the energy-conserving
//                          emission spectrum
// and skirt_dust_emission, which runs either the exact solver on every cell
// or the MLP surrogate (mlp.cu) with the exact solver as the fallback for
// cells outside the network's training hull.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <vector>

#include "async_copy.cuh"
#include "dfloat.cuh"
#include "skirt_internal.cuh"

namespace skirt {
namespace {

constexpr int NOUT = SKIRT_NEMIT;
constexpr int NB = SKIRT_NBANDS;
constexpr int NPOP = 3;
constexpr double T_REF = 30.0, T_LO = 3.0, T_HI = 2000.0;
const double DELTA[NPOP] = {-0.5, 0.0, 0.5};
const double BETA[NPOP] = {1.5, 2.0, 2.0};
// h c / k_B in micron kelvin from the exact SI constants
const double HCK_UM = 6.62607015e-34 * 299792458.0 / 1.380649e-23 * 1e6;

__constant__ double c_lnc[NPOP];        // ln c_i = -ln G_i(30 K)
__constant__ double c_Gref[NPOP];       // 1 / c_i
__constant__ double c_lnG_lo[NPOP];     // ln G_i(3 K)
__constant__ double c_lnG_hi[NPOP];     // ln G_i(2000 K)
__constant__ double c_h[NPOP], c_inv_h[NPOP];  // spacing of the table below in ln G_i, and its reciprocal
// 1/T and d(1/T)/d ln G_i times the spacing at NTAB values of ln G_i equally
// spaced over [ln G_i(3 K), ln G_i(2000 K)]: the start of the Newton solve (read
// through the L1 path); 8192 intervals, so that every 2^k-th point also spans
// the range
constexpr int NTAB = 8193;
__device__ double2 g_invT_tab[NPOP][NTAB];
// (256/ln 2 a_l, K_il) of slot s = i * NOUT + l as double-float pairs (the exact
// solve's terms), and the exponential's table
__device__ float4 g_slot[NPOP * NOUT];
__device__ float2 g_exp[DF_EXP_N];

struct HostModel {
    double lam[NOUT], W[NOUT], a[NOUT], K[NPOP][NOUT];
    double lnc[NPOP], Gref[NPOP], lnG_lo[NPOP], lnG_hi[NPOP], h[NPOP], inv_h[NPOP];
    double tab[NPOP][NTAB][2];
    float slot[NPOP * NOUT][4];
    float exp_tab[DF_EXP_N][2];
};

// v = hi + lo with hi = v rounded to binary32, lo = the rest rounded
void split_float(double v, float& hi, float& lo)
{
    hi = (float)v;
    lo = (float)(v - (double)hi);
}

// ln G_i at T = e^y and its derivative by y
double host_lnG(const HostModel& h, int i, double y, double& slope)
{
    const double T = std::exp(y);
    double g = 0.0, d = 0.0;
    for (int l = 0; l < NOUT; ++l) {
        const double x = h.a[l] / T;
        if (x > 700.0) continue;
        const double q = 1.0 / std::expm1(x);
        g += h.K[i][l] * q;
        d += h.K[i][l] * q * x * (1.0 + q);
    }
    slope = d / g;
    return std::log(g);
}

const HostModel& host_model()
{
    static HostModel h;
    static bool ready = false;
    if (!ready) {
        for (int l = 0; l < NOUT; ++l)  // log-spaced 1 .. 1000 micron
            h.lam[l] = std::pow(10.0, 3.0 * (double)l / (double)(NOUT - 1));
        for (int l = 0; l < NOUT; ++l) {
            const double left = l > 0 ? h.lam[l] - h.lam[l - 1] : 0.0;
            const double right = l < NOUT - 1 ? h.lam[l + 1] - h.lam[l] : 0.0;
            h.W[l] = 0.5 * (left + right);
            h.a[l] = HCK_UM / h.lam[l];
            for (int i = 0; i < NPOP; ++i)
                h.K[i][l] = h.W[l] * std::pow(h.lam[l] / 100.0, -BETA[i]) * std::pow(h.lam[l], -5.0);
        }
        for (int i = 0; i < NPOP; ++i) {
            if (i > 0 && BETA[i] == BETA[i - 1]) {  // the same G
                h.lnc[i] = h.lnc[i - 1];
                h.Gref[i] = h.Gref[i - 1];
                h.lnG_lo[i] = h.lnG_lo[i - 1];
                h.lnG_hi[i] = h.lnG_hi[i - 1];
                h.h[i] = h.h[i - 1];
                h.inv_h[i] = h.inv_h[i - 1];
                std::memcpy(h.tab[i], h.tab[i - 1], sizeof h.tab[i]);
                continue;
            }
            double slope;
            h.lnc[i] = -host_lnG(h, i, std::log(T_REF), slope);
            h.Gref[i] = std::exp(-h.lnc[i]);
            h.lnG_hi[i] = host_lnG(h, i, std::log(T_HI), slope);
            h.lnG_lo[i] = host_lnG(h, i, std::log(T_LO), slope);
            h.h[i] = (h.lnG_hi[i] - h.lnG_lo[i]) / (NTAB - 1);
            h.inv_h[i] = 1.0 / h.h[i];
            // ln T of every point by Newton from the extrapolated previous ones
            double y = std::log(T_LO), y1 = y, y2 = y;
            for (int k = 0; k < NTAB; ++k) {
                const double t = h.lnG_lo[i] + k * h.h[i];
                if (k == 1) y = y1 + h.h[i] / slope;
                if (k > 1) y = 2.0 * y1 - y2;
                for (int it = 0; it < 8; ++it) {
                    const double step = (t - host_lnG(h, i, y, slope)) / slope;
                    y += step;
                    // quadratic convergence: the next step would be below 1e-16
                    if (std::fabs(step) < 1e-8) break;
                }
                y2 = y1;
                y1 = y;
                h.tab[i][k][0] = std::exp(-y);
                h.tab[i][k][1] = -std::exp(-y) / slope * h.h[i];
            }
        }
        for (int i = 0; i < NPOP; ++i)
            for (int l = 0; l < NOUT; ++l) {
                float* q = h.slot[i * NOUT + l];
                split_float(h.a[l] * DF_Z_PER_X, q[0], q[1]);
                split_float(h.K[i][l], q[2], q[3]);
            }
        for (int j = 0; j < DF_EXP_N; ++j) {
            const dfl::df2 v = dfl::exp_table_entry(j);
            h.exp_tab[j][0] = v.hi;
            h.exp_tab[j][1] = v.lo;
        }
        ready = true;
    }
    return h;
}

// The model's tables on the current device: constants of the library, put there
// once per device (nine copies from pageable memory took 60 us of every call).
cudaError_t upload_model()
{
    static std::mutex mu;
    static bool done[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e) return e;
    std::lock_guard<std::mutex> lock(mu);
    if (dev >= 0 && dev < 64 && done[dev]) return cudaSuccess;
    const HostModel& h = host_model();
    if ((e = cudaMemcpyToSymbol(c_lnc, h.lnc, sizeof h.lnc))) return e;
    if ((e = cudaMemcpyToSymbol(c_Gref, h.Gref, sizeof h.Gref))) return e;
    if ((e = cudaMemcpyToSymbol(c_lnG_lo, h.lnG_lo, sizeof h.lnG_lo))) return e;
    if ((e = cudaMemcpyToSymbol(c_lnG_hi, h.lnG_hi, sizeof h.lnG_hi))) return e;
    if ((e = cudaMemcpyToSymbol(c_h, h.h, sizeof h.h))) return e;
    if ((e = cudaMemcpyToSymbol(c_inv_h, h.inv_h, sizeof h.inv_h))) return e;
    if ((e = cudaMemcpyToSymbol(g_invT_tab, h.tab, sizeof h.tab))) return e;
    if ((e = cudaMemcpyToSymbol(g_slot, h.slot, sizeof h.slot))) return e;
    if ((e = cudaMemcpyToSymbol(g_exp, h.exp_tab, sizeof h.exp_tab))) return e;
    // pageable copies may return before they have arrived; other streams use the tables next
    if ((e = cudaStreamSynchronize(cudaStreamLegacy))) return e;
    if (dev >= 0 && dev < 64) done[dev] = true;
    return cudaSuccess;
}

// vol: the cell volume; on an octree (leaf != NULL) the finest-lattice cell
// volume, times 8^(levels - level) for each leaf
__global__ void dust_mass_kernel(const float* __restrict__ kr, long long n, float vol, float* __restrict__ mass,
                                 const int4* __restrict__ leaf, int levels)
{
    for (long long m = (long long)blockIdx.x * blockDim.x + threadIdx.x; m < n; m += (long long)gridDim.x * blockDim.x)
        mass[m] = kr[m] * (leaf ? ldexpf(vol, 3 * (levels - leaf[m].w)) : vol);
}

// FP64 -> FP32 by truncation of the significand, on the integer pipe (GB300
// retires FP64 and conversion instructions slowly); values below the FP32
// normal range map to zero, values above it take the ordinary conversion.
__device__ __forceinline__ float narrow_trunc(double x)
{
    const unsigned long long u = (unsigned long long)__double_as_longlong(x);
    const int e = (int)((u >> 52) & 0x7FF) - 1023 + 127;
    if (e >= 255) return (float)x;
    if (e <= 0) return 0.f;
    return __uint_as_float((unsigned)(u >> 32 & 0x80000000u) | ((unsigned)e << 23) | (unsigned)((u >> 29) & 0x7FFFFFu));
}

// band b covers the input wavelengths [start[b], start[b+1]) (sorted input
// grid).  One cell per lane, 32 cells per warp pass.  The warp walks the
// input wavelengths in order in blocks of 32 columns; each block of its 32
// rows is copied to shared memory by asynchronous copies (one 256-byte row
// segment per instruction, coalesced), which keep the kernel at 64 registers
// and 16 warps per SM (a register-staged block took 148 registers, 12 warps
// per SM, and 18% longer).  Each lane sums its row's bands in wavelength
// order (FP64) and, as the walk passes each band's end, adds the band sum to
// the cell's total (FP64, band order): per cell about n_in/32 + 1 FP64 warp
// instructions, a floor near the HBM time on GB300; each lane's serial walk
// and the staging latency set the rest.  The walk adds each band's columns of
// a block in one inner loop (the next band end held in a register); 32 empty
// cells in a row skip their FP64 adds.  The features are formed in FP32 and
// leave through a shared-memory transpose as coalesced rows.
constexpr int BF_WARPS = 2;  // warps per block
static_assert(NB == 32, "32 bands");

__global__ void __launch_bounds__(32 * BF_WARPS) band_features_kernel(
    const double* __restrict__ A, long long ncell, int n_in, const int* __restrict__ start,
    const float* __restrict__ mass, float* __restrict__ features, double* __restrict__ total)
{
    __shared__ int s_start[NB + 1];
    __shared__ double s_tile[BF_WARPS][32][33];  // staged column block [row][column], one padding column
    __shared__ float s_band[BF_WARPS][32][33];   // band sums, then features [row][band]
    for (int b = threadIdx.x; b <= NB; b += blockDim.x) s_start[b] = start[b];
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double (*tile)[33] = s_tile[warp];
    float (*band)[33] = s_band[warp];
    for (long long base = ((long long)blockIdx.x * BF_WARPS + warp) * 32; base < ncell;
         base += (long long)gridDim.x * BF_WARPS * 32) {
        const int nrow = ncell - base < 32 ? (int)(ncell - base) : 32;
        int b = 0;
        double sb = 0.0, tot = 0.0;
        int nxt = s_start[1];  // the first column after band b
        bool live = false;     // warp-uniform: some staged block of these rows held a nonzero value
        for (int c0 = 0; c0 < n_in; c0 += 32) {
            const bool col_ok = c0 + lane < n_in;
            // the block's 32 row segments straight into shared memory (8-byte
            // asynchronous copies, one per lane and row: no register staging)
            __syncwarp();
#pragma unroll 8
            for (int rr = 0; rr < 32; ++rr) {
                if (rr < nrow && col_ok) {
                    const unsigned dst = (unsigned)__cvta_generic_to_shared(&tile[rr][lane]);
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst),
                                 "l"(A + (size_t)(base + rr) * n_in + c0 + lane) : "memory");
                } else {
                    tile[rr][lane] = 0.0;
                }
            }
            asm volatile("cp.async.wait_all;" ::: "memory");
            __syncwarp();
            const int cend = n_in - c0 < 32 ? n_in - c0 : 32;
            // a block that is zero on all 32 rows (a run of empty cells) adds nothing to
            // any band sum: the warp then skips its FP64 adds as a whole.  The test reads
            // the bits on the integer pipes and decides a real branch (a predicated-off
            // FP64 instruction would still hold the FP64 pipe for its full slot).  Once a
            // block of the 32 rows has held a nonzero value the rows are taken as live and
            // the later blocks are summed untested (cells are empty at every wavelength or
            // at few), which keeps the test's cost off the dense case.
            if (!live) {
                unsigned long long bits = 0ull;
                for (int jj = 0; jj < cend; ++jj)
                    bits |= (unsigned long long)__double_as_longlong(tile[lane][jj]);
                live = __any_sync(0xffffffffu, bits != 0ull);
            }
            if (live) {
                int jj = 0;
                while (jj < cend) {
                    // close the bands that end before this column (empty ones included)
                    while (b < NB && nxt <= c0 + jj) {
                        band[lane][b] = narrow_trunc(sb);
                        tot += sb;
                        sb = 0.0;
                        ++b;
                        nxt = b < NB ? s_start[b + 1] : 0x7fffffff;
                    }
                    // the columns of band b in this block, in order
                    const int seg = nxt - c0 < cend ? nxt - c0 : cend;
                    for (; jj < seg; ++jj) sb += tile[lane][jj];
                }
            } else {
                // the same closures, with no column to add
                while (b < NB && nxt <= c0 + cend - 1) {
                    band[lane][b] = narrow_trunc(sb);
                    tot += sb;
                    sb = 0.0;
                    ++b;
                    nxt = b < NB ? s_start[b + 1] : 0x7fffffff;
                }
            }
        }
        for (; b < NB; ++b) {
            band[lane][b] = narrow_trunc(sb);
            tot += sb;
            sb = 0.0;
        }
        const long long r = base + lane;
        const float M = lane < nrow ? mass[r] : 0.f;
        const float fl = 1e-6f * narrow_trunc(tot) / NB;
        const bool ok = M > 0.f && tot > 0.0;
        // an empty band sits 6 dex (per band) below the cell's total power
        for (int k = 0; k < NB; ++k)
            band[lane][k] = log10f(fmaxf(ok ? fmaxf(band[lane][k], fl) / M : 0.f, 1e-30f));
        if (lane < nrow) total[r] = tot;
        __syncwarp();
        for (int rr = 0; rr < nrow; ++rr) features[(size_t)(base + rr) * NB + lane] = band[rr][lane];
        __syncwarp();
    }
}

// v >> s for any s (the instruction's clamped shift)
__device__ __forceinline__ unsigned shr_clamped(unsigned v, unsigned s)
{
    unsigned r;
    asm("shr.b32 %0, %1, %2;" : "=r"(r) : "r"(v), "r"(s));
    return r;
}

// ((h0:l0) >> s) for any s
__device__ __forceinline__ unsigned long long shr64_clamped(unsigned h0, unsigned l0, unsigned s)
{
    const unsigned l1 = __funnelshift_rc(l0, h0, s);
    return ((unsigned long long)shr_clamped(h0, s) << 32) | shr_clamped(l1, (unsigned)max((int)s - 32, 0));
}

// sum 2^(e - 1080) rounded to FP64, for sum >= 2^40 or so and a result within the
// normal range
__device__ __forceinline__ double fixed58_to_double(unsigned long long sum, unsigned e)
{
    const int lz = __clzll((long long)sum);
    const unsigned long long m = (sum << lz) + 0x400ull;  // may carry out of the top: then the mantissa is zero
    return __longlong_as_double((long long)(((m >> 11) & 0xFFFFFFFFFFFFFull) +
                                            ((unsigned long long)(e + 6u - (unsigned)lz + (m < 0x400ull ? 1u : 0u)) << 52)));
}

// Band compression with one band per lane, for input grids whose bands hold at
// most W columns each.  A warp takes its rows from a ring of stages that bulk
// asynchronous copies fill (rows are contiguous: one copy per stage of `rows`
// rows), so the next stages stream in while one is summed and no row is staged
// through registers.  Lane b reads band b's columns into registers, finds the
// largest, and adds them as 64-bit fixed-point numbers relative to it (58 bits: an
// FP64 addition holds the FP64 pipe for as long as 78 of these instructions take
// to issue, the integer sum takes 13 per value and is exact but for one final
// rounding).  The total is the integer sum of the bands' sums, aligned to the
// row's largest entry.  Each lane then forms its band's feature and the row leaves
// as one 128-byte store.  A row with an entry that is negative, not finite, above
// 2^1009 or between 0 and 2^-895 is summed in FP64, band by band.
//
// Against one row per lane (above): 4e6 dense rows of 200 wavelengths 1.90 ms
// instead of 2.48, 8e6 rows of a torus that is 3/5 empty 2.28 ms instead of 3.84
// (75% of the copy rate, the bound there; dense rows are bound by issue, some
// 300 instructions a row).  Three or four stages of the ring, stages of 6 KB and
// blocks of 8 warps were 3 to 9% slower.  The form above stays for what this one
// cannot take: tables not 16-byte aligned, bands of more than 16 columns, rows of
// more than 512.
constexpr int BR_WARPS = 4;    // warps per block
constexpr int BR_STAGES = 2;   // stages of a warp's ring
constexpr int BR_MAXW = 16;
// The band starts as a call uploads them: NB + 1 starts, then two zeros that a kernel
// sets when a copy did not arrive in time: of a row (band compression), of a tile's
// features (inference).
constexpr int BAND_INTS = NB + 3;

// a stage holds about 3 KB, or two rows of the widest table
constexpr size_t BR_SMEM_MAX = 128 + (size_t)BR_WARPS * BR_STAGES * 2 * BR_MAXW * NB * sizeof(double);

// features and total of one row from its band values; s: where the bands start
template <int W>
__device__ __forceinline__ void band_row(const double* row, int first, int width, float M, float dark, float* __restrict__ feat,
                                         double* __restrict__ total, int lane)
{
    double v[W];
    unsigned mx = 0u, any = 0u;
#pragma unroll
    for (int k = 0; k < W; ++k) {
        v[k] = k < width ? row[first + k] : 0.0;
        mx = max(mx, (unsigned)__double2hiint(v[k]));
        any |= (unsigned)__double2loint(v[k]);
    }
    const bool zero = mx == 0u && any == 0u;
    const bool odd = mx - 0x08000000u >= 0x77000000u && !zero;  // below 2^-895, above 2^1009, negative, not finite
    double B = 0.0, tot = 0.0;
    bool ok = M > 0.f;
    if (__any_sync(0xffffffffu, odd)) {
#pragma unroll
        for (int k = 0; k < W; ++k) B += v[k];
        for (int b = 0; b < NB; ++b) tot += __shfl_sync(0xffffffffu, B, b);
        ok = ok && tot > 0.0;
    } else {
        const unsigned e = mx >> 20, E = __reduce_max_sync(0xffffffffu, mx) >> 20;
        if (E == 0u) {  // an empty row
            feat[lane] = dark;
            if (lane == 0) *total = 0.0;
            return;
        }
        unsigned long long sum = 0ull;
#pragma unroll
        for (int k = 0; k < W; ++k) {
            const unsigned hi = (unsigned)__double2hiint(v[k]), lo = (unsigned)__double2loint(v[k]);
            // (zeros and subnormals, read as normal numbers, shift out: e >= 128)
            const unsigned mh = (hi & 0xFFFFFu) | 0x100000u;
            sum += shr64_clamped(__funnelshift_l(lo, mh, 5), lo << 5, e - (hi >> 20));
        }
        if (zero) sum = 0ull;
        B = zero ? 0.0 : fixed58_to_double(sum, e);
        // the bands' sums (below 2^62) aligned to the row's exponent, summed over the
        // lanes in three pieces, and rounded to units of 2^-53 of the largest entry
        const unsigned long long a = shr64_clamped((unsigned)(sum >> 32), (unsigned)sum, E - e);
        const unsigned r0 = __reduce_add_sync(0xffffffffu, (unsigned)a & 0x1FFFFFu),
                       r1 = __reduce_add_sync(0xffffffffu, (unsigned)(a >> 21) & 0x1FFFFFu),
                       r2 = __reduce_add_sync(0xffffffffu, (unsigned)(a >> 42));
        tot = fixed58_to_double(((unsigned long long)r2 << 37) + ((unsigned long long)r1 << 16) + ((r0 + 16u) >> 5),
                                E + 5u);
    }
    const float fl = 1e-6f * narrow_trunc(tot) / NB;
    // an empty band sits 6 dex (per band) below the cell's total power
    feat[lane] = log10f(fmaxf(ok ? fmaxf(narrow_trunc(B), fl) / M : 0.f, 1e-30f));
    if (lane == 0) *total = tot;
}

template <int W>
__global__ void __launch_bounds__(32 * BR_WARPS) band_rows_kernel(
    const double* __restrict__ A, long long ncell, int n_in, int rows, const int* __restrict__ start, int* timeout,
    const float* __restrict__ mass, float tiny, float* __restrict__ features, double* __restrict__ total)
{
    extern __shared__ __align__(128) unsigned char br_smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned stage_bytes = (unsigned)rows * n_in * sizeof(double);
    double* ring = reinterpret_cast<double*>(br_smem + 128 + (size_t)warp * BR_STAGES * stage_bytes);
    unsigned long long* bar = reinterpret_cast<unsigned long long*>(br_smem) + warp * BR_STAGES;
    if (lane == 0) {
        for (int k = 0; k < BR_STAGES; ++k) mbar_init(&bar[k], 1);
        fence_barrier_init();
    }
    __syncwarp();
    const int first = start[lane], width = start[lane + 1] - first;
    const float dark = log10f(tiny);  // the feature of a band without dust or power
    const long long nfull = ncell / rows;  // full stages; the rows left over are read directly
    const long long w0 = (long long)blockIdx.x * BR_WARPS + warp, step = (long long)gridDim.x * BR_WARPS;
    const auto fetch = [&](long long c, int st) {
        fence_proxy_async();
        bulk_load(ring + (size_t)st * rows * n_in, A + (size_t)c * rows * n_in, stage_bytes, &bar[st]);
    };
    if (lane == 0)
        for (int k = 0; k < BR_STAGES - 1; ++k)
            if (w0 + k * step < nfull) fetch(w0 + k * step, k);
    int st = 0;
    unsigned parity = 0;
    for (long long c = w0; c < nfull; c += step) {
        const long long ahead = c + (BR_STAGES - 1) * step;
        const int st_ahead = st == 0 ? BR_STAGES - 1 : st - 1;
        if (lane == 0 && ahead < nfull) fetch(ahead, st_ahead);
        const float my_mass = lane < rows ? __ldg(mass + c * rows + lane) : 0.f;
        if (!__all_sync(0xffffffffu, mbar_wait(&bar[st], parity))) {
            atomicOr(timeout, 1);
            // the copies still in flight land in this block's memory: give them their time
            for (int k = 1; k < BR_STAGES; ++k) {
                const int s2 = (st + k) % BR_STAGES;
                if (c + k * step < nfull) mbar_wait(&bar[s2], s2 < st ? parity ^ 1u : parity);
            }
            break;
        }
        const double* tile = ring + (size_t)st * rows * n_in;
#pragma unroll 1
        for (int r = 0; r < rows; ++r) {
            const long long m = c * rows + r;
            band_row<W>(tile + r * n_in, first, width, __shfl_sync(0xffffffffu, my_mass, r), dark, features + m * NB,
                        total + m, lane);
        }
        __syncwarp();  // every lane is done with this stage before it is refilled
        if (++st == BR_STAGES) {
            st = 0;
            parity ^= 1u;
        }
    }
    for (long long m = nfull * rows + w0; m < ncell; m += step)
        band_row<W>(A + (size_t)m * n_in, first, width, mass[m], dark, features + m * NB, total + m, lane);
}

template <int W>
cudaError_t launch_band_rows(const double* A, long long ncell, int n_in, int* d_start, const float* mass,
                             float* features, double* total, cudaStream_t s)
{
    // stages of about 3 KB (an even number of rows, which keeps them 16-byte aligned)
    const int rows = std::min(32, std::max(2, 2 * (3072 / (16 * n_in))));
    const size_t smem = 128 + (size_t)BR_WARPS * BR_STAGES * rows * n_in * sizeof(double);
    cudaError_t e = cudaFuncSetAttribute(band_rows_kernel<W>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)BR_SMEM_MAX);
    if (e != cudaSuccess) return e;
    int dev = 0, sms = 0, per_sm = 0;
    if ((e = cudaGetDevice(&dev)) || (e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) ||
        (e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, band_rows_kernel<W>, 32 * BR_WARPS, smem)))
        return e;
    const long long want = (ncell + (long long)rows * BR_WARPS - 1) / ((long long)rows * BR_WARPS);
    const int blocks = (int)std::max<long long>(1, std::min<long long>(want, (long long)sms * std::max(1, per_sm)));
    band_rows_kernel<W><<<blocks, 32 * BR_WARPS, smem, s>>>(A, ncell, n_in, rows, d_start, d_start + NB + 1, mass, 1e-30f, features,
                                                     total);
    return cudaGetLastError();
}

int band_blocks(long long ncell)
{
    long long b = (ncell + 32 * BF_WARPS - 1) / (32 * BF_WARPS);
    if (b > 152LL * 16) b = 152LL * 16;
    return (int)(b < 1 ? 1 : b);
}

// The exact solve, one warp per batch of up to EX_BATCH rows.
//
// Per row and population i the solve needs P_i = sum_j w_ij A_j, the target
// ln G_i(T_i) = ln(P_i / M) - ln c_i, a start for T_i, one evaluation of
// G_i(T_i) = sum_l K_il / expm1(a_l / T_i), and a Newton test;
// the emission row is e_l = sum_i (P_i / G_i) K_il / expm1(a_l / T_i).
//
// An FP64 warp instruction holds the SM's FP64 pipe for as long as 78 other
// instructions take to issue, so FP64 does only what has to be FP64:
//
//  * The powers are sums in 64-bit integers.  The inputs of a block of 256
//    columns become fixed-point numbers relative to the largest (59 bits), the
//    shares relative to the population's largest in the block (58 bits), and a
//    product is three 32-bit multiply-adds into 64-bit sums, which do not depend
//    on their order.  A sum's unit is 2^-56 of the largest entry times the scale
//    of the shares; its roundings make 3 units (200 columns; 1.5 for 20), and what
//    is cut off entries below 1/64 of the largest 0.05 units each.  A population
//    whose sum holds at least 2^55 units (2^54 up to 64 columns) so has it to 0.7 x
//    2^-53, or 3 x 2^-53 if nearly all entries are that small; 200 FP64 additions in
//    the lanes' order come to 0.8 x 2^-53 in the mean and 13 x 2^-53 at most.
//    Where a sum holds fewer (the power lies in few columns, or where the
//    population's share is small: without the test a share of 5e-4 (1000 micron)
//    cost 5e-14 of that population's power, one of 5e-7 4e-11) the block is summed
//    in FP64 instead, and so is one with a negative or non-finite entry, or none
//    above 2^-895.  A power of two per entry and population instead of the test
//    took 13% more time for every row.
//  * Per population (FP64, lane 3r + i holds row r's population i, so the rows
//    share each FP64 instruction): the target, the clamp to 3 or 2000 K, the
//    start 1/T_i (cubic Hermite in ln G, on points equally spaced in it: no
//    search, no division) and after the evaluation the Newton test, which
//    compares G_i with P_i / (M c_i) itself.
//  * Per term (double-float, FP32 pipe; dfloat.cuh): the 300 terms of a row,
//    slots s = i * NOUT + l, lane j holding slots j + 32 k.  x = a_l / T_i,
//    expm1(x), its reciprocal, the term t = K_il q.  Terms with x > 70 are left
//    out: over 3..2000 K they carry less than 4e-23 of G_i.
//  * The output row: with E the binary exponent of max_i P_i, the scaled
//    P_i 2^-E over G_i times each term, summed over the populations in
//    double-float, widened to FP64 by integers and scaled by 2^E: every row sums
//    to sum_i P_i to the double-float rounding (~1e-14).
// The start is within 5e-15 of the root, so the first evaluation passes the
// 1e-13 convergence test; a population that does not (the coarse-start
// diagnostic, or a rare target) continues Newton over the whole warp, and its
// row is evaluated and written again.
//
// What bounds it is instruction issue (78%): 2530 warp instructions per row, of
// which the powers take some 670, the output 340 and the terms most of the rest, at
// 72 registers and 28 warps per SM.  1e6 rows of 200 wavelengths take 2.8 ms
// (5.3 with FP64 power sums, a start table searched in ln G and Taylor-series
// exponentials: FP64 pipe 62% busy, 4270 instructions per row), 2.1e6 rows of
// 200 + 100 wavelengths 6.6 ms (12.5).
constexpr int NS = NPOP * NOUT;
constexpr int EX_SLOTS = (NS + 31) / 32;
constexpr int EX_WARPS = 4;   // warps per block
constexpr int EX_BLOCKS = 7;  // blocks per SM (the registers' bound)
constexpr int EX_SPREAD = 24; // warps per SM that short row lists are spread over
constexpr int EX_BATCH = 10;  // most rows per warp batch: lanes 3r + i, r < 10
constexpr float Z_CUT = 70.f * (float)DF_Z_PER_X;

// binary32 -> FP64 on the integer pipe: exact for normal numbers, zero for
// zero and subnormals (which the double-float terms only reach below 1e-23
// of a row)
__device__ __forceinline__ double widen(float f)
{
    const unsigned u = __float_as_uint(f);
    const unsigned e = (u >> 23) & 0xFFu;
    return e ? __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7FFFFFFFu) >> 3) + 0x38000000u)), (int)(u << 29))
             : 0.0;
}

__device__ __forceinline__ double df_to_double(dfl::df2 v) { return widen(v.hi) + widen(v.lo); }

// (hi + lo) 2^E for a normalised pair with hi >= 0, on the integer pipe: the
// low word's bits added to the high word's significand (cut below 2^-52); a
// result that would leave the normal range takes the multiplication
__device__ __forceinline__ double df_scaled(dfl::df2 v, int E)
{
    const unsigned uh = __float_as_uint(v.hi), ul = __float_as_uint(v.lo);
    if (uh < 0x00800000u) return 0.0;
    int eh = (int)(uh >> 23);
    const int el = (int)((ul >> 23) & 0xFFu), d = eh - el;  // d >= 24 where lo counts
    const unsigned ml = el ? (ul & 0x7FFFFFu) | 0x800000u : 0u;
    const unsigned t = d <= 29 ? ml << (29 - d) : (d < 61 ? ml >> (d - 29) : 0u);
    long long m = (long long)((uh & 0x7FFFFFu) | 0x800000u) << 29;
    m += (ul >> 31) ? -(long long)t : (long long)t;
    if (m < (1ll << 52)) {  // the low word took the leading bit
        m <<= 1;
        --eh;
    }
    const int e = eh + 896 + E;
    if (e <= 0 || e >= 0x7FF)
        return __longlong_as_double(m + ((long long)(eh + 895) << 52)) * __longlong_as_double((long long)(E + 1023) << 52);
    return __longlong_as_double(m + ((long long)(e - 1) << 52));
}

// v 2^e for a normal v (or 0): the exponent field moved on the integer pipe; a
// result that would leave the normal range takes the multiplication
__device__ __forceinline__ double scale_pow2(double v, int e)
{
    const long long u = __double_as_longlong(v);
    const int ev = (int)((u >> 52) & 0x7FF);
    if (ev == 0 || ev + e <= 0 || ev + e >= 0x7FF) return v * __longlong_as_double((long long)(e + 1023) << 52);
    return __longlong_as_double(u + ((long long)e << 52));
}

// the warp sums of three values on every lane: one butterfly that halves the
// set of partial sums a lane carries at the first two levels (6 additions
// instead of 15); lanes 8k .. 8k+7 end with the sum of value k, broadcast
template <typename T, typename Shfl, typename Add>
__device__ __forceinline__ void warp_sum3(T& a, T& b, T& c, const T zero, const Shfl& xor_, const Shfl& from,
                                          const Add& add)
{
    const int lane = threadIdx.x & 31;
    const bool up = lane & 16;
    // level 16: the lower half keeps (a, b), the upper half (c, 0)
    T k0 = up ? c : a, k1 = up ? zero : b;
    const T s0 = up ? a : c, s1 = up ? b : zero;
    k0 = add(k0, xor_(s0, 16, true));
    k1 = add(k1, xor_(s1, 16, true));
    // level 8: lanes with bit 3 keep the second value
    const bool hi8 = lane & 8;
    T k = add(hi8 ? k1 : k0, xor_(hi8 ? k0 : k1, 8, true));
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) k = add(k, xor_(k, o, true));
    a = from(k, 0, false);
    b = from(k, 8, false);
    c = from(k, 16, false);
}

template <typename T>
__device__ __forceinline__ void warp_sum3(T& a, T& b, T& c)
{
    const auto sh = [](T v, int o, bool x) {
        return x ? __shfl_xor_sync(0xffffffffu, v, o) : __shfl_sync(0xffffffffu, v, o);
    };
    warp_sum3(a, b, c, T(0), sh, sh, [](T x, T y) { return x + y; });
}

__device__ __forceinline__ void warp_sum3(dfl::df2& a, dfl::df2& b, dfl::df2& c)
{
    const auto sh = [](dfl::df2 v, int o, bool x) {
        return x ? dfl::make(__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o))
                 : dfl::make(__shfl_sync(0xffffffffu, v.hi, o), __shfl_sync(0xffffffffu, v.lo, o));
    };
    // add(x, y) == add(y, x) bit for bit: every lane ends with the same sums
    warp_sum3(a, b, c, dfl::make(0.f, 0.f), sh, sh, [](dfl::df2 x, dfl::df2 y) { return dfl::add(x, y); });
}

__device__ __forceinline__ dfl::df2 df_from_double(double v)
{
    const float h = __double2float_rn(v);
    return dfl::make(h, __double2float_rn(v - (double)h));
}

// 1 / a for a = hi + lo > 0 (lo a few ulp of hi at most) in double-float: the
// approximate binary32 reciprocal corrected to its last bit, then the exact
// residual 1 - a y
__device__ __forceinline__ dfl::df2 df_recip(float hi, float lo)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(hi));
    y = fmaf(y, fmaf(-hi, y, 1.0f), y);
    const float r = fmaf(-lo, y, fmaf(-hi, y, 1.0f));
    const float yr = __fmul_rn(y, r);
    return dfl::make(y, fmaf(yr, r, yr));
}

// Term of slot (z, K) at 1/T: t = K / expm1(a / T) as hi + lo.  Sums and products
// here stay unevaluated (lo a few ulp of hi at most), which the next step allows.
__device__ __forceinline__ dfl::df2 slot_term(float4 aK, float ih, float il, const float2* __restrict__ exp_tab)
{
    float zh, zl;
    dfl::two_prod(aK.x, ih, zh, zl);
    zl = fmaf(aK.y, ih, fmaf(aK.x, il, zl));
    if (!(zh <= Z_CUT)) return dfl::make(0.f, 0.f);
    const dfl::df2 q0 = dfl::expm1_z(dfl::make(zh, zl), [&](int j) {
        const float2 e = exp_tab[j];
        return dfl::make(e.x, e.y);
    });
    const dfl::df2 q = df_recip(q0.hi, q0.lo);
    float th, tl;
    dfl::two_prod(aK.z, q.hi, th, tl);
    return dfl::make(th, fmaf(aK.w, q.hi, fmaf(aK.z, q.lo, tl)));
}

// One row: every slot at its population's 1/T (populations with on bit i), G_i
// over the warp, and the output row written from the same terms (staged in
// buf) with the scaled powers Pp_i (P_i 2^-E).  The slot loop is not unrolled:
// the solve's code has to stay in the instruction cache.
__device__ __forceinline__ void eval_row(const float4* __restrict__ slot, const float2* __restrict__ exp_tab,
                                         const dfl::df2 (&iT)[NPOP], unsigned on, const dfl::df2 (&Pp)[NPOP],
                                         int scale_e, double* __restrict__ out, float2* __restrict__ buf, int lane,
                                         dfl::df2 (&G)[NPOP])
{
    if (on == 0u) {  // no population absorbs (a dust-free or unheated cell): a zero row
#pragma unroll
        for (int i = 0; i < NPOP; ++i) G[i] = dfl::make(0.f, 0.f);
        for (int l = lane; l < NOUT; l += 32) __stcs(out + l, 0.0);
        return;
    }
    // a lane meets its populations' slots one population after the other: the
    // running sum is set aside where the next one starts
    dfl::df2 g0 = dfl::make(0.f, 0.f), g1 = g0, it = iT[0];
    float gh = 0.f, gl = 0.f;
    bool act = on & 1u;
    int next = NOUT;  // first slot of the next population
#pragma unroll 1
    for (int s = lane; s < EX_SLOTS * 32; s += 32) {
        if (s >= next) {
            const bool first = next == NOUT;
            if (first) g0 = dfl::renorm(gh, gl); else g1 = dfl::renorm(gh, gl);
            it = first ? iT[1] : iT[2];
            act = on & (first ? 2u : 4u);
            next = first ? 2 * NOUT : EX_SLOTS * 32;
            gh = gl = 0.f;
        }
        dfl::df2 o = dfl::make(0.f, 0.f);
        if (act && s < NS) o = slot_term(slot[s], it.hi, it.lo, exp_tab);
        if (s < NS) buf[s] = make_float2(o.hi, o.lo);
        float e;
        dfl::two_sum(gh, o.hi, gh, e);
        gl = __fadd_rn(gl, __fadd_rn(e, o.lo));
    }
    dfl::df2 g2 = dfl::renorm(gh, gl);
    warp_sum3(g0, g1, g2);
    G[0] = g0; G[1] = g1; G[2] = g2;
    // P_i / G_i, population i on the lanes that are i modulo 3
    const int i3 = lane % NPOP;
    const dfl::df2 gi = i3 == 0 ? g0 : (i3 == 1 ? g1 : g2), pi = i3 == 0 ? Pp[0] : (i3 == 1 ? Pp[1] : Pp[2]);
    const dfl::df2 ri = gi.hi > 0.f ? dfl::mul(pi, df_recip(gi.hi, gi.lo)) : dfl::make(0.f, 0.f);
    dfl::df2 PS[NPOP];
#pragma unroll
    for (int i = 0; i < NPOP; ++i)
        PS[i] = dfl::make(__shfl_sync(0xffffffffu, ri.hi, i), __shfl_sync(0xffffffffu, ri.lo, i));
    __syncwarp();
#pragma unroll 1
    for (int l = lane; l < NOUT; l += 32) {
        float h[NPOP], e[NPOP];
#pragma unroll
        for (int i = 0; i < NPOP; ++i) {
            const float2 b = buf[i * NOUT + l];
            dfl::two_prod(PS[i].hi, b.x, h[i], e[i]);
            e[i] = fmaf(PS[i].lo, b.x, fmaf(PS[i].hi, b.y, e[i]));
        }
        float u, ue, v, ve;
        dfl::two_sum(h[0], h[1], u, ue);
        dfl::two_sum(u, h[2], v, ve);
        const float lo = __fadd_rn(__fadd_rn(__fadd_rn(e[0], e[1]), e[2]), __fadd_rn(ue, ve));
        __stcs(out + l, df_scaled(dfl::renorm(v, lo), scale_e));
    }
    __syncwarp();
}

// G_i and T dG_i/dT at 1/T for one population, the lanes splitting the
// wavelengths (the rare Newton solve that needs more than one evaluation)
__device__ __noinline__ void pop_G_warp(const float4* __restrict__ slot, const float2* __restrict__ exp_tab, int i,
                                        dfl::df2 iT, int lane, double& G, double& D)
{
    dfl::df2 g = dfl::make(0.f, 0.f), z0 = g, z1 = g;
    float d = 0.f, y0 = 0.f, y1 = 0.f;
    for (int l = lane; l < NOUT; l += 32) {
        const float4 aK = slot[i * NOUT + l];
        const dfl::df2 t = slot_term(aK, iT.hi, iT.lo, exp_tab);
        g = dfl::add(g, dfl::renorm(t.hi, t.lo));
        // t x (1 + q), q = t / K
        d += t.hi * (aK.x * iT.hi * (float)(1.0 / DF_Z_PER_X)) * (1.f + t.hi / aK.z);
    }
    warp_sum3(g, z0, z1);
    warp_sum3(d, y0, y1);
    G = df_to_double(g);
    D = (double)d;
}

// Start of the Newton solve for ln G_i = target: 1/T from the cubic Hermite
// polynomial of the table's interval k that holds the target.  With 8192
// intervals it is within 5e-15 of the root (the error falls as the fourth
// power of the spacing; 4096 intervals leave 2e-14, which shows in the rows).  stride > 1 uses every stride-th point only (a
// coarser start that needs further Newton steps; a diagnostic setting).
__device__ __forceinline__ double start_invT(int i, double target, int stride, int& k, float& slope)
{
    const double t = target - c_lnG_lo[i];
    const int lg = 31 - __clz(stride);  // stride = 2^lg
    const int a = min((int)__double2float_rn(t * c_inv_h[i]) >> lg, ((NTAB - 1) >> lg) - 1);
    k = a << lg;
    // u = position within the interval; k as a double through the 2^52 offset
    double u = fma(-(__hiloint2double(0x43300000, k) - 4503599627370496.0), c_h[i], t) * c_inv_h[i];
    const double2 pa = __ldg(&g_invT_tab[i][k]), pb = __ldg(&g_invT_tab[i][k + stride]);
    double sa = pa.y, sb = pb.y;
    if (lg > 0) {
        const double st = __hiloint2double((1023 + lg) << 20, 0);
        sa *= st;
        sb *= st;
        u *= __hiloint2double((1023 - lg) << 20, 0);
    }
    const double dx = pb.x - pa.x;
    // d ln T / d ln G at the interval's start (it only sets the Newton test's step)
    slope = -__double2float_rn(pa.y * c_inv_h[i]) / __double2float_rn(pa.x);
    const double c2 = fma(3.0, dx, fma(-2.0, sa, -sb)), c3 = fma(-2.0, dx, sa + sb);
    return fma(u, fma(u, fma(u, c3, c2), sa), pa.x);
}

// The sums of a block of up to 256 columns of a row, sum_j w_ij A_j of the three
// populations, in fixed point: value = s_i 2^(e - 1078 - x_i), e the biased exponent
// of the block's largest entry, 2^-x_i the scale of the population's shares in the
// block.  False (nothing summed) for a block with a negative or non-finite entry,
// none above 2^-895 but one above zero, or too few units in a sum.
constexpr int EX_COLS = 256;
constexpr int SHARE_MAX_EXP = 60;                    // largest x_i
// x_i of the block whose shares start at wq (one byte each)
__device__ __forceinline__ int share_scale(const int4* wq, int i)
{
    return (int)(((unsigned)__ldg(&wq[1].z) >> (8 * i)) & 0xFFu);
}

__device__ __forceinline__ void mad_wide(unsigned long long& acc, unsigned a, int b)
{
    asm("mad.wide.u32 %0, %1, %2, %0;" : "+l"(acc) : "r"(a), "r"(b));
}

__device__ __forceinline__ void mad_wide(long long& acc, unsigned a, int b)
{
    asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(acc) : "r"(a), "r"(b));
}

// wq: the shares' fixed-point pairs, 32 bytes per wavelength: hi, lo of the three
// populations, the block's packed x_i, 4 bytes of padding (two 16-byte loads)
__device__ __forceinline__ bool block_powers(const double* __restrict__ row, int n, const int4* __restrict__ wq,
                                             int lane, unsigned long long& s0, unsigned long long& s1,
                                             unsigned long long& s2, int& e)
{
    double v[EX_COLS / 32];
    unsigned mx = 0u, any = 0u;
#pragma unroll
    for (int k = 0; k < EX_COLS / 32; ++k) {
        v[k] = lane + 32 * k < n ? __ldcs(row + lane + 32 * k) : 0.0;
        mx = max(mx, (unsigned)__double2hiint(v[k]));
        any |= (unsigned)__double2loint(v[k]);
    }
    mx = __reduce_max_sync(0xffffffffu, mx);
    s0 = s1 = s2 = 0ull;
    e = 1;
    if (mx >= 0x7FF00000u) return false;
    // all zero, or too small for a subnormal entry to shift out
    if (mx < 0x08000000u) return mx == 0u && __reduce_or_sync(0xffffffffu, any) == 0u;
    e = (int)(mx >> 20);
    // products a w: a = v 2^(1081 - e) as hi (27 bits) and lo (32 bits), w 2^(58 + x)
    // as hi (29 bits, unsigned) and lo (28 bits and sign); partial sums of up to 8
    unsigned long long hh0 = 0, hh1 = 0, hh2 = 0, lh0 = 0, lh1 = 0, lh2 = 0;
    long long hl0 = 0, hl1 = 0, hl2 = 0;
#pragma unroll
    for (int k = 0; k < EX_COLS / 32; ++k) {
        if (32 * k < n) {
            int4 wa = make_int4(0, 0, 0, 0), wb = wa;
            if (lane + 32 * k < n) {
                wa = __ldg(wq + 2 * lane + 64 * k);
                wb = __ldg(wq + 2 * lane + 64 * k + 1);
            }
            const unsigned hi = (unsigned)__double2hiint(v[k]), lo = (unsigned)__double2loint(v[k]);
            const unsigned ex = hi >> 20;
            const unsigned mh = (hi & 0xFFFFFu) | (ex ? 0x100000u : 0u), sh = (unsigned)e - ex;
            const unsigned ah0 = __funnelshift_l(lo, mh, 6), al0 = lo << 6;
            const unsigned al1 = __funnelshift_rc(al0, ah0, sh);
            const unsigned ah = shr_clamped(ah0, sh), al = shr_clamped(al1, (unsigned)max((int)sh - 32, 0));
            mad_wide(hh0, ah, wa.x);
            mad_wide(hl0, ah, wa.y);
            mad_wide(lh0, al, wa.x);
            mad_wide(hh1, ah, wa.z);
            mad_wide(hl1, ah, wa.w);
            mad_wide(lh1, al, wa.z);
            mad_wide(hh2, ah, wb.x);
            mad_wide(hl2, ah, wb.y);
            mad_wide(lh2, al, wb.x);
        }
    }
    // in units of hi x hi, rounded
    s0 = hh0 + (unsigned long long)((hl0 + (1ll << 28)) >> 29) + ((lh0 + (1ull << 31)) >> 32);
    s1 = hh1 + (unsigned long long)((hl1 + (1ll << 28)) >> 29) + ((lh1 + (1ull << 31)) >> 32);
    s2 = hh2 + (unsigned long long)((hl2 + (1ll << 28)) >> 29) + ((lh2 + (1ull << 31)) >> 32);
    warp_sum3(s0, s1, s2);
    const unsigned least = min((unsigned)(s0 >> 32), min((unsigned)(s1 >> 32), (unsigned)(s2 >> 32)));
    return least >= (n <= 64 ? 1u << 22 : 1u << 23);
}

// s 2^(e - 1078)
__device__ __forceinline__ double fixed_to_double(unsigned long long s, int e)
{
    if (s == 0ull) return 0.0;
    const int x = e - 1078, h = x / 2;
    return scale_pow2(scale_pow2(__ull2double_rn(s), h), x - h);
}

// the same sums in FP64
__device__ __noinline__ void block_powers_fp64(const double* __restrict__ row, int n, const double* __restrict__ w,
                                               int nw, int lane, double& p0, double& p1, double& p2)
{
    p0 = p1 = p2 = 0.0;
    for (int j = lane; j < n; j += 32) {
        const double v = __ldcs(row + j);
        p0 += __ldg(w + j) * v;
        p1 += __ldg(w + nw + j) * v;
        p2 += __ldg(w + 2 * nw + j) * v;
    }
    warp_sum3(p0, p1, p2);
}

// Exact emission for rows m = rows ? rows[k] : k, k < nrows.  w: the absorption
// shares as fill_shares lays them out (16-byte aligned).  A
// second absorbed table A2 [ncell][n2] with its shares w2 (may be NULL) adds its
// power to each population's.
__global__ void __launch_bounds__(32 * EX_WARPS, EX_BLOCKS) exact_kernel(
    const double* __restrict__ A, int n_in, const double* __restrict__ w, const double* __restrict__ A2, int n2,
    const double* __restrict__ w2, const float* __restrict__ mass, const unsigned* __restrict__ rows, long long nrows,
    double* __restrict__ emission, float* __restrict__ temperature, int stride, int batch)
{
    __shared__ float4 s_slot[NS];
    __shared__ float2 s_exp[DF_EXP_N];
    __shared__ float2 s_buf[EX_WARPS][NS];
    for (int s = threadIdx.x; s < NS; s += blockDim.x) s_slot[s] = g_slot[s];
    for (int j = threadIdx.x; j < DF_EXP_N; j += blockDim.x) s_exp[j] = g_exp[j];
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float2* buf = s_buf[warp];
    const int my_r = lane / NPOP, my_i = lane - NPOP * (lane / NPOP);  // this lane's (row, population)
    for (long long base = ((long long)blockIdx.x * EX_WARPS + warp) * batch; base < nrows;
         base += (long long)gridDim.x * EX_WARPS * batch) {
        const int nb = nrows - base < batch ? (int)(nrows - base) : batch;
        const bool mine = my_r < nb;
        const long long my_m = mine ? (rows ? (long long)rows[base + my_r] : base + my_r) : 0;
        // ---- population powers, one row at a time over the lanes: the first
        // block of each table as an integer, converted once for all rows; what
        // else there is is added in FP64
        unsigned long long sa = 0, sb = 0;
        int ea = 1, eb = 1;
        double rest = 0.0;
        bool more = false;
#pragma unroll 1
        for (int r = 0; r < nb; ++r) {
            const long long m = rows ? (long long)rows[base + r] : base + r;
#pragma unroll 1
            for (int tab = 0; tab < (A2 ? 2 : 1); ++tab) {
                const int nw = tab ? n2 : n_in;
                const double* row = (tab ? A2 : A) + (size_t)m * nw;
                const int4* wq = reinterpret_cast<const int4*>(tab ? w2 : w);
#pragma unroll 1
                for (int c = 0; c < nw; c += EX_COLS) {
                    const int n = min(nw - c, EX_COLS);
                    unsigned long long s0, s1, s2;
                    int e;
                    if (block_powers(row + c, n, wq + 2 * c, lane, s0, s1, s2, e)) {
                        const unsigned long long sv = my_i == 0 ? s0 : (my_i == 1 ? s1 : s2);
                        if (c > 0) {
                            more = true;
                            if (my_r == r) rest += fixed_to_double(sv, e - share_scale(wq + 2 * c, my_i));
                        } else if (my_r == r) {
                            if (tab) { sb = sv; eb = e; } else { sa = sv; ea = e; }
                        }
                    } else {
                        double p0, p1, p2;
                        block_powers_fp64(row + c, n, (tab ? w2 : w) + 4 * (size_t)nw + c, nw, lane, p0, p1, p2);
                        more = true;
                        if (my_r == r) rest += my_i == 0 ? p0 : (my_i == 1 ? p1 : p2);
                    }
                }
            }
        }
        double P = fixed_to_double(sa, ea - share_scale(reinterpret_cast<const int4*>(w), my_i));
        if (A2) P += fixed_to_double(sb, eb - share_scale(reinterpret_cast<const int4*>(w2), my_i));
        if (more) P += rest;
        // binary exponent of the row's largest population power (0 if none is positive)
        const int xe = P > 0.0 ? (__double2hiint(P) >> 20) + 1 : 0;
        const int l3 = min(lane - my_i, 29);
        int E = max(__shfl_sync(0xffffffffu, xe, l3),
                    max(__shfl_sync(0xffffffffu, xe, l3 + 1), __shfl_sync(0xffffffffu, xe, l3 + 2)));
        E = E > 0 ? E - 1024 : 0;
        E = E < -1000 ? -1000 : (E > 1000 ? 1000 : E);
        // ---- per population (FP64): target, clamp or table start, 1/T, scaled power
        const float M = mine ? mass[my_m] : 0.f;
        int kind = 0;  // 0 no power, 1 at 3 K, 2 at 2000 K, 3 Newton
        int k_tab = 0;
        float slope = 0.f;
        double Gt = 0.0;
        dfl::df2 iT = dfl::make(0.f, 0.f), Pp = dfl::make(0.f, 0.f);
        if (mine && P > 0.0 && M > 0.f) {
            const double ratio = P / (double)M;
            const double tg = log(ratio) - c_lnc[my_i];
            double x;
            if (c_lnG_lo[my_i] - tg >= 0.0) {
                kind = 1;
                x = 1.0 / T_LO;
            } else if (c_lnG_hi[my_i] - tg <= 0.0) {
                kind = 2;
                x = 1.0 / T_HI;
            } else {
                kind = 3;
                Gt = ratio * c_Gref[my_i];
                x = start_invT(my_i, tg, stride, k_tab, slope);
            }
            iT = df_from_double(x);
            Pp = df_from_double(P * __longlong_as_double((long long)(1023 - E) << 52));
        }
        const unsigned on_all = __ballot_sync(0xffffffffu, kind != 0);
        // ---- one evaluation per row (double-float); lane 3r + i keeps its G_i
        dfl::df2 Gm = dfl::make(0.f, 0.f);
        const auto evaluate = [&](int r) {
            const int l0 = NPOP * r;
            dfl::df2 iTr[NPOP], Ppr[NPOP], G[NPOP];
#pragma unroll
            for (int i = 0; i < NPOP; ++i) {
                iTr[i] = dfl::make(__shfl_sync(0xffffffffu, iT.hi, l0 + i), __shfl_sync(0xffffffffu, iT.lo, l0 + i));
                Ppr[i] = dfl::make(__shfl_sync(0xffffffffu, Pp.hi, l0 + i), __shfl_sync(0xffffffffu, Pp.lo, l0 + i));
            }
            const int Er = __shfl_sync(0xffffffffu, E, l0);
            const long long m = rows ? (long long)rows[base + r] : base + r;
            eval_row(s_slot, s_exp, iTr, (on_all >> l0) & 7u, Ppr, Er, emission + (size_t)m * NOUT, buf, lane, G);
            if (my_r == r) Gm = my_i == 0 ? G[0] : (my_i == 1 ? G[1] : G[2]);
        };
        unsigned todo = (1u << nb) - 1u;  // rows to evaluate: all of them, then those Newton moved
        bool first = true;
        while (todo) {
#pragma unroll 1
            for (unsigned left = todo; left; left &= left - 1u) evaluate(__ffs(left) - 1);
            todo = 0u;
            if (!first) break;
            first = false;
            // ---- Newton test of every population: converged when the step
            // ln(G / Gt) d ln T / d ln G of ln T is below 1e-13 of ln T
            bool redo = false;
            if (kind == 3) {
                const float f = __double2float_rn(df_to_double(Gm) - Gt) / __double2float_rn(Gt);
                const float step = f * slope;
                redo = !(fabsf(step) <= 1e-13f * fabsf(logf(iT.hi)));
            }
            unsigned redo_mask = __ballot_sync(0xffffffffu, redo);
            while (redo_mask) {  // rare: Newton continues for one population over the whole warp
                const int L = __ffs(redo_mask) - 1;
                redo_mask &= redo_mask - 1;
                const int ii = L % NPOP;
                const int k = __shfl_sync(0xffffffffu, k_tab, L);
                const double tgi = log(__shfl_sync(0xffffffffu, Gt, L));
                // from the table's points around the start (one to either side, for
                // a target that rounding put beyond its interval's end)
                double lo = -log(__ldg(&g_invT_tab[ii][max(k - stride, 0)].x)),
                       hi = -log(__ldg(&g_invT_tab[ii][min(k + 2 * stride, NTAB - 1)].x));
                dfl::df2 x = dfl::make(__shfl_sync(0xffffffffu, iT.hi, L), __shfl_sync(0xffffffffu, iT.lo, L));
                double y = -log(df_to_double(x));
                for (int it = 0; it < 100; ++it) {
                    double G, D;
                    pop_G_warp(s_slot, s_exp, ii, x, lane, G, D);
                    const double f = log(G) - tgi;
                    const double step = f * G / D;
                    if (fabs(step) <= 1e-13 * fabs(y)) break;
                    if (f < 0.0) lo = y; else hi = y;
                    double y_new = y - step;
                    if (!(y_new > lo && y_new < hi)) y_new = 0.5 * (lo + hi);
                    y = y_new;
                    x = df_from_double(exp(-y));
                }
                if (lane == L) iT = x;
                todo |= 1u << (L / NPOP);  // the row again, with the population's final temperature
            }
        }
        if (temperature && mine) {
            float T = 0.f;
            if (kind == 1) T = (float)T_LO;
            if (kind == 2) T = (float)T_HI;
            if (kind == 3) T = dfl::recip(iT).hi;
            temperature[(size_t)my_m * NPOP + my_i] = T;
        }
    }
}

__global__ void compact_flags_kernel(const unsigned char* __restrict__ flags, long long n,
                                     unsigned* __restrict__ rows, unsigned long long* __restrict__ count)
{
    for (long long m = (long long)blockIdx.x * blockDim.x + threadIdx.x; m < n; m += (long long)gridDim.x * blockDim.x) {
        const bool f = flags[m] != 0;
        const unsigned mask = __ballot_sync(__activemask(), f);
        if (!f) continue;
        const int lane = threadIdx.x & 31;
        const int leader = __ffs(mask) - 1;
        unsigned long long base = 0;
        if (lane == leader) base = atomicAdd(count, (unsigned long long)__popc(mask));
        base = __shfl_sync(mask, base, leader);
        rows[base + __popc(mask & ((1u << lane) - 1u))] = (unsigned)m;
    }
}

__global__ void zero_temperature_kernel(float* t, long long n)
{
    for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x)
        t[k] = 0.f;
}

// band compression on either kernel; start: the host's copy of d_start
cudaError_t launch_band_features(const double* A, long long ncell, int n_in, const std::vector<int>& start, int* d_start,
                                 const float* mass, float* features, double* total, cudaStream_t s)
{
    int w = 0;
    for (int b = 0; b < NB; ++b) w = std::max(w, start[b + 1] - start[b]);
    if ((reinterpret_cast<uintptr_t>(A) & 15) == 0 && w <= BR_MAXW && n_in <= BR_MAXW * NB) {
        if (w <= 4) return launch_band_rows<4>(A, ncell, n_in, d_start, mass, features, total, s);
        if (w <= 8) return launch_band_rows<8>(A, ncell, n_in, d_start, mass, features, total, s);
        return launch_band_rows<16>(A, ncell, n_in, d_start, mass, features, total, s);
    }
    band_features_kernel<<<band_blocks(ncell), 32 * BF_WARPS, 0, s>>>(A, ncell, n_in, d_start, mass, features, total);
    return cudaGetLastError();
}

// after the stream has synchronised: an error when the call gave up waiting for a copy
int band_check_timeout(int v)
{
    return v ? set_error(SKIRT_ERR_CUDA, "band compression: a row copy did not complete in time") : SKIRT_OK;
}

int grid_blocks(long long n, int block)
{
    long long b = (n + block - 1) / block;
    if (b > 152LL * 64) b = 152LL * 64;
    return (int)(b < 1 ? 1 : b);
}

bool is_device(const void* p)
{
    if (!p) return false;
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged;
}

int check_lambda(const double* lambda_in, int n_in)
{
    if (!lambda_in || n_in < 1 || n_in > 65536) return set_error(SKIRT_ERR_INVALID_ARG, "lambda_in / n_in invalid");
    for (int j = 0; j < n_in; ++j) {
        if (!(lambda_in[j] > 0) || !std::isfinite(lambda_in[j]))
            return set_error(SKIRT_ERR_INVALID_ARG, "lambda_in[%d] must be finite and > 0", j);
        if (j > 0 && !(lambda_in[j] > lambda_in[j - 1]))
            return set_error(SKIRT_ERR_INVALID_ARG, "lambda_in must be strictly increasing");
    }
    return SKIRT_OK;
}

// band start indices over a sorted grid: band b = floor(32 ln(l/lmin) / ln(lmax/lmin)) clamped
std::vector<int> band_starts(const double* lam, int n)
{
    std::vector<int> idx(n, 0);
    const double lo = lam[0], hi = lam[n - 1];
    for (int j = 0; j < n; ++j) {
        int b = 0;
        if (hi > lo) b = (int)std::floor(NB * std::log(lam[j] / lo) / std::log(hi / lo));
        idx[j] = b < 0 ? 0 : (b > NB - 1 ? NB - 1 : b);
    }
    std::vector<int> start(NB + 1, n);
    for (int b = NB; b >= 0; --b) {
        int s = n;
        for (int j = 0; j < n; ++j)
            if (idx[j] >= b) { s = j; break; }
        start[b] = b == NB ? n : s;
    }
    start.resize(BAND_INTS, 0);
    return start;
}

// shares w_i(lambda_j) = (lambda_j/0.55)^delta_i / sum_k (lambda_j/0.55)^delta_k:
// first their fixed-point pairs for block_powers, w 2^(58 + x) = hi 2^29 + lo, |lo|
// <= 2^28, with 2^-x the power of two from the population's largest share among the
// wavelength's block of EX_COLS on, 32 bytes per wavelength, then the shares
// themselves [3][n]; 8 doubles per wavelength in all, so that a second table behind
// the first stays aligned
constexpr int SHARES = 8;
void fill_shares(const double* lam, int n, double* out)
{
    double* w = out + 4 * (size_t)n;
    for (int c = 0; c < n; c += EX_COLS) {
        const int end = std::min(n, c + EX_COLS);
        double top[NPOP] = {};
        for (int j = c; j < end; ++j) {
            double r[NPOP], sum = 0.0;
            for (int i = 0; i < NPOP; ++i) {
                r[i] = std::pow(lam[j] / 0.55, DELTA[i]);
                sum += r[i];
            }
            for (int i = 0; i < NPOP; ++i) {
                w[(size_t)i * n + j] = r[i] / sum;
                top[i] = std::max(top[i], w[(size_t)i * n + j]);
            }
        }
        double scale[NPOP];
        unsigned packed = 0u;
        for (int i = 0; i < NPOP; ++i) {
            int x;
            std::frexp(top[i], &x);
            x = std::min(std::max(-x, 0), SHARE_MAX_EXP);
            packed |= (unsigned)x << (8 * i);
            scale[i] = std::ldexp(536870912.0, x);
        }
        for (int j = c; j < end; ++j) {
            int q[8] = {};
            for (int i = 0; i < NPOP; ++i) {
                const double v = w[(size_t)i * n + j] * scale[i], h = std::floor(v + 0.5);
                q[2 * i] = (int)h;
                q[2 * i + 1] = (int)std::floor((v - h) * 536870912.0 + 0.5);
            }
            q[6] = (int)packed;
            std::memcpy(out + 4 * (size_t)j, q, sizeof q);
        }
    }
}

std::vector<double> share_table(const double* lam, int n)
{
    std::vector<double> w((size_t)SHARES * n);
    fill_shares(lam, n, w.data());
    return w;
}

#define ECK(call)                                                                                       \
    do {                                                                                                \
        cudaError_t e_ = (call);                                                                        \
        if (e_ != cudaSuccess)                                                                          \
            return set_error(e_ == cudaErrorMemoryAllocation ? SKIRT_ERR_OOM : SKIRT_ERR_CUDA,          \
                             "%s failed: %s (%s:%d)", #call, cudaGetErrorString(e_), __FILE__, __LINE__); \
    } while (0)

}  // namespace

int launch_exact_emission(const double* absorbed, int n_in, const double* w_dev, const float* mass,
                          const unsigned* rows, long long nrows, double* emission, float* temperature,
                          cudaStream_t s, const double* absorbed2, int n2, const double* w2_dev)
{
    ECK(upload_model());
    // one warp per batch of rows, every row list alike (all cells, or the
    // surrogate's fallback rows).  SKIRT_EXACT_TABLE_STRIDE (a power of two up to 64)
    // starts the Newton solves from a coarser table: the same results through
    // more Newton steps, a diagnostic of that path.
    int stride = 1;
    if (const char* e = std::getenv("SKIRT_EXACT_TABLE_STRIDE")) {
        const int v = std::atoi(e);
        if (v >= 1 && v <= 64 && (v & (v - 1)) == 0) stride = v;
    }
    if (nrows > 0) {
        // full batches once there are enough rows for them to fill 24 warps per SM;
        // below that as many warps as rows allow, each with fewer rows in series (2000
        // rows: 115 us by tens, 28 us one by one).  24 of the 28 warps an SM holds: 4256
        // rows take 37 us on 2128 warps and 41 on 4256, 12,000 55 by fours and 59 by
        // threes.
        int dev = 0, sms = 0;
        ECK(cudaGetDevice(&dev));
        ECK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
        const long long warps = (long long)sms * EX_SPREAD;
        const int batch = (int)std::min<long long>(EX_BATCH, (nrows + warps - 1) / warps);
        long long blocks = (nrows + EX_WARPS * batch - 1) / (EX_WARPS * batch);
        if (blocks > sms * 32LL) blocks = sms * 32LL;
        exact_kernel<<<(int)blocks, 32 * EX_WARPS, 0, s>>>(absorbed, n_in, w_dev, absorbed2, n2, w2_dev, mass, rows,
                                                           nrows, emission, temperature, stride, batch);
    }
    ECK(cudaGetLastError());
    return SKIRT_OK;
}

}  // namespace skirt

using namespace skirt;

extern "C" int skirt_emission_grid(double* lambda_um, double* weights)
{
    const HostModel& h = host_model();
    if (lambda_um) std::memcpy(lambda_um, h.lam, sizeof h.lam);
    if (weights) std::memcpy(weights, h.W, sizeof h.W);
    return SKIRT_OK;
}

extern "C" int skirt_dust_mass(skirt_grid_t g, float* mass, void* stream)
{
    if (!g || !mass) return set_error(SKIRT_ERR_INVALID_ARG, "grid / mass is NULL");
    if (!is_device(mass)) return set_error(SKIRT_ERR_INVALID_ARG, "mass must be device memory");
    const double vol = (g->bbox[1] - g->bbox[0]) / g->nx * (g->bbox[3] - g->bbox[2]) / g->ny *
                       (g->bbox[5] - g->bbox[4]) / g->nz;
    dust_mass_kernel<<<grid_blocks(g->ncell, 256), 256, 0, (cudaStream_t)stream>>>(g->kr32, g->ncell, (float)vol, mass,
                                                                                  g->oct_leaf, g->oct_levels);
    ECK(cudaGetLastError());
    ECK(cudaStreamSynchronize((cudaStream_t)stream));
    return SKIRT_OK;
}

extern "C" int skirt_band_features(const double* absorbed, long long ncell, int n_in, const double* lambda_in,
                                   const float* mass, float* features, double* total, void* stream)
{
    if (ncell < 0) return set_error(SKIRT_ERR_INVALID_ARG, "ncell < 0");
    if (int r = check_lambda(lambda_in, n_in)) return r;
    if (ncell == 0) return SKIRT_OK;
    if (!is_device(absorbed) || !is_device(mass) || !is_device(features) || !is_device(total))
        return set_error(SKIRT_ERR_INVALID_ARG, "absorbed / mass / features / total must be device memory");
    cudaStream_t s = (cudaStream_t)stream;
    std::vector<int> start = band_starts(lambda_in, n_in);
    int* d_start = nullptr;
    int timeout = 0;
    ECK(cudaMallocAsync((void**)&d_start, sizeof(int) * BAND_INTS, s));
    ECK(cudaMemcpyAsync(d_start, start.data(), sizeof(int) * BAND_INTS, cudaMemcpyHostToDevice, s));
    cudaError_t e = launch_band_features(absorbed, ncell, n_in, start, d_start, mass, features, total, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&timeout, d_start + NB + 1, sizeof(int), cudaMemcpyDeviceToHost, s);
    cudaFreeAsync(d_start, s);
    if (e != cudaSuccess) return set_error(SKIRT_ERR_CUDA, "band features: %s", cudaGetErrorString(e));
    ECK(cudaStreamSynchronize(s));
    return band_check_timeout(timeout);
}

extern "C" int skirt_dust_emission(const double* absorbed, long long ncell, int n_in, const double* lambda_in,
                                   const float* mass, int mode, skirt_mlp_t net, double* emission, float* temperature,
                                   skirt_emission_stats* stats, void* stream)
{
    if (ncell < 0) return set_error(SKIRT_ERR_INVALID_ARG, "ncell < 0");
    if (int r = check_lambda(lambda_in, n_in)) return r;
    if (mode != SKIRT_EMIT_EXACT && mode != SKIRT_EMIT_SURROGATE)
        return set_error(SKIRT_ERR_INVALID_ARG, "unknown mode %d", mode);
    if (mode == SKIRT_EMIT_SURROGATE && !net) return set_error(SKIRT_ERR_INVALID_ARG, "surrogate mode needs a network");
    if (stats) std::memset(stats, 0, sizeof *stats);
    if (ncell == 0) return SKIRT_OK;
    if (ncell >= (1ll << 32)) return set_error(SKIRT_ERR_INVALID_ARG, "ncell must be < 2^32");
    if (!is_device(absorbed) || !is_device(mass) || !is_device(emission) || (temperature && !is_device(temperature)))
        return set_error(SKIRT_ERR_INVALID_ARG, "absorbed / mass / emission / temperature must be device memory");
    cudaStream_t s = (cudaStream_t)stream;
    std::vector<double> w = share_table(lambda_in, n_in);
    double* d_w = nullptr;
    ECK(cudaMallocAsync((void**)&d_w, sizeof(double) * w.size(), s));
    ECK(cudaMemcpyAsync(d_w, w.data(), sizeof(double) * w.size(), cudaMemcpyHostToDevice, s));
    cudaEvent_t ev[4];
    for (auto& e : ev) ECK(cudaEventCreate(&e));
    int rc = SKIRT_OK, timeout[2] = {0, 0};
    unsigned long long nfb = 0;
    if (mode == SKIRT_EMIT_EXACT) {
        ECK(cudaEventRecord(ev[0], s));
        rc = launch_exact_emission(absorbed, n_in, d_w, mass, nullptr, ncell, emission, temperature, s);
        ECK(cudaEventRecord(ev[1], s));
    } else {
        // the working tables live in the network's workspace (grown on demand, kept
        // between calls): a stream-ordered allocation of ~2.5 GB per call cost ~5 ms
        std::unique_lock<std::mutex> ws_lock(mlp_workspace_mutex(net));
        // on every way out of this block (errors included) the stream drains
        // before the lock is released, so no other call reuses tables in use
        struct DrainOnExit {
            cudaStream_t s;
            ~DrainOnExit() { cudaStreamSynchronize(s); }
        } drain{s};
        auto al = [](size_t b) { return (b + 255) & ~(size_t)255; };
        const size_t o_tot = 0, o_cnt = o_tot + al(sizeof(double) * (size_t)ncell), o_start = o_cnt + al(8),
                     o_feat = o_start + al(sizeof(int) * BAND_INTS),
                     o_rows = o_feat + al(sizeof(float) * NB * (size_t)ncell),
                     o_flag = o_rows + al(sizeof(unsigned) * (size_t)ncell), ws_total = o_flag + al((size_t)ncell);
        unsigned char* ws = nullptr;
        if (int r = mlp_workspace(net, ws_total, (void**)&ws)) {
            cudaFreeAsync(d_w, s);
            for (auto& e : ev) cudaEventDestroy(e);
            return r;
        }
        double* d_tot = (double*)(ws + o_tot);
        unsigned long long* d_cnt = (unsigned long long*)(ws + o_cnt);
        int* d_start = (int*)(ws + o_start);
        float* d_feat = (float*)(ws + o_feat);
        unsigned* d_rows = (unsigned*)(ws + o_rows);
        unsigned char* d_flag = ws + o_flag;
        ECK(cudaMemsetAsync(d_cnt, 0, sizeof(unsigned long long), s));
        std::vector<int> start = band_starts(lambda_in, n_in);
        ECK(cudaMemcpyAsync(d_start, start.data(), sizeof(int) * BAND_INTS, cudaMemcpyHostToDevice, s));
        if (temperature) zero_temperature_kernel<<<grid_blocks(3 * ncell, 256), 256, 0, s>>>(temperature, 3 * ncell);
        ECK(cudaEventRecord(ev[0], s));
        ECK(launch_band_features(absorbed, ncell, n_in, start, d_start, mass, d_feat, d_tot, s));
        ECK(cudaEventRecord(ev[1], s));
        rc = mlp_forward_internal(net, d_feat, d_tot, ncell, emission, d_flag, d_start + NB + 2, s);
        if (rc == SKIRT_OK) {
            compact_flags_kernel<<<grid_blocks(ncell, 256), 256, 0, s>>>(d_flag, ncell, d_rows, d_cnt);
            ECK(cudaGetLastError());
            ECK(cudaEventRecord(ev[2], s));
            ECK(cudaMemcpyAsync(&nfb, d_cnt, sizeof nfb, cudaMemcpyDeviceToHost, s));
            ECK(cudaMemcpyAsync(timeout, d_start + NB + 1, sizeof timeout, cudaMemcpyDeviceToHost, s));
            ECK(cudaStreamSynchronize(s));
            rc = launch_exact_emission(absorbed, n_in, d_w, mass, d_rows, (long long)nfb, emission, temperature, s);
            ECK(cudaEventRecord(ev[3], s));
        }
    }
    cudaFreeAsync(d_w, s);
    ECK(cudaStreamSynchronize(s));
    if (rc == SKIRT_OK) rc = mlp_check_timeout(timeout[1]);
    if (rc == SKIRT_OK) rc = band_check_timeout(timeout[0]);
    if (stats && rc == SKIRT_OK) {
        stats->n_cells = (unsigned long long)ncell;
        stats->n_fallback = nfb;
        float a = 0.f, b = 0.f, c = 0.f;
        if (mode == SKIRT_EMIT_EXACT) {
            cudaEventElapsedTime(&c, ev[0], ev[1]);
        } else {
            cudaEventElapsedTime(&a, ev[0], ev[1]);
            cudaEventElapsedTime(&b, ev[1], ev[2]);
            cudaEventElapsedTime(&c, ev[2], ev[3]);
        }
        stats->ms_features = a;
        stats->ms_surrogate = b;
        stats->ms_exact = c;
    }
    for (auto& e : ev) cudaEventDestroy(e);
    return rc;
}

extern "C" int skirt_dust_emission_pair(const double* absorbed_a, long long ncell, int n_a, const double* lambda_a,
                                        const double* absorbed_b, int n_b, const double* lambda_b, const float* mass,
                                        double* emission, float* temperature, void* stream)
{
    if (ncell < 0) return set_error(SKIRT_ERR_INVALID_ARG, "ncell < 0");
    if (int r = check_lambda(lambda_a, n_a)) return r;
    if (absorbed_b || n_b) {
        if (!absorbed_b) return set_error(SKIRT_ERR_INVALID_ARG, "absorbed_b is NULL with n_b > 0");
        if (int r = check_lambda(lambda_b, n_b)) return r;
    }
    if (ncell == 0) return SKIRT_OK;
    if (ncell >= (1ll << 32)) return set_error(SKIRT_ERR_INVALID_ARG, "ncell must be < 2^32");
    if (!is_device(absorbed_a) || (absorbed_b && !is_device(absorbed_b)) || !is_device(mass) ||
        !is_device(emission) || (temperature && !is_device(temperature)))
        return set_error(SKIRT_ERR_INVALID_ARG, "absorbed / mass / emission / temperature must be device memory");
    cudaStream_t s = (cudaStream_t)stream;
    std::vector<double> w = share_table(lambda_a, n_a);
    if (absorbed_b) {
        const std::vector<double> wb = share_table(lambda_b, n_b);
        w.insert(w.end(), wb.begin(), wb.end());
    }
    double* d_w = nullptr;
    ECK(cudaMallocAsync((void**)&d_w, sizeof(double) * w.size(), s));
    ECK(cudaMemcpyAsync(d_w, w.data(), sizeof(double) * w.size(), cudaMemcpyHostToDevice, s));
    int rc = launch_exact_emission(absorbed_a, n_a, d_w, mass, nullptr, ncell, emission, temperature, s, absorbed_b,
                                   absorbed_b ? n_b : 0, absorbed_b ? d_w + (size_t)SHARES * n_a : nullptr);
    cudaFreeAsync(d_w, s);
    ECK(cudaStreamSynchronize(s));
    return rc;
}

// ---------------------------------------------------------------------------
// ---------------------------------------------------------------------------
// Allocation-free exact emission.
//
// skirt_dust_emission allocates its per-call working table (the absorption
// share of every input wavelength for the three grain populations) with the
// stream-ordered allocator.  Some callers cannot allocate device memory at
// call time: a process whose framework allocator has already reserved the
// device memory it may use, or a loop with a fixed memory budget decided up
// front.  skirt_dust_emission_exact_static does the same exact solve with that
// table in the fixed array below instead (8 x 4096 doubles = 256 KiB, held by
// every device that loads the library until the process exits).
// ---------------------------------------------------------------------------
namespace {

constexpr int STATIC_MAX_NIN = 4096;
static __device__ __align__(256) double g_static_shares[SHARES * STATIC_MAX_NIN];

std::mutex g_static_mutex;
double* g_static_ptr[64] = {};  // device address of g_static_shares, per device ordinal
double g_static_host[SHARES * STATIC_MAX_NIN];  // host copy of the table (guarded by g_static_mutex)

}  // namespace

extern "C" int skirt_dust_emission_exact_static(const double* absorbed, long long ncell, int n_in,
                                                const double* lambda_in, const float* mass, double* emission,
                                                float* temperature, void* stream)
{
    if (ncell < 0) return set_error(SKIRT_ERR_INVALID_ARG, "ncell < 0");
    if (n_in > STATIC_MAX_NIN)
        return set_error(SKIRT_ERR_INVALID_ARG, "n_in = %d exceeds the static table's maximum of %d wavelengths",
                         n_in, STATIC_MAX_NIN);
    if (int r = check_lambda(lambda_in, n_in)) return r;
    if (ncell == 0) return SKIRT_OK;
    if (ncell >= (1ll << 32)) return set_error(SKIRT_ERR_INVALID_ARG, "ncell must be < 2^32");
    if (!is_device(absorbed) || !is_device(mass) || !is_device(emission) || (temperature && !is_device(temperature)))
        return set_error(SKIRT_ERR_INVALID_ARG, "absorbed / mass / emission / temperature must be device memory");
    int dev = 0;
    ECK(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return set_error(SKIRT_ERR_NO_DEVICE, "device ordinal %d out of range", dev);
    cudaStream_t s = (cudaStream_t)stream;
    double* shares = nullptr;
    {
        std::lock_guard<std::mutex> lock(g_static_mutex);
        // once per device, with that device current: the device address of the array
        if (!g_static_ptr[dev]) {
            void* p = nullptr;
            cudaError_t e = cudaGetSymbolAddress(&p, g_static_shares);
            if (e != cudaSuccess || !p)
                return set_error(SKIRT_ERR_CUDA, "cudaGetSymbolAddress: %s", cudaGetErrorString(e));
            g_static_ptr[dev] = (double*)p;
        }
        shares = g_static_ptr[dev];
        // the table is rewritten in full by every call (no part needs zeroing).  The copy
        // reads the shared host buffer, so it has to finish before another thread may
        // refill that buffer: the stream is synchronised before the lock is released
        // (CUDA does not promise that an asynchronous copy from pageable memory has
        // read its source when the call returns).
        fill_shares(lambda_in, n_in, g_static_host);
        ECK(cudaMemcpyAsync(shares, g_static_host, sizeof(double) * SHARES * n_in, cudaMemcpyHostToDevice, s));
        ECK(cudaStreamSynchronize(s));
    }
    int rc = launch_exact_emission(absorbed, n_in, shares, mass, nullptr, ncell, emission, temperature, s);
    ECK(cudaStreamSynchronize(s));
    return rc;
}
