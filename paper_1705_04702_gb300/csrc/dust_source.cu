// Dust-cell source (dust emission phase, Sect. 3.2): a packet at wavelength
// j starts in cell m with probability emission[m][j] / sum_m emission[m][j].
// This file builds, per wavelength, the cumulative distribution over the cells
// that the packets search (trace_device.cuh): the [cell][wavelength] emission
// table is transposed into [wavelength][cell] rows (the single-device
// counterpart of switching the table from row to column representation,
// Sect. 5.2) that hold the running sums within tiles of DUST_TILE cells, and a
// scan of the tiles' sums gives each tile's offset.  One pass over the table,
// one FP64 addition per entry, nothing normalised: a packet scales its uniform
// number by the wavelength's total instead.
//
// What bounds the pass is the table's traffic (3.4 GB at 128^3 cells and 100
// wavelengths, 0.5 ms) next to that addition (0.4 ms of the FP64 pipe, which
// adds 5e11 numbers a second); the former transpose, tile sums and full scan
// with normalisation (five FP64 operations per entry, four passes) took 4.2 ms
// there.
#include <cuda_runtime.h>

#include <cstring>
#include <vector>

#include "skirt_internal.cuh"

namespace skirt {
namespace {

constexpr int SCAN_T = 256;            // threads per scan block (8 tiles each)
constexpr int TILE = 8 * SCAN_T;       // tiles per scan step
constexpr int PW = 4;                  // warps per block of the prefix kernel

// One warp per tile of DUST_TILE cells and 32 wavelengths: lane = wavelength,
// the running sum goes through the cells in order, 32 of them at a time, and
// leaves transposed through shared memory (coalesced on both sides).  The
// table's values are checked on the integer pipe.  ROWS = false: the tiles'
// sums only.
template <bool ROWS>
__global__ void __launch_bounds__(32 * PW, 5) tile_prefix_kernel(const double* __restrict__ em, double* __restrict__ rows,
                                                              double* __restrict__ tsum, long long ncell, int nl,
                                                              long long ntiles, unsigned int* bad)
{
    __shared__ double sh[ROWS ? PW : 1][32][33];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    double (*s)[33] = sh[ROWS ? w : 0];
    const int j0 = blockIdx.y * 32, j = j0 + lane;
    const int nj = nl - j0 < 32 ? nl - j0 : 32;
    for (long long t = (long long)blockIdx.x * PW + w; t < ntiles; t += (long long)gridDim.x * PW) {
        double sum = 0.0;
        const long long end = (t + 1) * DUST_TILE < ncell ? (t + 1) * DUST_TILE : ncell;
        for (long long m0 = t * DUST_TILE; m0 < end; m0 += 32) {
            const int nr = end - m0 < 32 ? (int)(end - m0) : 32;
            const double* src = em + m0 * nl + j;
#pragma unroll
            for (int h = 0; h < 32; h += 16) {
                double v[16];
#pragma unroll
                for (int r = 0; r < 16; ++r)
                    v[r] = (h + r < nr && lane < nj) ? __ldcs(src + (size_t)(h + r) * nl) : 0.0;
#pragma unroll
                for (int r = 0; r < 16; ++r) {
                    if ((unsigned)__double2hiint(v[r]) >= 0x7FF00000u) {  // negative, infinite or NaN (or -0)
                        if (v[r] != 0.0) atomicOr(bad, 1u);
                        v[r] = 0.0;
                    }
                    sum += v[r];
                    if (ROWS) s[h + r][lane] = sum;
                }
            }
            if (ROWS) {
                __syncwarp();
                if (lane < nr) {
                    double* dst = rows + (size_t)j0 * ncell + m0 + lane;
#pragma unroll 8
                    for (int k = 0; k < nj; ++k) dst[(size_t)k * ncell] = s[lane][k];
                }
                __syncwarp();
            }
        }
        if (lane < nj) tsum[(size_t)j * ntiles + t] = sum;
    }
}

// inclusive scan of the 8*SCAN_T values held 8 per thread; returns the block total
__device__ double block_scan8(double v[8], double* sh)
{
#pragma unroll
    for (int i = 1; i < 8; ++i) v[i] += v[i - 1];
    double x = v[7];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        double y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) sh[w] = x;
    __syncthreads();
    if (w == 0) {
        double s = lane < SCAN_T / 32 ? sh[lane] : 0.0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            double y = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += y;
        }
        if (lane < SCAN_T / 32) sh[lane] = s;
    }
    __syncthreads();
    const double before = (w > 0 ? sh[w - 1] : 0.0) + (x - v[7]);
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] += before;
    const double total = sh[SCAN_T / 32 - 1];
    __syncthreads();
    return total;
}

// offsets off[j][0 .. ntiles] of one wavelength's tiles from their sums (one
// block per wavelength); off[j][ntiles] is the wavelength's total
__global__ void __launch_bounds__(SCAN_T) tile_offset_kernel(const double* __restrict__ tsum, double* __restrict__ off,
                                                             double* __restrict__ totals, long long ntiles)
{
    __shared__ double sh[SCAN_T / 32];
    const int j = blockIdx.x;
    const double* ts = tsum + (size_t)j * ntiles;
    double* o = off ? off + (size_t)j * (ntiles + 1) : nullptr;
    double carry = 0.0;
    if (o && threadIdx.x == 0) o[0] = 0.0;
    for (long long base = 0; base < ntiles; base += TILE) {
        double v[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const long long k = base + threadIdx.x * 8 + i;
            v[i] = k < ntiles ? ts[k] : 0.0;
        }
        const double total = block_scan8(v, sh);
        if (o) {
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const long long k = base + threadIdx.x * 8 + i;
                if (k < ntiles) o[k + 1] = carry + v[i];
            }
        }
        carry += total;
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        totals[j] = carry;
        if (o) o[ntiles] = carry;
    }
}

}  // namespace

int build_dust_cdf(skirt_grid_s* g, const double* emission, int nl, const uint64_t* npk, cudaStream_t s,
                   std::vector<double>* totals_out, bool rows_wanted)
{
    const long long ncell = g->ncell;
    const long long ntiles = (ncell + DUST_TILE - 1) / DUST_TILE;
    cudaError_t e;
    if (rows_wanted && (e = g->cdf.ensure(sizeof(double) * (size_t)nl * ncell)) != cudaSuccess)
        return set_error(SKIRT_ERR_OOM, "dust cdf: %s", cudaGetErrorString(e));
    const size_t aux = sizeof(double) * ((size_t)nl * (2 * ntiles + 1) + nl) + 256;
    if ((e = g->cdf_aux.ensure(aux)) != cudaSuccess) return set_error(SKIRT_ERR_OOM, "dust cdf aux: %s", cudaGetErrorString(e));
    double* off = (double*)g->cdf_aux.p;
    double* totals = off + (size_t)nl * (ntiles + 1);
    unsigned int* bad = (unsigned int*)(totals + nl);
    double* tsum = totals + nl + 1;
    if ((e = cudaMemsetAsync(bad, 0, sizeof(unsigned int), s)) != cudaSuccess)
        return set_error(SKIRT_ERR_CUDA, "memset: %s", cudaGetErrorString(e));
    const long long nb = (ntiles + PW - 1) / PW;
    const dim3 grid((unsigned)(nb < (1 << 20) ? nb : (1 << 20)), (unsigned)((nl + 31) / 32));
    if (rows_wanted)
        tile_prefix_kernel<true><<<grid, 32 * PW, 0, s>>>(emission, (double*)g->cdf.p, tsum, ncell, nl, ntiles, bad);
    else
        tile_prefix_kernel<false><<<grid, 32 * PW, 0, s>>>(emission, nullptr, tsum, ncell, nl, ntiles, bad);
    tile_offset_kernel<<<nl, SCAN_T, 0, s>>>(tsum, rows_wanted ? off : nullptr, totals, ntiles);
    if ((e = cudaGetLastError()) != cudaSuccess) return set_error(SKIRT_ERR_CUDA, "dust cdf kernels: %s", cudaGetErrorString(e));
    std::vector<double> h(nl + 1);
    if ((e = cudaMemcpyAsync(h.data(), totals, sizeof(double) * nl + sizeof(unsigned int), cudaMemcpyDeviceToHost, s)) !=
            cudaSuccess ||
        (e = cudaStreamSynchronize(s)) != cudaSuccess)
        return set_error(SKIRT_ERR_CUDA, "dust cdf totals: %s", cudaGetErrorString(e));
    unsigned int badv = 0;
    memcpy(&badv, h.data() + nl, sizeof badv);
    if (badv) return set_error(SKIRT_ERR_INVALID_ARG, "dust emission holds negative or non-finite values");
    for (int j = 0; j < nl; ++j)
        if (npk[j] > 0 && !(h[j] > 0.0 && isfinite(h[j])))
            return set_error(SKIRT_ERR_INVALID_ARG, "dust emission at wavelength %d is zero but has packets", j);
    if (totals_out) totals_out->assign(h.begin(), h.begin() + nl);
    return SKIRT_OK;
}

}  // namespace skirt
