// Device helpers shared by the FP64 and the mixed-precision trace kernels.
#pragma once

#include <cuda_runtime.h>
#include <math.h>

#include "skirt_internal.cuh"

namespace skirt {

enum { M_NONE = 0, M_DEPOSIT = 1, M_LOCATE = 2, M_PEEL = 3 };
enum {
    ST_NEW = 0,
    ST_START_DEP,
    ST_DEPOSIT_DONE,
    ST_LOCATE_DONE,
    ST_PEEL_DONE,
    ST_PEEL,  // start the peel-off towards the current instrument
    ST_AFTER_SCATTER,
    ST_END_PACKET,
};

// Henyey-Greenstein phase function, normalised to average 1 over the sphere.
template <typename R>
__device__ __forceinline__ R hg_phase(R g, R mu)
{
    const R den = (R)1 + g * g - (R)2 * g * mu;
    return ((R)1 - g * g) / (den * sqrt(den));
}

// Scattering-angle cosine by inversion of the HG cumulative distribution.
template <typename R>
__device__ __forceinline__ R hg_mu(R g, R u)
{
    if (fabs(g) < (R)1e-6) return (R)2 * u - (R)1;
    const R t = ((R)1 - g * g) / ((R)1 - g + (R)2 * g * u);
    const R mu = ((R)1 + g * g - t * t) / ((R)2 * g);
    return fmin(fmax(mu, (R)-1), (R)1);
}

// Direction at polar cosine mu and azimuth (sin, cos) = (sp, cp) around k.
template <typename R>
__device__ __forceinline__ void hg_rotate(R& k0, R& k1, R& k2, R mu, R sp, R cp)
{
    const R st = sqrt(fmax((R)1 - mu * mu, (R)0));
    R n0, n1, n2;
    if (fabs(k2) > (R)0.99999) {
        n0 = st * cp;
        n1 = st * sp;
        n2 = (k2 > (R)0) ? mu : -mu;
    } else {
        const R s = sqrt((R)1 - k2 * k2);
        n0 = st * (k0 * k2 * cp - k1 * sp) / s + k0 * mu;
        n1 = st * (k1 * k2 * cp + k0 * sp) / s + k1 * mu;
        n2 = -st * cp * s + k2 * mu;
    }
    k0 = n0;
    k1 = n1;
    k2 = n2;
}

// The dust-source cell of uniform number u (0 < u < 1) at wavelength lam: the
// first whose cumulative emission exceeds u times the total, found by bisecting
// the tiles' offsets and then the running sums of one tile.  All values are
// non-negative, so they compare as integers, off the FP64 pipe.
__device__ __forceinline__ long long dust_cell(const TraceArgs& A, int lam, double u)
{
    const double* off = A.cdf_off + (size_t)lam * (A.dust_tiles + 1);
    const double target = u * __ldg(off + A.dust_tiles);
    long long key = __double_as_longlong(target);
    long long a = 0, b = A.dust_tiles - 1;  // first tile that ends beyond the target
    while (a < b) {
        const long long mid = (a + b) >> 1;
        if (__double_as_longlong(__ldg(off + mid + 1)) > key) b = mid; else a = mid + 1;
    }
    const long long m0 = a * DUST_TILE;
    const double* row = A.cdf + (size_t)lam * A.ncell + m0;
    int lo = 0, hi = (int)(A.ncell - m0 < DUST_TILE ? A.ncell - m0 : DUST_TILE) - 1;
    key = __double_as_longlong(target - __ldg(off + a));
    // where rounding leaves nothing of the tile beyond the rest, its last emitting cell
    const long long last = __double_as_longlong(__ldg(row + hi));
    if (last <= key) key = last - 1;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (__double_as_longlong(__ldg(row + mid)) > key) hi = mid; else lo = mid + 1;
    }
    return m0 + lo;
}

// Cell index along one axis: floor((x - lo) / d) clamped to [0, n-1].
template <typename R>
__device__ __forceinline__ int cell_index(R x, R lo, R d, int n)
{
    const R f = floor((x - lo) / d);
    if (f < (R)0) return 0;
    if (f > (R)(n - 1)) return n - 1;
    return (int)f;
}

}  // namespace skirt
