// Photon-packet life cycle on the GPU, mixed form: FP32 cell traversal,
// directions, phase-function sampling and packet luminosity; FP64 cumulative
// optical depth, tallies and energy ledger.
//
// Same method as the FP64 form (Sect. 3.2 stellar emission phase: launch,
// peel-off towards every instrument, continuous absorption into the
// [cell, wavelength] table, forced scattering, life until a negligible
// luminosity is left; Sect. 1 for the techniques; Sect. 5.2 for the table
// layout and lock-free additions), organised for a GPU whose FP64 unit
// retires a warp instruction only every few dozen cycles per sub-partition:
// every FP64 or FP32<->FP64 conversion instruction a warp issues, even with
// one lane active, costs that much.  So:
//
//  * Warp-coherent stepping.  All lanes of a warp step one cell per round
//    whatever traversal they are in (deposit, forced-interaction search,
//    peel-off line of sight).  A lane whose traversal ended idles until fewer
//    than step_min lanes are still stepping; then the idle lanes handle
//    their events (launch, scattering, peel-off tally) together.
//  * Per cell crossing only FP32 arithmetic.  The optical depth of every
//    crossing is FP32 and the running optical depth is their error-free
//    double-float sum (Knuth two-sum: hi + lo, ~46-bit significand, exact
//    up to its final rounding); at every event it is formed as an FP64
//    value.  The sum depends only on the packet, never on the schedule.
//    Deposits are formed in FP32 and widened to FP64 by integer bit
//    operations for the reduction.
//  * Positions are double-float pairs (hi + lo, ~48 bits).  Face planes come
//    from exact per-grid tables; the distance from a start point to its first
//    faces and the snapping of an interaction point onto the plane through
//    which its cell was entered keep full relative precision for points deep
//    inside optically thick cells (~1/(kappa rho) from a face).  The
//    interaction cell found by the search is carried into the next
//    traversals.
//  * Per event, escaped / absorbed / scattered come from one
//    om = 1 - e^{-tau_path}, so they add up to the packet luminosity.
//  * Per-thread state used only at events lives in shared memory.
//
// What bounds it is instruction issue (71% of the cycles on the 256^3 disk),
// so the crossing is written for few warp instructions: the exit axis's next
// face is advanced under predicates from FP32 face indices, leaving the grid
// is tested by one distance comparison, the cell index moves by a signed
// stride, and no branch separates the traversal kinds.  The lanes handle
// events in one pass over the stages with a single copy of the traversal
// set-up and one random block per scattering, which also keeps the loop inside
// the instruction cache; the search for the interaction starts from the saved
// start of the deposit traversal it repeats.  Against selecting every operand
// by axis and setting traversals up inside each stage: 1e7 packets on the
// 256^3 disk 172 ms (259), 8e6 packets of 200 wavelengths on the 128^3 torus
// 117 ms (200), 3e6 packets on an octree of 8.3e5 leaves 58 ms (94; 40 with
// step_oct's later changes), the same
// histories bit for bit.  A crossing is now ~99 warp instructions for the
// lanes of a warp (27 of them the deposit's); events take a fifth of the
// instructions, run by 4 to 5 lanes at a time.
#include <cuda_runtime.h>
#include <math.h>

#include <type_traits>

#include "skirt_internal.cuh"
#include "trace_device.cuh"
#include "work_count.cuh"

namespace skirt {
namespace {

constexpr int MAXB = 256;       // threads per block of the mixed kernel (upper bound)
constexpr int ROUND = 8;        // cell crossings per stepping round between warp votes

// FP32 -> FP64 by IEEE-754 field manipulation on the integer pipe: exact for
// normal floats; zero and FP32 subnormals map to zero.
__device__ __forceinline__ double f2d(float f)
{
    const unsigned u = __float_as_uint(f);
    const unsigned ex = (u >> 23) & 0xFFu;
    const unsigned long long bits = ((unsigned long long)(u >> 31) << 63) |
                                    ((unsigned long long)(ex + 896u) << 52) |
                                    ((unsigned long long)(u & 0x7FFFFFu) << 29);
    return ex ? __longlong_as_double((long long)bits) : 0.0;
}

// FP32 -> FP64 for a positive normal float: the double's high word is the
// float's bits shifted right by 3 with the exponent re-biased by 1023 - 127,
// its low word the three mantissa bits shifted out.
__device__ __forceinline__ double f2d_pos(float f)
{
    const unsigned u = __float_as_uint(f);
    return __hiloint2double((int)((u >> 3) + 0x38000000u), (int)(u << 29));
}

// e^{-x} for x >= 0 as 2^{-x log2 e} with the PTX base-2 exponential
// (ex2.approx, relative error ~2^-22); the FP32 product x log2 e contributes
// an error of the same order as the FP32 rounding of x itself.  Results below
// the FP32 normal range flush to zero.
__device__ __forceinline__ float exp_neg(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(-1.4426950408889634f * x));
    return y;
}

// 1 - e^{-x} for x >= 0, accurate in relative terms: below 1/4 the Taylor
// series x (1 - x g(x)) with g(x) = 1/2! - x/3! + x^2/4! - ... - x^5/7!
// (Horner form with constant coefficients: six multiply-adds), whose first
// omitted term is below 4e-10 of the result; 1 - e^{-x} above, where no
// cancellation occurs.  Both branches are evaluated and selected.
__device__ __forceinline__ float one_minus_exp_neg(float x)
{
    const float g = fmaf(fmaf(fmaf(fmaf(fmaf(-1.f / 5040.f, x, 1.f / 720.f), x, -1.f / 120.f), x, 1.f / 24.f), x,
                         -1.f / 6.f), x, 0.5f);
    const float p = x * fmaf(g, -x, 1.f);
    const float q = 1.f - exp_neg(x);
    return x < 0.25f ? p : q;
}

// (hi, lo) += v, error-free: hi takes the rounded sum, lo collects the exact
// rounding errors (two-sum).
__device__ __forceinline__ void df_accumulate(float& hi, float& lo, float v)
{
    const float s = __fadd_rn(hi, v);
    const float bb = __fsub_rn(s, hi);
    const float e = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)), __fsub_rn(v, bb));
    hi = s;
    lo = __fadd_rn(lo, e);
}

// Double-float arithmetic (Knuth / Dekker error-free transformations), with
// round-to-nearest intrinsics so that nothing is contracted into an FMA.
__device__ __forceinline__ void df_add_prod(float& hi, float& lo, float a, float b)
{
    const float p = __fmul_rn(a, b);
    const float pe = fmaf(a, b, -p);
    const float s = __fadd_rn(hi, p);
    const float bb = __fsub_rn(s, hi);
    const float e = __fadd_rn(__fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)), __fsub_rn(p, bb)), __fadd_rn(lo, pe));
    hi = __fadd_rn(s, e);
    lo = __fsub_rn(e, __fsub_rn(hi, s));
}

__device__ __forceinline__ float df_diff(float2 f, float xh, float xl)
{
    return __fadd_rn(__fsub_rn(f.x, xh), __fsub_rn(f.y, xl));
}

// Integers 0 <= i < 2^23 and FP32 by the 2^23 offset: i + 2^23 has i in its
// low 23 bits.  Logical and FP32 instructions, where a conversion instruction
// would occupy a slow pipe (measured on the octree kernel, whose crossings
// held three float-to-int conversions: FP64/conversion pipe 64% active).
constexpr float TWO23 = 8388608.f;
constexpr int TWO23_BITS = 0x4B000000;
// floor(f) + 2^23 for 0 <= f < 2^23, as bits
__device__ __forceinline__ int floor_bits(float f) { return __float_as_int(__fadd_rd(f, TWO23)); }
__device__ __forceinline__ int floor_small(float f) { return floor_bits(f) & 0x7FFFFF; }

// Distance along the ray to face plane k (FP32 index) of one axis.
__device__ __forceinline__ float face_t(float k, float d, float lo, float x, float iv)
{
    return __fmul_rn(__fsub_rn(__fmaf_rn(k, d, lo), x), iv);
}

// Per-thread state used only at events, struct of arrays in shared memory.
struct Cold {
    double l_emit[MAXB], l_abs[MAXB], l_esc[MAXB], l_res[MAXB];
    unsigned long long q[MAXB];
    unsigned left[MAXB];                                        // packets left of the last queue refill
    unsigned c_dep[MAXB], c_loc[MAXB], c_peel[MAXB], c_scat[MAXB];  // emptied into the 64-bit counters
    float L0[MAXB], p_esc[MAXB], p_abs[MAXB], p_res[MAXB], p_peel[MAXB], om[MAXB], peel_w[MAXB], alb[MAXB];
    float xl0[MAXB], xl1[MAXB], xl2[MAXB];  // low words of the double-float position
    int lam[MAXB], nscat[MAXB], peel_i[MAXB];  // peel_i: instrument, + PEEL_SCATTER after a scattering
    unsigned pk[MAXB], ev[MAXB];
    unsigned ry[MAXB], rz[MAXB];            // the event's second and third random words
    // the deposit traversal's start, from which the search along the same ray
    // starts again: distances to the first faces, face indices (octree: lattice
    // corner), cell (node)
    float b_t0[MAXB], b_t1[MAXB], b_t2[MAXB];
    int b_k0[MAXB], b_k1[MAXB], b_k2[MAXB], b_m[MAXB];
    float b_kr[MAXB];
    // the search's interaction cell (octree: node; -1 before it is found), the
    // distance at which it was entered, the length inside it, how it was entered
    int f_m[MAXB], f_last[MAXB];
    float f_t[MAXB], f_s[MAXB];
};
constexpr int PEEL_SCATTER = 16;  // at most 16 instruments

__host__ __device__ constexpr size_t align16(size_t x) { return (x + 15) & ~(size_t)15; }

// An octree node's 32 bytes, fetched by one load: the children or the leaf, its
// density, and the nodes across its six faces.
struct OctRec {
    int ref;
    float kr;
    int nb[6];
};
__device__ __forceinline__ OctRec oct_load(const OctNode* p)
{
    OctRec r;
    int k;
    asm("ld.global.nc.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=r"(r.ref), "=r"(k), "=r"(r.nb[0]), "=r"(r.nb[1]), "=r"(r.nb[2]), "=r"(r.nb[3]), "=r"(r.nb[4]),
          "=r"(r.nb[5])
        : "l"(p));
    r.kr = __int_as_float(k);
    return r;
}

// Grid kinds.  G_CART: Cartesian, face indices held as FP32 integers (every
// dimension below 2^23, so that they stay exact); G_CART_BIG: Cartesian with a
// longer axis, face indices as integers; G_OCT: octree (Sect. 7.9), where the
// traversal state names a leaf (node, level, lattice corner) instead of a cell
// and a crossing reads the face neighbour and descends from it by the lattice
// cell of the entry point.
enum { G_CART = 0, G_CART_BIG = 1, G_OCT = 2 };

//
// LONG: the work counters are emptied at every event.  Only a run whose packets may
// make more than 2^32 crossings each needs it (counts_within_packet): in the other
// kernels that check, a few instructions per event, cost 2% of the disk and torus
// runs.
template <int G, bool LONG>
__global__ void __launch_bounds__(MAXB, 3) trace_mixed_kernel(const TraceArgs A)
{
    constexpr bool OCT = G == G_OCT, BIG = G == G_CART_BIG;
    extern __shared__ __align__(16) unsigned char smem[];
    InstrDev* sins = reinterpret_cast<InstrDev*>(smem);
    Cold& C = *reinterpret_cast<Cold*>(smem + align16(sizeof(InstrDev) * A.ninstr));
    for (int i = threadIdx.x; i < A.ninstr; i += blockDim.x) sins[i] = A.ins[i];
    const int t = threadIdx.x;
    C.l_emit[t] = C.l_abs[t] = C.l_esc[t] = C.l_res[t] = 0.0;
    C.q[t] = 0;
    C.left[t] = 0;
    C.c_dep[t] = C.c_loc[t] = C.c_peel[t] = C.c_scat[t] = 0;
    C.lam[t] = -1;
    __syncthreads();

    const float INF = __int_as_float(0x7f800000);
    const float* __restrict__ kr = A.kr32;
    const int step_min = A.step_min;

    // ---- stepping state (registers)
    int mode = M_NONE;
    // Cartesian: per axis the index of the next face (kf), its step (sf: +1, -1
    // or 0) and the cell-index stride of a crossing (st); octree: the leaf's
    // lattice corner (c, an integer in FP32) and minus the step (s)
    using KF = typename std::conditional<BIG, int, float>::type;
    KF kf0 = 0, kf1 = 0, kf2 = 0, sf0 = 0, sf1 = 0, sf2 = 0;
    int st0 = 0, st1 = 0, st2 = 0;
    float c0 = 0.f, c1 = 0.f, c2 = 0.f;
    int s0 = 0, s1 = 0, s2 = 0;
    float iv0 = 0.f, iv1 = 0.f, iv2 = 0.f, tn0 = 0.f, tn1 = 0.f, tn2 = 0.f, tcur = 0.f;
    float t_end = 0.f;               // Cartesian: no crossing before this distance leaves the grid
    float tau_h = 0.f, tau_l = 0.f;  // running optical depth of the traversal (double-float)
    float par = 0.f;                 // deposit: L (1 - albedo); search: interaction optical depth
    unsigned nsteps = 0;
    float last_dusty_end = 0.f;  // search: where the last dusty cell crossed ended
    int last = 0;        // search: how the current cell was entered (0: the start cell); Cartesian: the
                         // stride of the crossing, octree: 1 + the face's axis
    int cur_m = 0;       // index of the current cell
    float kr_cur = 0.f;  // its extinction coefficient (loaded one crossing ahead)
    double* dep_base = nullptr;  // the absorbed table at (cell 0, the packet's wavelength)
    // octree: the current leaf's node and level, the traversal direction, the
    // node of the interaction leaf
    const int OL = A.oct_levels;
    const OctNode* __restrict__ nodes = A.oct_nodes;
    bool started = false;  // per-wavelength schedule: this thread's packet is taken
    int onode = 0, olev = 0, pc_node = 0;
    // octree: the distance at which the ray leaves the current leaf, the axis of
    // that face, the node across it, and the way from the leaf's corner to the
    // entry point's lattice cell along that axis
    float oex = 0.f, odel = 0.f;
    int oax = 0, onb = 0;
    float v0 = 0.f, v1 = 0.f, v2 = 0.f;
    // ---- packet state (registers)
    int stage = ST_NEW;
    bool alive = true;
    int lam = 0;
    float krs = 0.f, gg = 0.f, L = 0.f;
    float x0 = 0.f, x1 = 0.f, x2 = 0.f;  // position, high words
    float k0 = 0.f, k1 = 0.f, k2 = 0.f;
    bool have_pc = false;
    int pc0 = 0, pc1 = 0, pc2 = 0;

    auto axis_cell = [&](float xh, float xl, float lo, float d, int n, const float2* f) {
        int c = (int)fminf(fmaxf(floorf((xh - lo) / d), 0.f), (float)(n - 1));
        if (c > 0 && df_diff(__ldg(f + c), xh, xl) > 0.f) --c;
        else if (c < n - 1 && df_diff(__ldg(f + c + 1), xh, xl) <= 0.f) ++c;
        return c;
    };

    // octree: enter the leaf holding the lattice cell (j0, j1, j2) (given as
    // 2^23 + j in FP32 bits), descending from `node` (a leaf, or a node of level
    // `lev`), whose record is q; q becomes the leaf's
    auto oct_enter = [&](OctRec& q, int node, int lev, int j0, int j1, int j2) {
        while (q.ref >= 0 && lev < OL) {
            ++lev;
            const int b = OL - lev;
            node = q.ref + (((j0 >> b) & 1) | (((j1 >> b) & 1) << 1) | (((j2 >> b) & 1) << 2));
            q = oct_load(nodes + node);
        }
        onode = node;
        olev = oct_leaf_level(q.ref);
        cur_m = oct_leaf_index(q.ref);
        kr_cur = q.kr;
        const int mask = (int)(~0u << (OL - olev));
        c0 = __int_as_float(j0 & mask) - TWO23;
        c1 = __int_as_float(j1 & mask) - TWO23;
        c2 = __int_as_float(j2 & mask) - TWO23;
    };

    // octree: where the ray leaves the current leaf, from its face distances and
    // its record (inside its parent, the node across a face is the sibling)
    auto oct_exit = [&](const OctRec& q) {
        oex = fminf(fminf(tn0, tn1), tn2);
        oax = (tn0 == oex) ? 0 : ((tn1 == oex) ? 1 : 2);
        const int ss = oax == 0 ? s0 : (oax == 1 ? s1 : s2);
        const int lo = oax == 0 ? q.nb[0] : (oax == 1 ? q.nb[2] : q.nb[4]);
        const int hi = oax == 0 ? q.nb[1] : (oax == 1 ? q.nb[3] : q.nb[5]);
        onb = ss < 0 ? hi : lo;
        odel = ss < 0 ? __int_as_float((127 + OL - olev) << 23) : -1.f;
    };

    // starts a traversal of kind m along (vx, vy, vz), whose reciprocals (zero
    // for zero components) are (i0, i1, i2), from the packet's position
    auto begin = [&](int m, float vx, float vy, float vz, float i0, float i1, float i2) {
        mode = m;
        const float2* __restrict__ fx = A.faces;
        const float2* __restrict__ fy = fx + (A.nx + 1);
        const float2* __restrict__ fz = fy + (A.ny + 1);
        const float l0 = C.xl0[t], l1 = C.xl1[t], l2 = C.xl2[t];
        if (!have_pc) {
            pc0 = axis_cell(x0, l0, A.lo_f[0], A.d_f[0], A.nx, fx);
            pc1 = axis_cell(x1, l1, A.lo_f[1], A.d_f[1], A.ny, fy);
            pc2 = axis_cell(x2, l2, A.lo_f[2], A.d_f[2], A.nz, fz);
            pc_node = 0;
            have_pc = true;
        }
        OctRec q;
        if constexpr (OCT) {
            q = oct_load(nodes + pc_node);
            oct_enter(q, pc_node, 0, TWO23_BITS | pc0, TWO23_BITS | pc1, TWO23_BITS | pc2);
            pc0 = floor_small(c0); pc1 = floor_small(c1); pc2 = floor_small(c2);
            pc_node = onode;
            v0 = vx; v1 = vy; v2 = vz;
        }
        const int g0 = vx > 0.f ? 1 : (vx < 0.f ? -1 : 0);
        const int g1 = vy > 0.f ? 1 : (vy < 0.f ? -1 : 0);
        const int g2 = vz > 0.f ? 1 : (vz < 0.f ? -1 : 0);
        iv0 = i0; iv1 = i1; iv2 = i2;
        // first faces from the exact face planes and the double-float position
        const int e = OCT ? 1 << (OL - olev) : 1;  // the cell's extent in lattice cells
        const int n0 = pc0 + (g0 > 0 ? e : 0), n1 = pc1 + (g1 > 0 ? e : 0), n2 = pc2 + (g2 > 0 ? e : 0);
        tn0 = g0 ? df_diff(__ldg(fx + n0), x0, l0) * iv0 : INF;
        tn1 = g1 ? df_diff(__ldg(fy + n1), x1, l1) * iv1 : INF;
        tn2 = g2 ? df_diff(__ldg(fz + n2), x2, l2) * iv2 : INF;
        tcur = 0.f;
        tau_h = tau_l = 0.f;
        nsteps = 0;
        if constexpr (OCT) {
            // minus the step: as a mask, all ones for a step up and zero or the low
            // bit (clear in a power of two) otherwise
            s0 = -g0; s1 = -g1; s2 = -g2;
            oct_exit(q);
        } else {
            kf0 = (KF)n0; kf1 = (KF)n1; kf2 = (KF)n2;
            sf0 = (KF)g0; sf1 = (KF)g1; sf2 = (KF)g2;
            st0 = g0 * A.cst[0];
            st1 = g1 * A.cst[1];
            st2 = g2 * A.cst[2];
            // the distance to each axis's last face by the crossing's own
            // formula: the crossing that leaves the grid lies at one of them
            const int m0 = g0 > 0 ? A.nx : 0, m1 = g1 > 0 ? A.ny : 0, m2 = g2 > 0 ? A.nz : 0;
            const float u0 = n0 == m0 ? tn0 : face_t((float)m0, A.d_f[0], A.lo_f[0], x0, iv0);
            const float u1 = n1 == m1 ? tn1 : face_t((float)m1, A.d_f[1], A.lo_f[1], x1, iv1);
            const float u2 = n2 == m2 ? tn2 : face_t((float)m2, A.d_f[2], A.lo_f[2], x2, iv2);
            t_end = fminf(g0 ? u0 : INF, fminf(g1 ? u1 : INF, g2 ? u2 : INF));
            cur_m = pc0 * A.cst[0] + pc1 * A.cst[1] + pc2 * A.cst[2];
            kr_cur = __ldg(kr + cur_m);
        }
    };

    // keeps the start of a deposit traversal for the search that follows it
    auto keep_start = [&]() {
        C.b_t0[t] = tn0; C.b_t1[t] = tn1; C.b_t2[t] = tn2;
        if constexpr (OCT) {
            C.b_k0[t] = __float_as_int(c0); C.b_k1[t] = __float_as_int(c1); C.b_k2[t] = __float_as_int(c2);
            C.b_m[t] = onode;
        } else {
            if constexpr (BIG) { C.b_k0[t] = kf0; C.b_k1[t] = kf1; C.b_k2[t] = kf2; }
            else { C.b_k0[t] = __float_as_int(kf0); C.b_k1[t] = __float_as_int(kf1); C.b_k2[t] = __float_as_int(kf2); }
            C.b_m[t] = cur_m;
            C.b_kr[t] = kr_cur;
        }
    };

    // starts the search: the same position and direction as the deposit
    // traversal just ended, so its direction state is still in place
    auto begin_search = [&]() {
        mode = M_LOCATE;
        tn0 = C.b_t0[t]; tn1 = C.b_t1[t]; tn2 = C.b_t2[t];
        if constexpr (OCT) {
            c0 = __int_as_float(C.b_k0[t]); c1 = __int_as_float(C.b_k1[t]); c2 = __int_as_float(C.b_k2[t]);
            onode = C.b_m[t];
            const OctRec q = oct_load(nodes + onode);
            olev = oct_leaf_level(q.ref);
            cur_m = oct_leaf_index(q.ref);
            kr_cur = q.kr;
            oct_exit(q);
        } else {
            if constexpr (BIG) { kf0 = C.b_k0[t]; kf1 = C.b_k1[t]; kf2 = C.b_k2[t]; }
            else { kf0 = __int_as_float(C.b_k0[t]); kf1 = __int_as_float(C.b_k1[t]); kf2 = __int_as_float(C.b_k2[t]); }
            cur_m = C.b_m[t];
            kr_cur = C.b_kr[t];
        }
        tcur = 0.f;
        tau_h = tau_l = 0.f;
        nsteps = 0;
        last = 0;
        last_dusty_end = 0.f;
        C.f_m[t] = -1;
    };

    // The work of one crossing in its cell, written without a branch per
    // traversal kind: a warp's lanes are nearly always in several kinds, so the
    // deposit's arithmetic is done by all of them and only its reduction is
    // predicated; only the end of a search, once per scattering, branches.  (In
    // the branched form the code after the branch ran once per kind.)
    auto cell_work = [&](int m, float tmin, float dtau, float krl) {
        const float tau_prev = tau_h + tau_l;
        const float dep = par * exp_neg(tau_prev) * one_minus_exp_neg(dtau);
        if (mode == M_DEPOSIT && dep >= 1.17549435e-38f)
            atomicAdd(reinterpret_cast<double*>(reinterpret_cast<char*>(dep_base) +
                                                (size_t)(unsigned)m * A.abs_cs8),
                      f2d_pos(dep));
        if (mode == M_LOCATE && krl > 0.f && tau_h + (tau_l + dtau) >= par) {
            C.f_m[t] = OCT ? onode : m;
            C.f_t[t] = tcur;
            C.f_s[t] = (par - tau_prev) / krl;  // distance inside the cell
            C.f_last[t] = last;
            mode = M_NONE;
        }
        last_dusty_end = krl > 0.f ? tmin : last_dusty_end;
        df_accumulate(tau_h, tau_l, dtau);
    };

    // One leaf crossing of an octree traversal.  The node across the exit face
    // is loaded before the crossing's work, all 32 bytes at once: its six
    // neighbours arrive with its density, so the next crossing's node is known
    // as soon as its exit face is.  (Loading the neighbour's index by itself
    // costs a second dependent access: the L1 share holds fewer lines than the
    // SM's lanes keep in use.)  The lattice corner stays in FP32, where the
    // entry point's clamp and floor, the alignment to the leaf (a mask on the
    // bits of c + 2^23) and the next faces need no conversion; the exit axis's
    // own lattice coordinate is set under its predicate, not by a branch.
    // 3e6 packets, 8.3e5 leaves: 57.2 -> 40.1 ms; 1e7 packets, 8.2e6 leaves
    // (nodes 2.4 times the L2): 417 -> 330 ms, the same histories.
    auto step_oct = [&]() {
        const float tmin = oex;
        const int nb = onb;
        const bool out = nb < 0;
        OctRec q = oct_load(nodes + max(nb, 0));
        const float ds = fmaxf(tmin - tcur, 0.f);
        const int m = cur_m;
        const float krl = kr_cur * krs;
        const float dtau = krl * ds;
        ++nsteps;
        cell_work(m, tmin, dtau, krl);
        const bool over = nsteps > (unsigned)A.oct_step_cap;
        if (mode != M_NONE) {
            if (out || over || tau_h > A.tau_cut) {
                if (!out && over) atomicOr(A.err, (unsigned)ERRBIT_PATH);
                mode = M_NONE;
            } else {
                tcur = tmin;
                last = oax + 1;
                // lattice cell of the entry point: across the exit face along its
                // axis, elsewhere the crossing point's cell kept within the current
                // leaf's cross-section
                const float em = __int_as_float((127 + OL - olev) << 23) - 1.f;  // the leaf's extent - 1
                const float p0 = (x0 + tmin * v0 - A.lo_f[0]) * A.id_f[0];
                const float p1 = (x1 + tmin * v1 - A.lo_f[1]) * A.id_f[1];
                const float p2 = (x2 + tmin * v2 - A.lo_f[2]) * A.id_f[2];
                float f0 = fminf(fmaxf(p0, c0), c0 + em);
                float f1 = fminf(fmaxf(p1, c1), c1 + em);
                float f2 = fminf(fmaxf(p2, c2), c2 + em);
                asm("{\n\t"
                    ".reg .pred p0, p1, p2;\n\t"
                    "setp.eq.s32 p0, %3, 0;\n\t"
                    "setp.eq.s32 p1, %3, 1;\n\t"
                    "setp.eq.s32 p2, %3, 2;\n\t"
                    "@p0 add.rn.f32 %0, %4, %7;\n\t"
                    "@p1 add.rn.f32 %1, %5, %7;\n\t"
                    "@p2 add.rn.f32 %2, %6, %7;\n\t"
                    "}"
                    : "+f"(f0), "+f"(f1), "+f"(f2)
                    : "r"(oax), "f"(c0), "f"(c1), "f"(c2), "f"(odel));
                // a neighbour that is not a leaf has the current level
                oct_enter(q, nb, olev, floor_bits(f0), floor_bits(f1), floor_bits(f2));
                const int en = (127 + OL - olev) << 23;  // the new leaf's extent: a power of two's bits
                tn0 = s0 ? face_t(c0 + __int_as_float(en & s0), A.d_f[0], A.lo_f[0], x0, iv0) : INF;
                tn1 = s1 ? face_t(c1 + __int_as_float(en & s1), A.d_f[1], A.lo_f[1], x1, iv1) : INF;
                tn2 = s2 ? face_t(c2 + __int_as_float(en & s2), A.d_f[2], A.lo_f[2], x2, iv2) : INF;
                oct_exit(q);
            }
        }
    };

    // one cell crossing of the current traversal (Cartesian)
    auto step = [&]() {
        // the exit axis (the first at the smallest distance), the next cell, and
        // the exit axis's next face.  Four instructions per axis under its
        // predicate take the place of selecting nine operands by axis.
        float tmin;
        int str;
        if constexpr (BIG) {
            tmin = fminf(tn0, fminf(tn1, tn2));
            if (tn0 == tmin) { str = st0; kf0 += sf0; tn0 = face_t((float)kf0, A.d_f[0], A.lo_f[0], x0, iv0); }
            else if (tn1 == tmin) { str = st1; kf1 += sf1; tn1 = face_t((float)kf1, A.d_f[1], A.lo_f[1], x1, iv1); }
            else { str = st2; kf2 += sf2; tn2 = face_t((float)kf2, A.d_f[2], A.lo_f[2], x2, iv2); }
        } else {
            asm("{\n\t"
                ".reg .pred p0, p1, p2;\n\t"
                "min.f32 %6, %1, %2;\n\t"
                "min.f32 %6, %0, %6;\n\t"
                "setp.eq.f32 p0, %0, %6;\n\t"
                "setp.eq.and.f32 p1, %1, %6, !p0;\n\t"
                "or.pred p2, p0, p1;\n\t"
                "selp.b32 %7, %24, %25, p1;\n\t"
                "selp.b32 %7, %23, %7, p0;\n\t"
                "@p0 add.rn.f32 %3, %3, %8;\n\t"
                "@p1 add.rn.f32 %4, %4, %9;\n\t"
                "@!p2 add.rn.f32 %5, %5, %10;\n\t"
                "@p0 fma.rn.f32 %0, %3, %11, %14;\n\t"
                "@p1 fma.rn.f32 %1, %4, %12, %15;\n\t"
                "@!p2 fma.rn.f32 %2, %5, %13, %16;\n\t"
                "@p0 sub.rn.f32 %0, %0, %17;\n\t"
                "@p1 sub.rn.f32 %1, %1, %18;\n\t"
                "@!p2 sub.rn.f32 %2, %2, %19;\n\t"
                "@p0 mul.rn.f32 %0, %0, %20;\n\t"
                "@p1 mul.rn.f32 %1, %1, %21;\n\t"
                "@!p2 mul.rn.f32 %2, %2, %22;\n\t"
                "}"
                : "+f"(tn0), "+f"(tn1), "+f"(tn2), "+f"(kf0), "+f"(kf1), "+f"(kf2), "=&f"(tmin), "=&r"(str)
                : "f"(sf0), "f"(sf1), "f"(sf2), "f"(A.d_f[0]), "f"(A.d_f[1]), "f"(A.d_f[2]), "f"(A.lo_f[0]),
                  "f"(A.lo_f[1]), "f"(A.lo_f[2]), "f"(x0), "f"(x1), "f"(x2), "f"(iv0), "f"(iv1), "f"(iv2), "r"(st0),
                  "r"(st1), "r"(st2));
        }
        // the next cell's density, requested before the current cell is
        // processed so that it arrives during this crossing's work
        const int mn = cur_m + str;
        const bool inside = tmin < t_end;
        float kr_next = 0.f;
        if (inside) kr_next = __ldg(kr + mn);
        const float ds = fmaxf(tmin - tcur, 0.f);
        const float krl = kr_cur * krs;
        const float dtau = krl * ds;
        ++nsteps;
        cell_work(cur_m, tmin, dtau, krl);
        last = str;
        tcur = tmin;
        cur_m = mn;
        kr_cur = kr_next;
        // Beyond tau = tau_cut (30) a line of sight transmits < e^-30 (1e-13) and a
        // deposit path has handed < e^-30 of the luminosity to its remaining
        // cells; 1 - e^-tau is 1 in FP32 from tau = 17 on, so the forced
        // scattering draw does not change: the traversal ends there (the search
        // never gets that far, since tau_int < 17 in FP32).
        if (!inside || tau_h > A.tau_cut) {
            // at the last face of an axis (its index has moved one beyond), a tie
            // with it, or a NaN
            const bool out = kf0 == (KF)(sf0 > 0 ? A.nx + 1 : -1) || kf1 == (KF)(sf1 > 0 ? A.ny + 1 : -1) ||
                             kf2 == (KF)(sf2 > 0 ? A.nz + 1 : -1);
            if (out || tau_h > A.tau_cut) mode = M_NONE;
            else kr_cur = __ldg(kr + mn);
        }
    };

    auto draw = [&](uint32_t event, uint32_t block) -> uint4 {
        return philox10(make_uint4(C.pk[t], (uint32_t)lam, event, (A.phase << 24) | block), A.key0, A.key1);
    };

    auto flush_ledger = [&]() {
        const int ll = C.lam[t];
        if (ll >= 0) {
            double* lg = A.ledger + 4 * (size_t)ll;
            atomicAdd(lg + 0, C.l_emit[t]);
            atomicAdd(lg + 1, C.l_abs[t]);
            atomicAdd(lg + 2, C.l_esc[t]);
            atomicAdd(lg + 3, C.l_res[t]);
        }
        C.l_emit[t] = C.l_abs[t] = C.l_esc[t] = C.l_res[t] = 0.0;
    };

    auto flush_counters = [&]() {
        atomicAdd(A.counters + 0, (unsigned long long)C.c_scat[t]);
        atomicAdd(A.counters + 1, (unsigned long long)C.c_dep[t]);
        atomicAdd(A.counters + 2, (unsigned long long)C.c_loc[t]);
        atomicAdd(A.counters + 3, (unsigned long long)C.c_peel[t]);
        C.c_dep[t] = C.c_loc[t] = C.c_peel[t] = C.c_scat[t] = 0;
    };

    // Event handling, from the end of a traversal to the start of the next, as
    // one pass over the stages in the order a packet meets them: the lanes of a
    // warp, whatever traversal they ended, share the code of the later stages
    // and one copy of the traversal set-up (the previous form set each
    // traversal up inside its own stage, five copies run by a few lanes each).
    // A lane goes round again only where no traversal came of a pass (a
    // peel-off of zero weight).
    auto events = [&]() {
        int need;
        do {
            need = M_NONE;
            if (stage == ST_PEEL_DONE) {
                if (count_add(C.c_peel[t], nsteps) && LONG) flush_counters();
                const int pk = C.peel_i[t], pi = pk & (PEEL_SCATTER - 1);
                const InstrDev& I = sins[pi];
                const float w = C.peel_w[t];
                if (w > 0.f) {
                    const float tobs = tau_h + tau_l;
                    const float flux = w * expf(-tobs) * I.flux_norm_f;
                    C.p_peel[t] += flux;
                    const float a = x0 * I.e1_f[0] + x1 * I.e1_f[1] + x2 * I.e1_f[2] +
                                    (C.xl0[t] * I.e1_f[0] + C.xl1[t] * I.e1_f[1] + C.xl2[t] * I.e1_f[2]);
                    const float b = x0 * I.e2_f[0] + x1 * I.e2_f[1] + x2 * I.e2_f[2] +
                                    (C.xl0[t] * I.e2_f[0] + C.xl1[t] * I.e2_f[1] + C.xl2[t] * I.e2_f[2]);
                    const float fa = (a + I.half_fov_f) * I.inv_dpx_f;
                    const float fb = (b + I.half_fov_f) * I.inv_dpx_f;
                    if (flux >= 1.17549435e-38f) {
                        // one FP64 reduction per peel-off (lanes of a warp rarely share a
                        // pixel; aggregating them measured no faster)
                        const float np = (float)I.npx;
                        if (fa >= 0.f && fa < np && fb >= 0.f && fb < np) {
                            const int pix = floor_small(fb) * I.npx + floor_small(fa);
                            atomicAdd(A.images + I.img_off + (long long)pix * A.nlambda + lam, f2d(flux));
                        } else {
                            atomicAdd(A.oof + (size_t)pi * A.nlambda + lam, f2d(flux));
                        }
                    }
                }
                C.peel_i[t] = pk + 1;
                stage = pi + 1 < A.ninstr ? ST_PEEL : (pk & PEEL_SCATTER ? ST_AFTER_SCATTER : ST_START_DEP);
            } else if (stage == ST_DEPOSIT_DONE) {
                if (count_add(C.c_dep[t], nsteps) && LONG) flush_counters();
                // om = 1 - e^{-tau_path}: from expm1 for small tau, from 1 - exp for
                // large tau, so that both om and 1 - om keep FP32 relative precision
                const float tf = tau_h + tau_l;
                float om, E;
                if (tf < 0.6931472f) { om = -expm1f(-tf); E = 1.f - om; }
                else { E = expf(-tf); om = 1.f - E; }
                C.p_esc[t] += L * E;
                C.p_abs[t] += L * (1.f - C.alb[t]) * om;
                // the path's optical depth is positive when its high word is a positive
                // normal number (the crossings' rounding errors in the low word are far
                // smaller); a sign bit means a NaN
                const int th = __float_as_int(tau_h);
                if (th < 0x00800000) {
                    if (th < 0) atomicOr(A.err, (unsigned)ERRBIT_NONFINITE);
                    L = 0.f;
                    C.nscat[t] = (int)C.ev[t] - 1;
                    stage = ST_END_PACKET;
                } else {
                    C.om[t] = om;
                    // forced scattering: tau_int from the exponential truncated at tau_path
                    const uint4 r = draw(C.ev[t], 0u);
                    C.ry[t] = r.y;
                    C.rz[t] = r.z;
                    par = -log1pf(-u01f(r.x) * om);
                    begin_search();
                    stage = ST_LOCATE_DONE;
                    break;
                }
            } else if (stage == ST_LOCATE_DONE) {
                if (count_add(C.c_loc[t], nsteps) && LONG) flush_counters();
                float l0 = C.xl0[t], l1 = C.xl1[t], l2 = C.xl2[t];
                const int fm = C.f_m[t];
                have_pc = fm >= 0;
                int axis = -1;  // of the face through which the interaction cell was entered
                float s = last_dusty_end;
                if (have_pc) {
                    s = C.f_s[t];
                    const int fl = C.f_last[t];
                    if constexpr (OCT) {
                        pc0 = c0; pc1 = c1; pc2 = c2;
                        pc_node = fm;
                        axis = fl - 1;
                    } else {
                        const unsigned row = (unsigned)fm / (unsigned)A.n_f, is = row / (unsigned)A.n_m;
                        const int jf = (int)((unsigned)fm - row * (unsigned)A.n_f);
                        const int jm = (int)(row - is * (unsigned)A.n_m);
                        pc0 = A.fast == 0 ? jf : jm;
                        pc1 = A.fast == 1 ? jf : (A.fast == 0 ? jm : (int)is);
                        pc2 = A.fast == 2 ? jf : (int)is;
                        // a stride names its axis, except along axes of one cell, which
                        // no crossing inside the grid runs along
                        if (fl != 0) axis = (fl == st0 && A.nx > 1) ? 0 : ((fl == st1 && A.ny > 1) ? 1 : 2);
                    }
                }
                if (axis >= 0) {
                    // entry point of the interaction cell, snapped onto the exact face plane
                    const float ft = C.f_t[t];
                    df_add_prod(x0, l0, ft, k0);
                    df_add_prod(x1, l1, ft, k1);
                    df_add_prod(x2, l2, ft, k2);
                    const int e = OCT ? 1 << (OL - olev) : 1;
                    const float ka = axis == 0 ? k0 : (axis == 1 ? k1 : k2);
                    const int ca = axis == 0 ? pc0 : (axis == 1 ? pc1 : pc2);
                    const int off = axis == 0 ? 0 : (axis == 1 ? A.nx + 1 : A.nx + 1 + A.ny + 1);
                    const float2 f = __ldg(A.faces + off + ca + (ka < 0.f ? e : 0));
                    if (axis == 0) { x0 = f.x; l0 = f.y; }
                    else if (axis == 1) { x1 = f.x; l1 = f.y; }
                    else { x2 = f.x; l2 = f.y; }
                }
                df_add_prod(x0, l0, s, k0);
                df_add_prod(x1, l1, s, k1);
                df_add_prod(x2, l2, s, k2);
                C.xl0[t] = l0; C.xl1[t] = l1; C.xl2[t] = l2;
                L = L * C.alb[t] * C.om[t];
                C.nscat[t] = (int)C.ev[t];
                if (L > 0.f && A.peel && A.ninstr > 0) {
                    C.peel_i[t] = PEEL_SCATTER;
                    stage = ST_PEEL;
                } else {
                    stage = ST_AFTER_SCATTER;
                }
            }

            if (stage == ST_AFTER_SCATTER) {
                if (L <= A.w_min_f * C.L0[t]) {
                    C.p_res[t] += L;
                    stage = ST_END_PACKET;
                } else if ((int)C.ev[t] >= A.max_events) {
                    atomicOr(A.err, (unsigned)ERRBIT_EVENT_CAP);
                    C.p_res[t] += L;
                    stage = ST_END_PACKET;
                } else {
                    // Henyey-Greenstein scattering: mu by inverse CDF, azimuth uniform
                    const float mu = hg_mu<float>(gg, u01f(C.ry[t]));
                    float sp, cp;
                    sincospif(2.f * u01f(C.rz[t]), &sp, &cp);
                    hg_rotate<float>(k0, k1, k2, mu, sp, cp);
                    stage = ST_START_DEP;
                }
            }

            if (stage == ST_END_PACKET) {
                C.c_scat[t] += (unsigned)C.nscat[t];
                if ((C.c_scat[t] | C.c_dep[t] | C.c_loc[t] | C.c_peel[t]) >> 30) flush_counters();
                const float pe = C.p_esc[t], pa = C.p_abs[t], pr = C.p_res[t], pp = C.p_peel[t];
                C.l_abs[t] += f2d(pa);
                C.l_esc[t] += f2d(pe);
                C.l_res[t] += f2d(pr);
                if (!isfinite(pe + pa + pr + pp)) atomicOr(A.err, (unsigned)ERRBIT_NONFINITE);
                const unsigned pk = C.pk[t] - (unsigned)__ldg(A.pk_first + lam);  // index within this call
                if (pk < (unsigned)A.nrec) {
                    double* rec = A.records + ((size_t)lam * A.nrec + pk) * SKIRT_REC_FIELDS;
                    rec[0] = (double)C.nscat[t];
                    rec[1] = f2d(pe);
                    rec[2] = f2d(pa);
                    rec[3] = f2d(pr);
                    rec[4] = f2d(pp);
                    rec[5] = f2d(x0) + f2d(C.xl0[t]);
                    rec[6] = f2d(x1) + f2d(C.xl1[t]);
                    rec[7] = f2d(x2) + f2d(C.xl2[t]);
                }
                stage = ST_NEW;
            }

            if (stage == ST_NEW) {
                if (C.left[t] == 0) {
                    if (!A.persistent) {
                        const unsigned long long q = (unsigned long long)blockIdx.x * blockDim.x + t;
                        if (started || q >= A.q_count) { alive = false; break; }
                        started = true;
                        C.q[t] = A.q_base + q;
                        C.left[t] = 1;
                    } else {
                        const unsigned mask = __activemask();
                        const int lane = t & 31;
                        const int leader = __ffs(mask) - 1;
                        const unsigned rank = __popc(mask & ((1u << lane) - 1u));
                        unsigned long long base = 0;
                        if (lane == leader)
                            base = atomicAdd(A.queue, (unsigned long long)__popc(mask) * (unsigned long long)A.chunk);
                        base = __shfl_sync(mask, base, leader);
                        const unsigned long long q = base + (unsigned long long)rank * A.chunk;
                        if (q >= A.total) { alive = false; break; }
                        C.q[t] = q;
                        C.left[t] = (unsigned)(A.total - q < (unsigned long long)A.chunk ? A.total - q : A.chunk);
                    }
                }
                C.left[t] -= 1;
                const unsigned long long qq = C.q[t]++;
                int ll = C.lam[t];
                if (ll < 0 || qq < __ldg(A.offsets + ll) || qq >= __ldg(A.offsets + ll + 1)) {
                    int a = 0, b = A.nlambda - 1;  // last wavelength whose offset <= qq
                    while (a < b) {
                        const int mid = (a + b + 1) >> 1;
                        if (__ldg(A.offsets + mid) <= qq) a = mid; else b = mid - 1;
                    }
                    flush_ledger();
                    ll = a;
                    C.lam[t] = ll;
                    C.alb[t] = __ldg(A.albedo_f + ll);
                    C.L0[t] = __ldg(A.L0_f + ll);
                }
                lam = ll;
                dep_base = A.absorbed + (size_t)lam * A.abs_ls;
                krs = __ldg(A.kscale_f + lam);
                gg = __ldg(A.g_f + lam);
                C.pk[t] = (unsigned)(qq - __ldg(A.offsets + lam) + __ldg(A.pk_first + lam));
                L = C.L0[t];
                C.p_esc[t] = C.p_abs[t] = C.p_res[t] = C.p_peel[t] = 0.f;
                C.ev[t] = 0;
                C.nscat[t] = 0;
                C.l_emit[t] += f2d(L);
                have_pc = false;
                float l0 = 0.f, l1 = 0.f, l2 = 0.f;

                // ---- launch (Sect. 3.2)
                bool isotropic = true;
                if (A.src_kind == SKIRT_SRC_BEAM || A.src_kind == SKIRT_SRC_POINT) {
                    x0 = A.src_df[0].x; x1 = A.src_df[1].x; x2 = A.src_df[2].x;
                    l0 = A.src_df[0].y; l1 = A.src_df[1].y; l2 = A.src_df[2].y;
                    if (A.src_kind == SKIRT_SRC_BEAM) {
                        k0 = A.src_dir_f[0]; k1 = A.src_dir_f[1]; k2 = A.src_dir_f[2];
                        isotropic = false;
                    }
                } else if (A.src_kind == SKIRT_SRC_DISK) {
                    const float hR = (float)A.h_R, hz = (float)A.h_z;
                    for (uint32_t tries = 0;; ++tries) {
                        const uint4 r = draw(0u, tries == 0 ? 0u : tries + 1u);
                        const float u0 = u01f(r.x), u1 = u01f(r.y), u2 = u01f(r.z), u3 = u01f(r.w);
                        const float Rr = -hR * (logf(u0) + logf(u1));
                        const float z = (u2 < 0.5f) ? hz * logf(2.f * u2) : -hz * logf(2.f * (1.f - u2));
                        float sp, cp;
                        sincospif(2.f * u3, &sp, &cp);
                        x0 = A.src_df[0].x + Rr * cp;
                        x1 = A.src_df[1].x + Rr * sp;
                        x2 = A.src_df[2].x + z;
                        if (x0 >= A.lo_f[0] && x0 <= A.hi_f[0] && x1 >= A.lo_f[1] && x1 <= A.hi_f[1] &&
                            x2 >= A.lo_f[2] && x2 <= A.hi_f[2])
                            break;
                        if (tries + 1 >= 64) {
                            atomicOr(A.err, (unsigned)ERRBIT_SOURCE);
                            x0 = A.src_df[0].x; x1 = A.src_df[1].x; x2 = A.src_df[2].x;
                            break;
                        }
                    }
                } else {  // SKIRT_SRC_DUST
                    const uint4 r = draw(0u, 0u);
                    const long long a = dust_cell(A, lam, f2d(u01f(r.x)));
                    float side = 1.f;  // the cell's extent in lattice cells
                    if constexpr (OCT) {
                        // uniform point in the leaf's box; its leaf is found again
                        // from the position
                        const int4 lf = __ldg(&A.oct_leaf[a]);
                        pc0 = lf.x; pc1 = lf.y; pc2 = lf.z;
                        side = (float)(1 << (OL - lf.w));
                    } else {
                        pc0 = (int)(a % A.nx);
                        pc1 = (int)((a / A.nx) % A.ny);
                        pc2 = (int)(a / ((long long)A.nx * A.ny));
                    }
                    const float2* fx = A.faces;
                    const float2* fy = fx + (A.nx + 1);
                    const float2* fz = fy + (A.ny + 1);
                    const float2 f0 = __ldg(fx + pc0), f1 = __ldg(fy + pc1), f2 = __ldg(fz + pc2);
                    x0 = f0.x; l0 = f0.y;
                    x1 = f1.x; l1 = f1.y;
                    x2 = f2.x; l2 = f2.y;
                    df_add_prod(x0, l0, u01f(r.y), side * A.d_f[0]);
                    df_add_prod(x1, l1, u01f(r.z), side * A.d_f[1]);
                    df_add_prod(x2, l2, u01f(r.w), side * A.d_f[2]);
                    have_pc = !OCT;
                }
                C.xl0[t] = l0; C.xl1[t] = l1; C.xl2[t] = l2;
                stage = ST_START_DEP;
                if (isotropic) {
                    const uint4 r = draw(0u, 1u);
                    const float mu = 2.f * u01f(r.x) - 1.f;
                    const float st = sqrtf(fmaxf(1.f - mu * mu, 0.f));
                    float sp, cp;
                    sincospif(2.f * u01f(r.y), &sp, &cp);
                    k0 = st * cp; k1 = st * sp; k2 = mu;
                    if (A.peel && A.ninstr > 0) {
                        C.peel_i[t] = 0;
                        stage = ST_PEEL;
                    }
                }
            }

            float w0 = k0, w1 = k1, w2 = k2, i0 = 0.f, i1 = 0.f, i2 = 0.f;  // the traversal to start
            if (stage == ST_PEEL) {
                const int pk = C.peel_i[t];
                const InstrDev& I = sins[pk & (PEEL_SCATTER - 1)];
                float w = L;  // isotropic emission: phase factor 1
                if (pk & PEEL_SCATTER) {
                    const float mu = k0 * I.kobs_f[0] + k1 * I.kobs_f[1] + k2 * I.kobs_f[2];
                    w = L * hg_phase<float>(gg, mu);
                }
                C.peel_w[t] = w;
                stage = ST_PEEL_DONE;
                nsteps = 0;
                if (w > 0.f) {
                    need = M_PEEL;
                    w0 = I.kobs_f[0]; w1 = I.kobs_f[1]; w2 = I.kobs_f[2];
                    i0 = I.ikobs_f[0]; i1 = I.ikobs_f[1]; i2 = I.ikobs_f[2];
                }
            } else if (stage == ST_START_DEP) {
                C.ev[t] += 1;
                par = L * (1.f - C.alb[t]);
                need = M_DEPOSIT;
                i0 = k0 != 0.f ? 1.f / k0 : 0.f;
                i1 = k1 != 0.f ? 1.f / k1 : 0.f;
                i2 = k2 != 0.f ? 1.f / k2 : 0.f;
                stage = ST_DEPOSIT_DONE;
            }
            if (need != M_NONE) {
                begin(need, w0, w1, w2, i0, i1, i2);
                if (need == M_DEPOSIT) keep_start();
            }
        } while (need == M_NONE);
    };

    for (;;) {
        const bool stepping = mode != M_NONE;
        const unsigned sm = __ballot_sync(0xffffffffu, stepping);
        const unsigned wm = __ballot_sync(0xffffffffu, !stepping && alive);
        if (!(sm | wm)) break;
        if (sm && (__popc(sm) >= step_min || !wm)) {
            // the barrier makes the lanes meet after every crossing: without it
            // the rare branches of a crossing leave parts of the warp running
            // their crossings apart (15 of 26 stepping lanes at a time)
#pragma unroll 1
            for (int r = 0; r < ROUND; ++r) {
                if (mode != M_NONE) {
                    if constexpr (OCT) step_oct();
                    else step();
                }
                __syncwarp();
            }
            continue;
        }
        if (!stepping && alive) events();
    }

    flush_ledger();
    flush_counters();
}

}  // namespace

size_t trace_mixed_smem_bytes(int ninstr, int block)
{
    (void)block;
    return align16(sizeof(InstrDev) * ninstr) + sizeof(Cold);
}

namespace {

using MixedKernel = void (*)(TraceArgs);

MixedKernel mixed_kernel(int kind, bool long_counts)
{
    if (kind == G_OCT) return long_counts ? trace_mixed_kernel<G_OCT, true> : trace_mixed_kernel<G_OCT, false>;
    if (kind == G_CART) return long_counts ? trace_mixed_kernel<G_CART, true> : trace_mixed_kernel<G_CART, false>;
    return long_counts ? trace_mixed_kernel<G_CART_BIG, true> : trace_mixed_kernel<G_CART_BIG, false>;
}

cudaError_t set_smem_limit(MixedKernel k)
{
    return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)trace_mixed_smem_bytes(16, MAXB));
}

}  // namespace

cudaError_t launch_trace_mixed(const TraceArgs& a, int block, int grid, cudaStream_t s)
{
    if (block > MAXB || block % 32) return cudaErrorInvalidValue;
    const int kind = a.oct_levels > 0 ? G_OCT
                                      : (a.nx < (1 << 23) && a.ny < (1 << 23) && a.nz < (1 << 23) ? G_CART : G_CART_BIG);
    const unsigned long long line = (unsigned long long)a.nx + a.ny + a.nz + 8;  // (of an octree: its crossing bound)
    const MixedKernel k = mixed_kernel(kind, counts_within_packet(a.max_events, a.ninstr, line));
    cudaError_t e = set_smem_limit(k);
    if (e != cudaSuccess) return e;
    k<<<grid, block, trace_mixed_smem_bytes(a.ninstr, block), s>>>(a);
    return cudaGetLastError();
}

cudaError_t trace_mixed_occupancy(int block, int* blocks_per_sm, bool octree)
{
    if (block > MAXB || block % 32) {
        *blocks_per_sm = 0;
        return cudaSuccess;
    }
    const MixedKernel k = mixed_kernel(octree ? G_OCT : G_CART, false);
    cudaError_t e = set_smem_limit(k);
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k, block, trace_mixed_smem_bytes(16, block));
}

}  // namespace skirt
