// Photon-packet life cycle on the GPU, plain FP64 form: every quantity FP64.
// The mixed form lives in trace_mixed.cu.
//
// Method (arXiv:1705.04702): Sect. 3.2 (stellar emission phase: packets per
// wavelength, Monte Carlo launch / interaction sampling, peel-off to every
// instrument on each scattering, continuous absorption into the absorbed
// table, life until a negligible luminosity is left); Sect. 1 (peel-off,
// continuous absorption, forced scattering); Sect. 5.2 (absorbed table
// element (cell, wavelength) at cell * N_lambda + wavelength, updated with
// lock-free atomic additions -- here native FP64 reductions in L2); Sect. 7.9
// (octree dust grid: a cell crossing steps from a leaf to the leaf across its
// exit face, through the precomputed face neighbour and a descent by the
// lattice cell of the entry point).
//
// What bounds it is the FP64 pipe (83% active): a warp instruction
// holds it for some 20 cycles of the SM, whatever its active lanes.  So the lanes
// of a warp step together, peel-offs in some rounds and deposits and searches in
// others (a deposit crossing costs three times a peel-off's FP64 instructions),
// and handle their events together when few of them are stepping; and FP64 does
// only what has to be FP64.  Distances and optical depths are compared as integers
// (none is negative), face planes come from a table, the search starts from the
// saved start of the deposit traversal it repeats, and the deposits of a path take
// e^{-tau} once per round of crossings and carry what each cell leaves of it in
// between.  A peel-off crossing is 5 or 6 FP64 instructions, a deposit crossing
// 18 in thin cells.  3e5 packets of 3 wavelengths on a 97^3 disk take 37 ms, 36 to
// 39 by their seed (132 with one state machine per lane, every crossing 12 FP64
// instructions and two exponentials more per deposit, at 5 of 32 lanes).
#include <cuda_runtime.h>
#include <math.h>

#include <type_traits>

#include "skirt_internal.cuh"
#include "trace_device.cuh"
#include "work_count.cuh"

namespace skirt {
namespace {

// Lanes of one kind stepping below which a warp handles its idle lanes' events, and
// crossings between warp votes (and between evaluations of e^{-tau}).  The case
// named above with 8 / 24: 39 ms; 8 / 16: 43, 16 / 16: 48, 8 / 32: 43, 12 / 16: 46
// (deposits as they were before take(); with it 8 / 24: 39.1, 8 / 16: 43.2).
constexpr int FP64_STEP_MIN = 8;
constexpr int FP64_ROUND = 24;
constexpr int FP64_MAXB = 512;     // threads per block (upper bound)

// Per-thread state used only at events, in shared memory: arrays of blockDim.x.
enum {
    D_L_EMIT, D_L_ABS, D_L_ESC, D_L_RES,   // ledger of the current wavelength
    D_L0, D_P_ESC, D_P_ABS, D_P_RES, D_P_PEEL, D_OM, D_PEEL_W, D_ALB, D_LABS,
    D_B_T0, D_B_T1, D_B_T2,                // start of the deposit traversal: distances to its first faces
    D_NUM
};
enum {
    I_C_DEP, I_C_LOC, I_C_PEEL, I_C_SCAT,  // emptied into the 64-bit counters (count_add)
    I_LAM, I_NSCAT, I_PEEL_I, I_PK, I_EV, I_RY, I_RZ, I_LEFT, I_QLO, I_QHI,
    I_B_0, I_B_1, I_B_2, I_B_M,            // start of the deposit traversal: cell (lattice corner) and index (node)
    I_NUM
};
constexpr int PEEL_SCATTER = 16;  // added to the instrument's index after a scattering (at most 16 instruments)

__device__ __forceinline__ long long bits(double v) { return __double_as_longlong(v); }
// v, or 0 where its sign bit is set
__device__ __forceinline__ double clip0(double v) { return __double2hiint(v) < 0 ? 0.0 : v; }

// What a cell of optical depth x >= 0 takes of the power par, which becomes what is
// left: par (1 - e^{-x}).
//  x < 1/16: the Taylor series x (1 - x/2 + ... + x^8/9!), whose first omitted term
//    is below 4e-18 of the result.
//  x < 1/2: the same at x/8, then three doublings f(2y) = 2 f(y) - f(y)^2 with f kept
//    as y + s, y exact and s a few hundredths of it: 1.3 x 2^-53 off at most and
//    0.45 in the mean, as expm1 is (doubling f itself: 3.6 and 0.8), for 10
//    instructions beyond the series that the lanes in thin cells run anyway.
//  Beyond: par less what was taken would carry that product's rounding e^x times as
//    large (behind x = 37 none of par's digits is left), so what is left is par e^{-x}
//    by itself.
// Either way a crossing adds at most 2 x 2^-53 to par's relative error.  3e5 packets
// of 3 wavelengths on a 97^3 disk: 35.4 ms, against 36.7 with -expm1(-x) from 1/16 on
// and par - dep throughout; with expm1 between 1/16 and 1/2 39.1, with par formed
// afresh from tau behind every half optical depth 40.4.
__device__ __forceinline__ double take(double x, double& par)
{
    if (bits(x) >= 0x3FE0000000000000ll) {
        const double e = exp(-x), dep = par * (1.0 - e);
        par *= e;
        return dep;
    }
    const bool mid = bits(x) >= 0x3FB0000000000000ll;
    const double y = mid ? __longlong_as_double(bits(x) - (3ll << 52)) : x, q = y * y;
    double p = fma(y, 1.0 / 362880.0, -1.0 / 40320.0);
    p = fma(y, p, 1.0 / 5040.0);
    p = fma(y, p, -1.0 / 720.0);
    p = fma(y, p, 1.0 / 120.0);
    p = fma(y, p, -1.0 / 24.0);
    p = fma(y, p, 1.0 / 6.0);
    p = fma(y, p, -0.5);
    double f = fma(q, p, y);
    if (mid) {
        double s = q * p;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            f = __longlong_as_double(bits(y) + ((long long)k << 52)) + s;
            s = fma(-f, f, s + s);
        }
        f = x + s;
    }
    const double dep = par * f;
    par -= dep;
    return dep;
}

template <bool OCT>
__global__ void __launch_bounds__(FP64_MAXB) trace_kernel(const TraceArgs A)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int t = threadIdx.x, nt = blockDim.x;
    InstrDev* sins = reinterpret_cast<InstrDev*>(smem_raw);
    double* cd = reinterpret_cast<double*>(smem_raw + sizeof(InstrDev) * A.ninstr);
    int* ci = reinterpret_cast<int*>(cd + (size_t)D_NUM * nt);
    const auto D = [&](int k) -> double& { return cd[k * nt + t]; };
    const auto I = [&](int k) -> int& { return ci[k * nt + t]; };
    for (int i = threadIdx.x; i < A.ninstr; i += blockDim.x) sins[i] = A.ins[i];
    D(D_L_EMIT) = D(D_L_ABS) = D(D_L_ESC) = D(D_L_RES) = 0.0;
    I(I_C_DEP) = I(I_C_LOC) = I(I_C_PEEL) = I(I_C_SCAT) = 0;
    I(I_LAM) = -1;
    I(I_LEFT) = I(I_QLO) = I(I_QHI) = 0;
    __syncthreads();

    const int NL = A.nlambda;
    const int nx = A.nx, ny = A.ny, nz = A.nz;
    const double INF = __longlong_as_double(0x7ff0000000000000ll);
    const double* __restrict__ faces = A.faces64;  // x [nx+1], y [ny+1], z [nz+1]

    // ---- traversal state: origin (x0, x1, x2), direction in its reciprocals
    int mode = M_NONE;
    int c0 = 0, c1 = 0, c2 = 0;
    int s0 = 0, s1 = 0, s2 = 0;
    double iv0 = 0, iv1 = 0, iv2 = 0;
    double tn0 = 0, tn1 = 0, tn2 = 0;  // distance to the next face on each axis
    double tcur = 0;
    double tau = 0.0;                  // optical depth along this traversal
    double par = 0.0;                  // deposit: L (1 - albedo) e^{-tau}; search: interaction optical depth
    double taken = 0.0;                // deposit: what the cells have taken, the ledger's absorbed power
    double s_found = 0, last_dusty_end = 0;
    bool found = false;
    unsigned nsteps = 0;
    int cur_m = 0;                     // the current cell (octree: leaf) and its extinction coefficient
    double kr_cur = 0;
    // octree: the current leaf's node and level (c0..c2: its lattice corner), the
    // direction of the traversal
    const int OL = A.oct_levels;
    int onode = 0, olev = 0;
    double v0 = 0, v1 = 0, v2 = 0;

    // ---- packet state
    int stage = ST_NEW;
    bool alive = true, started = false;
    int lam = 0;
    double L = 0.0;
    double x0 = 0, x1 = 0, x2 = 0;     // position
    double k0 = 0, k1 = 0, k2 = 0;     // direction
    double krs = 0, gg = 0;
    bool unit = false;                 // krs is 1
    bool have_pc = false;              // pc0..pc2 (octree: pc_node) is the position's cell
    int pc0 = 0, pc1 = 0, pc2 = 0, pc_node = 0;

    // octree: the leaf holding lattice cell (j0, j1, j2), found by descending
    // from `node` (a node of level `lev`, or a leaf)
    auto oct_enter = [&](int node, int lev, int j0, int j1, int j2) {
        int r = __ldg(&A.oct_nodes[node].ref);
        while (r >= 0 && lev < OL) {
            ++lev;
            const int b = OL - lev;
            node = r + (((j0 >> b) & 1) | (((j1 >> b) & 1) << 1) | (((j2 >> b) & 1) << 2));
            r = __ldg(&A.oct_nodes[node].ref);
        }
        onode = node;
        olev = oct_leaf_level(r);
        cur_m = oct_leaf_index(r);
        kr_cur = (double)__ldg(&A.oct_nodes[node].kr);
        const int mask = ~((1 << (OL - olev)) - 1);
        c0 = j0 & mask;
        c1 = j1 & mask;
        c2 = j2 & mask;
    };

    // distances to the faces through which the current cell (of e lattice cells
    // per axis) can be left
    auto set_faces = [&](int e) {
        const double* fy = faces + (nx + 1);
        const double* fz = fy + (ny + 1);
        tn0 = s0 ? clip0((__ldg(faces + c0 + (s0 > 0 ? e : 0)) - x0) * iv0) : INF;
        tn1 = s1 ? clip0((__ldg(fy + c1 + (s1 > 0 ? e : 0)) - x1) * iv1) : INF;
        tn2 = s2 ? clip0((__ldg(fz + c2 + (s2 > 0 ? e : 0)) - x2) * iv2) : INF;
    };

    // starts a traversal of kind m along (vx, vy, vz), whose reciprocals (zero
    // for zero components) are (i0, i1, i2), from the packet's position
    auto begin = [&](int m, double vx, double vy, double vz, double i0, double i1, double i2) {
        mode = m;
        if (!have_pc) {
            pc0 = cell_index<double>(x0, A.lo[0], A.d[0], nx);
            pc1 = cell_index<double>(x1, A.lo[1], A.d[1], ny);
            pc2 = cell_index<double>(x2, A.lo[2], A.d[2], nz);
            pc_node = 0;
            have_pc = true;
        }
        s0 = vx > 0.0 ? 1 : (vx < 0.0 ? -1 : 0);
        s1 = vy > 0.0 ? 1 : (vy < 0.0 ? -1 : 0);
        s2 = vz > 0.0 ? 1 : (vz < 0.0 ? -1 : 0);
        iv0 = i0; iv1 = i1; iv2 = i2;
        if (OCT) {
            oct_enter(pc_node, 0, pc0, pc1, pc2);
            pc0 = c0; pc1 = c1; pc2 = c2;
            pc_node = onode;
            v0 = vx; v1 = vy; v2 = vz;
            set_faces(1 << (OL - olev));
        } else {
            c0 = pc0; c1 = pc1; c2 = pc2;
            cur_m = (c2 * ny + c1) * nx + c0;
            kr_cur = __ldg(A.kr64 + cur_m);
            set_faces(1);
        }
        tcur = 0.0;
        tau = 0.0;
        nsteps = 0;
    };

    // one cell crossing (PEEL: of a peel-off; otherwise of a deposit or a search)
    auto step = [&](auto kind) {
        constexpr bool PEEL = decltype(kind)::value;
        const long long b0 = bits(tn0), b1 = bits(tn1), b2 = bits(tn2);
        const int axis = b0 <= b1 ? (b0 <= b2 ? 0 : 2) : (b1 <= b2 ? 1 : 2);
        const double tnext = axis == 0 ? tn0 : (axis == 1 ? tn1 : tn2);
        const int sa = axis == 0 ? s0 : (axis == 1 ? s1 : s2);
        const int ca = axis == 0 ? c0 : (axis == 1 ? c1 : c2);
        const int na = axis == 0 ? nx : (axis == 1 ? ny : nz);
        // what the crossing leads to, requested before the crossing's work
        int nb = 0, mn = 0;
        bool out;
        double kr_next = 0.0;
        if (OCT) {
            nb = __ldg(&A.oct_nodes[onode].nb[2 * axis + (sa > 0)]);
            out = nb < 0;  // the exit face lies on the root box
        } else {
            out = (unsigned)(ca + sa) >= (unsigned)na;
            mn = cur_m + sa * (axis == 0 ? 1 : (axis == 1 ? nx : nx * ny));
            if (!out) kr_next = __ldg(A.kr64 + mn);
        }
        const double ds = clip0(tnext - tcur);
        double krl = kr_cur;
        if (!unit) krl *= krs;
        const double dtau = krl * ds;
        const double tau_n = tau + dtau;
        ++nsteps;
        if (PEEL) {
        } else if (mode == M_DEPOSIT) {
            if (bits(dtau) > 0) {
                const double dep = take(dtau, par);
                if (bits(dep) > 0) {
                    atomicAdd(A.absorbed + ((size_t)cur_m * A.abs_cs + (size_t)lam * A.abs_ls), dep);
                    taken += dep;
                }
            }
        } else if (bits(krl) > 0) {
            if (bits(tau_n) >= bits(par)) {
                s_found = tcur + (par - tau) / krl;
                found = true;
                mode = M_NONE;
                return;  // the current cell stays
            }
            last_dusty_end = tnext;
        }
        tau = tau_n;
        if (out) {
            mode = M_NONE;
            return;
        }
        tcur = tnext;
        if (OCT) {
            if (nsteps > (unsigned)A.oct_step_cap) {
                atomicOr(A.err, (unsigned)ERRBIT_PATH);
                mode = M_NONE;
                return;
            }
            // lattice cell of the entry point into the next leaf: across the exit
            // face along `axis`; along the other axes the cell of the crossing
            // point, kept within the current leaf's cross-section
            const int osz = 1 << (OL - olev);
            int j[3];
            const int cc[3] = {c0, c1, c2};
            const double oo[3] = {x0, x1, x2}, vv[3] = {v0, v1, v2};
#pragma unroll
            for (int b = 0; b < 3; ++b) {
                if (b == axis) {
                    j[b] = sa > 0 ? cc[b] + osz : cc[b] - 1;
                } else {
                    const double f = floor((oo[b] + tnext * vv[b] - A.lo[b]) / A.d[b]);
                    j[b] = f < (double)cc[b] ? cc[b] : (f > (double)(cc[b] + osz - 1) ? cc[b] + osz - 1 : (int)f);
                }
            }
            // a neighbour that is not a leaf has the current level
            oct_enter(nb, olev, j[0], j[1], j[2]);
            set_faces(1 << (OL - olev));
        } else {
            cur_m = mn;
            kr_cur = kr_next;
            const int cn = ca + sa;
            const int off = axis == 0 ? 0 : (axis == 1 ? nx + 1 : nx + 1 + ny + 1);
            const double xa = axis == 0 ? x0 : (axis == 1 ? x1 : x2);
            const double iva = axis == 0 ? iv0 : (axis == 1 ? iv1 : iv2);
            const double tnew = clip0((__ldg(faces + off + cn + (sa > 0)) - xa) * iva);
            c0 = axis == 0 ? cn : c0;
            c1 = axis == 1 ? cn : c1;
            c2 = axis == 2 ? cn : c2;
            tn0 = axis == 0 ? tnew : tn0;
            tn1 = axis == 1 ? tnew : tn1;
            tn2 = axis == 2 ? tnew : tn2;
        }
    };

    auto flush_ledger = [&]() {
        const int ll = I(I_LAM);
        if (ll >= 0) {
            double* lg = A.ledger + 4 * (size_t)ll;
            atomicAdd(lg + 0, D(D_L_EMIT));
            atomicAdd(lg + 1, D(D_L_ABS));
            atomicAdd(lg + 2, D(D_L_ESC));
            atomicAdd(lg + 3, D(D_L_RES));
        }
        D(D_L_EMIT) = D(D_L_ABS) = D(D_L_ESC) = D(D_L_RES) = 0.0;
    };

    auto flush_counters = [&]() {
        atomicAdd(A.counters + 0, (unsigned long long)(unsigned)I(I_C_SCAT));
        atomicAdd(A.counters + 1, (unsigned long long)(unsigned)I(I_C_DEP));
        atomicAdd(A.counters + 2, (unsigned long long)(unsigned)I(I_C_LOC));
        atomicAdd(A.counters + 3, (unsigned long long)(unsigned)I(I_C_PEEL));
        I(I_C_DEP) = I(I_C_LOC) = I(I_C_PEEL) = I(I_C_SCAT) = 0;
    };

    auto draw = [&](uint32_t event, uint32_t block) -> uint4 {
        return philox10(make_uint4((unsigned)I(I_PK), (uint32_t)lam, event, (A.phase << 24) | block), A.key0, A.key1);
    };

    // Event handling: one pass over the stages in the order a packet meets them,
    // from the end of a traversal to the start of the next.  A lane goes round
    // again only where no traversal came of a pass (a peel-off of zero weight).
    auto events = [&]() {
        int need;
        const auto count = [&](int which, unsigned n) {
            unsigned c = (unsigned)I(which);
            const bool full = count_add(c, n);
            I(which) = (int)c;
            return full;
        };
        do {
            need = M_NONE;
            bool full = false;  // a work counter is to be emptied
            if (stage == ST_PEEL_DONE) {
                full = count(I_C_PEEL, nsteps);
                const int pk = I(I_PEEL_I), pi = pk & (PEEL_SCATTER - 1);
                const InstrDev& S = sins[pi];
                const double w = D(D_PEEL_W);
                if (w > 0.0) {
                    const double flux = w * exp(-tau) * S.flux_norm;
                    D(D_P_PEEL) += flux;
                    const double a = x0 * S.e1[0] + x1 * S.e1[1] + x2 * S.e1[2];
                    const double b = x0 * S.e2[0] + x1 * S.e2[1] + x2 * S.e2[2];
                    const double fa = floor((a + S.half_fov) * S.inv_dpx);
                    const double fb = floor((b + S.half_fov) * S.inv_dpx);
                    if (fa >= 0.0 && fa < (double)S.npx && fb >= 0.0 && fb < (double)S.npx) {
                        const long long pix = (long long)fb * S.npx + (long long)fa;
                        atomicAdd(A.images + S.img_off + pix * NL + lam, flux);
                    } else {
                        atomicAdd(A.oof + (size_t)pi * NL + lam, flux);
                    }
                }
                I(I_PEEL_I) = pk + 1;
                stage = pi + 1 < A.ninstr ? ST_PEEL : (pk & PEEL_SCATTER ? ST_AFTER_SCATTER : ST_START_DEP);
            } else if (stage == ST_DEPOSIT_DONE) {
                count(I_C_DEP, nsteps);  // emptied, if need be, behind the search that follows
                // what the path takes; stored here, on every lane's way: formed only in the
                // branch that uses it, it made runs with long packets a quarter slower (1.3e5
                // packets of 7 wavelengths, 110^3 disk: 32 ms, 25.3 this way)
                const double om = -expm1(-tau);
                D(D_OM) = om;
                D(D_P_ESC) += L * exp(-tau);
                D(D_P_ABS) += taken;
                if (!(tau > 0.0)) {
                    if (!(tau == 0.0)) atomicOr(A.err, (unsigned)ERRBIT_NONFINITE);
                    L = 0.0;
                    I(I_NSCAT) = I(I_EV) - 1;
                    stage = ST_END_PACKET;
                } else {
                    // forced scattering: tau_int from the exponential truncated at tau_path
                    const uint4 r = draw((unsigned)I(I_EV), 0u);
                    I(I_RY) = (int)r.y;
                    I(I_RZ) = (int)r.z;
                    par = -log1p(-(double)u01f(r.x) * om);
                    // the search: position and direction of the deposit traversal just
                    // ended, from its start
                    mode = M_LOCATE;
                    tn0 = D(D_B_T0); tn1 = D(D_B_T1); tn2 = D(D_B_T2);
                    c0 = I(I_B_0); c1 = I(I_B_1); c2 = I(I_B_2);
                    if (OCT) {
                        oct_enter(I(I_B_M), 0, c0, c1, c2);
                    } else {
                        cur_m = I(I_B_M);
                        kr_cur = __ldg(A.kr64 + cur_m);
                    }
                    tcur = 0.0;
                    tau = 0.0;
                    nsteps = 0;
                    found = false;
                    last_dusty_end = 0.0;
                    stage = ST_LOCATE_DONE;
                    break;
                }
            } else if (stage == ST_LOCATE_DONE) {
                full = count(I_C_LOC, nsteps) || count(I_C_DEP, 0u);
                const double s = found ? s_found : last_dusty_end;
                x0 += s * k0;
                x1 += s * k1;
                x2 += s * k2;
                have_pc = found;
                if (found) {
                    pc0 = c0; pc1 = c1; pc2 = c2;
                    pc_node = onode;
                }
                L = L * D(D_ALB) * D(D_OM);
                I(I_NSCAT) = I(I_EV);
                if (L > 0.0 && A.peel && A.ninstr > 0) {
                    I(I_PEEL_I) = PEEL_SCATTER;
                    stage = ST_PEEL;
                } else {
                    stage = ST_AFTER_SCATTER;
                }
            }

            if (stage == ST_AFTER_SCATTER) {
                if (L <= A.w_min * D(D_L0)) {
                    D(D_P_RES) += L;
                    stage = ST_END_PACKET;
                } else if (I(I_EV) >= A.max_events) {
                    atomicOr(A.err, (unsigned)ERRBIT_EVENT_CAP);
                    D(D_P_RES) += L;
                    stage = ST_END_PACKET;
                } else {
                    // Henyey-Greenstein scattering: mu by inverse CDF, azimuth uniform
                    const double mu = hg_mu<double>(gg, (double)u01f((unsigned)I(I_RY)));
                    double sp, cp;
                    sincospi(2.0 * (double)u01f((unsigned)I(I_RZ)), &sp, &cp);
                    hg_rotate<double>(k0, k1, k2, mu, sp, cp);
                    stage = ST_START_DEP;
                }
            }

            if (stage == ST_END_PACKET) full = count(I_C_SCAT, (unsigned)I(I_NSCAT)) || full || count(I_C_DEP, 0u);
            if (full) flush_counters();
            if (stage == ST_END_PACKET) {
                const double pe = D(D_P_ESC), pa = D(D_P_ABS), pr = D(D_P_RES), pp = D(D_P_PEEL);
                D(D_L_ABS) += pa;
                D(D_L_ESC) += pe;
                D(D_L_RES) += pr;
                if (!isfinite(pe + pa + pr + pp)) atomicOr(A.err, (unsigned)ERRBIT_NONFINITE);
                const uint32_t li = (uint32_t)I(I_PK) - (uint32_t)__ldg(A.pk_first + lam);  // index within this call
                if (li < (uint32_t)A.nrec) {
                    double* rec = A.records + ((size_t)lam * A.nrec + li) * SKIRT_REC_FIELDS;
                    rec[0] = (double)I(I_NSCAT);
                    rec[1] = pe;
                    rec[2] = pa;
                    rec[3] = pr;
                    rec[4] = pp;
                    rec[5] = x0;
                    rec[6] = x1;
                    rec[7] = x2;
                }
                stage = ST_NEW;
            }

            if (stage == ST_NEW) {
                if (I(I_LEFT) == 0) {
                    unsigned long long q;
                    if (!A.persistent) {
                        q = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x;
                        if (started || q >= A.q_count) { alive = false; break; }
                        started = true;
                        q += A.q_base;
                        I(I_LEFT) = 1;
                    } else {
                        // warp-aggregated refill from the global work queue
                        const unsigned mask = __activemask();
                        const int lane = threadIdx.x & 31;
                        const int leader = __ffs(mask) - 1;
                        const unsigned rank = __popc(mask & ((1u << lane) - 1u));
                        unsigned long long base = 0;
                        if (lane == leader)
                            base = atomicAdd(A.queue, (unsigned long long)__popc(mask) * (unsigned long long)A.chunk);
                        base = __shfl_sync(mask, base, leader);
                        q = base + (unsigned long long)rank * A.chunk;
                        if (q >= A.total) { alive = false; break; }
                        I(I_LEFT) = (int)(A.total - q < (unsigned long long)A.chunk ? A.total - q : A.chunk);
                    }
                    I(I_QLO) = (int)(unsigned)q;
                    I(I_QHI) = (int)(unsigned)(q >> 32);
                }
                I(I_LEFT) -= 1;
                const unsigned long long qq = ((unsigned long long)(unsigned)I(I_QHI) << 32) | (unsigned)I(I_QLO);
                I(I_QLO) = (int)(unsigned)(qq + 1);
                I(I_QHI) = (int)(unsigned)((qq + 1) >> 32);
                int ll = I(I_LAM);
                if (ll < 0 || qq < __ldg(A.offsets + ll) || qq >= __ldg(A.offsets + ll + 1)) {
                    int a = 0, b = NL - 1;  // last wavelength whose offset <= qq
                    while (a < b) {
                        const int mid = (a + b + 1) >> 1;
                        if (__ldg(A.offsets + mid) <= qq) a = mid; else b = mid - 1;
                    }
                    flush_ledger();
                    ll = a;
                    I(I_LAM) = ll;
                    D(D_ALB) = __ldg(A.albedo + ll);
                    D(D_L0) = __ldg(A.L0 + ll);
                }
                lam = ll;
                krs = __ldg(A.kscale + lam);
                unit = bits(krs) == 0x3FF0000000000000ll;
                gg = __ldg(A.g + lam);
                I(I_PK) = (int)(uint32_t)(qq - __ldg(A.offsets + lam) + __ldg(A.pk_first + lam));
                L = D(D_L0);
                D(D_P_ESC) = D(D_P_ABS) = D(D_P_RES) = D(D_P_PEEL) = 0.0;
                I(I_EV) = 0;
                I(I_NSCAT) = 0;
                D(D_L_EMIT) += L;
                have_pc = false;

                // ---- launch (Sect. 3.2): position from the source, isotropic direction
                bool isotropic = true;
                if (A.src_kind == SKIRT_SRC_BEAM) {
                    x0 = A.src_pos[0]; x1 = A.src_pos[1]; x2 = A.src_pos[2];
                    k0 = A.src_dir[0]; k1 = A.src_dir[1]; k2 = A.src_dir[2];
                    isotropic = false;
                } else if (A.src_kind == SKIRT_SRC_DISK) {
                    for (uint32_t tries = 0;; ++tries) {
                        const uint4 r = draw(0u, tries == 0 ? 0u : tries + 1u);
                        const double u0 = u01f(r.x), u1 = u01f(r.y), u2 = u01f(r.z), u3 = u01f(r.w);
                        const double Rr = -A.h_R * (log(u0) + log(u1));
                        const double z = (u2 < 0.5) ? A.h_z * log(2.0 * u2) : -A.h_z * log(2.0 * (1.0 - u2));
                        double sp, cp;
                        sincospi(2.0 * u3, &sp, &cp);
                        x0 = A.src_pos[0] + Rr * cp;
                        x1 = A.src_pos[1] + Rr * sp;
                        x2 = A.src_pos[2] + z;
                        const bool inside = x0 >= A.lo[0] && x0 <= A.hi[0] && x1 >= A.lo[1] && x1 <= A.hi[1] &&
                                            x2 >= A.lo[2] && x2 <= A.hi[2];
                        if (inside) break;
                        if (tries + 1 >= 64) {
                            atomicOr(A.err, (unsigned)ERRBIT_SOURCE);
                            x0 = A.src_pos[0]; x1 = A.src_pos[1]; x2 = A.src_pos[2];
                            break;
                        }
                    }
                } else if (A.src_kind == SKIRT_SRC_DUST) {
                    const uint4 r = draw(0u, 0u);
                    const long long a = dust_cell(A, lam, (double)u01f(r.x));
                    if (OCT) {
                        // uniform point in the leaf's box
                        const int4 lf = __ldg(&A.oct_leaf[a]);
                        const double side = (double)(1 << (OL - lf.w));
                        x0 = A.lo[0] + ((double)lf.x + (double)u01f(r.y) * side) * A.d[0];
                        x1 = A.lo[1] + ((double)lf.y + (double)u01f(r.z) * side) * A.d[1];
                        x2 = A.lo[2] + ((double)lf.z + (double)u01f(r.w) * side) * A.d[2];
                    } else {
                        const int ix = (int)(a % nx), iy = (int)((a / nx) % ny), iz = (int)(a / ((long long)nx * ny));
                        x0 = A.lo[0] + ((double)ix + (double)u01f(r.y)) * A.d[0];
                        x1 = A.lo[1] + ((double)iy + (double)u01f(r.z)) * A.d[1];
                        x2 = A.lo[2] + ((double)iz + (double)u01f(r.w)) * A.d[2];
                    }
                } else {
                    x0 = A.src_pos[0]; x1 = A.src_pos[1]; x2 = A.src_pos[2];
                }
                stage = ST_START_DEP;
                if (isotropic) {
                    const uint4 r = draw(0u, 1u);
                    const double mu = 2.0 * (double)u01f(r.x) - 1.0;
                    const double st = sqrt(fmax(1.0 - mu * mu, 0.0));
                    double sp, cp;
                    sincospi(2.0 * (double)u01f(r.y), &sp, &cp);
                    k0 = st * cp; k1 = st * sp; k2 = mu;
                    if (A.peel && A.ninstr > 0) {
                        I(I_PEEL_I) = 0;
                        stage = ST_PEEL;
                    }
                }
            }

            double w0 = k0, w1 = k1, w2 = k2, i0 = 0.0, i1 = 0.0, i2 = 0.0;  // the traversal to start
            if (stage == ST_PEEL) {
                const int pk = I(I_PEEL_I);
                const InstrDev& S = sins[pk & (PEEL_SCATTER - 1)];
                double w = L;  // isotropic emission: phase factor 1
                if (pk & PEEL_SCATTER) {
                    const double mu = k0 * S.kobs[0] + k1 * S.kobs[1] + k2 * S.kobs[2];
                    w = L * hg_phase<double>(gg, mu);
                }
                D(D_PEEL_W) = w;
                stage = ST_PEEL_DONE;
                nsteps = 0;
                if (w > 0.0) {
                    need = M_PEEL;
                    w0 = S.kobs[0]; w1 = S.kobs[1]; w2 = S.kobs[2];
                    i0 = S.ikobs[0]; i1 = S.ikobs[1]; i2 = S.ikobs[2];
                }
            } else if (stage == ST_START_DEP) {
                I(I_EV) += 1;
                par = L * (1.0 - D(D_ALB));
                D(D_LABS) = par;
                taken = 0.0;
                need = M_DEPOSIT;
                i0 = k0 != 0.0 ? 1.0 / k0 : 0.0;
                i1 = k1 != 0.0 ? 1.0 / k1 : 0.0;
                i2 = k2 != 0.0 ? 1.0 / k2 : 0.0;
                stage = ST_DEPOSIT_DONE;
            }
            if (need != M_NONE) {
                begin(need, w0, w1, w2, i0, i1, i2);
                if (need == M_DEPOSIT) {
                    D(D_B_T0) = tn0; D(D_B_T1) = tn1; D(D_B_T2) = tn2;
                    I(I_B_0) = c0; I(I_B_1) = c1; I(I_B_2) = c2;
                    I(I_B_M) = OCT ? onode : cur_m;
                }
            }
        } while (need == M_NONE);
    };

    // FP64_ROUND crossings of the lanes in one kind of traversal
    auto round = [&](auto kind) {
        constexpr bool PEEL = decltype(kind)::value;
#pragma unroll 1
        for (int r = 0; r < FP64_ROUND; ++r) {
            if (PEEL ? mode == M_PEEL : (mode == M_DEPOSIT || mode == M_LOCATE)) step(kind);
            __syncwarp();
        }
    };

    for (;;) {
        const unsigned pm = __ballot_sync(0xffffffffu, mode == M_PEEL);
        const unsigned dm = __ballot_sync(0xffffffffu, mode == M_DEPOSIT || mode == M_LOCATE);
        const unsigned wm = __ballot_sync(0xffffffffu, mode == M_NONE && alive);
        if (!(pm | dm | wm)) break;
        const int np = __popc(pm), nd = __popc(dm);
        if (max(np, nd) >= FP64_STEP_MIN || !wm) {
            if (np >= nd) {
                round(std::true_type{});
            } else {
                // e^{-tau} afresh, so that the roundings of at most a round's deposits stand
                // between it and a deposit
                if (mode == M_DEPOSIT && bits(tau) > 0) par = D(D_LABS) * exp(-tau);
                __syncwarp();
                round(std::false_type{});
            }
            continue;
        }
        if (mode == M_NONE && alive) events();
    }

    flush_ledger();
    flush_counters();
}

// SED = sum over the pixels of every image plus the out-of-frame peel-offs.
// images of instrument q are [npx*npx][nlambda]; thread (lambda lane, row
// group) sums a strided set of pixel rows for one wavelength column.
__global__ void sed_finalize_kernel(const double* __restrict__ img, const double* __restrict__ oof,
                                    double* __restrict__ sed, long long npix, int nlambda, int q, double sign)
{
    __shared__ double part[8][33];
    const int lam = blockIdx.x * 32 + threadIdx.x;
    const int rg = threadIdx.y;
    double s = 0.0;
    if (lam < nlambda)
        for (long long p = (long long)blockIdx.y * 8 + rg; p < npix; p += (long long)gridDim.y * 8)
            s += img[p * nlambda + lam];
    part[rg][threadIdx.x] = s;
    __syncthreads();
    if (rg == 0 && lam < nlambda) {
        double t = 0.0;
        for (int r = 0; r < 8; ++r) t += part[r][threadIdx.x];
        t *= sign;
        if (blockIdx.y == 0 && oof) t += oof[(size_t)q * nlambda + lam];
        atomicAdd(sed + (size_t)q * nlambda + lam, t);
    }
}

__global__ void f32_to_f64_kernel(const float* __restrict__ in, double* __restrict__ out, long long n,
                                  unsigned int* bad)
{
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        const float v = in[i];
        if (!(v >= 0.0f) || !isfinite(v)) atomicOr(bad, 1u);
        out[i] = (double)v;
    }
}

}  // namespace

size_t trace_smem_bytes(int ninstr, int block)
{
    return sizeof(InstrDev) * (size_t)ninstr + (sizeof(double) * D_NUM + sizeof(int) * I_NUM) * (size_t)block;
}

static cudaError_t set_smem_limit()
{
    const int bytes = (int)trace_smem_bytes(16, FP64_MAXB);
    cudaError_t e = cudaFuncSetAttribute(trace_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(trace_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}

cudaError_t launch_trace(const TraceArgs& a, int precision, int block, int grid, cudaStream_t s)
{
    if (precision == SKIRT_PREC_MIXED) return launch_trace_mixed(a, block, grid, s);
    cudaError_t e = set_smem_limit();
    if (e != cudaSuccess) return e;
    const size_t smem = trace_smem_bytes(a.ninstr, block);
    if (a.oct_levels > 0)
        trace_kernel<true><<<grid, block, smem, s>>>(a);
    else
        trace_kernel<false><<<grid, block, smem, s>>>(a);
    return cudaGetLastError();
}

cudaError_t trace_occupancy(int precision, int block, int* blocks_per_sm, bool octree)
{
    if (precision == SKIRT_PREC_MIXED) return trace_mixed_occupancy(block, blocks_per_sm, octree);
    cudaError_t e = set_smem_limit();
    if (e != cudaSuccess) return e;
    const size_t smem = trace_smem_bytes(16, block);
    return octree ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, trace_kernel<true>, block, smem)
                  : cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, trace_kernel<false>, block, smem);
}

CellOrder cell_order(int nx, int ny, int nz, int fast)
{
    CellOrder o;
    o.n[0] = nx; o.n[1] = ny; o.n[2] = nz;
    o.fast = fast;
    const int mid = fast == 0 ? 1 : 0, slow = fast == 2 ? 1 : 2;
    o.n_f = o.n[fast];
    o.n_m = o.n[mid];
    o.st[fast] = 1;
    o.st[mid] = o.n_f;
    o.st[slow] = (int)((long long)o.n_f * o.n_m);  // below the number of cells (< 2^31) if any axis is longer than one cell
    return o;
}

namespace {

// the API's cell number of number c in order o
__device__ __forceinline__ unsigned api_cell(unsigned c, const CellOrder& o)
{
    if (o.fast == 0) return c;
    const unsigned row = c / (unsigned)o.n_f, jf = c - row * (unsigned)o.n_f;
    const unsigned js = row / (unsigned)o.n_m, jm = row - js * (unsigned)o.n_m;
    const unsigned y = o.fast == 1 ? jf : js, z = o.fast == 2 ? jf : js;  // the middle axis is x
    return (z * (unsigned)o.n[1] + y) * (unsigned)o.n[0] + jm;
}

// out[c][l] (+)= in[l][c], 32 x 32 tiles through shared memory (one padding
// column): coalesced reads along the cells and writes along the wavelengths.
__global__ void transpose_absorbed_kernel(const double* __restrict__ in, double* __restrict__ out, long long ncell,
                                          int nl, int add, const CellOrder o)
{
    __shared__ double tile[32][33];
    const long long c0 = (long long)blockIdx.x * 32;
    const int l0 = blockIdx.y * 32;
    for (int k = threadIdx.y; k < 32; k += blockDim.y) {
        const long long c = c0 + threadIdx.x;
        const int l = l0 + k;
        tile[k][threadIdx.x] = (c < ncell && l < nl) ? in[(size_t)l * ncell + c] : 0.0;
    }
    __syncthreads();
    for (int k = threadIdx.y; k < 32; k += blockDim.y) {
        const long long c = c0 + k;
        const int l = l0 + threadIdx.x;
        if (c < ncell && l < nl) {
            const long long m = o.fast ? (long long)api_cell((unsigned)c, o) : c;
            double* p = out + (size_t)m * nl + l;
            *p = add ? *p + tile[threadIdx.x][k] : tile[threadIdx.x][k];
        }
    }
}

// Reordering between the API's cell order (x fastest) and order o (axis o.fast
// fastest), in 32 x 32 tiles of (x, fast axis) at one position of the third
// axis: coalesced on both sides.  TO_API: out[api][lambda] (+)=
// in[lambda][o], wavelength blockIdx.y of nl; otherwise out[o] = in[api].
template <bool TO_API, typename T>
__global__ void reorder_cells_kernel(const T* __restrict__ in, T* __restrict__ out, const CellOrder o,
                                     long long ncell, int nl, int add)
{
    __shared__ T tile[32][33];
    const int fa = o.fast, ta = 3 - fa;  // the fastest axis (1 or 2) and the third one
    const int nx = o.n[0], nf = o.n[fa], nt = o.n[ta];
    const size_t api_f = fa == 1 ? (size_t)nx : (size_t)nx * o.n[1], api_t = fa == 1 ? (size_t)nx * o.n[1] : (size_t)nx;
    const size_t o_x = (size_t)o.st[0], o_t = (size_t)o.st[ta];
    const long long tx = (nx + 31) / 32, tf = (nf + 31) / 32, total = tx * tf * nt;
    const int l = blockIdx.y;
    for (long long b = blockIdx.x; b < total; b += gridDim.x) {
        const int x0 = (int)(b % tx) * 32, f0 = (int)((b / tx) % tf) * 32, it = (int)(b / (tx * tf));
        for (int k = threadIdx.y; k < 32; k += blockDim.y) {
            const int x = x0 + (TO_API ? k : (int)threadIdx.x), f = f0 + (TO_API ? (int)threadIdx.x : k);
            if (x < nx && f < nf)
                tile[k][threadIdx.x] = TO_API ? in[(size_t)l * ncell + f + x * o_x + it * o_t]
                                              : in[x + f * api_f + it * api_t];
        }
        __syncthreads();
        for (int k = threadIdx.y; k < 32; k += blockDim.y) {
            const int x = x0 + (TO_API ? (int)threadIdx.x : k), f = f0 + (TO_API ? k : (int)threadIdx.x);
            if (x < nx && f < nf) {
                const T v = tile[threadIdx.x][k];
                if constexpr (TO_API) {
                    T* p = out + (x + f * api_f + it * api_t) * nl + l;
                    *p = add ? *p + v : v;
                } else {
                    out[f + x * o_x + it * o_t] = v;
                }
            }
        }
        __syncthreads();
    }
}

int reorder_blocks(const CellOrder& o)
{
    const long long b = (long long)((o.n[0] + 31) / 32) * ((o.n[o.fast] + 31) / 32) * o.n[3 - o.fast];
    return (int)(b < 65536 ? b : 65536);
}

}  // namespace

cudaError_t launch_transpose_absorbed(const double* in, double* out, long long ncell, int nlambda, bool add,
                                      const CellOrder& o, cudaStream_t s)
{
    if (o.fast != 0 && nlambda < 4) {
        // too few wavelengths for the tiles below: 32-byte runs of the output from four on
        reorder_cells_kernel<true, double><<<dim3(reorder_blocks(o), nlambda), dim3(32, 8), 0, s>>>(in, out, o, ncell,
                                                                                                    nlambda, add ? 1 : 0);
        return cudaGetLastError();
    }
    const long long bx = (ncell + 31) / 32;
    if (bx > 0x7fffffffLL) return cudaErrorInvalidValue;
    transpose_absorbed_kernel<<<dim3((unsigned)bx, (unsigned)((nlambda + 31) / 32)), dim3(32, 8), 0, s>>>(
        in, out, ncell, nlambda, add ? 1 : 0, o);
    return cudaGetLastError();
}

cudaError_t launch_reorder_density(const float* in, float* out, const CellOrder& o, cudaStream_t s)
{
    reorder_cells_kernel<false, float><<<reorder_blocks(o), dim3(32, 8), 0, s>>>(
        in, out, o, (long long)o.n[0] * o.n[1] * o.n[2], 1, 0);
    return cudaGetLastError();
}

cudaError_t launch_sed_finalize(const double* images, const double* oof, double* sed, int ninstr,
                                const int* npx_host, int nlambda, double sign, cudaStream_t s)
{
    long long off = 0;
    for (int q = 0; q < ninstr; ++q) {
        const long long npix = (long long)npx_host[q] * npx_host[q];
        dim3 block(32, 8);
        long long rows = (npix + 7) / 8;
        int gy = (int)(rows < 256 ? rows : 256);
        if (gy < 1) gy = 1;
        dim3 grid((nlambda + 31) / 32, gy);
        sed_finalize_kernel<<<grid, block, 0, s>>>(images + off, oof, sed, npix, nlambda, q, sign);
        off += npix * nlambda;
    }
    return cudaGetLastError();
}

cudaError_t launch_f32_to_f64(const float* in, double* out, long long n, unsigned int* bad, cudaStream_t s)
{
    long long blocks = (n + 255) / 256;
    if (blocks > 65536) blocks = 65536;
    if (blocks < 1) blocks = 1;
    f32_to_f64_kernel<<<(int)blocks, 256, 0, s>>>(in, out, n, bad);
    return cudaGetLastError();
}

}  // namespace skirt
