// gks_stencil.cu -- the gas-kinetic stencil of one S2O4 stage on sm_103a.
//
// Per stage and per direction d (x, y, z):
//   face_eq      one thread per tangential position of the extended face box,
//                marching along d with the differences around a cell (FP32C:
//                the 5 cells) in registers: WENO5-JS (Sec. 2, Jiang-Shu)
//                left/right states from one paired evaluation per cell, the
//                equilibrium state Q0 from the half Maxwellians (u>0 from the
//                left, u<0 from the right), and the quartic normal slope of Q0.
//   face_flux    (large FP32C grids: x and y) linear quartic reconstruction of
//                Q0 and its normal slope to the 2x2 Gauss points (Sec. 2, Eq.
//                (x_example)) and the gas-kinetic flux F0 and its time
//                derivative F1 at each point (Sec. 2, Eq. (flux); Appendix),
//                averaged with weights 1/4 and stored per face. FP32C: warps
//                marching along t2 with the t1-pass rows in registers; FP64 and
//                double-single: persistent blocks on 32x8 face tiles loaded by
//                TMA, the t1 pass in shared memory. The flux of FP32 and
//                double-single arithmetic runs at two Gauss points at once on
//                packed pairs.
//   flux_update  large FP32C grids: the z-face flux, walking z per tile column,
//                fused with the divergence (Eq. (finite)) and the two-stage
//                fourth-order combination of every cell; the others: the
//                update over the stored fluxes of all three directions. Stage
//                2 also prepares the next step (FP32 input, max |U|^2 for the
//                CFL step).
// Small grids run the three directions of face_eq and of face_flux as one
// launch each.
//
// All arithmetic runs in the working type R: double for GKS_FP64, float for
// GKS_FP32C. The reconstruction works on rho - off (off = rho_ref in FP32C,
// 0 in FP64), so the large constant pressure theta * rho_ref never enters an
// FP32 difference; it cancels exactly between the two faces of a cell.
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "gks_bounds.cuh"
#include "gks_device.cuh"
#include "gks_internal.h"

namespace gks {
namespace {

using namespace dev;

// ---------------------------------------------------------------- ghosts --

template <typename R>
struct GhostArgs {
    R *w;
    long np;
    int n[3], P[3];
    int bc[3][2];
    R off, csound;
    R uin[3];
    long nz, ny, nx;   // ghosts of the z, y and x layers (in that order of thread ranges)
    // dt of the step (first launch of a step), by the first thread
    Scalars *scal;
    double cfl, dt_fixed, hmin, cs64;
};

// dt from the largest |U|^2, which it clears.
__device__ __forceinline__ void set_dt(Scalars *scal, double cfl, double dt_fixed, double hmin, double csound)
{
    const double umax = sqrt(__longlong_as_double((long long)scal->maxu2_bits));
    double dt;
    if (dt_fixed > 0.0) {
        dt = dt_fixed;
        const double num = dt * (umax + csound) / hmin;
        scal->cfl_number = num;
        if (cfl > 0.0 && !(num <= cfl)) atomicOr(&scal->flags, FLAG_CFL);
    } else {
        dt = cfl * hmin / (umax + csound);
        scal->cfl_number = cfl;
        if (!isfinite(dt)) atomicOr(&scal->flags, FLAG_NONFINITE);
    }
    scal->dt = dt;
    scal->maxu2_bits = 0ull;
}

// The ghosts of axis d at index g (inside [0, n) for an interior index): the
// source index and the change of the source's value that the boundary makes.
template <typename R>
__device__ __forceinline__ int ghost_source(const GhostArgs<R> &A, int d, int g)
{
    const int n = A.n[d];
    if (g >= 0 && g < n) return g;
    const int bc = A.bc[d][g < 0 ? 0 : 1];
    if (bc == GKS_BC_PERIODIC) {
        const int r = g % n;
        return r < 0 ? r + n : r;
    }
    if (bc == GKS_BC_NOSLIP || bc == GKS_BC_SLIP) return g < 0 ? -1 - g : 2 * n - 1 - g;
    return g < 0 ? 0 : n - 1;
}
template <typename R>
__device__ __forceinline__ void ghost_value(const GhostArgs<R> &A, int d, int g, R q[4])
{
    if (g >= 0 && g < A.n[d]) return;
    const int s = g < 0 ? 0 : 1, bc = A.bc[d][s];
    if (bc == GKS_BC_NOSLIP) {
        q[1] = -q[1]; q[2] = -q[2]; q[3] = -q[3];
    } else if (bc == GKS_BC_SLIP) {
        if (d == 0) q[1] = -q[1];
        else if (d == 1) q[2] = -q[2];
        else q[3] = -q[3];
    } else if (bc == GKS_BC_INFLOW) {
        // density from the outgoing isothermal Riemann invariant of cell 1
        const R r1 = A.off + q[0];
        const R un1 = (d == 0 ? q[1] : (d == 1 ? q[2] : q[3])) / r1;
        const R x = (s == 0 ? R(1) : R(-1)) * (A.uin[d] - un1) / A.csound;
        const R ex = exp(x);
        const R rg = r1 * ex;
        q[0] = q[0] * ex + A.off * expm1(x);   // rg - off
        q[1] = rg * A.uin[0];
        q[2] = rg * A.uin[1];
        q[3] = rg * A.uin[2];
    }
}

// All ghost cells in one launch. The fill is defined axis by axis (x, then y
// and z over the ghosts of the axes before, which gives the edges and
// corners); a ghost of several axes is the interior source cell of all of them
// with each axis's change applied in that order, so no ghost waits for
// another one. Consecutive threads take cells that are contiguous in memory (a
// row of the z or y layers, the 2G x ghosts of a row). One launch in place of
// three, and the step's dt with the first: 384x256x256 121 -> 48 us a step,
// 128^3 54 -> 21, 32^3 37 -> 14. An exchange side's ghosts are left to the
// copy from the neighbouring slab.
template <typename R>
__global__ void __launch_bounds__(256) ghost_kernel(const __grid_constant__ GhostArgs<R> A)
{
    long t = blockIdx.x * 256L + threadIdx.x;
    if (t == 0 && A.scal) set_dt(A.scal, A.cfl, A.dt_fixed, A.hmin, A.cs64);
    int i, j, k;
    if (t < A.nz) {
        const long r = t / A.P[0];
        i = (int)(t - r * A.P[0]) - G;
        const long l = r / A.P[1];
        j = (int)(r - l * A.P[1]) - G;
        k = l < G ? (int)l - G : A.n[2] + (int)l - G;
    } else if ((t -= A.nz) < A.ny) {
        const long r = t / A.P[0];
        i = (int)(t - r * A.P[0]) - G;
        const int l = (int)(r % (2 * G));
        k = (int)(r / (2 * G));
        j = l < G ? l - G : A.n[1] + l - G;
    } else if ((t -= A.ny) < A.nx) {
        const long r = t / (2 * G);
        const int l = (int)(t - r * 2 * G);
        i = l < G ? l - G : A.n[0] + l - G;
        j = (int)(r % A.n[1]);
        k = (int)(r / A.n[1]);
    } else {
        return;
    }
    if ((i < 0 && A.bc[0][0] == GKS_BC_EXCHANGE) || (i >= A.n[0] && A.bc[0][1] == GKS_BC_EXCHANGE)) return;
    const int is = ghost_source(A, 0, i), js = ghost_source(A, 1, j), ks = ghost_source(A, 2, k);
    const long lg = (long)(i + G) + (long)A.P[0] * ((long)(j + G) + (long)A.P[1] * (k + G));
    const long ls = (long)(is + G) + (long)A.P[0] * ((long)(js + G) + (long)A.P[1] * (ks + G));
    if (!in_bounds(lg, A.np) || !in_bounds(ls, A.np)) return;
    R q[4];
#pragma unroll
    for (int v = 0; v < 4; ++v) q[v] = A.w[v * A.np + ls];
    ghost_value(A, 0, i, q);
    ghost_value(A, 1, j, q);
    ghost_value(A, 2, k, q);
#pragma unroll
    for (int v = 0; v < 4; ++v) A.w[v * A.np + lg] = q[v];
}

template <typename R>
void ghost_impl(const Ctx &c, R *w, bool with_dt)
{
    GhostArgs<R> A;
    A.w = w;
    A.np = c.np;
    for (int e = 0; e < 3; ++e) {
        A.n[e] = c.n[e];
        A.P[e] = c.P[e];
        A.bc[e][0] = c.bc[e][0];
        A.bc[e][1] = c.bc[e][1];
        A.uin[e] = (R)c.inflow[1 + e];
    }
    A.off = (R)c.off;
    A.csound = (R)c.csound;
    A.nz = 2L * G * c.P[0] * c.P[1];
    A.ny = 2L * G * c.P[0] * c.n[2];
    A.nx = 2L * G * c.n[1] * c.n[2];
    A.scal = with_dt ? c.scal : nullptr;
    A.cfl = c.cfl;
    A.dt_fixed = c.dt_fixed;
    A.hmin = c.hmin;
    A.cs64 = c.csound;
    mark(c, K_GHOST, 1);
    ghost_kernel<R><<<(unsigned)((A.nz + A.ny + A.nx + 255) / 256), 256, 0, c.stream>>>(A);
    mark(c, K_GHOST, 0);
}

// ------------------------------------------------------------ face state --

// Storage type of the face boxes and face fluxes between kernels: double-
// single pairs when the arithmetic is double-single (no conversion between
// the kernels), else the state's type.
template <typename R, typename C>
using Mid = typename std::conditional<std::is_same<C, dsf>::value, dsf, R>::type;

template <typename R, typename C = R>
struct FaceEqArgs {
    const R *w;      // working state, 4 arrays of np
    long np;
    Mid<R, C> *fq;   // 8 arrays of nfq
    long nfq;
    const R *ihf;    // inverse centre distance at faces of axis d
    int n1, n2;      // interior cells along t1, t2
    int e1p;         // row stride of the face box (n1 + 4 rounded up to 4)
    long sd, s1, s2; // element strides along d, t1, t2
    int cn, c1, c2;  // state component of the normal / t1 / t2 momentum
    int nf, K;       // faces along d, faces per thread of the marching kernel
    Phys<C> ph;      // in the compute type
};

// Blocks of the face-state kernels (ALL: of the launch of all directions):
// threads, blocks that fit on an SM, and how few of them keep it as busy. FP32
// with 64, 128, 256 threads: 1.82, 1.82, 1.88 ms a step of 384x256x256;
// double-single with 64 and 256 1.07 and 1.00 ms on 96^3, 0.076 and 0.108 in the
// launch of all directions of 32^3, whose few blocks spread better when small.
// FP64: 12 warps at 168 registers are what the FP64 pipe's latency needs (16 at
// 128 registers spill, 3.42 against 3.14 ms).
template <typename C, bool ALL>
constexpr int kEqThreads = ALL || std::is_same<C, double>::value ? 64 : std::is_same<C, dsf>::value ? 256 : 128;
template <typename C, bool ALL>
constexpr int kEqBlocks = std::is_same<C, float>::value ? (ALL ? 8 : 6) : std::is_same<C, dsf>::value ? (ALL ? 8 : 2) : 6;
template <typename C, bool ALL>
constexpr int kEqBusy = std::is_same<C, float>::value ? (ALL ? 1 : 6) : std::is_same<C, dsf>::value ? (ALL ? 6 : 2) : 5;

// Marching variant: each thread walks K consecutive faces along d at one
// tangential position of the extended face box, with the differences around
// the current cell in registers (WenoMarch). Per cell it forms both face
// values of WENO5 from one set of smoothness indicators; face f takes the
// right-face value of cell f-1 and the left-face value of cell f. Launched
// for FP64 grids in FP64 arithmetic; FP32 grids and double-single arithmetic
// take the packed variants below, which march the same way.
__device__ __forceinline__ void face_eq_march(const FaceEqArgs<double, double> &A, int2 blk)
{
    int a, b;
    const int f0 = blk.y * A.K;
    if (!face_position((unsigned)blk.x * blockDim.x + threadIdx.x, A.n1, A.n2, a, b) || f0 >= A.nf) return;
    const int f1 = min(f0 + A.K, A.nf);
    const long base = (long)(a + G) * A.s1 + (long)(b + G) * A.s2;   // cell index along d = -G
    // cells f0-3 .. f1+1 are read, faces f0 .. f1-1 written
    if (!in_bounds(base + (long)(f0 - 3 + G) * A.sd, A.np) || !in_bounds(base + (long)(f1 + 1 + G) * A.sd, A.np) ||
        !in_bounds(((long)f0 * (A.n2 + 4) + (b + 2)) * A.e1p + (a + 2), A.nfq) ||
        !in_bounds(((long)(f1 - 1) * (A.n2 + 4) + (b + 2)) * A.e1p + (a + 2), A.nfq))
        return;
    const double *pc[4] = {A.w + base, A.w + (long)A.cn * A.np + base, A.w + (long)A.c1 * A.np + base,
                           A.w + (long)A.c2 * A.np + base};
    // cells f0-3 .. f0 start the march at cell f0-1, cell f0+1 completes it
    WenoMarch<double> w[4];
    double Qprev[4];
#pragma unroll
    for (int v = 0; v < 4; ++v) {
        const double *p = pc[v] + (long)(f0 - 3 + G) * A.sd;
        w[v].start(__ldg(p), __ldg(p + A.sd), __ldg(p + 2 * A.sd), __ldg(p + 3 * A.sd));
        double l;
        w[v].push(__ldg(p + 4 * A.sd), Qprev[v], l);
    }
    // the cell entering the march, loaded one face ahead
    double nxt[4];
#pragma unroll
    for (int v = 0; v < 4; ++v) nxt[v] = __ldg(pc[v] + (long)(f0 + 2 + G) * A.sd);
    for (int f = f0; f < f1; ++f) {
        const double ihf = A.ihf[f];
        const long o = ((long)f * (A.n2 + 4) + (b + 2)) * A.e1p + (a + 2);
        double e[4];
#pragma unroll
        for (int v = 0; v < 4; ++v) e[v] = nxt[v];
        if (f + 1 < f1) {
            // cell f + 3 <= nf + 1 = n + 2: inside the ghost layers
#pragma unroll
            for (int v = 0; v < 4; ++v) nxt[v] = __ldg(pc[v] + (long)(f + 3 + G) * A.sd);
        }
        double Ql[4], Qr[4], Q0[4];
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            A.fq[(4 + v) * A.nfq + o] = w[v].slope() * ihf;
            Ql[v] = Qprev[v];
            w[v].push(e[v], Qprev[v], Qr[v]);
        }
        face_equilibrium(A.ph, Ql, Qr, Q0);
#pragma unroll
        for (int v = 0; v < 4; ++v) A.fq[v * A.nfq + o] = Q0[v];
    }
}

// face_eq_march for FP32 grids on packed pairs: WENO5 of the
// components paired as (rho, m_n) and (m_t1, m_t2), the half-space terms of
// the left and right states as one pair, the normal slopes paired like the
// components. Unrolled by two so that the window shifts cost no moves.
//
// SEG (the x faces, whose cells are consecutive along the march but a row
// apart across t1): a warp's lanes are 4 consecutive march segments of K
// faces times 8 positions, so that the rows a warp walks (8 per component
// instead of 32) stay in L1 for the K faces that reuse each sector; a store
// of the face box still writes 4 whole sectors (8 rows of 4 segments).
template <bool SEG>
__device__ __forceinline__ void face_eq_f2(const FaceEqArgs<float, float> &A, int2 blk)
{
    const int t = threadIdx.x;
    int a, b;
    const int f0 = SEG ? (blk.y * 4 + ((t >> 3) & 3)) * A.K : blk.y * A.K;
    const unsigned pos = SEG ? blk.x * (blockDim.x / 4) + (t >> 5) * 8 + (t & 7) : blk.x * blockDim.x + t;
    if (!face_position(pos, A.n1, A.n2, a, b) || f0 >= A.nf) return;
    const int f1 = min(f0 + A.K, A.nf);
    const long base = (long)(a + G) * A.s1 + (long)(b + G) * A.s2;   // cell index along d = -G
    // cells f0-3 .. f1+1 are read, faces f0 .. f1-1 written
    if (!in_bounds(base + (long)(f0 - 3 + G) * A.sd, A.np) || !in_bounds(base + (long)(f1 + 1 + G) * A.sd, A.np) ||
        !in_bounds(((long)f0 * (A.n2 + 4) + (b + 2)) * A.e1p + (a + 2), A.nfq) ||
        !in_bounds(((long)(f1 - 1) * (A.n2 + 4) + (b + 2)) * A.e1p + (a + 2), A.nfq))
        return;
    const float *pc[4] = {A.w + base, A.w + (long)A.cn * A.np + base, A.w + (long)A.c1 * A.np + base,
                          A.w + (long)A.c2 * A.np + base};
    float2 *fq = reinterpret_cast<float2 *>(A.fq);   // component pairs (see tile_t1_pass_f2)
    // cells f0-3 .. f0 start the march at cell f0-1, cell f0+1 completes it
    WenoWindow w[2];
    f2 Qprev[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        f2 v[5], l;
#pragma unroll
        for (int k = 0; k < 5; ++k) {
            const long o = (long)(f0 - 3 + k + G) * A.sd;
            v[k] = f2(__ldg(pc[2 * q] + o), __ldg(pc[2 * q + 1] + o));
        }
        w[q].start(v[0], v[1], v[2], v[3]);
        w[q].push(v[4], Qprev[q], l);
    }
    // the cell entering the march, loaded one face ahead
    float nxt[4];
#pragma unroll
    for (int v = 0; v < 4; ++v) nxt[v] = __ldg(pc[v] + (long)(f0 + 2 + G) * A.sd);
#pragma unroll 2
    for (int f = f0; f < f1; ++f) {
        const f2 s(A.ihf[f] * float(1.0 / 12.0));
        const long o = ((long)f * (A.n2 + 4) + (b + 2)) * A.e1p + (a + 2);
        const f2 e[2] = {f2(nxt[0], nxt[1]), f2(nxt[2], nxt[3])};
        if (f + 1 < f1) {
            // cell f + 3 <= nf + 1 = n + 2: inside the ghost layers
#pragma unroll
            for (int v = 0; v < 4; ++v) nxt[v] = __ldg(pc[v] + (long)(f + 3 + G) * A.sd);
        }
        f2 Ql[2], Qr[2], Q0[2];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            fq[(2 + q) * A.nfq + o] = (w[q].slope12() * s).v;
            Ql[q] = Qprev[q];
            w[q].push(e[q], Qprev[q], Qr[q]);
        }
        face_equilibrium2(A.ph, Ql, Qr, Q0);
#pragma unroll
        for (int q = 0; q < 2; ++q) fq[q * A.nfq + o] = Q0[q].v;
    }
}

// face_eq_march for FP64 grids in double-single arithmetic on packed
// pairs: WENO5 of the components paired as (rho, m_n) and (m_t1, m_t2), the
// half-space terms of the left and right states as one pair, the normal
// slopes paired like the components.
__device__ __forceinline__ void face_eq_ds2(const FaceEqArgs<double, dsf> &A, int2 blk)
{
    int a, b;
    const int f0 = blk.y * A.K;
    if (!face_position((unsigned)blk.x * blockDim.x + threadIdx.x, A.n1, A.n2, a, b) || f0 >= A.nf) return;
    const int f1 = min(f0 + A.K, A.nf);
    const long base = (long)(a + G) * A.s1 + (long)(b + G) * A.s2;   // cell index along d = -G
    // cells f0-3 .. f1+1 are read, faces f0 .. f1-1 written
    if (!in_bounds(base + (long)(f0 - 3 + G) * A.sd, A.np) || !in_bounds(base + (long)(f1 + 1 + G) * A.sd, A.np) ||
        !in_bounds(((long)f0 * (A.n2 + 4) + (b + 2)) * A.e1p + (a + 2), A.nfq) ||
        !in_bounds(((long)(f1 - 1) * (A.n2 + 4) + (b + 2)) * A.e1p + (a + 2), A.nfq))
        return;
    const double *pc[4] = {A.w + base, A.w + (long)A.cn * A.np + base, A.w + (long)A.c1 * A.np + base,
                           A.w + (long)A.c2 * A.np + base};
    // cells f0-3 .. f0 start the march at cell f0-1, cell f0+1 completes it
    WenoMarch<dsf2> w[2];
    dsf2 Qprev[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        dsf2 v[5], l;
#pragma unroll
        for (int k = 0; k < 5; ++k) {
            const long o = (long)(f0 - 3 + k + G) * A.sd;
            v[k] = dsf2(to_ds(__ldg(pc[2 * q] + o)), to_ds(__ldg(pc[2 * q + 1] + o)));
        }
        w[q].start(v[0], v[1], v[2], v[3]);
        w[q].push(v[4], Qprev[q], l);
    }
    // the cell entering the march, loaded one face ahead
    double nxt[4];
#pragma unroll
    for (int v = 0; v < 4; ++v) nxt[v] = __ldg(pc[v] + (long)(f0 + 2 + G) * A.sd);
    for (int f = f0; f < f1; ++f) {
        const dsf2 ihf(to_ds(A.ihf[f]));
        const long o = ((long)f * (A.n2 + 4) + (b + 2)) * A.e1p + (a + 2);
        double e[4];
#pragma unroll
        for (int v = 0; v < 4; ++v) e[v] = nxt[v];
        if (f + 1 < f1) {
            // cell f + 3 <= nf + 1 = n + 2: inside the ghost layers
#pragma unroll
            for (int v = 0; v < 4; ++v) nxt[v] = __ldg(pc[v] + (long)(f + 3 + G) * A.sd);
        }
        dsf2 Ql[2], Qr[2], Q0[2];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const dsf2 dq = w[q].slope() * ihf;
            A.fq[(4 + 2 * q) * A.nfq + o] = dq.lane(0);
            A.fq[(5 + 2 * q) * A.nfq + o] = dq.lane(1);
            Ql[q] = Qprev[q];
            w[q].push(dsf2(to_ds(e[2 * q]), to_ds(e[2 * q + 1])), Qprev[q], Qr[q]);
        }
        face_equilibrium_ds2(A.ph, Ql, Qr, Q0);
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            A.fq[(2 * q) * A.nfq + o] = Q0[q].lane(0);
            A.fq[(2 * q + 1) * A.nfq + o] = Q0[q].lane(1);
        }
    }
}

// Blocks of a face plane with `threads` threads (FP32 x faces: 4 segments a
// warp, a quarter of the positions).
inline int face_eq_plane(bool seg, int threads, int n1, int n2)
{
    const int per = seg ? threads / 4 : threads;
    return (int)(((long)(n1 + 4) * (n2 + 4) + per - 1) / per);
}
// Blocks of the face-state launch of one direction, along the plane and the march.
template <typename R, typename C, bool ALL>
dim3 face_eq_blocks(const FaceEqArgs<R, C> &E, int d)
{
    const bool seg = std::is_same<C, float>::value && d == 0;
    const int k = seg ? 4 * E.K : E.K;
    return dim3(face_eq_plane(seg, kEqThreads<C, ALL>, E.n1, E.n2), (E.nf + k - 1) / k);
}

// Faces per thread of the marching face-state kernels, for the directions of
// one launch: of all lengths of the march that cut the faces into equal
// segments, the one with the least work on the busiest SM, K faces and about
// one to start the window for each of its blocks; fewer blocks than fit, and a
// last wave of fewer than kEqBusy, take as long as those. (Halving a fixed
// length until the launch had two blocks to an SM left 680 FP64 blocks of
// 128^3 on 152 SMs.) The x segments of FP32 grids are 4 or 8 faces: whole
// sectors, 4 of them a line; 9 faces, which fill the blocks better, took 0.39
// against 0.36 ms a step of 256x128x128. Face state of a step with this rule and
// face_position, before and now: FP64 128^3 8.94 -> 6.61 ms and 32^3 0.349 ->
// 0.181, double-single 96^3 1.41 -> 1.00. FP32C waits on its loads and takes the
// halved length as well: 1.82 and 1.82 ms on 384x256x256, 0.359 and 0.356 on
// 256x128x128, 0.207 and 0.214 on 128^3.
template <typename R, typename C, bool ALL>
void march_faces(FaceEqArgs<R, C> *E, const int *dir, int nd)
{
    constexpr bool F32 = std::is_same<C, float>::value;
    constexpr long fit = kEqBlocks<C, ALL>, busy = kEqBusy<C, ALL>;
    const int sms = sm_count();
    long best = -1;
    for (int K = 4; K <= 128; ++K) {
        long blocks = 0;
        int most = 0, k[3];
        for (int i = 0; i < nd; ++i) {
            const bool seg = F32 && dir[i] == 0;
            const int per = seg ? 4 : 1, Ks = seg ? (K < 8 ? 4 : 8) : K;
            const int S = (E[i].nf + per * Ks - 1) / (per * Ks);
            k[i] = seg ? Ks : (E[i].nf + S - 1) / S;
            blocks += (long)face_eq_plane(seg, kEqThreads<C, ALL>, E[i].n1, E[i].n2) * S;
            most = std::max(most, k[i]);
        }
        const long m = (blocks + sms - 1) / sms, last = m % fit;   // of the busiest SM, in its last wave
        const long waves = m <= fit ? fit : m - last + (last ? std::max(last, busy) : 0);
        const long cost = waves * (most + (F32 && !ALL && dir[0] == 0 ? 2 : 1));
        if (best < 0 || cost < best) {
            best = cost;
            for (int i = 0; i < nd; ++i) E[i].K = k[i];
        }
    }
}

template <bool SEG>
__global__ void __launch_bounds__(kEqThreads<float, false>, kEqBlocks<float, false>)
    face_eq_f2_kernel(FaceEqArgs<float, float> A)
{
    face_eq_f2<SEG>(A, make_int2(blockIdx.x, blockIdx.y));
}
template <typename C>
__global__ void __launch_bounds__(kEqThreads<C, false>, kEqBlocks<C, false>)
    face_eq_kernel(const __grid_constant__ FaceEqArgs<double, C> A)
{
    const int2 blk = make_int2(blockIdx.x, blockIdx.y);
    if constexpr (std::is_same<C, dsf>::value)
        face_eq_ds2(A, blk);
    else
        face_eq_march(A, blk);
}

template <typename R, typename C>
void launch_face_eq(FaceEqArgs<R, C> E, int d, cudaStream_t stream)
{
    march_faces<R, C, false>(&E, &d, 1);
    const dim3 g = face_eq_blocks<R, C, false>(E, d);
    if constexpr (std::is_same<C, float>::value) {
        if (d == 0)
            face_eq_f2_kernel<true><<<g, kEqThreads<C, false>, 0, stream>>>(E);
        else
            face_eq_f2_kernel<false><<<g, kEqThreads<C, false>, 0, stream>>>(E);
    } else {
        face_eq_kernel<C><<<g, kEqThreads<C, false>, 0, stream>>>(E);
    }
}

// The face states of all three directions in one launch (small grids, whose
// three face boxes are kept apart): blocks of x, then y, then z.
template <typename R, typename C>
struct FaceEq3 {
    FaceEqArgs<R, C> d[3];
    int gx[3], first[4];   // blocks of a face plane of each direction, its first block
};
template <typename R, typename C>
__global__ void __launch_bounds__(kEqThreads<C, true>, kEqBlocks<C, true>)
    face_eq_all_kernel(const __grid_constant__ FaceEq3<R, C> E)
{
    int b = blockIdx.x;
    const int d = b < E.first[1] ? 0 : (b < E.first[2] ? 1 : 2);
    b -= E.first[d];
    const int2 blk = make_int2(b % E.gx[d], b / E.gx[d]);
    if constexpr (std::is_same<C, float>::value) {
        if (d == 0)
            face_eq_f2<true>(E.d[0], blk);
        else
            face_eq_f2<false>(E.d[d], blk);
    } else if constexpr (std::is_same<C, dsf>::value) {
        face_eq_ds2(E.d[d], blk);
    } else {
        face_eq_march(E.d[d], blk);
    }
}

// ------------------------------------------------------------- face flux --

template <typename R, typename C = R>
struct FluxArgs {
    Mid<R, C> *ff;   // 8 arrays of nff (0..3 F0, 4..7 F1, global components)
    long nff;
    void *gp;        // FP64 only, may be null: the 64 Gauss-point inputs per face (stride ngp)
    long ngp;
    int gp32;        // gp holds float (else double)
    const R *ih1, *ih2;  // inverse cell widths along t1, t2 (padded index)
    int n1, n2, nf;
    int gcomp[4];        // global component of local component 0..3
    Phys<C> ph;          // in the compute type
    Scalars *scal;
};

// The launch of ND directions: one (index 0), or all three of a small grid.
template <int ND>
struct FluxMaps {
    CUtensorMap d[ND];
};
template <typename R, typename C, int ND>
struct FluxLaunch {
    FluxArgs<R, C> A[ND];
    int L[ND];          // t2 rows per segment (march), unused by the tile kernel
    int first[ND + 1];  // first work item of each direction
};

// The face averages 1/4 sum of the Gauss-point fluxes: of F0, and of F1 from
// the sum of -F1 (gk_flux).
__device__ __forceinline__ double face_avg(double s) { return s * 0.25; }
__device__ __forceinline__ float face_avg(float s) { return s * 0.25f; }
__device__ __forceinline__ dsf face_avg(dsf s) { return scale_pow2(s, 0.25f); }
__device__ __forceinline__ double face_avg_neg(double s) { return s * -0.25; }
__device__ __forceinline__ float face_avg_neg(float s) { return s * -0.25f; }
__device__ __forceinline__ dsf face_avg_neg(dsf s) { return scale_pow2(s, -0.25f); }

// The t2 pass of component v at column (tx, ty) of the tile, t1 Gauss point
// m: values and t2 slopes of Q0, values of the t1 slopes and of the normal
// slope at the two t2 Gauss points -g, +g (k = 0, 1); the density's slopes
// negated, as gk_flux takes them.
template <int V>
__device__ __forceinline__ void t2_pass(const double *st, int m, const int ro[5], double q[2], double dn[2], double d1[2],
                                        double d2[2])
{
    using R = double;
    constexpr bool NEG = V == 0;
    const R *x = st + (V * 4 + m) * ST_ROWS;
    const R *y = st + (V * 4 + 2 + m) * ST_ROWS;
    const R *z = st + (16 + V * 2 + m) * ST_ROWS;
    tan_val_der<R, NEG>(x[ro[0]], x[ro[1]], x[ro[2]], x[ro[3]], x[ro[4]], q[0], q[1], d2[0], d2[1]);
    tan_val_direct<R, NEG>(y[ro[0]], y[ro[1]], y[ro[2]], y[ro[3]], y[ro[4]], d1[0], d1[1]);
    tan_val_direct<R, NEG>(z[ro[0]], z[ro[1]], z[ro[2]], z[ro[3]], z[ro[4]], dn[0], dn[1]);
}

// t2 pass at each t1 Gauss point m, then the flux at (m, -g), (m, +g): the
// sums of F0 and of -F1 over the 4 Gauss points of a face, whose 5 rows of t1
// results stand at st + ro[i].
// GP (the recorded steps of the adjoint) with gp set: the inputs of Gauss
// point g = 2m + n (Q0 with its density as rho; normal slope, t1 and t2
// slopes; 4 components each) go to gp[(16 g + k) ngp + face], as double or
// (gp32) rounded to float.
template <bool NEED_F0, bool GP = false>
__device__ __forceinline__ void tile_gauss_flux(const FluxPhys<double> &ph, const double *st, const int ro[5], double ih1,
                                                double ih2, double acc0[4], double acc1[4], void *gp = nullptr,
                                                int gp32 = 0, long ngp = 0, long face = 0)
{
#pragma unroll
    for (int v = 0; v < 4; ++v) acc0[v] = acc1[v] = 0.0;
#pragma unroll
    for (int m = 0; m < 2; ++m) {
        double t[4][4][2];   // [Q0, normal slope, t1 slope, t2 slope][component][t2 Gauss point]
        t2_pass<0>(st, m, ro, t[0][0], t[1][0], t[2][0], t[3][0]);
        t2_pass<1>(st, m, ro, t[0][1], t[1][1], t[2][1], t[3][1]);
        t2_pass<2>(st, m, ro, t[0][2], t[1][2], t[2][2], t[3][2]);
        t2_pass<3>(st, m, ro, t[0][3], t[1][3], t[2][3], t[3][3]);
        if constexpr (GP) {
            if (gp) {
#pragma unroll
                for (int nn = 0; nn < 2; ++nn) {
                    const long o = (long)(16 * (2 * m + nn)) * ngp + face;
#pragma unroll
                    for (int k = 0; k < 16; ++k) {
                        // the density's slopes are recorded unnegated
                        const double x = k >= 4 && k % 4 == 0 ? -t[k / 4][k % 4][nn] : t[k / 4][k % 4][nn];
                        if (!gp32)
                            ((double *)gp)[o + k * ngp] = x;
                        else
                            ((float *)gp)[o + k * ngp] = (float)x;
                    }
                }
            }
        }
#pragma unroll
        for (int nn = 0; nn < 2; ++nn) {
            double q[4][4], F0[4], nF1[4];
#pragma unroll
            for (int k = 0; k < 4; ++k)
#pragma unroll
                for (int v = 0; v < 4; ++v) q[k][v] = t[k][v][nn];
            gk_flux<double, NEED_F0>(ph, q[0], q[1], q[2], q[3], ih1, ih2, F0, nF1);
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                if (NEED_F0) acc0[v] += F0[v];
                acc1[v] += nF1[v];
            }
        }
    }
}

// The flux of face (tx, ty) of a 32 x 8 tile in FP32 (the fused z kernel): the
// t2 pass, then the two t2 Gauss points of each t1 Gauss point as one packed
// evaluation; the sums of F0 and -F1 over the 4 Gauss points, in the order of
// march_face (the same bits).
template <bool NEED_F0>
__device__ __forceinline__ void tile_gauss_flux_f2(const FluxPhys<f2> &ph, const float2 *st, int tx, int ty, float ih1,
                                                   float ih2, float acc0[4], float acc1[4])
{
#pragma unroll
    for (int m = 0; m < 2; ++m) {
        f2 Qv[4], Dn[4], D1[4], D2[4];   // the two t2 Gauss points -g, +g in the lanes
        t2_pass_f2<true>(st, m, tx, ty, Qv, Dn, D1, D2);
        f2 F0[4], F1[4];
        gk_flux<f2, NEED_F0>(ph, Qv, Dn, D1, D2, f2(ih1), f2(ih2), F0, F1);
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            if (NEED_F0) {
                const float s = F0[v].v.x + F0[v].v.y;
                acc0[v] = m == 0 ? s : acc0[v] + s;
            }
            const float s = F1[v].v.x + F1[v].v.y;
            acc1[v] = m == 0 ? s : acc1[v] + s;
        }
    }
}

// tile_gauss_flux for double-single arithmetic (no Gauss-point output): the
// same t2 pass, the flux at the two t2 Gauss points of each t1 Gauss point
// as one evaluation on packed double-single pairs.
template <int V>
__device__ __forceinline__ void t2_pass_ds2(const dsf *st, int m, const int ro[5], dsf2 &q, dsf2 &dn, dsf2 &d1, dsf2 &d2)
{
    constexpr bool NEG = V == 0;
    const dsf *x = st + (V * 4 + m) * ST_ROWS;
    const dsf *y = st + (V * 4 + 2 + m) * ST_ROWS;
    const dsf *z = st + (16 + V * 2 + m) * ST_ROWS;
    dsf p[5], D[4];
#pragma unroll
    for (int i = 0; i < 5; ++i) p[i] = x[ro[i]];
#pragma unroll
    for (int i = 0; i < 4; ++i) D[i] = p[i + 1] - p[i];
    ds_val_der<NEG>(p[2], D, q, d2);
#pragma unroll
    for (int i = 0; i < 5; ++i) p[i] = y[ro[i]];
    d1 = ds_val_direct<NEG>(p);
#pragma unroll
    for (int i = 0; i < 5; ++i) p[i] = z[ro[i]];
    dn = ds_val_direct<NEG>(p);
}
template <bool NEED_F0>
__device__ __forceinline__ void tile_gauss_flux_ds2(const FluxPhys<dsf2> &ph, const dsf *st, const int ro[5], dsf ih1,
                                                    dsf ih2, dsf acc0[4], dsf acc1[4])
{
    dsf2 s0[4], s1[4];   // the t2 Gauss points -g, +g in the lanes
#pragma unroll
    for (int m = 0; m < 2; ++m) {
        dsf2 Qv[4], Dn[4], D1[4], D2[4];
        t2_pass_ds2<0>(st, m, ro, Qv[0], Dn[0], D1[0], D2[0]);
        t2_pass_ds2<1>(st, m, ro, Qv[1], Dn[1], D1[1], D2[1]);
        t2_pass_ds2<2>(st, m, ro, Qv[2], Dn[2], D1[2], D2[2]);
        t2_pass_ds2<3>(st, m, ro, Qv[3], Dn[3], D1[3], D2[3]);
        dsf2 F0[4], F1[4];
        gk_flux<dsf2, NEED_F0>(ph, Qv, Dn, D1, D2, dsf2(ih1), dsf2(ih2), F0, F1);
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            if (NEED_F0) s0[v] = m == 0 ? F0[v] : s0[v] + F0[v];
            s1[v] = m == 0 ? F1[v] : s1[v] + F1[v];
        }
    }
#pragma unroll
    for (int v = 0; v < 4; ++v) {
        if (NEED_F0) acc0[v] = s0[v].lane(0) + s0[v].lane(1);
        acc1[v] = s1[v].lane(0) + s1[v].lane(1);
    }
}

// Persistent: each block takes a run of consecutive tiles, t2 fastest; the face
// box of a tile is dead once its t1 pass is in shared memory, so the next
// tile's face box is fetched by TMA into the same buffer while the Gauss
// points of the current one are computed (one buffer: more blocks per SM).
// A tile that follows its neighbour along t2 finds its first 4 rows of t1
// results there (the rows are a ring of SQ_H, turned by TY a tile) and passes
// only the 8 others, a third less of the t1 operations in kernels that the FP64
// pipe (85 % busy) or the issue of double-single bounds: x and y fluxes of a step
// of 128^3 FP64 11.2 -> 10.4 ms, of 96^3 double-single 1.22 -> 1.13 ms.
struct TilePos {
    int t, d, f, a0, b0;   // tile, direction, face plane, first face along t1 and t2
};

template <typename R, typename C, bool NEED_F0, bool GP, int ND>
__global__ void __launch_bounds__(256, std::is_same<C, dsf>::value ? 2 : 1)
    face_flux_kernel(const __grid_constant__ FluxMaps<ND> maps, FluxLaunch<R, C, ND> F)
{
    static_assert(sizeof(C) == sizeof(R), "the t1-pass rows share the storage size");
    using M = Mid<R, C>;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    M *sq = reinterpret_cast<M *>(smem_raw);             // face-box tile (SQ_N)
    C *st = reinterpret_cast<C *>(sq + SQ_N);
    uint64_t *bar = reinterpret_cast<uint64_t *>(st + ST_N);
    const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * TX + tx;
    // runs of equal length, the first blocks (one to an SM) one tile more
    const int run = F.first[ND] / (int)gridDim.x, more = F.first[ND] % (int)gridDim.x, blk = blockIdx.x;
    const int t0 = blk * run + min(blk, more), tend = t0 + run + (blk < more);
    const uint32_t bytes = (uint32_t)(SQ_N * sizeof(R));
    auto tile = [&](int t) {
        TilePos p;
        p.t = t;
        p.d = ND == 1 ? 0 : (t < F.first[1] ? 0 : (t < F.first[ND - 1] ? 1 : ND - 1));
        const FluxArgs<R, C> &A = F.A[p.d];
        const int NA = (A.n1 + TX - 1) / TX, NB = (A.n2 + TY - 1) / TY;
        const int l = t - F.first[p.d], r = l / NB;
        p.b0 = (l - r * NB) * TY;
        p.f = r / NA;
        p.a0 = (r - p.f * NA) * TX;
        return p;
    };
    auto load = [&](const TilePos &p) {
        if (tid == 0 && p.t < tend)
            tma_load_tile(&maps.d[p.d], sq, &bar[0], p.a0, p.b0, p.f, bytes);
    };
    if (tid == 0) {
        mbar_init(&bar[0], 1);
        mbar_fence_init();
    }
    __syncthreads();
    TilePos cur = tile(t0);
    load(cur);
    int off = 0;   // ring row of the tile's first row
    for (int k = 0; cur.t < tend; ++k) {
        const TilePos nxt = tile(cur.t + 1);
        const FluxArgs<R, C> &A = F.A[cur.d];
        const bool ok = mbar_wait(&bar[0], (uint32_t)(k & 1));
        if (__syncthreads_or(!ok)) {
            if (tid == 0) atomicOr(&A.scal->flags, FLAG_TIMEOUT);
            return;
        }
        const bool next_to = k > 0 && cur.b0 > 0;   // the last tile's neighbour
        off = next_to ? ring_row(off + TY) : 0;
        tile_t1_pass(sq, st, tid, next_to ? TY : SQ_H, off);
        __syncthreads();
        // the face box is free: fetch the next tile's while this one's Gauss
        // points are computed
        if (tid == 0) fence_proxy_async();
        load(nxt);

        const int a = cur.a0 + tx, b = cur.b0 + ty;
        if (a < A.n1 && b < A.n2) {
            const C ih1 = cvt<C>(__ldg(A.ih1 + a + G)), ih2 = cvt<C>(__ldg(A.ih2 + b + G));
            C acc0[4], acc1[4];
            int ro[5];
#pragma unroll
            for (int i = 0; i < 5; ++i) ro[i] = ring_row(ty + i + off) * TX + tx;
            const long o = ((long)cur.f * A.n2 + b) * A.n1 + a;
            if constexpr (std::is_same<C, dsf>::value)
                tile_gauss_flux_ds2<NEED_F0>(flux_phys_ds2(A.ph), st, ro, ih1, ih2, acc0, acc1);
            else
                tile_gauss_flux<NEED_F0, GP>(flux_phys(A.ph), st, ro, ih1, ih2, acc0, acc1, A.gp, A.gp32, A.ngp,
                                             o);
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                if (!in_bounds(o, A.nff)) break;
                if (NEED_F0) A.ff[A.gcomp[v] * A.nff + o] = face_avg(acc0[v]);
                A.ff[(4 + A.gcomp[v]) * A.nff + o] = face_avg_neg(acc1[v]);
            }
        }
        cur = nxt;
        __syncthreads();   // st and this buffer are free again
    }
}

// ---- FP32C face fluxes: a march along t2 in registers ----
//
// A warp owns 32 faces along t1 and walks a segment of t2 rows of one face
// plane. Per row it forms the t1 pass of the 8 face-box values at both t1
// Gauss points (the lanes of a pair) and keeps the last 5 rows of the 24
// results in registers; every row then completes the t2 stencil of the face
// two rows back, whose flux is evaluated at both t1 Gauss points at once. The
// face box arrives by TMA, 5 rows (all components) at a time, into the warp's
// own two buffers: no block barrier, and the t1 rows never go through shared
// memory. The tile kernel that this replaces (32 x 16 faces, t1 rows in shared
// memory) was held by shared-memory traffic and issue: 528 B and 718
// instructions a face (stage 2) against 200 B here, and it redid the t1 pass
// of 4 rows per 16 (here per segment).
constexpr int RB = 5;                                  // rows per TMA box, and of the register window
constexpr int kMarchStage = 4 * RB * 2 * SQ_W;         // floats of one box: 4 component pairs x 5 rows x 36 columns
constexpr int kMarchWarps = 8;                         // warps per block at most
constexpr size_t march_smem_bytes(int warps)
{
    return (size_t)warps * (2 * kMarchStage * sizeof(float) + 2 * sizeof(uint64_t));
}

struct MarchWin {
    f2 v[4][RB], d[4][RB], n[4][RB];   // Q0, its t1 slope, the normal slope: [component][row slot], t1 Gauss points
};

// t1 pass of row `j` of a box (columns lane .. lane + 4) into window slot J.
template <int J>
__device__ __forceinline__ void march_row(const float2 *box, int lane, MarchWin &w)
{
    constexpr float o1 = float(0.20046884346862007), o2 = float(0.028065638085606807);
    constexpr float e1 = float(0.41697519441472974), e2 = float(0.032075014954979206);
    constexpr float w0 = float(-1.0 / 4320.0 + 0.028065638085606807), w1 = float(1.0 / 1080.0 - 0.20046884346862007);
    constexpr float w2 = float(719.0 / 720.0);
    constexpr float w3 = float(1.0 / 1080.0 + 0.20046884346862007), w4 = float(-1.0 / 4320.0 - 0.028065638085606807);
#pragma unroll
    for (int P = 0; P < 2; ++P) {
        float2 x[5];
#pragma unroll
        for (int k = 0; k < 5; ++k) x[k] = box[(P * RB + J) * SQ_W + lane + k];
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            float q[5];
#pragma unroll
            for (int k = 0; k < 5; ++k) q[k] = c ? x[k].y : x[k].x;
            const float d1 = __fmaf_rn(q[2], -2.0f, __fadd_rn(q[3], q[1]));
            const float d2 = __fmaf_rn(q[2], -2.0f, __fadd_rn(q[4], q[0]));
            const float a1 = __fsub_rn(q[3], q[1]), a2 = __fsub_rn(q[4], q[0]);
            // tan_val_der with the two Gauss points in the lanes
            const float E = __fmaf_rn(d1, float(1.0 / 1080.0), __fmaf_rn(d2, float(-1.0 / 4320.0), q[2]));
            const float O = __fmaf_rn(a1, o1, __fmul_rn(a2, -o2));
            const float Do = __fmaf_rn(a1, float(2.0 / 3.0), __fmul_rn(a2, float(-1.0 / 12.0)));
            const float De = __fmaf_rn(d1, e1, __fmul_rn(d2, -e2));
            w.v[2 * P + c][J] = fma(f2(O), f2(-1.0f, 1.0f), f2(E));
            w.d[2 * P + c][J] = fma(f2(De), f2(-1.0f, 1.0f), f2(Do));
        }
#pragma unroll
        for (int k = 0; k < 5; ++k) x[k] = box[((2 + P) * RB + J) * SQ_W + lane + k];
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            float q[5];
#pragma unroll
            for (int k = 0; k < 5; ++k) q[k] = c ? x[k].y : x[k].x;
            w.n[2 * P + c][J] = fma(f2(q[4]), f2(w0, w4), fma(f2(q[3]), f2(w1, w3),
                                fma(f2(q[2]), f2(w2, w2), fma(f2(q[1]), f2(w3, w1), f2(q[0]) * f2(w4, w0)))));
        }
    }
}

// t2 pass over the window whose newest row is in slot J, and the flux of the
// face two rows back: the sums of F0 and -F1 over its 4 Gauss points.
template <int J, bool NEED_F0>
__device__ __forceinline__ void march_face(const FluxPhys<f2> &ph, const MarchWin &w, f2 ih1, f2 ih2, float acc0[4],
                                           float acc1[4])
{
    constexpr int r0 = (J + 1) % RB, r1 = (J + 2) % RB, r2 = (J + 3) % RB, r3 = (J + 4) % RB, r4 = J;
    f2 q[2][4], dn[2][4], d1[2][4], d2[2][4];   // [t2 Gauss point][component]
#pragma unroll
    for (int v = 0; v < 4; ++v) {
        if (v == 0) {
            tan_val_der<f2, true>(w.v[v][r0], w.v[v][r1], w.v[v][r2], w.v[v][r3], w.v[v][r4], q[0][v], q[1][v], d2[0][v],
                                  d2[1][v]);
            tan_val_direct<f2, true>(w.d[v][r0], w.d[v][r1], w.d[v][r2], w.d[v][r3], w.d[v][r4], d1[0][v], d1[1][v]);
            tan_val_direct<f2, true>(w.n[v][r0], w.n[v][r1], w.n[v][r2], w.n[v][r3], w.n[v][r4], dn[0][v], dn[1][v]);
        } else {
            tan_val_der<f2>(w.v[v][r0], w.v[v][r1], w.v[v][r2], w.v[v][r3], w.v[v][r4], q[0][v], q[1][v], d2[0][v],
                            d2[1][v]);
            tan_val_direct<f2>(w.d[v][r0], w.d[v][r1], w.d[v][r2], w.d[v][r3], w.d[v][r4], d1[0][v], d1[1][v]);
            tan_val_direct<f2>(w.n[v][r0], w.n[v][r1], w.n[v][r2], w.n[v][r3], w.n[v][r4], dn[0][v], dn[1][v]);
        }
    }
    f2 s0[4], s1[4];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        f2 F0[4], F1[4];
        gk_flux<f2, NEED_F0>(ph, q[k], dn[k], d1[k], d2[k], ih1, ih2, F0, F1);
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            if (NEED_F0) s0[v] = k == 0 ? F0[v] : s0[v] + F0[v];
            s1[v] = k == 0 ? F1[v] : s1[v] + F1[v];
        }
    }
#pragma unroll
    for (int v = 0; v < 4; ++v) {
        if (NEED_F0) acc0[v] = s0[v].v.x + s0[v].v.y;
        acc1[v] = s1[v].v.x + s1[v].v.y;
    }
}

// Position of a warp in its work: item (direction, face plane, t2 segment, t1
// tile), box k of the item's n boxes; a0, b0 its first face along t1 and t2,
// be the end.
struct MarchPos {
    int it, d, k, n, f, a0, b0, be;
};

template <bool NEED_F0, int ND>
__global__ void __launch_bounds__(32 * kMarchWarps, 1)
    face_flux_march_kernel(const __grid_constant__ FluxMaps<ND> maps, FluxLaunch<float, float, ND> F)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    float *buf = reinterpret_cast<float *>(smem_raw) + warp * 2 * kMarchStage;
    uint64_t *bar = reinterpret_cast<uint64_t *>(smem_raw + (size_t)nw * 2 * kMarchStage * sizeof(float)) + 2 * warp;
    const int nitems = F.first[ND], step = gridDim.x * nw;
    auto item = [&](int it) {
        MarchPos p;
        p.d = ND == 1 ? 0 : (it < F.first[1] ? 0 : (it < F.first[ND - 1] ? 1 : ND - 1));
        const FluxArgs<float, float> &A = F.A[p.d];
        const int L = F.L[p.d], NA = (A.n1 + TX - 1) / TX, NS = (A.n2 + L - 1) / L;
        const int l = it - F.first[p.d], r = l / NA, sg = r % NS;
        p.it = it;
        p.k = 0;
        p.f = r / NS;
        p.a0 = (l - r * NA) * TX;
        p.b0 = sg * L;
        p.be = min(p.b0 + L, A.n2);
        p.n = (p.be - p.b0 + 4 + RB - 1) / RB;
        return p;
    };
    auto load = [&](const MarchPos &p, int s) {
        if (lane == 0 && p.it < nitems)
            tma_load_tile(&maps.d[p.d], buf + s * kMarchStage, &bar[s], 2 * p.a0, p.b0 + p.k * RB, p.f,
                          (uint32_t)(kMarchStage * sizeof(float)));
    };
    auto next = [&](const MarchPos &p) {
        MarchPos q = p;
        if (++q.k >= q.n) q = item(p.it + step);
        return q;
    };
    if (lane == 0) {
        mbar_init(&bar[0], 1);
        mbar_init(&bar[1], 1);
        mbar_fence_init();
    }
    __syncwarp();
    MarchPos cur = item(blockIdx.x * nw + warp), ahead = cur;
    load(ahead, 0);
    if (ahead.it < nitems) ahead = next(ahead);
    load(ahead, 1);
    const FluxPhys<f2> ph = flux_phys_f2(F.A[0].ph);
    MarchWin w;
    for (int cnt = 0; cur.it < nitems; ++cnt) {
        const FluxArgs<float, float> &A = F.A[cur.d];
        const int s = cnt & 1;
        const int a = cur.a0 + lane, b = cur.b0 + cur.k * RB - 4;   // face that the box's first row completes
        const bool in = a < A.n1;
        const f2 ih1(in ? __ldg(A.ih1 + a + G) : 0.0f);
        if (__any_sync(0xffffffffu, !mbar_wait(&bar[s], (uint32_t)((cnt >> 1) & 1)))) {
            if (lane == 0) atomicOr(&A.scal->flags, FLAG_TIMEOUT);
            mbar_wait(&bar[s ^ 1], (uint32_t)(((cnt + 1) >> 1) & 1));   // the copy in flight, with the same limit
            return;
        }
        const float2 *box = reinterpret_cast<const float2 *>(buf + s * kMarchStage);
        auto row = [&](auto jc) {
            constexpr int J = decltype(jc)::value;
            march_row<J>(box, lane, w);
            const int bf = b + J;
            if (bf >= cur.b0 && bf < cur.be) {
                float acc0[4], acc1[4];
                march_face<J, NEED_F0>(ph, w, ih1, f2(__ldg(A.ih2 + bf + G)), acc0, acc1);
                const long o = ((long)cur.f * A.n2 + bf) * A.n1 + a;
                if (in && in_bounds(o, A.nff)) {
#pragma unroll
                    for (int v = 0; v < 4; ++v) {
                        if (NEED_F0) A.ff[A.gcomp[v] * A.nff + o] = face_avg(acc0[v]);
                        A.ff[(4 + A.gcomp[v]) * A.nff + o] = face_avg_neg(acc1[v]);
                    }
                }
            }
        };
        row(std::integral_constant<int, 0>{});
        row(std::integral_constant<int, 1>{});
        row(std::integral_constant<int, 2>{});
        row(std::integral_constant<int, 3>{});
        row(std::integral_constant<int, 4>{});
        // the box is read: fetch the one after the next into it
        cur = next(cur);
        if (ahead.it < nitems) ahead = next(ahead);
        __syncwarp();
        fence_proxy_async();
        load(ahead, s);
    }
}

// Rows per march segment: S segments of L = ceil(n2 / S) rows; the busiest
// warp's rows are least (the priming rows of a segment cost their t1 pass,
// about one face together), over up to 64 segments. On large grids this picks
// long segments with even rounds of the warps (128^3: 19 rows, 3612 items for
// 3 x 1216 warps), in the launch of all directions of 32^3, with a third of the
// warps for each, 3 rows (363 items for 405 warps).
int march_segment(int na, int nf, int n2, int warps)
{
    double best = -1.0;
    int bestL = n2;
    for (int S = 1; S <= 64 && S <= n2; ++S) {
        const int L = (n2 + S - 1) / S, Sa = (n2 + L - 1) / L;
        const long items = (long)na * nf * Sa;
        const double cost = (double)((items + warps - 1) / warps) * (L + 1.0);
        if (best < 0.0 || cost < best) {
            best = cost;
            bestL = L;
        }
    }
    return bestL;
}

// ------------------------------------------------- z flux + stage update --

constexpr int kMaxPrepBoxes = 8;   // forcing boxes the fused prep can leave out
constexpr int kUpdZ = 4;           // planes per block of the stage update

template <typename R, typename M = R>
struct UpdArgs {
    const M *ffx, *ffy, *ffz;     // face fluxes of the x, y and z directions (8 arrays each; no z in the fused kernel)
    long nffx, nffy, nffz;
    const R *ihx, *ihy, *ihz;     // inverse cell widths (padded index)
    int nx, ny, nz, P0, P1;
    long np;
    const void *w0;   // stage 1: state (FP64 W / FP32C hi,lo)
    void *wk1;        // stage 1 output W* (R)
    void *pbuf;       // P
    void *state;      // stage 2 output
    R off;
    R fb[3];
    // stage 2, optional: the next step's prep (FP32C: the FP32 input into
    // wk0n; max |U|^2 over the cells outside the forcing boxes into scal)
    int prep;
    float *wk0n;
    int nbox;
    int box[kMaxPrepBoxes][3][2];
    int advance;      // stage 2: t += dt (the last launch of a step without forcing)
    Scalars *scal;
};

__device__ __forceinline__ void add_comp(float &hi, float &lo, float d)
{
    // error-free two-sum of hi + d, then renormalise (hi, lo + err)
    const float s = hi + d;
    const float bp = s - hi;
    const float e = (hi - (s - bp)) + (d - bp);
    const float l = lo + e;
    const float h2 = s + l;
    lo = l - (h2 - s);
    hi = h2;
}

// Stage update of one cell from the differences of its face fluxes along x,
// y, z (high minus low face, global components; entries 0..3 hold F0, used
// in stage 1 only, entries 4..7 hold F1):
//   L = -sum_d dF0_d / h_d, Lt = -sum_d dF1_d / h_d,
//   stage 1: W* = W + dt/2 L + dt^2/8 Lt, P = W + dt L + dt^2/6 Lt,
//   stage 2: W = P + dt^2/3 Lt(W*) + dt f_body.
// Returns false when a written value is not finite (stage 2).
// Double-single arithmetic on an FP64 grid: the same update with the state
// split into double-single (exact to 48 bits) and the results composed back
// into FP64.
template <int STAGE>
__device__ __forceinline__ bool update_cell_ds(const UpdArgs<double, dsf> &A, long lin, double dt, const dsf dx[],
                                               const dsf dy[], const dsf dz[], dsf ihx, dsf ihy, dsf ihz,
                                               const double s0[4], double o0[4])
{
    const dsf h = to_ds(dt), h2 = h * h;
    bool bad = false;
#pragma unroll
    for (int v = 0; v < 4; ++v) {
        const dsf Lt = -(dx[4 + v] * ihx + dy[4 + v] * ihy + dz[4 + v] * ihz);
        const dsf w = to_ds(s0[v]);
        if (STAGE == 1) {
            const dsf L = -(dx[v] * ihx + dy[v] * ihy + dz[v] * ihz);
            ((double *)A.wk1)[v * A.np + lin] = to_double(w + (scale_pow2(h, 0.5f) * L + scale_pow2(h2, 0.125f) * Lt));
            ((double *)A.pbuf)[v * A.np + lin] = to_double(w + (h * L + (h2 / dsf(6.0)) * Lt));
        } else {
            dsf inc = (h2 / dsf(3.0)) * Lt;
            if (v > 0) inc += h * to_ds((double)A.fb[v - 1]);
            const double wn = to_double(w + inc);
            ((double *)A.state)[v * A.np + lin] = wn;
            bad |= !isfinite(wn);
            o0[v] = wn;
        }
    }
    return !bad;
}

template <typename R, int STAGE>
__device__ __forceinline__ bool update_cell(const UpdArgs<R> &A, long lin, double dt, const R dx[], const R dy[],
                                            const R dz[], R ihx, R ihy, R ihz, const R s0[4], const R s1[4],
                                            R o0[4], R o1[4])
{
    const R dtr = (R)dt;
    bool bad = false;
#pragma unroll
    for (int v = 0; v < 4; ++v) {
        const R Lt = -fma(dz[4 + v], ihz, fma(dy[4 + v], ihy, dx[4 + v] * ihx));
        if (STAGE == 1) {
            const R L = -fma(dz[v], ihz, fma(dy[v], ihy, dx[v] * ihx));
            if constexpr (std::is_same<R, double>::value) {
                const double w = s0[v];
                ((double *)A.wk1)[v * A.np + lin] = w + fma(0.5 * dt, L, 0.125 * dt * dt * Lt);
                ((double *)A.pbuf)[v * A.np + lin] = w + fma(dt, L, dt * dt / 6.0 * Lt);
            } else {
                float hi = s0[v], lo = s1[v];
                const float offv = v == 0 ? A.off : 0.0f;
                ((float *)A.wk1)[v * A.np + lin] = ((hi - offv) + lo) + fma(0.5f * dtr, L, 0.125f * dtr * dtr * Lt);
                add_comp(hi, lo, fma(dtr, L, dtr * dtr * (1.0f / 6.0f) * Lt));
                ((float *)A.pbuf)[v * A.np + lin] = hi;
                ((float *)A.pbuf)[(4 + v) * A.np + lin] = lo;
            }
        } else {
            if constexpr (std::is_same<R, double>::value) {
                double w = fma(dt * dt / 3.0, Lt, s0[v]);
                if (v > 0) w = fma(dt, (double)A.fb[v - 1], w);
                ((double *)A.state)[v * A.np + lin] = w;
                bad |= !isfinite(w);
                o0[v] = w;
            } else {
                float hi = s0[v], lo = s1[v];
                float inc = dtr * dtr * (1.0f / 3.0f) * Lt;
                if (v > 0) inc = fma(dtr, A.fb[v - 1], inc);
                add_comp(hi, lo, inc);
                ((float *)A.state)[v * A.np + lin] = hi;
                ((float *)A.state)[(4 + v) * A.np + lin] = lo;
                bad |= !isfinite(hi) || !isfinite(lo);
                o0[v] = hi;
                o1[v] = lo;
            }
        }
    }
    return !bad;
}

constexpr int SX_H = TX + 1, SX_W = TY + 1;   // x-face slab of a tile in shared memory (padded)

constexpr int SY_H = TY + 1;                  // y-face slab of a tile: the TY + 1 face rows of its cells

constexpr size_t flux_update_smem_bytes(int nc)
{
    return flux_smem_bytes<float>() + (size_t)nc * (SX_H * SX_W + SY_H * TX) * sizeof(float);
}

// z-direction face flux fused with the stage update (FP32C). Work items are
// (z segment, tile column) pairs, segment-major, taken round-robin by the
// persistent blocks, so that the blocks resident at one time march through
// the same z range of neighbouring columns (their tile halos and the x-face
// rows they read are shared through L2). Inside an item a block walks the
// segment's z-faces in order: F(f) - F(f-1) of the column is formed in
// registers and cell f-1 is updated at once; the first face of an item
// (the last face of the previous segment) only primes F. The x-face fluxes
// of the cell plane (x-fastest reads of a y-fastest array) and its y-face
// fluxes are copied asynchronously into shared slabs at the start of the
// tile (the x slab padded against bank conflicts), so that no register waits
// on them during the flux; the state of the thread's cell is loaded into
// registers (nothing reads it before the update).
struct ZWalk {
    int it, f, fe, f0;   // item, face, end face (exclusive), first (priming) face of the item
    int a0, b0;          // first cell of the item's tile column along x, y
};

// Item it: its segment and tile column, decoded once per item (not per face).
__device__ __forceinline__ ZWalk zwalk_item(int it, int ncol, int NA, int L, int nf)
{
    const int sgm = it / ncol, col = it - sgm * ncol, cb = col / NA;
    ZWalk z;
    z.it = it;
    z.f0 = sgm > 0 ? sgm * L - 1 : 0;
    z.f = z.f0;
    z.fe = min((sgm + 1) * L, nf);
    z.a0 = (col - cb * NA) * TX;
    z.b0 = cb * TY;
    return z;
}

template <int STAGE>
__global__ void __launch_bounds__(256, 2)
    flux_update_kernel(const __grid_constant__ CUtensorMap tmap, FluxArgs<float, float> A, UpdArgs<float> U, int seg)
{
    using R = float;
    using M = float;
    constexpr bool NEED_F0 = STAGE == 1;
    constexpr int NC = STAGE == 1 ? 8 : 4, C0 = STAGE == 1 ? 0 : 4;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    float2 *sq = reinterpret_cast<float2 *>(smem_raw);   // face-box tile (SQ_N floats), refilled after its t1 pass
    float2 *st = sq + SQ_N / 2;
    uint64_t *bar = reinterpret_cast<uint64_t *>(st + ST_N / 2);
    M *sx = reinterpret_cast<M *>(bar + 2);               // [NC][SX_H][SX_W]
    M *sy = sx + NC * SX_H * SX_W;                        // [NC][SY_H][TX]
    const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * TX + tx;
    const int NA = (A.n1 + TX - 1) / TX, NB = (A.n2 + TY - 1) / TY, nf = A.nf, L = seg;
    const int ncol = NA * NB, nitems = ncol * ((nf + L - 1) / L);
    if ((int)blockIdx.x >= nitems) return;
    const uint32_t bytes = (uint32_t)(SQ_N * sizeof(R));
    ZWalk cur = zwalk_item(blockIdx.x, ncol, NA, L, nf);
    if (tid == 0) {
        mbar_init(&bar[0], 1);
        mbar_fence_init();
    }
    __syncthreads();
    if (tid == 0) tma_load_tile(&tmap, sq, &bar[0], 2 * cur.a0, cur.b0, cur.f, bytes);
    const double dt = A.scal->dt;
    bool bad = false;
    float mx = 0.0f;   // stage 2 with prep: max |U|^2 of this thread's cells outside the forcing boxes
    M P0[4], P1[4];   // F0, F1 of the previous face of this column (storage type: the
                      // differences of neighbouring faces telescope exactly)
    for (int k = 0; cur.it < nitems; ++k) {
        ZWalk nxt = cur;
        if (++nxt.f >= nxt.fe) nxt = zwalk_item(cur.it + gridDim.x, ncol, NA, L, nf);
        const int f = cur.f, a0 = cur.a0, b0 = cur.b0;
        const bool upd = f > cur.f0;
        if (upd) {
            // x-face fluxes of cell plane z = f-1: faces a0 .. a0+32, rows b0 .. b0+7.
            // Thread: row y = b0 + (tid & 7), face a0 + tid/8 of every component;
            // the 8 threads with tid/8 = 0 also take face a0 + 32.
            const int yy = tid & 7, xf = tid >> 3;
            if (b0 + yy < U.ny) {
                const long sxf = (long)U.nz * U.ny;   // stride between x-faces
                const long g0 = ((long)(a0 + xf) * U.nz + (f - 1)) * U.ny + b0 + yy;
                const M *src = U.ffx + C0 * U.nffx + g0;
                if (a0 + xf <= U.nx && in_bounds(g0, U.nffx)) {
#pragma unroll
                    for (int c = 0; c < NC; ++c) cp_async(sx + (c * SX_H + xf) * SX_W + yy, src + c * U.nffx);
                }
                if (xf == 0 && a0 + 32 <= U.nx && in_bounds(g0 + 32 * sxf, U.nffx)) {
#pragma unroll
                    for (int c = 0; c < NC; ++c)
                        cp_async(sx + (c * SX_H + 32) * SX_W + yy, src + c * U.nffx + 32 * sxf);
                }
            }
            // y-face fluxes of the plane: faces b0 .. b0+8 along y, columns a0 .. a0+31.
            // Thread: column a0 + tx, face row ty of every component; face row 8 of
            // component ty.
            if (a0 + tx < U.nx) {
                const long g1 = ((long)(b0 + ty) * U.nz + (f - 1)) * U.nx + a0 + tx;
                const M *src = U.ffy + C0 * U.nffy + g1;
                if (b0 + ty <= U.ny && in_bounds(g1, U.nffy)) {
#pragma unroll
                    for (int c = 0; c < NC; ++c) cp_async(sy + (c * SY_H + ty) * TX + tx, src + c * U.nffy);
                }
                const long g8 = g1 + (long)(TY - ty) * U.nz * U.nx;   // face row b0 + 8
                if (ty < NC && b0 + TY <= U.ny && in_bounds(g8, U.nffy))
                    cp_async(sy + (ty * SY_H + TY) * TX + tx, U.ffy + (C0 + ty) * U.nffy + g8);
            }
            cp_async_commit();
        }
        // the state of this thread's cell, loaded now so that it arrives
        // during the flux computation
        const int a = a0 + tx, b = b0 + ty;
        const bool in = a < A.n1 && b < A.n2;
        // inverse widths (x, y of the flux and the update; z of the update),
        // loaded with the prefetch so that their latency overlaps it
        R ih1 = R(0), ih2 = R(0), ihz = R(0);
        if (in) {
            ih1 = __ldg(A.ih1 + a + G);
            ih2 = __ldg(A.ih2 + b + G);
            if (upd) ihz = __ldg(U.ihz + f - 1 + G);
        }
        R s0[4], s1[4];
        long lin = 0;
        bool cell_ok = true;
        if (upd && in) {
            const int z = f - 1;
            lin = (long)(a + G) + (long)U.P0 * ((long)(b + G) + (long)U.P1 * (z + G));
            cell_ok = in_bounds(lin, U.np);
            if (cell_ok) {
                const R *src = (const R *)(STAGE == 1 ? U.w0 : U.pbuf);
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                    s0[v] = __ldg(src + v * U.np + lin);
                    s1[v] = __ldg(src + (4 + v) * U.np + lin);
                }
            }
        }
        const bool ok = mbar_wait(&bar[0], (uint32_t)(k & 1));
        if (__syncthreads_or(!ok)) {
            cp_async_wait_all();
            if (tid == 0) atomicOr(&A.scal->flags, FLAG_TIMEOUT);
            __syncthreads();
            return;
        }
        tile_t1_pass_f2(sq, st, tid);
        __syncthreads();
        // the face box is free: fetch the next tile's during this one's flux
        if (tid == 0 && nxt.it < nitems) {
            fence_proxy_async();
            tma_load_tile(&tmap, sq, &bar[0], 2 * nxt.a0, nxt.b0, nxt.f, bytes);
        }

        M F0[4], F1[4];
        if (in) {
            float G0[4], G1[4];
            tile_gauss_flux_f2<NEED_F0>(flux_phys_f2(A.ph), st, tx, ty, ih1, ih2, G0, G1);
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                F0[v] = NEED_F0 ? face_avg(G0[v]) : 0.0f;
                F1[v] = face_avg_neg(G1[v]);
            }
        }
        if (upd) {
            cp_async_wait_all();
            __syncthreads();   // the x-face slab of every thread is in place
            if (in && cell_ok) {
                const int z = f - 1;
                M dx[8], dy[8], dz[8];
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    dx[C0 + c] = sx[(c * SX_H + tx + 1) * SX_W + ty] - sx[(c * SX_H + tx) * SX_W + ty];
                    dy[C0 + c] = sy[(c * SY_H + ty + 1) * TX + tx] - sy[(c * SY_H + ty) * TX + tx];
                }
                // local frame of a z-face: (rho, m_z, m_x, m_y); global (rho, m_x, m_y, m_z)
                constexpr int loc[4] = {0, 2, 3, 1};
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                    if (NEED_F0) dz[v] = F0[loc[v]] - P0[loc[v]];
                    dz[4 + v] = F1[loc[v]] - P1[loc[v]];
                }
                R o0[4], o1[4];
                bad |= !update_cell<R, STAGE>(U, lin, dt, dx, dy, dz, ih1, ih2, ihz, s0, s1, o0, o1);
                if (STAGE == 2 && U.prep) {
                    bool boxed = false;
                    for (int q = 0; q < U.nbox; ++q)
                        boxed |= a >= U.box[q][0][0] && a <= U.box[q][0][1] && b >= U.box[q][1][0] &&
                                 b <= U.box[q][1][1] && z >= U.box[q][2][0] && z <= U.box[q][2][1];
#pragma unroll
                    for (int v = 0; v < 4; ++v) U.wk0n[v * U.np + lin] = (o0[v] - (v == 0 ? U.off : 0.0f)) + o1[v];
                    if (!boxed) mx = max_u2f(mx, cell_u2f(o0, o1));
                }
            }
        }
        if (in) {
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                P0[v] = F0[v];
                P1[v] = F1[v];
            }
        }
        cur = nxt;
        __syncthreads();   // st, the face buffer and the slabs are free again
    }
    if (STAGE == 2 && bad) atomicOr(&A.scal->flags, FLAG_NONFINITE);
    if (STAGE == 2 && U.prep) block_max_to((double)mx, &A.scal->maxu2_bits);
    if (STAGE == 2 && U.advance && blockIdx.x == 0 && tid == 0) U.scal->t = U.scal->t + dt;
}

// Stage update of every cell from the stored fluxes of all its faces (FP64
// grids, and the small FP32C grids whose directions run together). A block
// takes 32 x 8 columns of kUpdZ planes, a thread one cell per plane; the
// x-face fluxes (y fastest in memory) arrive through a padded shared slab, the
// y- and z-face fluxes and the state straight from memory: bound by memory.
// FP64 kernels: the fused form needs 218 registers and recomputes the first
// face of each z segment (z faces and update of a 96^3 step 2.89 -> 2.70 ms
// apart). Large FP32C grids stay fused: 2.75 ms apart against 2.44 ms on
// 384x256x256, where the z-face fluxes' way through memory costs more than the
// tile kernel's shared memory.
template <typename R, typename C, int STAGE>
__global__ void __launch_bounds__(256) update_kernel(const __grid_constant__ UpdArgs<R, Mid<R, C>> U, int planes)
{
    using M = Mid<R, C>;
    constexpr int NC = STAGE == 1 ? 8 : 4, C0 = STAGE == 1 ? 0 : 4;
    __shared__ M sx[2][NC][SX_H][SX_W];
    const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * TX + tx;
    const int a0 = blockIdx.x * TX, b0 = blockIdx.y * TY, zb = blockIdx.z * planes, ze = min(zb + planes, U.nz);
    const int a = a0 + tx, b = b0 + ty;
    const bool in = a < U.nx && b < U.ny;
    const double dt = U.scal->dt;
    R ihx = R(0), ihy = R(0);
    if (in) {
        ihx = __ldg(U.ihx + a + G);
        ihy = __ldg(U.ihy + b + G);
    }
    // x faces a0 .. a0+32 of rows b0 .. b0+7 of plane z: thread row b0 + (tid &
    // 7), face a0 + tid/8; the 8 threads with tid/8 = 0 also take face a0 + 32
    auto slab = [&](int z, int s) {
        const int yy = tid & 7, xf = tid >> 3;
        if (b0 + yy < U.ny) {
            const long sxf = (long)U.nz * U.ny;
            const long g0 = ((long)(a0 + xf) * U.nz + z) * U.ny + b0 + yy;
            if (a0 + xf <= U.nx && in_bounds(g0, U.nffx)) {
#pragma unroll
                for (int c = 0; c < NC; ++c) cp_async(&sx[s][c][xf][yy], U.ffx + (C0 + c) * U.nffx + g0);
            }
            if (xf == 0 && a0 + 32 <= U.nx && in_bounds(g0 + 32 * sxf, U.nffx)) {
#pragma unroll
                for (int c = 0; c < NC; ++c) cp_async(&sx[s][c][32][yy], U.ffx + (C0 + c) * U.nffx + g0 + 32 * sxf);
            }
        }
        cp_async_commit();
    };
    bool bad = false;
    double mx = 0.0;
    float mxf = 0.0f;
    slab(zb, 0);
    for (int z = zb, s = 0; z < ze; ++z, s ^= 1) {
        const long lin = (long)(a + G) + (long)U.P0 * ((long)(b + G) + (long)U.P1 * (z + G));
        const long iy = ((long)b * U.nz + z) * U.nx + a, sy = (long)U.nz * U.nx;
        const long iz = ((long)z * U.ny + b) * U.nx + a, sz = (long)U.ny * U.nx;
        const bool ok = in && in_bounds(lin, U.np) && in_bounds(iy + sy, U.nffy) && in_bounds(iz + sz, U.nffz);
        M dx[8], dy[8], dz[8];
        R s0[4], s1[4];
        if (ok) {
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                const int k = C0 + c;
                dy[k] = U.ffy[k * U.nffy + iy + sy] - U.ffy[k * U.nffy + iy];
                dz[k] = U.ffz[k * U.nffz + iz + sz] - U.ffz[k * U.nffz + iz];
            }
            const R *src = (const R *)(STAGE == 1 ? U.w0 : U.pbuf);
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                s0[v] = src[v * U.np + lin];
                s1[v] = std::is_same<R, double>::value ? R(0) : src[(4 + v) * U.np + lin];
            }
        }
        cp_async_wait_all();
        __syncthreads();   // the slab of plane z is in place, that of z - 1 has been read
        if (z + 1 < ze) slab(z + 1, s ^ 1);
        if (!ok) continue;
#pragma unroll
        for (int c = 0; c < NC; ++c) dx[C0 + c] = sx[s][c][tx + 1][ty] - sx[s][c][tx][ty];
        const R ihz = __ldg(U.ihz + z + G);
        R o0[4], o1[4];
        if constexpr (std::is_same<C, dsf>::value)
            bad |= !update_cell_ds<STAGE>(U, lin, dt, dx, dy, dz, to_ds(ihx), to_ds(ihy), to_ds(ihz), s0, o0);
        else
            bad |= !update_cell<R, STAGE>(U, lin, dt, dx, dy, dz, ihx, ihy, ihz, s0, s1, o0, o1);
        if (STAGE == 2 && U.prep) {
            bool boxed = false;
            for (int q = 0; q < U.nbox; ++q)
                boxed |= a >= U.box[q][0][0] && a <= U.box[q][0][1] && b >= U.box[q][1][0] && b <= U.box[q][1][1] &&
                         z >= U.box[q][2][0] && z <= U.box[q][2][1];
            if constexpr (std::is_same<R, double>::value) {
                if (!boxed) mx = max_u2(mx, cell_u2(o0));
            } else {
#pragma unroll
                for (int v = 0; v < 4; ++v) U.wk0n[v * U.np + lin] = (o0[v] - (v == 0 ? U.off : 0.0f)) + o1[v];
                if (!boxed) mxf = max_u2f(mxf, cell_u2f(o0, o1));
            }
        }
    }
    if (STAGE == 2 && bad) atomicOr(&U.scal->flags, FLAG_NONFINITE);
    if (STAGE == 2 && U.prep) block_max_to(std::is_same<R, double>::value ? mx : (double)mxf, &U.scal->maxu2_bits);
    if (STAGE == 2 && U.advance && blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0 && tid == 0)
        U.scal->t = U.scal->t + dt;
}

template <typename K>
int persistent_grid(K kernel, size_t smem)
{
    int dev = 0, sms = 0, per = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, TX * TY, smem);
    return (per > 0 ? per : 1) * (sms > 0 ? sms : 1);
}

// Blocks of the persistent face-flux kernels (FP32C: one block per SM), found
// once per kernel; GP (the Gauss-point output of the adjoint's recorded steps)
// exists in FP64 arithmetic only.
template <typename R, typename C, int STAGE, bool GP, int ND>
int flux_blocks()
{
    static const int n = [] {
        if constexpr (std::is_same<C, float>::value) {
            cudaFuncSetAttribute(face_flux_march_kernel<STAGE == 1, ND>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)march_smem_bytes(kMarchWarps));
            return sm_count();
        } else {
            return persistent_grid(face_flux_kernel<R, C, STAGE == 1, GP, ND>, flux_smem_bytes<R>());
        }
    }();
    return n;
}

// z-faces per segment of the fused z kernel: the length L that minimises the
// steps of the busiest block, ceil(items / G) x (L + 1 priming face), with
// items = columns x ceil(nf / L), over 1 to 64 segments.
int z_segment(int ncol, int nf, int G)
{
    long best = -1;
    int bestL = nf;
    for (int S = 1; S <= 64 && S <= nf; ++S) {
        const int L = (nf + S - 1) / S, Sa = (nf + L - 1) / L;
        const long items = (long)ncol * Sa;
        const long cost = (items + G - 1) / G * (L + (Sa > 1 ? 1 : 0));
        if (best < 0 || cost < best) {
            best = cost;
            bestL = L;
        }
    }
    return bestL;
}

// Arguments of the face-state kernel of direction d on working array w.
template <typename R, typename C>
FaceEqArgs<R, C> face_eq_args(const Ctx &c, int d, const R *w, const Phys<C> &ph)
{
    const long stride[3] = {1, (long)c.P[0], (long)c.P[0] * c.P[1]};
    const int t1 = tan1(d), t2 = tan2(d);
    FaceEqArgs<R, C> E;
    E.w = w;
    E.np = c.np;
    E.fq = (Mid<R, C> *)c.fq[d];
    E.nfq = c.nfq;
    E.ihf = (const R *)c.ihf[d];
    E.n1 = c.n[t1];
    E.n2 = c.n[t2];
    E.e1p = c.e1p[d];
    E.sd = stride[d];
    E.s1 = stride[t1];
    E.s2 = stride[t2];
    E.cn = 1 + d;
    E.c1 = 1 + t1;
    E.c2 = 1 + t2;
    E.ph = ph;
    E.nf = c.n[d] + 1;
    E.K = 1;
    return E;
}

// Arguments of the face flux of direction d.
template <typename R, typename C>
FluxArgs<R, C> flux_args(const Ctx &c, int d, const Phys<C> &ph)
{
    const int t1 = tan1(d), t2 = tan2(d);
    FluxArgs<R, C> F;
    F.ff = (Mid<R, C> *)c.ff[d];
    F.nff = c.nff[d];
    F.ih1 = (const R *)c.ih[t1];
    F.ih2 = (const R *)c.ih[t2];
    F.n1 = c.n[t1];
    F.n2 = c.n[t2];
    F.nf = c.n[d] + 1;
    F.gcomp[0] = 0;
    F.gcomp[1] = 1 + d;
    F.gcomp[2] = 1 + t1;
    F.gcomp[3] = 1 + t2;
    F.ph = ph;
    F.scal = c.scal;
    F.gp = std::is_same<C, double>::value ? c.gp_dir[d] : nullptr;
    F.ngp = c.ngp;
    F.gp32 = c.gp_bytes == 4;
    return F;
}

// The face fluxes of ND directions (their arguments in F.A).
template <typename R, typename C, int STAGE, bool GP, int ND>
void launch_flux(const FluxMaps<ND> &maps, FluxLaunch<R, C, ND> &F, cudaStream_t stream)
{
    const int G1 = flux_blocks<R, C, STAGE, GP, ND>();
    F.first[0] = 0;
    for (int k = 0; k < ND; ++k) {
        const FluxArgs<R, C> &A = F.A[k];
        const int na = (A.n1 + TX - 1) / TX;
        if (std::is_same<C, float>::value) {
            F.L[k] = march_segment(na, A.nf, A.n2, kMarchWarps * G1 / ND);
            F.first[k + 1] = F.first[k] + na * A.nf * ((A.n2 + F.L[k] - 1) / F.L[k]);
        } else {
            F.first[k + 1] = F.first[k] + na * ((A.n2 + TY - 1) / TY) * A.nf;
        }
    }
    const int items = F.first[ND];
    if constexpr (std::is_same<C, float>::value) {
        // few items: fewer warps per block, so that they spread over the SMs
        const int nw = std::min(kMarchWarps, (items + G1 - 1) / G1), g = std::min(G1, (items + nw - 1) / nw);
        face_flux_march_kernel<STAGE == 1, ND><<<g, 32 * nw, march_smem_bytes(nw), stream>>>(maps, F);
    } else {
        face_flux_kernel<R, C, STAGE == 1, GP, ND>
            <<<std::min(items, G1), dim3(TX, TY), flux_smem_bytes<R>(), stream>>>(maps, F);
    }
}

template <typename R, typename C, int STAGE>
UpdArgs<R, Mid<R, C>> update_args(const Ctx &c)
{
    UpdArgs<R, Mid<R, C>> U;
    U.ffx = (const Mid<R, C> *)c.ff[0];
    U.ffy = (const Mid<R, C> *)c.ff[1];
    U.ffz = (const Mid<R, C> *)c.ff[2];
    U.nffx = c.nff[0];
    U.nffy = c.nff[1];
    U.nffz = c.nff[2];
    U.ihx = (const R *)c.ih[0];
    U.ihy = (const R *)c.ih[1];
    U.ihz = (const R *)c.ih[2];
    U.nx = c.n[0];
    U.ny = c.n[1];
    U.nz = c.n[2];
    U.P0 = c.P[0];
    U.P1 = c.P[1];
    U.np = c.np;
    U.w0 = c.state;
    U.wk1 = c.wk1;
    U.pbuf = c.pbuf;
    U.state = c.state;
    U.off = (R)c.off;
    for (int a = 0; a < 3; ++a) U.fb[a] = (R)c.fbody[a];
    U.prep = STAGE == 2 && c.prep_next && c.nprep_box <= kMaxPrepBoxes;
    U.wk0n = c.prec == GKS_FP32C ? (float *)c.wk0 : nullptr;
    U.nbox = U.prep ? c.nprep_box : 0;
    for (int q = 0; q < U.nbox; ++q)
        for (int e = 0; e < 3; ++e)
            for (int k = 0; k < 2; ++k) U.box[q][e][k] = c.prep_box[q][e][k];
    U.advance = STAGE == 2 && c.advance;
    U.scal = c.scal;
    return U;
}

template <typename R, typename C, int STAGE>
void launch_update(const Ctx &c)
{
    // planes per block: the grid's z extent stays within its 65535 blocks
    int planes = kUpdZ;
    while ((c.n[2] + planes - 1) / planes > 65535) planes *= 2;
    const dim3 g((c.n[0] + TX - 1) / TX, (c.n[1] + TY - 1) / TY, (c.n[2] + planes - 1) / planes);
    mark(c, K_FLUX_UPDATE, 1);
    update_kernel<R, C, STAGE><<<g, dim3(TX, TY), 0, c.stream>>>(update_args<R, C, STAGE>(c), planes);
    mark(c, K_FLUX_UPDATE, 0);
}

// z faces of a large FP32C grid: flux and the stage update of every cell.
template <int STAGE>
void launch_flux_update(const Ctx &c, const FluxArgs<float, float> &F)
{
    constexpr size_t su = flux_update_smem_bytes(STAGE == 1 ? 8 : 4);
    static const int G1 = persistent_grid(flux_update_kernel<STAGE>, su);
    const int ncol = ((F.n1 + TX - 1) / TX) * ((F.n2 + TY - 1) / TY), seg = z_segment(ncol, F.nf, G1);
    const long nitems = (long)ncol * ((F.nf + seg - 1) / seg);
    mark(c, K_FLUX_UPDATE, 1);
    flux_update_kernel<STAGE><<<(int)std::min(nitems, (long)G1), dim3(TX, TY), su, c.stream>>>(
        c.tmap[2], F, update_args<float, float, STAGE>(c), seg);
    mark(c, K_FLUX_UPDATE, 0);
}

template <typename R, typename C, int STAGE, bool GP>
void stage_impl(const Ctx &c)
{
    const Phys<C> ph = make_phys<C>(c);
    const R *w = (const R *)(STAGE == 1 ? c.wk0 : c.wk1);
    auto map = [&](int d) -> const CUtensorMap & { return std::is_same<C, float>::value ? c.tmapM[d] : c.tmap[d]; };
    if (c.small) {
        // all directions at once: their face boxes have buffers of their own
        FaceEq3<R, C> E;
        const int dirs[3] = {0, 1, 2};
        for (int d = 0; d < 3; ++d) E.d[d] = face_eq_args<R, C>(c, d, w, ph);
        march_faces<R, C, true>(E.d, dirs, 3);
        E.first[0] = 0;
        for (int d = 0; d < 3; ++d) {
            const dim3 g = face_eq_blocks<R, C, true>(E.d[d], d);
            E.gx[d] = g.x;
            E.first[d + 1] = E.first[d] + g.x * g.y;
        }
        mark(c, K_FACE_EQ, 1);
        face_eq_all_kernel<R, C><<<E.first[3], kEqThreads<C, true>, 0, c.stream>>>(E);
        mark(c, K_FACE_EQ, 0);
        FluxMaps<3> maps;
        FluxLaunch<R, C, 3> F;
        for (int d = 0; d < 3; ++d) {
            maps.d[d] = map(d);
            F.A[d] = flux_args<R, C>(c, d, ph);
        }
        mark(c, K_FACE_FLUX, 1);
        launch_flux<R, C, STAGE, GP, 3>(maps, F, c.stream);
        mark(c, K_FACE_FLUX, 0);
        launch_update<R, C, STAGE>(c);
        return;
    }
    for (int d = 0; d < 3; ++d) {
        mark(c, K_FACE_EQ, 1);
        launch_face_eq(face_eq_args<R, C>(c, d, w, ph), d, c.stream);
        mark(c, K_FACE_EQ, 0);
        FluxMaps<1> maps;
        FluxLaunch<R, C, 1> F;
        maps.d[0] = map(d);
        F.A[0] = flux_args<R, C>(c, d, ph);
        if constexpr (std::is_same<C, float>::value)
            if (d == 2) {
                launch_flux_update<STAGE>(c, F.A[0]);
                return;
            }
        const int grp = d < 2 ? K_FACE_FLUX : K_FLUX_UPDATE;
        mark(c, grp, 1);
        launch_flux<R, C, STAGE, GP, 1>(maps, F, c.stream);
        mark(c, grp, 0);
    }
    launch_update<R, C, STAGE>(c);
}

// ----------------------------------------------------- prep, CFL, misc --

constexpr int kPrepZ = 8;      // z planes per block of the state upload
constexpr int kPrepBoxZ = 2;   // z planes per block of the prep of a box

// Interior cells [lo, hi) of up to kMaxPrepBoxes boxes, one per blockIdx.z
// layer of nz blocks.
struct PrepBoxes {
    int3 lo[kMaxPrepBoxes], hi[kMaxPrepBoxes];
    int nz;
};

// Start of a step: the largest |U|^2 over the interior cells (for the CFL
// time step) and, for FP32C, the FP32 reconstruction input hi + lo (density
// as rho - off), over boxes of interior cells (the whole interior, or the
// forcing boxes after the forcing: one launch for all of them and 2 planes per
// block, 3 x 13.8 -> 8 us on the boxes of a 221x83x91 rotor with tower and
// nacelle). One atomicMax per block; cells in two boxes get the same values
// twice.
template <int PREC>
__global__ void __launch_bounds__(256) prep_cfl_kernel(const void *__restrict__ S, float *__restrict__ wk, long np,
                                                       const __grid_constant__ PrepBoxes B, int planes, int P0, int P1,
                                                       float off, Scalars *scal, int advance)
{
    if (advance && blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0 && threadIdx.x == 0 && threadIdx.y == 0)
        scal->t = scal->t + scal->dt;   // the last launch of a step with forcing
    const int q = blockIdx.z / B.nz;
    const int3 lo = B.lo[q], hi = B.hi[q];
    const int i = lo.x + blockIdx.x * 32 + threadIdx.x, j = lo.y + blockIdx.y * 8 + threadIdx.y;
    const int k0 = lo.z + (blockIdx.z - q * B.nz) * planes, k1 = min(k0 + planes, hi.z);
    if (lo.x + (int)blockIdx.x * 32 >= hi.x || lo.y + (int)blockIdx.y * 8 >= hi.y || k0 >= hi.z) return;   // whole blocks
    double mx = 0.0;
    float mxf = 0.0f;
    if (i < hi.x && j < hi.y) {
        for (int k = k0; k < k1; ++k) {
            const long lin = (long)(i + G) + (long)P0 * ((long)(j + G) + (long)P1 * (k + G));
            if (PREC == GKS_FP64) {
                const double *__restrict__ W = (const double *)S;
                double w[4];
#pragma unroll
                for (int v = 0; v < 4; ++v) w[v] = W[v * np + lin];
                mx = max_u2(mx, cell_u2(w));
            } else {
                const float *__restrict__ W = (const float *)S;
                float h[4], l[4];
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                    h[v] = W[v * np + lin];
                    l[v] = W[(4 + v) * np + lin];
                }
#pragma unroll
                for (int v = 0; v < 4; ++v) wk[v * np + lin] = (h[v] - (v == 0 ? off : 0.0f)) + l[v];
                mxf = max_u2f(mxf, cell_u2f(h, l));
            }
        }
    }
    block_max_to(PREC == GKS_FP64 ? mx : (double)mxf, &scal->maxu2_bits);
}

__global__ void dt_kernel(Scalars *scal, double cfl, double dt_fixed, double hmin, double csound)
{
    set_dt(scal, cfl, dt_fixed, hmin, csound);
}

__global__ void advance_kernel(Scalars *scal) { scal->t = scal->t + scal->dt; }


// Compact FP64 state -> the padded state (FP32C: hi = fl32(q), lo =
// fl32(q - hi)), kPrepZ planes per block. With scal set it also does the
// work of prep_cfl on the new state (FP32 input into wk for FP32C, max
// |U|^2 into scal; FP32C takes the max over the FP32 values of cell_u2,
// whose order and NaN the conversion to double keeps).
__global__ void __launch_bounds__(256) scatter_kernel(int prec, const double *__restrict__ src, void *S, long np,
                                                      int nx, int ny, int nz, int P0, int P1, float *wk, float off,
                                                      Scalars *scal)
{
    const int i = blockIdx.x * 32 + threadIdx.x, j = blockIdx.y * 8 + threadIdx.y;
    const int k0 = blockIdx.z * kPrepZ, k1 = min(k0 + kPrepZ, nz);
    const long N = (long)nx * ny * nz;
    double mx = 0.0;
    float mxf = 0.0f;
    if (i < nx && j < ny) {
        // the next plane's values are loaded while this one's are stored
        double qn[4];
#pragma unroll
        for (int v = 0; v < 4; ++v) qn[v] = k0 < k1 ? src[v * N + i + (long)nx * (j + (long)ny * k0)] : 0.0;
        for (int k = k0; k < k1; ++k) {
            const long lin = (long)(i + G) + (long)P0 * ((long)(j + G) + (long)P1 * (k + G));
            double q[4];
            float h[4], l[4];
#pragma unroll
            for (int v = 0; v < 4; ++v) q[v] = qn[v];
            if (k + 1 < k1) {
                const long cn = i + (long)nx * (j + (long)ny * (k + 1));
#pragma unroll
                for (int v = 0; v < 4; ++v) qn[v] = src[v * N + cn];
            }
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                if (prec == GKS_FP64) {
                    ((double *)S)[v * np + lin] = q[v];
                } else {
                    split_hi_lo(q[v], h[v], l[v]);
                    ((float *)S)[v * np + lin] = h[v];
                    ((float *)S)[(4 + v) * np + lin] = l[v];
                }
            }
            if (scal) {
                if (prec == GKS_FP64) {
                    mx = max_u2(mx, cell_u2(q));
                } else {
#pragma unroll
                    for (int v = 0; v < 4; ++v) wk[v * np + lin] = (h[v] - (v == 0 ? off : 0.0f)) + l[v];
                    mxf = max_u2f(mxf, cell_u2f(h, l));
                }
            }
        }
    }
    if (scal) block_max_to(prec == GKS_FP64 ? mx : (double)mxf, &scal->maxu2_bits);
}

template <int PREC>
__global__ void __launch_bounds__(256) gather_kernel(const void *S, double *dst, long np, int nx, int ny, int nz,
                                                     int P0, int P1)
{
    const int i = blockIdx.x * 32 + threadIdx.x, j = blockIdx.y * 8 + threadIdx.y, k = blockIdx.z;
    if (i >= nx || j >= ny) return;
    const long N = (long)nx * ny * nz;
    const long ci = i + (long)nx * (j + (long)ny * k);
    const long lin = (long)(i + G) + (long)P0 * ((long)(j + G) + (long)P1 * (k + G));
    if (PREC == GKS_FP64) {
        const double *W = (const double *)S;
#pragma unroll
        for (int v = 0; v < 4; ++v) dst[v * N + ci] = W[v * np + lin];
    } else {
        const float *W = (const float *)S;
        float h[4], l[4];
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            h[v] = W[v * np + lin];
            l[v] = W[(4 + v) * np + lin];
        }
#pragma unroll
        for (int v = 0; v < 4; ++v) dst[v * N + ci] = compose_hi_lo(h[v], l[v]);
    }
}

// a / b in FP64 from a double-single reciprocal r0 of b (within 2^-44): one
// correction of the quotient by its remainder, 3 FP64 operations in place of
// the library division's 9 or so (within one ulp of it).
__device__ __forceinline__ double quotient(double a, double b, double r0)
{
    const double q = __dmul_rn(a, r0);
    return fma(fma(-q, b, a), r0, q);
}
// Whether b and its reciprocal are far from the ends of the FP32 exponents.
__device__ __forceinline__ bool rcp_range(unsigned int e) { return e >= 27u && e <= 227u; }

// 1 / (h + l) as a double, within 2^-44, for h in the range of rcp_range.
__device__ __forceinline__ double rcp_ds(float h, float l)
{
    const float r = rcp_approx(h);
    const float e = __fmaf_rn(-l, r, __fmaf_rn(-h, r, 1.0f));
    const float s = __fmul_rn(e, r);
    const float rh = __fadd_rn(r, s);
    return compose_hi_lo(rh, __fsub_rn(s, __fsub_rn(rh, r)));
}

// Sum of FP32 values with the rounding errors of the first two levels kept:
// a + b + c holds the sum to about 2^-70 of its largest partial sum.
struct Sum3 {
    f2 a, b, c;
    __device__ __forceinline__ void add(f2 x)
    {
        const dsf2 t = two_sum(a, x), u = two_sum(b, t.lo);
        a = t.hi;
        b = u.hi;
        c += u.lo;
    }
    __device__ __forceinline__ void add_low(f2 x)
    {
        const dsf2 u = two_sum(b, x);
        b = u.hi;
        c += u.lo;
    }
};

// FP64 sums of mass, momentum and kinetic energy: a block walks (32 x 8
// columns) x (kDiagZ planes) pieces of the grid in a fixed order, a thread one
// column of a piece; per-block partial sums, then one block adds the partials
// in order (deterministic). GB300 runs FP64 at 1/64 of its FP32 rate, so what
// counts is FP64 operations per cell (34 when every value was converted,
// weighted by its cell volume and the energy divided out: 1.49 ms on 25.2M
// cells against 0.12 ms of memory traffic). FP32C: the widths along z are
// equal to 1e-12 (ZU), so mass and momentum are summed unweighted in FP32 with
// their rounding errors kept (Sum3) and weighted once per column, the widths'
// differences from the column's first one added as an FP32 correction; only
// the energy stays FP64 per cell, 7 operations with a double-single
// reciprocal of the density: 0.54 ms. A stretched z and FP64 grids weight each
// value by its plane's width (a multiply-add each).
constexpr int kDiagZ = 16;

template <int PREC, bool ZU>
__global__ void __launch_bounds__(256) diag_partial_kernel(const void *S, long np, int nx, int ny, int nz, int P0,
                                                           int P1, const double *hx, const double *hy,
                                                           const double *hz, double *partials)
{
    __shared__ double sh[5][256];
    __shared__ float dz[kDiagZ];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int NA = (nx + 31) / 32, NB = (ny + 7) / 8, NC = (nz + kDiagZ - 1) / kDiagZ;
    const long nitems = (long)NA * NB * NC;
    double s[5] = {0, 0, 0, 0, 0};
    for (long it = blockIdx.x; it < nitems; it += gridDim.x) {
        const long r = it / NA;
        const int i = (int)(it - r * NA) * 32 + tx, j = (int)(r % NB) * 8 + ty;
        const int k0 = (int)(r / NB) * kDiagZ, nk = min(kDiagZ, nz - k0);
        if (ZU && PREC == GKS_FP32C) {
            __syncthreads();
            if ((int)threadIdx.x < nk) dz[threadIdx.x] = (float)(hz[k0 + threadIdx.x + G] - hz[k0 + G]);
            __syncthreads();
        }
        if (i >= nx || j >= ny) continue;
        const double area = hx[i + G] * hy[j + G], h0 = hz[k0 + G];
        const long lin0 = (long)(i + G) + (long)P0 * ((long)(j + G) + (long)P1 * (k0 + G)), sz = (long)P0 * P1;
        double t[5] = {0, 0, 0, 0, 0};   // the column's sums over z, times the widths
        bool finite = true;
        if (PREC == GKS_FP64) {
            const double *W = (const double *)S;
            for (int k = 0; k < nk; ++k) {
                double q[4];
#pragma unroll
                for (int v = 0; v < 4; ++v) q[v] = W[v * np + lin0 + k * sz];
                const double w = hz[k0 + k + G], m2 = fma(q[1], q[1], fma(q[2], q[2], q[3] * q[3]));
                const int hw = __double2hiint(q[0]), e = ((hw >> 20) & 0x7ff) - 896;
                double u;
                if (e > 52 && e <= 227) {
                    // the top 24 bits of rho as a float, the rest as its low part
                    // (a normal float down to 2^-74)
                    const float f = __uint_as_float((hw & 0x80000000u) | ((unsigned int)e << 23) | ((hw & 0xfffffu) << 3) |
                                                    ((unsigned int)__double2loint(q[0]) >> 29));
                    const float g = __fmul_rn(__uint2float_rn((unsigned int)__double2loint(q[0]) & 0x1fffffffu),
                                              __uint_as_float((unsigned int)(e - 52) << 23));
                    u = quotient(m2, q[0], rcp_ds(f, copysignf(g, f)));
                } else {
                    u = m2 / q[0];
                }
#pragma unroll
                for (int v = 0; v < 4; ++v) t[v] = fma(w, q[v], t[v]);
                t[4] = fma(w, u, t[4]);
            }
        } else {
            const float *W = (const float *)S;
            const f2 z(0.0f);
            Sum3 a[2] = {{z, z, z}, {z, z, z}};
            f2 dc[2] = {z, z};
            float de = 0.0f;
#pragma unroll 2
            for (int k = 0; k < nk; ++k) {
                float h[4], l[4];
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                    h[v] = W[v * np + lin0 + k * sz];
                    l[v] = W[(4 + v) * np + lin0 + k * sz];
                }
                double m2 = 0.0;
#pragma unroll
                for (int v = 1; v < 4; ++v) {
                    const double m = compose_hi_lo(h[v], l[v]);
                    m2 = fma(m, m, m2);
                }
                const double rho = compose_hi_lo(h[0], l[0]);
                const double u = rcp_range((__float_as_uint(h[0]) >> 23) & 0xffu) ? quotient(m2, rho, rcp_ds(h[0], l[0]))
                                                                                  : m2 / rho;
                if (ZU) {
                    const f2 d(dz[k]);
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        const f2 x(h[2 * q], h[2 * q + 1]);
                        a[q].add(x);
                        a[q].add_low(f2(l[2 * q], l[2 * q + 1]));
                        dc[q] = fma(d, x, dc[q]);
                    }
                    de = __fmaf_rn(dz[k], __fmul_rn(__fmaf_rn(h[1], h[1], __fmaf_rn(h[2], h[2], h[3] * h[3])),
                                                    rcp_approx(h[0])), de);
                    t[4] += u;
                } else {
                    const double w = hz[k0 + k + G];
                    t[0] = fma(w, rho, t[0]);
#pragma unroll
                    for (int v = 1; v < 4; ++v) t[v] = fma(w, compose_hi_lo(h[v], l[v]), t[v]);
                    t[4] = fma(w, u, t[4]);
                }
            }
            if (ZU) {
                finite = isfinite(de) && isfinite(a[0].a.v.x) && isfinite(a[0].a.v.y) && isfinite(a[1].a.v.x) &&
                         isfinite(a[1].a.v.y);
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    t[2 * q] = fma(h0, ((double)a[q].a.v.x + (double)a[q].b.v.x) + (double)a[q].c.v.x, (double)dc[q].v.x);
                    t[2 * q + 1] =
                        fma(h0, ((double)a[q].a.v.y + (double)a[q].b.v.y) + (double)a[q].c.v.y, (double)dc[q].v.y);
                }
                t[4] = fma(h0, t[4], (double)de);
            }
        }
        if (!finite || !isfinite(t[4])) {
            // an infinity, a NaN or an FP32 overflow: the column in plain FP64
            for (int q = 0; q < 5; ++q) t[q] = 0.0;
            for (int k = 0; k < nk; ++k) {
                const double w = hz[k0 + k + G];
                double q[4];
                for (int v = 0; v < 4; ++v) {
                    const long l = v * np + lin0 + k * sz;
                    q[v] = PREC == GKS_FP64 ? ((const double *)S)[l]
                                            : (double)((const float *)S)[l] + (double)((const float *)S)[4 * np + l];
                    t[v] += w * q[v];
                }
                t[4] += w * ((q[1] * q[1] + q[2] * q[2] + q[3] * q[3]) / q[0]);
            }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) s[q] = fma(area, t[q], s[q]);
        s[4] = fma(0.5 * area, t[4], s[4]);
    }
#pragma unroll
    for (int q = 0; q < 5; ++q) sh[q][threadIdx.x] = s[q];
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w)
#pragma unroll
            for (int q = 0; q < 5; ++q) sh[q][threadIdx.x] += sh[q][threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x < 5) partials[blockIdx.x * 8 + threadIdx.x] = sh[threadIdx.x][0];
}

__global__ void __launch_bounds__(256) diag_final_kernel(const double *partials, int nparts, double *out)
{
    __shared__ double sh[5][256];
    double s[5] = {0, 0, 0, 0, 0};
    for (int b = threadIdx.x; b < nparts; b += blockDim.x)
#pragma unroll
        for (int q = 0; q < 5; ++q) s[q] += partials[b * 8 + q];
#pragma unroll
    for (int q = 0; q < 5; ++q) sh[q][threadIdx.x] = s[q];
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w)
#pragma unroll
            for (int q = 0; q < 5; ++q) sh[q][threadIdx.x] += sh[q][threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x < 5) out[threadIdx.x] = sh[threadIdx.x][0];
}

__global__ void __launch_bounds__(256) fill_rest_kernel(int prec, void *S, long np, int nx, int ny,
                                                        int nz, int P0, int P1)
{
    const int i = blockIdx.x * 32 + threadIdx.x, j = blockIdx.y * 8 + threadIdx.y, k = blockIdx.z;
    if (i >= nx || j >= ny) return;
    const long lin = (long)(i + G) + (long)P0 * ((long)(j + G) + (long)P1 * (k + G));
    if (prec == GKS_FP64)
        ((double *)S)[lin] = 1.0;
    else
        ((float *)S)[lin] = 1.0f;
}

// Copy the stored component arrays (4 doubles or 8 floats per cell) between
// the padded state and a compact interior array (x fastest).
template <typename T>
__global__ void __launch_bounds__(256) raw_copy_kernel(T *S, T *cpt, int narr, long np, int nx, int ny,
                                                       int nz, int P0, int P1, int to_compact)
{
    const int i = blockIdx.x * 32 + threadIdx.x, j = blockIdx.y * 8 + threadIdx.y, k = blockIdx.z;
    if (i >= nx || j >= ny) return;
    const long N = (long)nx * ny * nz;
    const long ci = i + (long)nx * (j + (long)ny * k);
    const long lin = (long)(i + G) + (long)P0 * ((long)(j + G) + (long)P1 * (k + G));
    for (int a = 0; a < narr; ++a) {
        if (to_compact)
            cpt[a * N + ci] = S[a * np + lin];
        else
            S[a * np + lin] = cpt[a * N + ci];
    }
}

}  // namespace

namespace {
bool prep_boxes(const Ctx &c, const int (*box)[3][2], int n, int planes, int advance)
{
    PrepBoxes B;
    int nb = 0, gx = 0, gy = 0;
    B.nz = 0;
    for (int q = 0; q < n && nb < kMaxPrepBoxes; ++q) {
        const int3 lo = make_int3(box[q][0][0], box[q][1][0], box[q][2][0]);
        const int3 hi = make_int3(box[q][0][1] + 1, box[q][1][1] + 1, box[q][2][1] + 1);
        if (hi.x <= lo.x || hi.y <= lo.y || hi.z <= lo.z) continue;
        B.lo[nb] = lo;
        B.hi[nb++] = hi;
        gx = std::max(gx, (hi.x - lo.x + 31) / 32);
        gy = std::max(gy, (hi.y - lo.y + 7) / 8);
        B.nz = std::max(B.nz, (hi.z - lo.z + planes - 1) / planes);
    }
    if (!nb) return false;
    const dim3 blk(32, 8), g(gx, gy, B.nz * nb);
    const int grp = c.prec == GKS_FP32C ? K_PREP : K_CFL;
    mark(c, grp, 1);
    if (c.prec == GKS_FP32C)
        prep_cfl_kernel<GKS_FP32C><<<g, blk, 0, c.stream>>>(c.state, (float *)c.wk0, c.np, B, planes, c.P[0], c.P[1],
                                                           (float)c.off, c.scal, advance);
    else
        prep_cfl_kernel<GKS_FP64><<<g, blk, 0, c.stream>>>(c.state, nullptr, c.np, B, planes, c.P[0], c.P[1], 0.0f,
                                                          c.scal, advance);
    mark(c, grp, 0);
    return true;
}
}  // namespace

bool launch_prep_boxes(const Ctx &c, const int (*box)[3][2], int n, bool advance)
{
    // planes per block: the grid's z extent stays within its 65535 blocks
    int planes = kPrepBoxZ;
    while ((long)((c.n[2] + planes - 1) / planes) * kMaxPrepBoxes > 65535) planes *= 2;
    return prep_boxes(c, box, n, planes, advance);
}

void launch_prep(const Ctx &c)
{
    const int box[1][3][2] = {{{0, c.n[0] - 1}, {0, c.n[1] - 1}, {0, c.n[2] - 1}}};
    int planes = kPrepZ;
    while ((c.n[2] + planes - 1) / planes > 65535) planes *= 2;
    prep_boxes(c, box, 1, planes, 0);
}

void launch_ghost(const Ctx &c, void *w, bool with_dt)
{
    if (c.prec == GKS_FP64)
        ghost_impl<double>(c, (double *)w, with_dt);
    else
        ghost_impl<float>(c, (float *)w, with_dt);
}

// ------------------------------------------------------------ slab groups --

// One thread per element of the G x-planes: (component, row, plane) with
// row = the (y, z) position over the padded P1 x P2 rows.
template <typename T>
__global__ void __launch_bounds__(256) halo_copy_kernel(const T *__restrict__ src, long np_src, int P0_src, int i_src,
                                                        T *__restrict__ dst, long np_dst, int P0_dst, int i_dst,
                                                        long rows)
{
    const long t = blockIdx.x * (long)blockDim.x + threadIdx.x;
    const long per = rows * G;
    if (t >= 4 * per) return;
    const int v = (int)(t / per);
    const long r = t - v * per, row = r / G;
    const int l = (int)(r - row * G);
    const long is = (long)(i_src + l) + (long)P0_src * row, id = (long)(i_dst + l) + (long)P0_dst * row;
    if (!in_bounds(is, np_src) || !in_bounds(id, np_dst)) return;
    dst[v * np_dst + id] = src[v * np_src + is];
}

void launch_halo_copy(const Ctx &src, const void *w_src, int side_src, const Ctx &dst, void *w_dst, int side_dst)
{
    // padded x index of the first plane: the interior planes next to the
    // low side start at G, next to the high side at n; the ghost planes of
    // the low side start at 0, of the high side at n + G
    const int i_src = side_src == 0 ? G : src.n[0];
    const int i_dst = side_dst == 0 ? 0 : dst.n[0] + G;
    const long rows = (long)src.P[1] * src.P[2];
    const long nt = 4 * rows * G;
    const int grid = (int)((nt + 255) / 256);
    mark(dst, K_GHOST, 1);
    if (src.prec == GKS_FP64)
        halo_copy_kernel<double><<<grid, 256, 0, dst.stream>>>((const double *)w_src, src.np, src.P[0], i_src,
                                                                (double *)w_dst, dst.np, dst.P[0], i_dst, rows);
    else
        halo_copy_kernel<float><<<grid, 256, 0, dst.stream>>>((const float *)w_src, src.np, src.P[0], i_src,
                                                               (float *)w_dst, dst.np, dst.P[0], i_dst, rows);
    mark(dst, K_GHOST, 0);
}

struct GroupScal {
    Scalars *p[64];
};

__global__ void group_max_u2_kernel(GroupScal g, int n)
{
    unsigned long long m = 0ull;   // bits of non-negative doubles order like the values
    for (int s = 0; s < n; ++s) m = max(m, g.p[s]->maxu2_bits);
    for (int s = 0; s < n; ++s) g.p[s]->maxu2_bits = m;
}

void launch_group_max_u2(Scalars *const *scal, int n, cudaStream_t stream)
{
    GroupScal g;
    for (int s = 0; s < n && s < 64; ++s) g.p[s] = scal[s];
    group_max_u2_kernel<<<1, 1, 0, stream>>>(g, n);
}

// FP32C: the forward face state of direction d from the FP32 working array
// w into the face box c.fq (the reverse recomputes it instead of storing it).
void launch_face_state32(const Ctx &c, int d, const float *w)
{
    launch_face_eq(face_eq_args<float, float>(c, d, w, make_phys<float>(c)), d, c.stream);
}

void launch_stage(const Ctx &c, int stage)
{
    if (c.prec == GKS_FP64 && c.gp_dir[0])
        stage == 1 ? stage_impl<double, double, 1, true>(c) : stage_impl<double, double, 2, true>(c);
    else if (c.prec == GKS_FP64 && c.fp64_ds)
        stage == 1 ? stage_impl<double, dsf, 1, false>(c) : stage_impl<double, dsf, 2, false>(c);
    else if (c.prec == GKS_FP64)
        stage == 1 ? stage_impl<double, double, 1, false>(c) : stage_impl<double, double, 2, false>(c);
    else
        stage == 1 ? stage_impl<float, float, 1, false>(c) : stage_impl<float, float, 2, false>(c);
}

void launch_cfl(const Ctx &c)
{
    mark(c, K_MISC, 1);
    dt_kernel<<<1, 1, 0, c.stream>>>(c.scal, c.cfl, c.dt_fixed, c.hmin, c.csound);
    mark(c, K_MISC, 0);
}

void launch_advance(const Ctx &c)
{
    mark(c, K_MISC, 1);
    advance_kernel<<<1, 1, 0, c.stream>>>(c.scal);
    mark(c, K_MISC, 0);
}

void launch_scatter_state(const Ctx &c, const double *d_src)
{
    dim3 blk(32, 8), g((c.n[0] + 31) / 32, (c.n[1] + 7) / 8, (c.n[2] + kPrepZ - 1) / kPrepZ);
    scatter_kernel<<<g, blk, 0, c.stream>>>(c.prec, d_src, c.state, c.np, c.n[0], c.n[1], c.n[2], c.P[0], c.P[1],
                                            nullptr, 0.0f, nullptr);
}

void launch_scatter_state_prep(const Ctx &c, const double *d_src)
{
    cudaMemsetAsync(&c.scal->maxu2_bits, 0, sizeof(unsigned long long), c.stream);
    dim3 blk(32, 8), g((c.n[0] + 31) / 32, (c.n[1] + 7) / 8, (c.n[2] + kPrepZ - 1) / kPrepZ);
    scatter_kernel<<<g, blk, 0, c.stream>>>(c.prec, d_src, c.state, c.np, c.n[0], c.n[1], c.n[2], c.P[0], c.P[1],
                                            c.prec == GKS_FP32C ? (float *)c.wk0 : nullptr, (float)c.off, c.scal);
}

void launch_gather_state(const Ctx &c, double *d_dst)
{
    dim3 blk(32, 8), g((c.n[0] + 31) / 32, (c.n[1] + 7) / 8, c.n[2]);
    if (c.prec == GKS_FP64)
        gather_kernel<GKS_FP64><<<g, blk, 0, c.stream>>>(c.state, d_dst, c.np, c.n[0], c.n[1], c.n[2], c.P[0], c.P[1]);
    else
        gather_kernel<GKS_FP32C><<<g, blk, 0, c.stream>>>(c.state, d_dst, c.np, c.n[0], c.n[1], c.n[2], c.P[0], c.P[1]);
}

void launch_fill_rest(const Ctx &c)
{
    dim3 blk(32, 8), g((c.n[0] + 31) / 32, (c.n[1] + 7) / 8, c.n[2]);
    fill_rest_kernel<<<g, blk, 0, c.stream>>>(c.prec, c.state, c.np, c.n[0], c.n[1], c.n[2], c.P[0],
                                              c.P[1]);
}

void launch_raw_copy(const Ctx &c, void *compact, int to_compact)
{
    dim3 blk(32, 8), g((c.n[0] + 31) / 32, (c.n[1] + 7) / 8, c.n[2]);
    if (c.prec == GKS_FP64)
        raw_copy_kernel<double><<<g, blk, 0, c.stream>>>((double *)c.state, (double *)compact, 4, c.np,
                                                         c.n[0], c.n[1], c.n[2], c.P[0], c.P[1],
                                                         to_compact);
    else
        raw_copy_kernel<float><<<g, blk, 0, c.stream>>>((float *)c.state, (float *)compact, 8, c.np,
                                                        c.n[0], c.n[1], c.n[2], c.P[0], c.P[1],
                                                        to_compact);
}

// FP32 values as FP64: out[i] = a[i] (+ b[i]) (+ off0 for i < n0), i < n; in
// integer operations (4 x 4.6M hi and lo: 35 -> 20 us).
__global__ void __launch_bounds__(256) widen_kernel(const float *a, const float *b, double *out, long n, long n0,
                                                     double off0)
{
    for (long i = blockIdx.x * 256L + threadIdx.x; i < n; i += (long)gridDim.x * 256L) {
        double v = compose_hi_lo(a[i], b ? b[i] : 0.0f);
        if (i < n0) v += off0;
        out[i] = v;
    }
}

void launch_widen(const Ctx &c, const float *a, const float *b, double *out, long n, long n0, double off0)
{
    mark(c, K_MISC, 1);
    const long nb = (n + 255) / 256;
    widen_kernel<<<(int)(nb < 16L * sm_count() ? nb : 16L * sm_count()), 256, 0, c.stream>>>(a, b, out, n, n0, off0);
    mark(c, K_MISC, 0);
}

void launch_diagnostics(const Ctx &c, double *d_out5)
{
    const long items = (long)((c.n[0] + 31) / 32) * ((c.n[1] + 7) / 8) * ((c.n[2] + kDiagZ - 1) / kDiagZ);
    const int nb = (int)std::min(items, (long)std::min(kMaxPartials, 4 * sm_count()));
    auto kernel = c.prec == GKS_FP64 ? diag_partial_kernel<GKS_FP64, false>
                  : c.uniform[2]     ? diag_partial_kernel<GKS_FP32C, true>
                                     : diag_partial_kernel<GKS_FP32C, false>;
    kernel<<<nb, 256, 0, c.stream>>>(c.state, c.np, c.n[0], c.n[1], c.n[2], c.P[0], c.P[1], c.h64[0], c.h64[1], c.h64[2],
                                     c.partials);
    diag_final_kernel<<<1, 256, 0, c.stream>>>(c.partials, nb, d_out5);
}

int bounds_flag_stencil() { return bounds_flag_take(); }

}  // namespace gks
