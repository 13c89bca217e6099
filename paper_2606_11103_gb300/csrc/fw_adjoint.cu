// Gradients of a receiver functional by the discrete adjoint of the time
// step (Sec. 2.1, Sec. 3.3 discretisation), with forward states recomputed
// from checkpoints.
//
// Functional: L = sum_{r,col} G[r][col] trace[r][col].  Parameters:
//  * c(x) through K dt = rho c^2 dt (pressure update and the volume-source
//    gain K dt / dx^D); dt, the absorbing profile and the relaxation sets
//    are held fixed;
//  * alpha0(x) through a per-voxel factor s(x) = alpha0(x) / alpha0_class on
//    every d of the voxel's class (kappa, alpha at the class values), taken
//    at s = 1: dL/dalpha0 = dL/ds / alpha0;
//  * maps of the absorbing layer are inherited from the nearest interior
//    cell: the gradient folds them back onto the cells they came from.
//
// The adjoint of one time step is reverse-mode differentiation of the two
// sweeps of fw_kernels.cuh, in the kernels' own variables (memory variables
// of the divergence side summed over directions; r the tissue ramp of the cell,
// 1 outside the absorbing layer):
//   pressure: psi2' = b2 psi2 + r a2 div, stp = div/kappa2 + sum (psi2 + psi2')/2
//             + absorbing, p' = p - K dt stp,  div = sum_d D-_d v_d;
//   velocity: psi1' = b1 psi1 + r a1 g, st = g/kappa1 + sum (psi1 + psi1')/2
//             + absorbing, v' = v - dtr st,  g = D+_d p;
// with (D+)^T = -D- and (D-)^T = -D+ for zero values beyond the grid.
// A reverse step is two kernels, one thread per quad of four x points, every
// operand read straight from memory:
//   k_adj_pressure: the update of the pressure adjoint by the later step's
//       adjoint of g_d (-D-), then the pressure adjoint (gives that of q_d);
//   k_adj_velocity: the velocity adjoint (a stencil of the adjoint of q_d;
//       gives that of g_d);
// the first also takes the transpose of injection and recording on its tile.
// Gradients accumulate in FP64.
// The linear system only (no nonlinear factor); FP32 and FP64 media.
#include "fw_internal.h"
#include "fw_launch.cuh"

#include <algorithm>
#include <cmath>
#include <initializer_list>
#include <vector>

namespace fwgb {
cudaError_t launch_advance(int *d_it, int n, bool pdl, cudaStream_t s);
void *workspace_take(fw_medium *m, size_t bytes);
void workspace_give(fw_medium *m, void *p, size_t bytes);
size_t state_image_bytes(const fw_medium *m);
cudaError_t image_step_f32(const fw_medium *m, const StepImages &im, const int *zero, int it, bool record, bool pdl,
                           cudaStream_t s);
cudaError_t image_step_f64(const fw_medium *m, const StepImages &im, const int *zero, int it, bool record, bool pdl,
                           cudaStream_t s);
}  // namespace fwgb

using namespace fwgb;

namespace {

constexpr int kDStride = 16;   // derivative table per class: dA1[4], dB1[4], dA2[4], dB2[4]

// adjoint state: p, v_d, the memory variables of both sides and of the absorbing layer
template <typename R> struct AdjState {
    R *lp, *lv[3], *lpsi1[kMaxMech][3], *lpsi2[kMaxMech], *lpsi1p[3], *lpsi2p[3];
};

template <typename R> struct AdjArgs {
    int nx, ny, nz, px;
    long long plane;
    R c1, c2, c3, c4, dt;
    int wabs;          // absorbing width (0: none) and 1 / length of the tissue ramp
    R inv_lr;
    AdjState<R> L;     // adjoint state, updated in place from after the step to before it
    // forward state before the step (f) and velocity after it (fv1)
    const R *fp, *fpsi1[kMaxMech][3], *fpsi2[kMaxMech], *fpsi2p[3];
    const R *fv1[3];
    // maps and tables
    const R *kdt, *rho;
    const uint16_t *cls;
    const R *lut, *dlut;
    const R *pdh[3], *pah[3], *pdi[3], *pai[3];   // absorbing profile at half / integer points
    R *Q[3], *Gd[3];   // adjoints of q_d (this step) and of g_d (the later step, then this one)
    R *gsp;            // this step's pressure-side term of the gradient with respect to the d factor
    double *gk, *gs;
    // transpose of injection and recording by the pressure kernel's CTAs: their
    // cells' entries (IoEntry), ordered by tile (off null: none)
    const int *off;
    const IoEntry *ent;
    const R *waves, *G;        // source waveforms; dL/dtraces [receiver][n_col]
    const int *wave_of;
    int wave_len, n_col;
    int it, col;               // the step; trace column of the step before it (-1: not recorded)
    double inv_dxd;
};

// A thread's quad: coordinates, row lengths and strides per kernel axis
struct AdjPos {
    int c[3], n[3];
    long long st[3], i;
    unsigned tile;     // of the entries of sources and receivers
    bool on;
};

// CTAs of the reverse step: the tiles of the sweeps' sources and receivers
template <typename R, int DIM> struct AdjCta {
    static constexpr int BX = (DIM == 3 ? kTile3W : kTileW) / 4, BY = DIM == 3 ? tile3_rows(sizeof(R)) : kTileH;
};

template <typename R, int DIM> __device__ __forceinline__ AdjPos adj_pos(const AdjArgs<R> &A)
{
    constexpr int BX = AdjCta<R, DIM>::BX, BY = AdjCta<R, DIM>::BY;
    const unsigned gx = (unsigned)(A.nx + 4 * BX - 1) / (4 * BX);
    unsigned r = blockIdx.x / gx;
    AdjPos P;
    P.c[0] = 4 * (int)((blockIdx.x % gx) * BX + threadIdx.x);
    if (DIM == 3) {
        const unsigned gy = (unsigned)(A.ny + BY - 1) / BY;
        P.c[1] = (int)(r % gy) * BY + threadIdx.y;
        P.c[2] = (int)(r / gy);
        P.tile = ((r % gy) * gx + blockIdx.x % gx) * (unsigned)A.nz + r / gy;
    } else {
        P.c[1] = 0;
        P.c[2] = (int)r * BY + threadIdx.y;
        P.tile = blockIdx.x;
    }
    P.n[0] = A.nx; P.n[1] = A.ny; P.n[2] = A.nz;
    P.st[0] = 1; P.st[1] = A.px; P.st[2] = A.plane;
    P.on = P.c[0] < A.nx && P.c[1] < A.ny && P.c[2] < A.nz;
    P.i = (long long)P.c[2] * A.plane + (long long)P.c[1] * A.px + P.c[0];
    return P;
}

// staggered difference of f along axis ax at the quad's cells, zero beyond the
// grid: forward (at + 1/2) or backward
template <typename R, int ax, bool FORWARD>
__device__ __forceinline__ void adj_diff(const AdjArgs<R> &A, const AdjPos &P, const R *f, R (&out)[4])
{
    if (ax == 0) {
        R w[12], t[4];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const int x = P.c[0] + 4 * (k - 1);
            ld4_or_zero(f + P.i + 4 * (k - 1), x >= 0 && x < A.px, t);
#pragma unroll
            for (int e = 0; e < 4; ++e) w[4 * k + e] = t[e];
        }
        quad_diff_x(A, w, FORWARD ? 5 : 4, out);
    } else {
        R t[8][4];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int d = j - (FORWARD ? 3 : 4), c = P.c[ax] + d;
            ld4_or_zero(f + P.i + d * P.st[ax], c >= 0 && c < P.n[ax], t[j]);
        }
        quad_diff(A, t, out);
    }
}

// coefficients of one cell: 1/kappa (two parts), a, b and their derivatives by
// the factor on d
template <typename R, int NM> struct CellCoef {
    R ik, il, a[4], b[4], da[4], db[4];
    __device__ __forceinline__ void load(const AdjArgs<R> &A, int cls, int side)
    {
        lut2(A.lut, cls, side == 1 ? kLutIk1 : kLutIk2, ik, il);
        lut4(A.lut, cls, side == 1 ? kLutA1 : kLutA2, a);
        lut4(A.lut, cls, side == 1 ? kLutB1 : kLutB2, b);
        const R *d = A.dlut + (size_t)cls * kDStride + (side == 1 ? 0 : 8);
        Io<R>::ldg(d, da);
        Io<R>::ldg(d + 4, db);
    }
};

// tissue-mechanism strength of the cell e of the quad (the forward sweeps' ramp)
template <typename R>
__device__ __forceinline__ R adj_ramp(const AdjArgs<R> &A, const AdjPos &P, int e)
{
    const R s = fmax(fmax(layer_depth<R>(P.c[0] + e, A.nx, A.wabs), layer_depth<R>(P.c[1], A.ny, A.wabs)),
                     layer_depth<R>(P.c[2], A.nz, A.wabs));
    return ramp_of(s, A.inv_lr);
}

template <typename R, int DIM> __device__ __forceinline__ bool adj_in_layer(const AdjArgs<R> &A, const AdjPos &P, int ax)
{
    if (A.wabs <= 0 || (DIM == 2 && ax == 1)) return false;
    const int c = P.c[ax], last = ax == 0 ? c + 3 : c;
    return c < A.wabs || last >= P.n[ax] - A.wabs;
}

// Lines of the arrays a kernel reads late, on their way into L2 from its first
// instructions on (no registers held): 128^3, N = 2, one gradient 10.2 -> 9.8 ms
__device__ __forceinline__ void prefetch(const void *p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

__device__ __forceinline__ void add4(double *p, const double (&v)[4])
{
    double2 *q = reinterpret_cast<double2 *>(p);
    const double2 a = q[0], b = q[1];
    q[0] = make_double2(a.x + v[0], a.y + v[1]);
    q[1] = make_double2(b.x + v[2], b.y + v[3]);
}

// What bounds both kernels: DRAM and L2 traffic of one pass over the adjoint
// state, the forward images and the FP64 accumulators (about 220 bytes per
// point in 2D with three mechanisms); so there is no tile with recomputed
// halos: the adjoints of q_d and g_d go through global scratch (8 to 24 bytes
// per point each way, mostly L2 hits from one kernel to the next).
// Registers are held to four CTAs of 128 threads per SM in FP32.
template <typename R, int DIM, int NM>
__device__ __forceinline__ void adj_pressure_quad(const AdjArgs<R> &A, const AdjPos &P, const uint16_t (&cls)[4],
                                                  const R (&kd)[4])
{
    R lp[4], q[3][4], div[4], d[4];
#pragma unroll
    for (int ax = 0; ax < 3; ++ax)
        if (DIM == 3 || ax != 1) prefetch(A.fv1[ax] + P.i);
#pragma unroll
    for (int m = 0; m < NM; ++m) {
        prefetch(A.L.lpsi2[m] + P.i);
        prefetch(A.fpsi2[m] + P.i);
    }
    prefetch(A.gk + P.i);
    Io<R>::ld(A.L.lp + P.i, lp);
    adj_diff<R, 0, false>(A, P, A.Gd[0], d);
#pragma unroll
    for (int e = 0; e < 4; ++e) div[e] = d[e];
    if (DIM == 3) {
        adj_diff<R, 1, false>(A, P, A.Gd[1], d);
#pragma unroll
        for (int e = 0; e < 4; ++e) div[e] += d[e];
    }
    adj_diff<R, 2, false>(A, P, A.Gd[2], d);
#pragma unroll
    for (int e = 0; e < 4; ++e) lp[e] = P.c[0] + e < A.nx ? lp[e] - (div[e] + d[e]) : R(0);
    adj_diff<R, 0, false>(A, P, A.fv1[0], q[0]);
    adj_diff<R, 2, false>(A, P, A.fv1[2], q[2]);
    if (DIM == 3) adj_diff<R, 1, false>(A, P, A.fv1[1], q[1]);
#pragma unroll
    for (int e = 0; e < 4; ++e) div[e] = DIM == 3 ? q[0][e] + q[2][e] + q[1][e] : q[0][e] + q[2][e];
    R ln[NM][4], old[NM][4];
#pragma unroll
    for (int m = 0; m < NM; ++m) {
        Io<R>::ld(A.L.lpsi2[m] + P.i, ln[m]);
        Io<R>::ld(A.fpsi2[m] + P.i, old[m]);
    }
    const bool in[3] = {adj_in_layer<R, DIM>(A, P, 0), adj_in_layer<R, DIM>(A, P, 1), adj_in_layer<R, DIM>(A, P, 2)};
    R Q[4], gsp[4], stp[4], lst[4], ik[4];
    CellCoef<R, NM> C;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        if (e == 0 || cls[e] != cls[e - 1]) C.load(A, cls[e], 2);
        ik[e] = C.ik;
        const R r = in[0] || in[1] || in[2] ? adj_ramp(A, P, e) : R(1);
        lst[e] = -kd[e] * lp[e];
        const R rdiv = r * div[e], half = R(0.5) * lst[e];
        R lq = R(0), mem = R(0), gs = R(0);
#pragma unroll
        for (int m = 0; m < NM; ++m) {
            const R t = ln[m][e] + half, o = old[m][e];
            lq += C.a[m] * t;
            mem += o + (C.b[m] * o + C.a[m] * rdiv);
            gs += (C.db[m] * o + C.da[m] * rdiv) * t;
            ln[m][e] = C.b[m] * t + half;
        }
        Q[e] = fma(C.ik, lst[e], fma(C.il, lst[e], r * lq));
        stp[e] = fma(C.ik, div[e], fma(C.il, div[e], R(0.5) * mem));
        gsp[e] = gs;
    }
    pdl_launch();
    Io<R>::st(A.L.lp + P.i, lp);
#pragma unroll
    for (int m = 0; m < NM; ++m) Io<R>::st(A.L.lpsi2[m] + P.i, ln[m]);
    Io<R>::st(A.gsp + P.i, gsp);
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
        if (DIM == 2 && ax == 1) continue;
        R Qa[4] = {Q[0], Q[1], Q[2], Q[3]};
        if (in[ax]) {
            R a[4], b[4], lpn[4], po[4];
            if (ax == 0) quad_layer_ab(ik, A.pdi[0] + P.c[0], A.pai[0] + P.c[0], A.dt, a, b);
            else if (A.pdi[ax][P.c[ax]] > R(0))
                quad_layer_ab(ik, A.pdi[ax][P.c[ax]], A.pai[ax][P.c[ax]], A.dt, a, b);
            else b[0] = b[1] = b[2] = b[3] = R(2);
            Io<R>::ld(A.L.lpsi2p[ax] + P.i, lpn);
            Io<R>::ld(A.fpsi2p[ax] + P.i, po);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                if (!(b[e] <= R(1)) || P.c[0] + e >= A.nx) continue;   // zero profile, dead lane
                Qa[e] += a[e] * (lpn[e] + R(0.5) * lst[e]);
                stp[e] += R(0.5) * (R(1) + b[e]) * po[e] + R(0.5) * a[e] * q[ax][e];
                lpn[e] = b[e] * lpn[e] + R(0.5) * (R(1) + b[e]) * lst[e];
            }
            Io<R>::st(A.L.lpsi2p[ax] + P.i, lpn);
        }
        Io<R>::st(A.Q[ax] + P.i, Qa);
    }
    double gk[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) gk[e] = double(-stp[e] * lp[e]);
    add4(A.gk + P.i, gk);
}

template <typename R, int DIM, int NM>
__global__ void __launch_bounds__(AdjCta<R, DIM>::BX * AdjCta<R, DIM>::BY, sizeof(R) == 4 ? 4 : 1) k_adj_pressure(const __grid_constant__ AdjArgs<R> A)
{
    const AdjPos P = adj_pos<R, DIM>(A);
    uint16_t cls[4];
    R kd[4];
    int first = 0, last = 0;
    if (P.on) {
        quad_classes(__ldg(reinterpret_cast<const uint2 *>(A.cls + P.i)), cls);
        Io<R>::ldg(A.kdt + P.i, kd);
    }
    if (A.off) {
        first = __ldg(A.off + P.tile);
        last = __ldg(A.off + P.tile + 1);
    }
    pdl_wait();
    if (P.on) adj_pressure_quad<R, DIM, NM>(A, P, cls, kd);
    if (first >= last) return;
    // Transpose of injection and recording on the tile's cells, once their
    // pressure adjoint and source-gain gradient are stored: the gradient of the
    // gain of step it, then the adjoint of the earlier step's receiver.  (As a
    // kernel of its own 5 to 8 us per reverse step, 1 to 4 thousand sources.)
    __syncthreads();
    constexpr int BX = AdjCta<R, DIM>::BX, BY = AdjCta<R, DIM>::BY;
    for (int j = first + threadIdx.y * BX + threadIdx.x; j < last; j += BX * BY) {
        const IoEntry e = A.ent[j];
        const R l = A.L.lp[e.cell];
        if (e.src >= 0 && A.it < A.wave_len)
            A.gk[e.cell] += double(A.waves[(size_t)A.wave_of[e.src] * A.wave_len + A.it]) * double(l) * A.inv_dxd;
        if (e.rcv >= 0 && A.col >= 0) A.L.lp[e.cell] = l + A.G[(size_t)e.rcv * A.n_col + A.col];
    }
}

// velocity adjoint along ax; adds its terms to gs
template <typename R, int DIM, int NM, int ax>
__device__ __forceinline__ void adj_velocity_axis(const AdjArgs<R> &A, const AdjPos &P, const uint16_t (&cls)[4],
                                                  const R (&own)[4], const R (&rr)[4], R (&gs)[4])
{
    R lv[4], dq[4], g[4], nxt[4], ln[NM][4], old[NM][4], lg[4], lst[4], ik[4];
    Io<R>::ld(A.L.lv[ax] + P.i, lv);
#pragma unroll
    for (int m = 0; m < NM; ++m) {
        Io<R>::ld(A.L.lpsi1[m][ax] + P.i, ln[m]);
        Io<R>::ld(A.fpsi1[m][ax] + P.i, old[m]);
    }
    adj_diff<R, ax, true>(A, P, A.Q[ax], dq);
    adj_diff<R, ax, true>(A, P, A.fp, g);
    if (ax == 0) {
        nxt[0] = own[1]; nxt[1] = own[2]; nxt[2] = own[3];
        nxt[3] = P.c[0] + 4 < A.nx ? __ldg(A.rho + P.i + 4) : own[3];
    } else {
        ld4_or_zero(A.rho + P.i + P.st[ax], P.c[ax] + 1 < P.n[ax], nxt);
    }
    CellCoef<R, NM> C;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const bool live = P.c[0] + e < A.nx;
        if (ax == 0 ? P.c[0] + e + 1 >= A.nx : P.c[ax] + 1 >= P.n[ax]) nxt[e] = own[e];
        if (e == 0 || cls[e] != cls[e - 1]) C.load(A, cls[e], 1);
        ik[e] = C.ik;
        lv[e] = live ? lv[e] - dq[e] : R(0);
        lst[e] = live ? div_face(-A.dt, fma(R(0.5), nxt[e], R(0.5) * own[e])) * lv[e] : R(0);
        const R rg = live ? rr[e] * g[e] : R(0), half = R(0.5) * lst[e];
        R lq = R(0);
#pragma unroll
        for (int m = 0; m < NM; ++m) {
            const R t = ln[m][e] + half, o = old[m][e];
            lq += C.a[m] * t;
            gs[e] += (C.db[m] * o + C.da[m] * rg) * t;
            ln[m][e] = C.b[m] * t + half;
        }
        lg[e] = fma(C.ik, lst[e], fma(C.il, lst[e], rr[e] * lq));
    }
    Io<R>::st(A.L.lv[ax] + P.i, lv);
#pragma unroll
    for (int m = 0; m < NM; ++m) Io<R>::st(A.L.lpsi1[m][ax] + P.i, ln[m]);
    if (adj_in_layer<R, DIM>(A, P, ax)) {
        R a[4], b[4], lpn[4];
        if (ax == 0) quad_layer_ab(ik, A.pdh[0] + P.c[0], A.pah[0] + P.c[0], A.dt, a, b);
        else if (A.pdh[ax][P.c[ax]] > R(0)) quad_layer_ab(ik, A.pdh[ax][P.c[ax]], A.pah[ax][P.c[ax]], A.dt, a, b);
        else b[0] = b[1] = b[2] = b[3] = R(2);
        Io<R>::ld(A.L.lpsi1p[ax] + P.i, lpn);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            if (!(b[e] <= R(1)) || P.c[0] + e >= A.nx) continue;
            lg[e] += a[e] * (lpn[e] + R(0.5) * lst[e]);
            lpn[e] = b[e] * lpn[e] + R(0.5) * (R(1) + b[e]) * lst[e];
        }
        Io<R>::st(A.L.lpsi1p[ax] + P.i, lpn);
    }
    Io<R>::st(A.Gd[ax] + P.i, lg);
}

template <typename R, int DIM, int NM>
__global__ void __launch_bounds__(AdjCta<R, DIM>::BX * AdjCta<R, DIM>::BY, sizeof(R) == 4 ? 4 : 1) k_adj_velocity(const __grid_constant__ AdjArgs<R> A)
{
    const AdjPos P = adj_pos<R, DIM>(A);
    uint16_t cls[4];
    R own[4], gs[4], rr[4] = {R(1), R(1), R(1), R(1)};
    if (P.on) {
        quad_classes(__ldg(reinterpret_cast<const uint2 *>(A.cls + P.i)), cls);
        Io<R>::ldg(A.rho + P.i, own);
    }
    pdl_wait();
    if (!P.on) return;
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
        if (DIM == 2 && ax == 1) continue;
        prefetch(A.L.lv[ax] + P.i);
        prefetch(A.Q[ax] + P.i);
#pragma unroll
        for (int m = 0; m < NM; ++m) {
            prefetch(A.L.lpsi1[m][ax] + P.i);
            prefetch(A.fpsi1[m][ax] + P.i);
        }
    }
    prefetch(A.fp + P.i);
    prefetch(A.gs + P.i);
    // the pressure side's terms: in 2D they start the step's sum, in 3D (three
    // axes' terms more) the two sides add up in FP64 (128^3, N = 2: 9.58 ->
    // 9.68 ms per gradient of 48 steps; loaded at the end 9.74)
    if (DIM == 3) {
        prefetch(A.gsp + P.i);
        gs[0] = gs[1] = gs[2] = gs[3] = R(0);
    } else {
        Io<R>::ld(A.gsp + P.i, gs);
    }
    if (adj_in_layer<R, DIM>(A, P, 0) || adj_in_layer<R, DIM>(A, P, 1) || adj_in_layer<R, DIM>(A, P, 2))
#pragma unroll
        for (int e = 0; e < 4; ++e) rr[e] = adj_ramp(A, P, e);
    adj_velocity_axis<R, DIM, NM, 0>(A, P, cls, own, rr, gs);
    if (DIM == 3) adj_velocity_axis<R, DIM, NM, 1>(A, P, cls, own, rr, gs);
    R gp[4];
    if (DIM == 3) Io<R>::ld(A.gsp + P.i, gp);
    adj_velocity_axis<R, DIM, NM, 2>(A, P, cls, own, rr, gs);
    pdl_launch();
    double g[4] = {double(gs[0]), double(gs[1]), double(gs[2]), double(gs[3])};
    if (DIM == 3) {
#pragma unroll
        for (int e = 0; e < 4; ++e) g[e] += double(gp[e]);
    }
    add4(A.gs + P.i, g);
}

// adjoints of the last step's receivers (trace column col), before the first
// reverse step
template <typename R>
__global__ void k_adj_receivers(R *lp, const IoEntry *ent, int n, const R *G, int n_col, int col)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j < n && ent[j].rcv >= 0) lp[ent[j].cell] += G[(size_t)ent[j].rcv * n_col + col];
}

// internal gradients -> the user's grid (transpose of the layer inheritance)
template <typename R>
__global__ void k_grad_fold(const double *gk, const double *gs, const R *rho, const R *c, double dt, int nx,
                            int ny, int nz, int px, int w, double *uc, double *us)
{
    const long long n = (long long)nx * ny * nz;
    for (long long j = blockIdx.x * (long long)blockDim.x + threadIdx.x; j < n;
         j += (long long)gridDim.x * blockDim.x) {
        const int x = int(j % nx);
        const long long r = j / nx;
        const int y = int(r % ny), z = int(r / ny);
        auto clampw = [w](int cc, int n_) {
            if (w <= 0) return cc;
            int lo = min(w, n_ - 1), hi = max(n_ - 1 - w, 0);
            if (lo > hi) lo = hi = n_ / 2;
            return min(max(cc, lo), hi);
        };
        const int sx = clampw(x, nx), sy = ny > 1 ? clampw(y, ny) : y, sz = clampw(z, nz);
        const long long i = r * px + x;
        const long long t = ((long long)sz * ny + sy) * nx + sx;
        const double gc = gk[i] * 2.0 * double(rho[i]) * double(c[i]) * dt;
        if (gc != 0.0) atomicAdd(&uc[t], gc);
        if (gs[i] != 0.0) atomicAdd(&us[t], gs[i]);
    }
}

template <typename D>
__global__ void k_grad_out(const double *uc, const double *us, const float *a0f, const double *a0d, long long n,
                           D *gc, D *ga)
{
    for (long long j = blockIdx.x * (long long)blockDim.x + threadIdx.x; j < n;
         j += (long long)gridDim.x * blockDim.x) {
        if (gc) gc[j] = D(uc[j]);
        if (ga) {
            double g = us[j];
            if (a0f || a0d) {
                const double a = a0f ? double(a0f[j]) : a0d[j];
                g = a > 0.0 ? g / a : 0.0;
            }
            ga[j] = D(g);
        }
    }
}

template <typename R, int DIM, int NM>
cudaError_t launch_reverse_n(const AdjArgs<R> &A, int side, bool pdl, cudaStream_t s)
{
    constexpr int BX = AdjCta<R, DIM>::BX, BY = AdjCta<R, DIM>::BY;
    const unsigned gx = (unsigned)(A.nx + 4 * BX - 1) / (4 * BX);
    const unsigned rows = DIM == 3 ? (unsigned)(A.ny + BY - 1) / BY * (unsigned)A.nz : (unsigned)(A.nz + BY - 1) / BY;
    return launch_kernel(side == 2 ? k_adj_pressure<R, DIM, NM> : k_adj_velocity<R, DIM, NM>, dim3(gx * rows),
                         dim3(BX, BY), 0, s, pdl, A);
}

// one half of a reverse step (side 2: pressure, 1: velocity); instances per
// dimension and number of mechanisms (their loops unroll)
template <typename R>
cudaError_t launch_reverse(const AdjArgs<R> &A, int ndim, int nmech, int side, bool pdl, cudaStream_t s)
{
    const bool d3 = ndim == 3;
    switch (nmech) {
    case 1: return d3 ? launch_reverse_n<R, 3, 1>(A, side, pdl, s) : launch_reverse_n<R, 2, 1>(A, side, pdl, s);
    case 2: return d3 ? launch_reverse_n<R, 3, 2>(A, side, pdl, s) : launch_reverse_n<R, 2, 2>(A, side, pdl, s);
    case 3: return d3 ? launch_reverse_n<R, 3, 3>(A, side, pdl, s) : launch_reverse_n<R, 2, 3>(A, side, pdl, s);
    default: return d3 ? launch_reverse_n<R, 3, 4>(A, side, pdl, s) : launch_reverse_n<R, 2, 4>(A, side, pdl, s);
    }
}

int nblocks(long long n) { return (int)std::min<long long>((n + 255) / 256, 152LL * 16); }

// All device buffers of one gradient in one block: sized first (p null), then
// placed in the medium's workspace
struct Buf {
    void *p = nullptr;
    size_t bytes, at = 0;
    explicit Buf(size_t b) : bytes(b) {}
    Buf(const Buf &) = delete;
    Buf &operator=(const Buf &) = delete;
};

struct Workspace {
    fw_medium *m;
    cudaStream_t s;
    void *p = nullptr;
    size_t bytes = 0;
    Workspace(fw_medium *m_, cudaStream_t s_) : m(m_), s(s_) {}
    Workspace(const Workspace &) = delete;
    Workspace &operator=(const Workspace &) = delete;
    ~Workspace()
    {
        if (p) cudaStreamSynchronize(s);   // nothing of this call may still run in it
        workspace_give(m, p, bytes);
    }
    bool place(std::initializer_list<Buf *> bufs)
    {
        for (Buf *b : bufs) {
            b->at = bytes;
            bytes += (b->bytes + 255) / 256 * 256;
        }
        p = workspace_take(m, bytes);
        for (Buf *b : bufs)
            if (p && b->bytes) b->p = static_cast<char *>(p) + b->at;
        return p != nullptr;
    }
};

#define ADJ_CK(call)                                   \
    do {                                               \
        if ((call) != cudaSuccess) {                   \
            cudaGetLastError();                        \
            return FW_ERR_CUDA;                        \
        }                                              \
    } while (0)

// derivatives of a, b (Eqs. relaxation_a / relaxation_b) with respect to a
// factor s on d, at s = 1:
//   db/ds = -(d dt / kappa) b,
//   da/ds = d alpha (b - 1) / (d + kappa alpha)^2 + d / (kappa (d + kappa alpha)) db/ds
void dab(double d, double al, double ka, double dt, double &da, double &db)
{
    const double b = std::exp(-(d / ka + al) * dt);
    db = -(d * dt / ka) * b;
    da = d * al * (b - 1.0) / ((d + ka * al) * (d + ka * al)) + d / (ka * (d + ka * al)) * db;
}

// The recomputation's side stream and the events between it and the caller's
// stream; on every way out, both streams finish before the buffers go.
struct SideStream {
    cudaStream_t main = nullptr, side = nullptr;
    std::vector<cudaEvent_t> ev;
    SideStream() = default;
    SideStream(const SideStream &) = delete;
    SideStream &operator=(const SideStream &) = delete;
    ~SideStream()
    {
        if (side) {
            cudaStreamSynchronize(side);
            cudaStreamDestroy(side);
        }
        if (main) cudaStreamSynchronize(main);
        for (cudaEvent_t e : ev) cudaEventDestroy(e);
    }
};

template <typename R>
int gradient_impl(fw_medium *m, int n_steps, int K, const void *G, const void *alpha0, void *grad_c, void *grad_a,
                  int as_f64, cudaStream_t s)
{
    const size_t vol = m->vol, n_user = (size_t)m->NX * m->NY * m->NZ;
    const size_t SB = state_image_bytes(m);
    const int n_ck = (n_steps + K - 1) / K;
    const int seg_len = std::min(K, n_steps);
    char *slab = static_cast<char *>(m->slab);
    auto off = [slab](const void *p) { return (size_t)(static_cast<const char *>(p) - slab); };

    // segment images: the states after steps k0 .. k1-2 of a segment (the state
    // before it is its checkpoint, the state after it the next checkpoint)
    Buf lam(SB), ck((size_t)n_ck * SB), fin(SB);
    Buf seg0((size_t)std::max(seg_len - 1, 1) * SB), seg1(n_ck > 1 ? (size_t)std::max(seg_len - 1, 1) * SB : 0);
    // scratch: adjoints of q_d and g_d per axis, the pressure side's gradient term
    const size_t n_scratch = 2 * (size_t)m->ndim + 1;
    Buf scratch(n_scratch * vol * sizeof(R)), gacc(2 * vol * sizeof(double)),
        uacc(2 * n_user * sizeof(double));
    const size_t nG = (size_t)m->n_rcv * m->n_rec;
    Buf dG(nG * sizeof(R)), dA0(alpha0 ? n_user * (as_f64 ? 8 : 4) : 0);
    Buf dlut((size_t)m->n_classes * kDStride * sizeof(R)), zero(256);   // zero: step counter of the image steps
    const size_t eb = as_f64 ? 8 : 4;
    Buf out(2 * n_user * eb);
    Workspace ws(m, s);
    if (!ws.place({&lam, &ck, &fin, &seg0, &seg1, &scratch, &gacc, &uacc, &dG, &dA0, &dlut, &zero, &out}))
        return FW_ERR_NOMEM;
    ADJ_CK(cudaMemsetAsync(zero.p, 0, 256, s));
    ADJ_CK(cudaMemsetAsync(lam.p, 0, SB, s));
    ADJ_CK(cudaMemsetAsync(scratch.p, 0, n_scratch * vol * sizeof(R), s));
    ADJ_CK(cudaMemsetAsync(gacc.p, 0, 2 * vol * sizeof(double), s));
    ADJ_CK(cudaMemsetAsync(uacc.p, 0, 2 * n_user * sizeof(double), s));
    // receiver weights in the field type
    if (nG) {
        if (as_f64 == (sizeof(R) == 8)) {
            ADJ_CK(cudaMemcpyAsync(dG.p, G, nG * sizeof(R), cudaMemcpyDefault, s));
        } else {
            std::vector<R> h(nG);
            if (as_f64) {
                std::vector<double> t(nG);
                ADJ_CK(cudaMemcpy(t.data(), G, nG * 8, cudaMemcpyDefault));
                for (size_t k = 0; k < nG; ++k) h[k] = R(t[k]);
            } else {
                std::vector<float> t(nG);
                ADJ_CK(cudaMemcpy(t.data(), G, nG * 4, cudaMemcpyDefault));
                for (size_t k = 0; k < nG; ++k) h[k] = R(t[k]);
            }
            ADJ_CK(cudaMemcpyAsync(dG.p, h.data(), nG * sizeof(R), cudaMemcpyHostToDevice, s));
            ADJ_CK(cudaStreamSynchronize(s));
        }
    }
    if (alpha0) ADJ_CK(cudaMemcpyAsync(dA0.p, alpha0, n_user * (as_f64 ? 8 : 4), cudaMemcpyDefault, s));
    {
        std::vector<R> h((size_t)m->n_classes * kDStride, R(0));
        for (int c = 0; c < m->n_classes; ++c) {
            const fw_relax_params &p = m->classes[c];
            for (int k = 0; k < p.n_mech; ++k) {
                double da, db;
                dab(p.d1[k], p.alpha1[k], p.kappa1, m->dt, da, db);
                h[(size_t)c * kDStride + k] = R(da);
                h[(size_t)c * kDStride + 4 + k] = R(db);
                dab(p.d2[k], p.alpha2[k], p.kappa2, m->dt, da, db);
                h[(size_t)c * kDStride + 8 + k] = R(da);
                h[(size_t)c * kDStride + 12 + k] = R(db);
            }
        }
        ADJ_CK(cudaMemcpyAsync(dlut.p, h.data(), h.size() * sizeof(R), cudaMemcpyHostToDevice, s));
        ADJ_CK(cudaStreamSynchronize(s));
    }

    // ---- forward run ----
    // The adjoint begins with the last two segments, whose images have buffers of
    // their own (segs): their states are kept as the forward run passes them, by
    // image steps, and only the segments before them are recomputed.
    // (128 steps, K = 32: 62 recomputed steps instead of 124.)
    const long long it0 = m->step;
    const int n_run = std::max(0, n_ck - 2);      // segments run in place, recomputed later
    char *segs[2] = {static_cast<char *>(seg0.p), static_cast<char *>(seg1.p)};
    auto ck_at = [&](int si) { return static_cast<char *>(ck.p) + (size_t)si * SB; };
    // One step from image rd to image wr (memory variables in the state type:
    // FP32 or FP64 storage, the only ones fw_gradient accepts)
    auto image_step = [&](const char *rd, char *wr, int k, bool record, bool pdl, cudaStream_t st) -> cudaError_t {
        const StepImages im{rd, (long long)(wr - rd)};
        const int *z = static_cast<const int *>(zero.p);
        return sizeof(R) == 8 ? image_step_f64(m, im, z, (int)(it0 + k), record, pdl, st)
                              : image_step_f32(m, im, z, (int)(it0 + k), record, pdl, st);
    };
    // image steps do not write the padding of a row, and read it as zero
    if (m->px != m->NX)
        for (Buf *b : {&ck, &fin, &seg0, &seg1})
            if (b->p) ADJ_CK(cudaMemsetAsync(b->p, 0, b->bytes, s));
    // The last image becomes the medium's state.  Steps write the absorbing-layer
    // memories inside the layer only and nothing between the arrays: there it
    // starts with what the medium holds (a copy of 16 MiB at 1024^2, of the whole
    // image where the arrays' size leaves gaps between them).
    const size_t state_end = off(m->d_it);
    const size_t unwritten = vol * sizeof(R) % 256 ? 0 : m->psi1p[0] ? off(m->psi1p[0]) : state_end;
    if (unwritten < state_end)
        ADJ_CK(cudaMemcpyAsync(static_cast<char *>(fin.p) + unwritten, slab + unwritten, state_end - unwritten,
                               cudaMemcpyDeviceToDevice, s));
    for (int si = 0; si < n_ck; ++si) {
        const int k0 = si * K, k1 = std::min(n_steps, k0 + K);
        if (si <= n_run) ADJ_CK(cudaMemcpyAsync(ck_at(si), slab, SB, cudaMemcpyDeviceToDevice, s));
        if (si < n_run) {
            int rc = fw_run(m, k1 - k0, s);
            if (rc) return rc;
            continue;
        }
        const char *rd = ck_at(si);
        for (int k = k0; k < k1; ++k) {
            char *wr = k + 1 < k1 ? segs[si & 1] + (size_t)(k - k0) * SB
                                  : (si + 1 < n_ck ? ck_at(si + 1) : static_cast<char *>(fin.p));
            ADJ_CK(image_step(rd, wr, k, true, true, s));
            rd = wr;
        }
    }

    // ---- kernel arguments (pointers into images are set per step) ----
    AdjArgs<R> A{};
    A.nx = m->NX; A.ny = m->NY; A.nz = m->NZ; A.px = m->px;
    A.plane = (long long)m->plane;
    const double cm[4] = {1225.0 / 1024.0, -245.0 / 3072.0, 49.0 / 5120.0, -5.0 / 7168.0};
    A.c1 = R(cm[0] / m->dx); A.c2 = R(cm[1] / m->dx); A.c3 = R(cm[2] / m->dx); A.c4 = R(cm[3] / m->dx);
    A.dt = R(m->dt);
    A.wabs = m->wabs;
    A.inv_lr = m->wabs > 0 ? R(1) / R(m->g.transition > 0 ? m->g.transition : 0.5 * m->g.pml) : R(0);
    // the adjoint state's fields at the medium's offsets inside a state-sized buffer
    auto state_in = [&](void *buf) {
        char *L = static_cast<char *>(buf);
        AdjState<R> S{};
        S.lp = reinterpret_cast<R *>(L + off(m->p));
        for (int ax = 0; ax < 3; ++ax) {
            S.lv[ax] = m->v[ax] ? reinterpret_cast<R *>(L + off(m->v[ax])) : nullptr;
            S.lpsi1p[ax] = m->psi1p[ax] ? reinterpret_cast<R *>(L + off(m->psi1p[ax])) : nullptr;
            S.lpsi2p[ax] = m->psi2p[ax] ? reinterpret_cast<R *>(L + off(m->psi2p[ax])) : nullptr;
            for (int k = 0; k < m->nmech; ++k)
                S.lpsi1[k][ax] = m->psi1[k][ax] ? reinterpret_cast<R *>(L + off(m->psi1[k][ax])) : nullptr;
        }
        for (int k = 0; k < m->nmech; ++k) S.lpsi2[k] = reinterpret_cast<R *>(L + off(m->psi2[k]));
        return S;
    };
    A.L = state_in(lam.p);
    R *next = static_cast<R *>(scratch.p);
    for (int ax = 0; ax < 3; ++ax) {
        const bool layer = m->psi1p[ax] != nullptr;
        A.pdh[ax] = layer ? static_cast<const R *>(m->prof[ax][0]) : nullptr;
        A.pah[ax] = layer ? static_cast<const R *>(m->prof[ax][1]) : nullptr;
        A.pdi[ax] = layer ? static_cast<const R *>(m->prof[ax][2]) : nullptr;
        A.pai[ax] = layer ? static_cast<const R *>(m->prof[ax][3]) : nullptr;
        if (!m->v[ax]) continue;
        A.Q[ax] = next;
        A.Gd[ax] = next + vol;
        next += 2 * vol;
    }
    A.gsp = next;
    A.kdt = static_cast<const R *>(m->kdt);
    A.rho = static_cast<const R *>(m->rho);
    A.cls = m->cls;
    A.lut = static_cast<const R *>(m->lut);
    A.dlut = static_cast<const R *>(dlut.p);
    A.gk = static_cast<double *>(gacc.p);
    A.gs = static_cast<double *>(gacc.p) + vol;
    const double inv_dxd = 1.0 / std::pow(m->dx, m->ndim);
    // trace column of time step it, -1 where it is not recorded
    auto column = [m](long long it) {
        return m->n_rcv > 0 && it % m->decim == 0 && it / m->decim < m->n_rec ? (int)(it / m->decim) : -1;
    };
    if (m->n_ent > 0) {
        A.off = m->io_off;
        A.ent = static_cast<const IoEntry *>(m->ent_buf);
        A.waves = static_cast<const R *>(m->waves);
        A.wave_of = m->wave_of;
        A.wave_len = m->n_src > 0 ? m->wave_len : 0;
        A.G = static_cast<const R *>(dG.p);
        A.n_col = m->n_rec;
        A.inv_dxd = inv_dxd;
        const int col = column(it0 + n_steps - 1);
        if (col >= 0) {
            k_adj_receivers<R><<<(m->n_ent + 255) / 256, 256, 0, s>>>(A.L.lp, A.ent, m->n_ent, A.G, A.n_col, col);
            ADJ_CK(cudaGetLastError());
        }
    }

    // ---- reverse sweep, one checkpoint segment at a time ----
    // The recomputation of segment si - 1 (a side stream, into the other of two
    // image buffers) runs beside the adjoint of segment si: the adjoint reads
    // only the images and the medium's maps, never the medium's state.
    SideStream ss;
    ss.main = s;
    ADJ_CK(cudaStreamCreateWithFlags(&ss.side, cudaStreamNonBlocking));
    cudaEvent_t ev_start, rec_done[2], rev_done[2], side_done;
    for (cudaEvent_t *e : {&ev_start, &rec_done[0], &rec_done[1], &rev_done[0], &rev_done[1], &side_done}) {
        ADJ_CK(cudaEventCreateWithFlags(e, cudaEventDisableTiming));
        ss.ev.push_back(*e);
    }
    bool rev_recorded[2] = {false, false};
    // images after steps k0 .. k1-2 of segment si into segs[si & 1]: each step
    // reads the image before it (the checkpoint first) and writes the next
    auto recompute = [&](int si) -> int {
        const int k0 = si * K, k1 = std::min(n_steps, k0 + K);
        const char *rd = ck_at(si);
        for (int k = k0; k < k1 - 1; ++k) {
            char *wr = segs[si & 1] + (size_t)(k - k0) * SB;
            if (image_step(rd, wr, k, false, k > k0, ss.side) != cudaSuccess) return FW_ERR_CUDA;
            rd = wr;
        }
        return FW_OK;
    };
    ADJ_CK(cudaEventRecord(ev_start, s));   // the forward run and the checkpoints
    ADJ_CK(cudaStreamWaitEvent(ss.side, ev_start, 0));
    for (int si = n_ck - 1; si >= 0; --si) {
        const int k0 = si * K, k1 = std::min(n_steps, k0 + K);
        if (si < n_run) ADJ_CK(cudaStreamWaitEvent(s, rec_done[si & 1], 0));
        if (si >= 1 && si - 1 < n_run) {
            // segs[(si - 1) & 1] was last read by the adjoint of segment si + 1
            if (rev_recorded[(si + 1) & 1]) ADJ_CK(cudaStreamWaitEvent(ss.side, rev_done[(si + 1) & 1], 0));
            int rc = recompute(si - 1);
            if (rc) return rc;
            ADJ_CK(cudaEventRecord(rec_done[(si - 1) & 1], ss.side));
        }
        const char *ck_si = ck_at(si);
        // image j of the segment: the state after step k0 + j - 1
        auto image = [&](int j) -> const char * {
            if (j == 0) return ck_si;
            if (j == k1 - k0) return si + 1 < n_ck ? ck_si + SB : static_cast<const char *>(fin.p);
            return segs[si & 1] + (size_t)(j - 1) * SB;
        };
        for (int k = k1 - 1; k >= k0; --k) {
            const long long it = it0 + k;
            const char *F = image(k - k0), *F1 = image(k - k0 + 1);
            A.fp = reinterpret_cast<const R *>(F + off(m->p));
            for (int ax = 0; ax < 3; ++ax) {
                A.fv1[ax] = m->v[ax] ? reinterpret_cast<const R *>(F1 + off(m->v[ax])) : nullptr;
                A.fpsi2p[ax] = m->psi2p[ax] ? reinterpret_cast<const R *>(F + off(m->psi2p[ax])) : nullptr;
                for (int q = 0; q < m->nmech; ++q)
                    A.fpsi1[q][ax] = m->psi1[q][ax] ? reinterpret_cast<const R *>(F + off(m->psi1[q][ax])) : nullptr;
            }
            for (int q = 0; q < m->nmech; ++q) A.fpsi2[q] = reinterpret_cast<const R *>(F + off(m->psi2[q]));
            // a segment's first kernel follows an event of the side stream: no early start
            A.it = (int)it;
            A.col = k > 0 ? column(it - 1) : -1;
            ADJ_CK(launch_reverse<R>(A, m->ndim, m->nmech, 2, k < k1 - 1, s));
            ADJ_CK(launch_reverse<R>(A, m->ndim, m->nmech, 1, true, s));
        }
        ADJ_CK(cudaEventRecord(rev_done[si & 1], s));
        rev_recorded[si & 1] = true;
        ADJ_CK(cudaGetLastError());
    }
    ADJ_CK(cudaEventRecord(side_done, ss.side));
    ADJ_CK(cudaStreamWaitEvent(s, side_done, 0));
    // leave the medium at the end of the forward run: the fields of the last
    // image, the step counter past the image steps (images hold no counters; the
    // monitor has followed every step)
    ADJ_CK(cudaMemcpyAsync(slab, fin.p, state_end, cudaMemcpyDeviceToDevice, s));
    ADJ_CK(launch_advance(m->d_it, n_steps - n_run * K, false, s));
    m->step = it0 + n_steps;

    // ---- fold onto the user's grid and convert ----
    double *uc = static_cast<double *>(uacc.p), *us = uc + n_user;
    k_grad_fold<R><<<nblocks((long long)n_user), 256, 0, s>>>(A.gk, A.gs, A.rho, static_cast<const R *>(m->cdev),
                                                            m->dt, m->NX, m->NY, m->NZ, m->px, m->wabs, uc, us);
    ADJ_CK(cudaGetLastError());
    const float *a0f = alpha0 && !as_f64 ? static_cast<const float *>(dA0.p) : nullptr;
    const double *a0d = alpha0 && as_f64 ? static_cast<const double *>(dA0.p) : nullptr;
    if (as_f64) {
        double *o = static_cast<double *>(out.p);
        k_grad_out<double><<<nblocks((long long)n_user), 256, 0, s>>>(uc, us, a0f, a0d, (long long)n_user,
                                                                    grad_c ? o : nullptr, grad_a ? o + n_user : nullptr);
    } else {
        float *o = static_cast<float *>(out.p);
        k_grad_out<float><<<nblocks((long long)n_user), 256, 0, s>>>(uc, us, a0f, a0d, (long long)n_user,
                                                                   grad_c ? o : nullptr, grad_a ? o + n_user : nullptr);
    }
    ADJ_CK(cudaGetLastError());
    if (grad_c) ADJ_CK(cudaMemcpyAsync(grad_c, out.p, n_user * eb, cudaMemcpyDefault, s));
    if (grad_a)
        ADJ_CK(cudaMemcpyAsync(grad_a, static_cast<char *>(out.p) + n_user * eb, n_user * eb, cudaMemcpyDefault, s));
    ADJ_CK(cudaStreamSynchronize(s));
    m->last_stream = s;
    return FW_OK;
}

}  // namespace

extern "C" int fw_gradient(fw_medium *m, int n_steps, int checkpoint_every, const void *G, const void *alpha0,
                           void *grad_c, void *grad_alpha0, int as_f64, void *stream)
{
    if (!m || n_steps < 1 || (m->n_rcv > 0 && !G)) return FW_ERR_ARG;
    if (m->sticky) return m->sticky;
    if (m->nonlinear) return FW_ERR_UNSUPPORTED;
    if (m->time_order == 4) return FW_ERR_UNSUPPORTED;   // the transpose of the per-cell time-space weights is not built
    if (m->storage != FW_STORE_F32 && m->storage != FW_STORE_F64) return FW_ERR_UNSUPPORTED;
    if (m->NY > 65535 || m->NZ > 65535) return FW_ERR_UNSUPPORTED;   // the call's documented limit
    int K = checkpoint_every > 0 ? checkpoint_every : std::max(1, (int)std::lround(std::sqrt((double)n_steps)));
    K = std::min(K, n_steps);
    cudaStream_t s = (cudaStream_t)stream;
    if (cudaStreamSynchronize(m->last_stream) != cudaSuccess) {
        cudaGetLastError();
        return FW_ERR_CUDA;
    }
    return m->storage == FW_STORE_F64 ? gradient_impl<double>(m, n_steps, K, G, alpha0, grad_c, grad_alpha0, as_f64, s)
                                      : gradient_impl<float>(m, n_steps, K, G, alpha0, grad_c, grad_alpha0, as_f64, s);
}
