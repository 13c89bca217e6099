// Sweeps of 2D grids (kernel axes x and depth): one thread per quad of four
// consecutive x points, no march along the depth (the 3D sweeps' form).  A
// marching CTA walks its rows one after the other: on a 256^2 grid 32 CTAs of
// 64 threads did all the work (27 us per step, 6.3 us now).
//
// Small grids (k_velocity_plane, k_pressure_plane): bound by launches and by
// the latency of one pass of loads, so every stream is read straight into
// registers, all loads of a thread independent of each other; rows above and
// below are shared through L1 by the four rows of a CTA and through L2 by
// neighbouring CTAs.  Also FP64 media and image steps.
// Large FP32-state grids (k_velocity_tiles, k_pressure_tiles): bound by DRAM;
// see there.  The dispatch and its measurements are in fw_launch.cuh.
#pragma once

#include "fw_kernels.cuh"

namespace fwgb {

// position of a thread's quad; gx CTAs along x (a flat grid: depths beyond
// the grid's y limit stay possible)
struct PlanePos {
    int x0, z;
    bool on;
    long long row;
};

template <int BY, typename R> __device__ __forceinline__ PlanePos plane_pos(const Geo<R> &G, int gx)
{
    PlanePos P;
    P.x0 = 4 * (int)((blockIdx.x % gx) * (kTileW / 4) + threadIdx.x);
    P.z = (int)(blockIdx.x / gx) * BY + threadIdx.y;
    P.on = P.x0 < G.nx && P.z < G.nz;
    P.row = (long long)P.z * G.px + P.x0;
    return P;
}

// eight rows z + lo .. z + lo + 7 of f at this quad, zero outside the grid
template <typename SS, typename R>
__device__ __forceinline__ void plane_rows(const SS *f, const Geo<R> &G, const PlanePos &P, int lo, R (&t)[8][4])
{
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const int zz = P.z + lo + j;
        ld4_or_zero(f + P.row + (long long)(lo + j) * G.px, zz >= 0 && zz < G.nz, t[j]);
    }
}

// twelve values x0 - 4 .. x0 + 7 of row z of f (own: the middle four)
template <typename SS, typename R>
__device__ __forceinline__ void plane_row12(const SS *f, const Geo<R> &G, const PlanePos &P, const R (&own)[4], R (&w)[12])
{
    R l[4], r[4];
    ld4_or_zero(f + P.row - 4, P.x0 >= 4, l);
    ld4_or_zero(f + P.row + 4, P.x0 + 4 < G.px, r);
#pragma unroll
    for (int i = 0; i < 4; ++i) { w[i] = l[i]; w[i + 4] = own[i]; w[i + 8] = r[i]; }
}

// tissue strength of the quad's cells
template <typename R>
__device__ __forceinline__ void plane_ramp(const Geo<R> &G, const PlanePos &P, R (&rr)[4])
{
    const R sz = layer_depth<R>(P.z, G.nz, G.wabs), inv_lr = R(1) / G.lr;
#pragma unroll
    for (int e = 0; e < 4; ++e) rr[e] = ramp_of(fmax(layer_depth<R>(P.x0 + e, G.nx, G.wabs), sz), inv_lr);
}

// The absorbing mechanism along ax (0 or 2) of the quad: ik its cells'
// 1 / kappa, g the derivative, pp the memory; its term is added to st
template <typename R>
__device__ __forceinline__ void plane_layer(const R *const (&pd)[3], const R *const (&pa)[3], const R (&ik)[4], R dt,
                                            int ax, const PlanePos &P, const R (&g)[4], R (&pp)[4], R (&st)[4])
{
    R a[4], b[4], w[4] = {R(0.5), R(0.5), R(0.5), R(0.5)};
    if (ax == 0) {
        quad_layer_ab(ik, pd[0] + P.x0, pa[0] + P.x0, dt, a, b);
        quad_layer_weights(b, w);
    } else {
        const R d = pd[2][P.z];
        if (!(d > R(0))) return;
        quad_layer_ab(ik, d, pa[2][P.z], dt, a, b);
    }
    quad_layer(a, b, w, g, pp, st);
}

// Time-space stencil (see vel_gradient_ts): gradient of p at the two faces of
// the quad's cells; q rows z-3 .. z+4, w columns x0-4 .. x0+7, pm4 / pp4
// column x0+4 of rows z-1 / z+1, ppm1 column x0-1 of row z+1
template <typename R>
__device__ __forceinline__ void vel_gradient_ts_plane(const Geo<R> &G, const R (&kd)[4], const R (&rho)[4],
                                                      const R (&q)[8][4], const R (&w)[12], R pm4, R pp4, R ppm1,
                                                      int x0, R (&g)[3][4])
{
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const R r2 = x0 + e < G.nx ? kd[e] * G.r2s * rcp_face(rho[e]) : R(0);
        R a[4], b;
        ts_weights(G, r2, a, b);
        const R qm1 = e < 3 ? q[2][e + 1] : pm4, qp1 = e < 3 ? q[4][e + 1] : pp4, pl = e > 0 ? q[4][e - 1] : ppm1;
        g[0][e] = a[0] * (w[e + 5] - w[e + 4]) + a[1] * (w[e + 6] - w[e + 3]) + a[2] * (w[e + 7] - w[e + 2]) +
                  a[3] * (w[e + 8] - w[e + 1]) + b * ((qm1 - q[2][e]) + (qp1 - q[4][e]));
        g[2][e] = a[0] * (q[4][e] - q[3][e]) + a[1] * (q[5][e] - q[2][e]) + a[2] * (q[6][e] - q[1][e]) +
                  a[3] * (q[7][e] - q[0][e]) + b * ((pl - w[e + 3]) + (qp1 - w[e + 5]));
    }
}

// ... and the divergence terms (see pres_divergence_ts): qz rows z-4 .. z+3 of
// v_z, w columns x0-4 .. x0+7 of v_x, up / dn v_x of rows z-1 / z+1 (um1 / dm1
// column x0-1), v_z of columns x0-1 (l0, l1) and x0+4 (r0, r1) of rows z, z-1
template <typename R>
__device__ __forceinline__ void pres_divergence_ts_plane(const Geo<R> &G, const R (&kd)[4], const R (&rh)[4],
                                                         const R (&qz)[8][4], const R (&w)[12], const R (&up)[4],
                                                         const R (&dn)[4], R um1, R dm1, R l0, R l1, R r0, R r1,
                                                         int x0, R (&qd)[3][4])
{
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const R r2 = x0 + e < G.nx ? kd[e] * G.r2s * rcp_face(rh[e]) : R(0);
        R a[4], b;
        ts_weights(G, r2, a, b);
        const R X0 = (up[e] - (e > 0 ? up[e - 1] : um1)) + (dn[e] - (e > 0 ? dn[e - 1] : dm1));
        const R a0 = e > 0 ? qz[4][e - 1] : l0, a1 = e > 0 ? qz[3][e - 1] : l1;
        const R b0 = e < 3 ? qz[4][e + 1] : r0, b1 = e < 3 ? qz[3][e + 1] : r1;
        qd[0][e] = a[0] * (w[e + 4] - w[e + 3]) + a[1] * (w[e + 5] - w[e + 2]) + a[2] * (w[e + 6] - w[e + 1]) +
                   a[3] * (w[e + 7] - w[e + 0]) + b * X0;
        qd[2][e] = a[0] * (qz[4][e] - qz[3][e]) + a[1] * (qz[5][e] - qz[2][e]) + a[2] * (qz[6][e] - qz[1][e]) +
                   a[3] * (qz[7][e] - qz[0][e]) + b * ((a0 - a1) + (b0 - b1));
    }
}

// -dt / face density along x and z (the mean of the two cells; a last face has
// its own cell's); dead lanes (x >= nx) get no drive, so that their memory
// variables and v stay exactly 0
template <typename R>
__device__ __forceinline__ void vel_faces_plane(const Geo<R> &G, const R (&own)[4], R (&nx1)[4], R (&nz1)[4], int x0,
                                                int z, R (&g)[3][4], R (&dtr)[3][4])
{
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        if (x0 + e + 1 >= G.nx) nx1[e] = own[e];
        if (z + 1 >= G.nz) nz1[e] = own[e];
        const R ho = R(0.5) * own[e];
        dtr[0][e] = div_face(-G.dt, fma(R(0.5), nx1[e], ho));
        dtr[2][e] = div_face(-G.dt, fma(R(0.5), nz1[e], ho));
        if (x0 + e >= G.nx) g[0][e] = g[2][e] = dtr[0][e] = dtr[2][e] = R(0);
    }
}

// divergence of the quad's cells, nothing in dead lanes
template <typename R>
__device__ __forceinline__ void pres_div_plane(const Geo<R> &G, int x0, R (&qd)[3][4], R (&div)[4])
{
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        if (x0 + e >= G.nx) qd[0][e] = qd[2][e] = R(0);
        div[e] = qd[0][e] + qd[2][e];
    }
}

// CTAs per SM the registers are held to: five of 128 threads with up to two
// mechanisms (360x992, 720 CTAs, one wave instead of two: 13.0 -> 10.6 us per
// step), four above (five spill: 512^2, N = 4, 10.7 -> 11.5 us)
template <typename R, int NM, bool TS> constexpr int plane_ctas()
{
    return sizeof(R) == 4 ? (NM <= 2 && !TS ? 5 : 4) : 1;
}

// Velocity sweep: v_x, v_z and the memory variables of the gradient side
template <typename R, typename SS, typename SP, int NM, int BY, bool TS>
__global__ void __launch_bounds__(32 * BY, plane_ctas<R, NM, TS>())
k_velocity_plane(const __grid_constant__ VelArgs<R, SS, SP> A, int gx)
{
    const Geo<R> &G = A.g;
    const PlanePos P = plane_pos<BY>(G, gx);
    if (!P.on) {
        pdl_wait();
        return;
    }
    const long long row = P.row;
    const int x0 = P.x0, z = P.z;

    // maps and tables first, then (after the wait) every stream of the quad
    R q[8][4], w[12], own[4], nx1[4], nz1[4], vv[2][4], ps[2][NM][4];
    const uint2 cl = __ldg(reinterpret_cast<const uint2 *>(A.cls + row));
    Io<SS>::ldg(A.rho + row, own);
    ld4_or_zero(A.rho + row + G.px, z + 1 < G.nz, nz1);
    nx1[0] = own[1]; nx1[1] = own[2]; nx1[2] = own[3];
    nx1[3] = ldz1<SS, R>(A.rho + row + 4, x0 + 4 < G.nx);
    uint16_t cls4[4];
    quad_classes(cl, cls4);
    QuadCoef<R, NM> C;
    C.load(A.lut, cls4, kLutA1, kLutB1, kLutIk1);
    pdl_wait();
    pdl_launch();
    plane_rows(A.p, G, P, -3, q);
    plane_row12(A.p, G, P, q[3], w);
#pragma unroll
    for (int ax = 0; ax < 2; ++ax) {
        Io<SS>::ld(A.v[2 * ax] + row, vv[ax]);
#pragma unroll
        for (int m = 0; m < NM; ++m) Io<SP>::ld(A.psi[m][2 * ax] + row, ps[ax][m]);
    }

    R g[3][4], dtr[3][4];
    if (TS) {   // the time-space stencil (see vel_gradient_ts)
        R kd[4];
        Io<SS>::ldg(A.kdt + row, kd);
        const bool up = z >= 1, dn = z + 1 < G.nz, rt = x0 + 4 < G.px;
        vel_gradient_ts_plane(G, kd, own, q, w, ldz1<SS, R>(A.p + row - G.px + 4, up && rt),
                              ldz1<SS, R>(A.p + row + G.px + 4, dn && rt),
                              ldz1<SS, R>(A.p + row + G.px - 1, dn && x0 >= 1), x0, g);
    } else {
        quad_diff_x(G, w, 5, g[0]);
        quad_diff(G, q, g[2]);
    }
    vel_faces_plane(G, own, nx1, nz1, x0, z, g, dtr);
    const bool in[3] = {G.wabs > 0 && (x0 < G.wabs || x0 + 3 >= G.nx - G.wabs), false,
                        G.wabs > 0 && (z < G.wabs || z >= G.nz - G.wabs)};
    R rr[4] = {R(1), R(1), R(1), R(1)};
    if (in[0] || in[2]) plane_ramp(G, P, rr);
#pragma unroll
    for (int ax = 0; ax < 3; ax += 2) {
        R(&v)[4] = vv[ax / 2], (&pa)[NM][4] = ps[ax / 2], stv[4];
        quad_stretch<R, NM>(C, g[ax], rr, G.hs1, pa, stv);
        if (in[ax]) {
            R pp[4];
            Io<SS>::ld(A.psip[ax] + row, pp);
            plane_layer(A.pd, A.pa, C.ik, G.dt, ax, P, g[ax], pp, stv);
            Io<SS>::st(wr_at(A.psip[ax] + row, A.wofs), pp);
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) unpair(v, h, p_fma(pair(dtr[ax], h), pair(stv, h), pair(v, h)));
        Io<SS>::st(wr_at(A.v[ax] + row, A.wofs), v);
#pragma unroll
        for (int m = 0; m < NM; ++m) Io<SP>::st(wr_at(A.psi[m][ax] + row, A.wofs), pa[m]);
    }
}

// Pressure sweep: p, the memory variables of the divergence side, the monitor
template <typename R, typename SS, typename SP, int NM, int BY, bool NL, bool TS>
__global__ void __launch_bounds__(32 * BY, plane_ctas<R, NM, TS>())
k_pressure_plane(const __grid_constant__ PresArgs<R, SS, SP> A, int gx)
{
    const Geo<R> &G = A.g;
    const PlanePos P = plane_pos<BY>(G, gx);
    PMax<R> pmax;
    int io0 = 0, io1 = 0;                          // this tile's sources and receivers
    if (A.io.off) {
        io0 = __ldg(A.io.off + blockIdx.x);
        io1 = __ldg(A.io.off + blockIdx.x + 1);
    }
    if (!P.on) {
        pdl_wait();
    } else {
        const long long row = P.row;
        const int x0 = P.x0, z = P.z;
        R qz[8][4], w[12], own[4], kd[4], bd[4], pv[4], ps[NM][4];
        const uint2 cl = __ldg(reinterpret_cast<const uint2 *>(A.cls + row));
        Io<SS>::ldg(A.kdt + row, kd);
        if (NL) Io<SS>::ldg(A.b2dt + row, bd);
        uint16_t cls4[4];
        quad_classes(cl, cls4);
        QuadCoef<R, NM> C;
        C.load(A.lut, cls4, kLutA2, kLutB2, kLutIk2);
        pdl_wait();
        pdl_launch();
        plane_rows(A.v[2], G, P, -4, qz);
        Sm<SS>::ld(A.v[0] + row, own);
        plane_row12(A.v[0], G, P, own, w);
        Io<SS>::ld(A.p + row, pv);
#pragma unroll
        for (int m = 0; m < NM; ++m) Io<SP>::ld(A.psi[m] + row, ps[m]);
        R qd[3][4];
        if (TS) {   // the time-space stencil (see pres_divergence_ts)
            R rh[4], up[4], dn[4];
            Io<SS>::ldg(A.rho + row, rh);
            const bool okm = z >= 1, okp = z + 1 < G.nz, lf = x0 >= 1, rt = x0 + 4 < G.px;
            ld4_or_zero(A.v[0] + row - G.px, okm, up);
            ld4_or_zero(A.v[0] + row + G.px, okp, dn);
            pres_divergence_ts_plane(
                G, kd, rh, qz, w, up, dn, ldz1<SS, R>(A.v[0] + row - G.px - 1, okm && lf),
                ldz1<SS, R>(A.v[0] + row + G.px - 1, okp && lf), ldz1<SS, R>(A.v[2] + row - 1, lf),
                ldz1<SS, R>(A.v[2] + row - G.px - 1, lf && okm), ldz1<SS, R>(A.v[2] + row + 4, rt),
                ldz1<SS, R>(A.v[2] + row - G.px + 4, rt && okm), x0, qd);
        } else {
            quad_diff_x(G, w, 4, qd[0]);
            quad_diff(G, qz, qd[2]);
        }
        R div[4], stp[4];
        pres_div_plane(G, x0, qd, div);
        const bool in[3] = {G.wabs > 0 && (x0 < G.wabs || x0 + 3 >= G.nx - G.wabs), false,
                            G.wabs > 0 && (z < G.wabs || z >= G.nz - G.wabs)};
        R rr[4] = {R(1), R(1), R(1), R(1)};
        if (in[0] || in[2]) plane_ramp(G, P, rr);
        quad_stretch<R, NM>(C, div, rr, G.hs2, ps, stp);
#pragma unroll
        for (int m = 0; m < NM; ++m) Io<SP>::st(wr_at(A.psi[m] + row, A.wofs), ps[m]);
#pragma unroll
        for (int ax = 0; ax < 3; ax += 2) {
            if (!in[ax]) continue;
            R pp[4];
            Io<SS>::ld(A.psip[ax] + row, pp);
            plane_layer(A.pd, A.pa, C.ik, G.dt, ax, P, qd[ax], pp, stp);
            Io<SS>::st(wr_at(A.psip[ax] + row, A.wofs), pp);
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const R fac = NL ? fma(bd[e], pv[e], kd[e]) : kd[e];
            pv[e] = fma(-fac, stp[e], pv[e]);
            pmax.see(pv[e]);
        }
        Io<SS>::st(wr_at(A.p + row, A.wofs), pv);
    }
    if (io0 < io1) tile_io(A.io, wr_at(A.p, A.wofs), io0, io1, threadIdx.y * 32 + threadIdx.x, 32 * BY, A.mon);
    record_max(A.mon, pmax);
}

// ---------------------------------------------------------------------------
// large FP32-state grids: tiles staged by TMA

// A tile is 128 x 4 points, one quad per thread.  A CTA walks a short run of
// tiles down a strip of 128 columns and keeps NS - 1 of them in flight ahead
// of the one it computes, each with its halos in one box per stream; nothing
// is carried from tile to tile but the coefficients of the last classes.
constexpr int kTileN = kTileW * kTileH;
static_assert(kTileW == 4 * 32, "a warp per row: walk_tiles, tile_io");

constexpr size_t pad128(size_t b) { return (b + 127) / 128 * 128; }

template <typename SP, int NM, bool TS> struct VelTile {
    static constexpr int SW = kTileW + 8, SH = kTileH + 7, RW = kTileW + 4;
    static constexpr size_t o_v = 0;
    static constexpr size_t o_psi = o_v + 2 * kTileN * 4;
    static constexpr size_t o_cls = o_psi + (size_t)NM * 2 * kTileN * sizeof(SP);
    static constexpr size_t o_kv = o_cls + kTileN * 2;
    static constexpr size_t o_sp = o_kv + (TS ? kTileN * 4 : 0);
    static constexpr size_t o_sr = o_sp + pad128(SW * SH * 4);
    static constexpr size_t stage = o_sr + pad128(RW * (kTileH + 1) * 4);
};

template <typename SP, int NM, bool NL, bool TS> struct PresTile {
    static constexpr int XW = kTileW + 8, XH = kTileH + (TS ? 2 : 0), ZW = kTileW + (TS ? 8 : 0), ZH = kTileH + 7;
    static constexpr size_t o_p = 0;
    static constexpr size_t o_kd = o_p + kTileN * 4;
    static constexpr size_t o_bd = o_kd + kTileN * 4;
    static constexpr size_t o_rh = o_bd + (NL ? kTileN * 4 : 0);
    static constexpr size_t o_psi = o_rh + (TS ? kTileN * 4 : 0);
    static constexpr size_t o_cls = o_psi + (size_t)NM * kTileN * sizeof(SP);
    static constexpr size_t o_vx = o_cls + kTileN * 2;
    static constexpr size_t o_vz = o_vx + pad128(XW * XH * 4);
    static constexpr size_t stage = o_vz + pad128(ZW * ZH * 4);
};

// The walk of a CTA over its run of tiles (gx strips, n_rows tiles per strip):
// load(warp, position, stage, barrier) arms the barrier with the bytes of the
// warp's share of a tile's copies and issues them NS - 1 tiles ahead,
// body(position, stage, wait) computes it in all, after() follows it.  Waits are
// bounded; after a timeout the sweep is flagged on the monitor.
template <int NS, size_t STAGE, typename Load, typename Body, typename After>
__device__ __forceinline__ void walk_tiles(unsigned char *smem, int gx, int run, int n_rows, Monitor *mon, const Load &load,
                                           const Body &body, const After &after)
{
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + NS * STAGE);
    const bool lead = threadIdx.x == 0 && threadIdx.y < 3;   // three warps issue a share of the copies each
    if (threadIdx.x == 0 && threadIdx.y == 0) {
        for (int b = 0; b < NS; ++b) mbar_init(bars + b, 3);
        mbar_fence_init();
    }
    __syncthreads();
    const int xb = (int)(blockIdx.x % gx) * kTileW, r0 = (int)(blockIdx.x / gx) * run;
    const int n = min(run, n_rows - r0);
    auto issue = [&](int i) {
        if (!lead || i >= n) return;
        fence_proxy_async_smem();
        load(threadIdx.y, xb, (r0 + i) * kTileH, smem + (i % NS) * STAGE, bars + i % NS);
    };
    pdl_wait();
    for (int i = 0; i < NS - 1; ++i) issue(i);
    bool timed_out = false;
    for (int i = 0; i < n; ++i) {
        if (i > 0) __syncthreads();        // tile i - 1 is done with the stage that tile i + NS - 1 takes
        issue(i + NS - 1);
        if (i + 1 == n) pdl_launch();
        body(xb, (r0 + i) * kTileH, smem + (i % NS) * STAGE, [&] {
            if (!timed_out && !mbar_wait_bounded(bars + i % NS, (unsigned)(i / NS) & 1u)) timed_out = true;
        });
        after();
    }
    if (timed_out) {
        // record it and give the copies in flight one more bounded chance to
        // land before the CTA's shared memory is released
        atomicExch(&mon->timeout, 1);
        for (int j = max(0, n - NS); j < n; ++j) mbar_wait_bounded(bars + j % NS, (unsigned)(j / NS) & 1u);
    }
}

template <typename SP, int NM, bool TS, int NS>
__global__ void __launch_bounds__(128, 3)
k_velocity_tiles(const __grid_constant__ VelArgs<float, float, SP> A, const __grid_constant__ VelMaps M, int gx,
                 int run, int n_rows)
{
    using L = VelTile<SP, NM, TS>;
    extern __shared__ __align__(128) unsigned char smem[];
    const Geo<float> &G = A.g;
    const int tx = threadIdx.x, ty = threadIdx.y, e0 = ty * kTileW + 4 * tx;
    QuadCoef<float, NM> C;
    uint2 key = make_uint2(0xffffffffu, 0xffffffffu);
    auto load = [&](int w, int xb, int zb, unsigned char *st, uint64_t *bar) {
        if (w == 0) {
            mbar_expect_tx(bar, (unsigned)((L::SW * L::SH + L::RW * (kTileH + 1) + (TS ? kTileN : 0)) * 4 + kTileN * 2));
            tma_load_3d(st + L::o_sp, &M.p_halo, xb - 4, 0, zb - 3, bar);
            tma_load_3d(st + L::o_sr, &M.rho_halo, xb, 0, zb, bar);
            tma_load_3d(st + L::o_cls, &M.cls, xb, 0, zb, bar);
            if (TS) tma_load_3d(st + L::o_kv, &M.kdt, xb, 0, zb, bar);
            return;
        }
        const int s = w - 1;
        mbar_expect_tx(bar, (unsigned)(kTileN * (4 + NM * sizeof(SP))));
        tma_load_3d(st + L::o_v + s * kTileN * 4, &M.v[2 * s], xb, 0, zb, bar);
#pragma unroll
        for (int m = 0; m < NM; ++m)
            tma_load_3d(st + L::o_psi + (2 * m + s) * kTileN * sizeof(SP), &M.psi[m][2 * s], xb, 0, zb, bar);
    };
    walk_tiles<NS, L::stage>(smem, gx, run, n_rows, A.mon, load, [&](int xb, int zb, unsigned char *st, auto wait) {
        PlanePos P;
        P.x0 = xb + 4 * tx;
        P.z = zb + ty;
        P.on = P.x0 < G.nx && P.z < G.nz;
        P.row = (long long)P.z * G.px + P.x0;
        const int x0 = P.x0, z = P.z;
        const bool in[3] = {P.on && G.wabs > 0 && (x0 < G.wabs || x0 + 3 >= G.nx - G.wabs), false,
                            P.on && G.wabs > 0 && (z < G.wabs || z >= G.nz - G.wabs)};
        float pp[3][4];                    // absorbing-layer memory, on its way while the tile lands
#pragma unroll
        for (int ax = 0; ax < 3; ax += 2)
            if (in[ax]) Io<float>::ld(A.psip[ax] + P.row, pp[ax]);
        wait();
        if (!P.on) return;
        const float *sp = reinterpret_cast<const float *>(st + L::o_sp) + ty * L::SW + 4 * tx;   // row z - 3, column x0 - 4
        const float *sr = reinterpret_cast<const float *>(st + L::o_sr) + ty * L::RW + 4 * tx;
        const uint2 cl = *reinterpret_cast<const uint2 *>(reinterpret_cast<const uint16_t *>(st + L::o_cls) + e0);
        uint16_t cls4[4];
        quad_classes(cl, cls4);
        if (cl.x != key.x || cl.y != key.y) {
            C.load(A.lut, cls4, kLutA1, kLutB1, kLutIk1);
            key = cl;
        }
        float q[8][4], w[12], own[4], nx1[4], nz1[4], g[3][4], dtr[3][4];
#pragma unroll
        for (int r = 0; r < 8; ++r) Sm<float>::ld(sp + r * L::SW + 4, q[r]);
        Sm<float>::ld12(sp + 3 * L::SW, w);
        Sm<float>::ld(sr, own);
        Sm<float>::ld(sr + L::RW, nz1);
        nx1[0] = own[1]; nx1[1] = own[2]; nx1[2] = own[3]; nx1[3] = sr[4];
        if (TS) {
            float kd[4];
            Sm<float>::ld(reinterpret_cast<const float *>(st + L::o_kv) + e0, kd);
            const float pm4 = sp[2 * L::SW + 8], pp4 = sp[4 * L::SW + 8], ppm1 = sp[4 * L::SW + 3];
            vel_gradient_ts_plane(G, kd, own, q, w, pm4, pp4, ppm1, x0, g);
        } else {
            quad_diff_x(G, w, 5, g[0]);
            quad_diff(G, q, g[2]);
        }
        vel_faces_plane(G, own, nx1, nz1, x0, z, g, dtr);
        float rr[4] = {1.0f, 1.0f, 1.0f, 1.0f};
        if (in[0] || in[2]) plane_ramp(G, P, rr);
#pragma unroll
        for (int ax = 0; ax < 3; ax += 2) {
            float vv[4], ps[NM][4], stv[4];
            Sm<float>::ld(reinterpret_cast<const float *>(st + L::o_v) + (ax / 2) * kTileN + e0, vv);
#pragma unroll
            for (int m = 0; m < NM; ++m)
                Sm<SP>::ld(reinterpret_cast<const SP *>(st + L::o_psi) + (2 * m + ax / 2) * kTileN + e0, ps[m]);
            quad_stretch<float, NM>(C, g[ax], rr, G.hs1, ps, stv);
            if (in[ax]) {
                plane_layer(A.pd, A.pa, C.ik, G.dt, ax, P, g[ax], pp[ax], stv);
                Io<float>::st(A.psip[ax] + P.row, pp[ax]);
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) unpair(vv, h, p_fma(pair(dtr[ax], h), pair(stv, h), pair(vv, h)));
            Io<float>::st(A.v[ax] + P.row, vv);
#pragma unroll
            for (int m = 0; m < NM; ++m) Io<SP>::st(A.psi[m][ax] + P.row, ps[m]);
        }
    }, [] {});
}

template <typename SP, int NM, bool NL, bool TS, int NS>
__global__ void __launch_bounds__(128, TS ? 3 : 4)
k_pressure_tiles(const __grid_constant__ PresArgs<float, float, SP> A, const __grid_constant__ PresMaps M, int gx,
                 int run, int n_rows)
{
    using L = PresTile<SP, NM, NL, TS>;
    extern __shared__ __align__(128) unsigned char smem[];
    const Geo<float> &G = A.g;
    const int tx = threadIdx.x, ty = threadIdx.y, e0 = ty * kTileW + 4 * tx;
    QuadCoef<float, NM> C;
    uint2 key = make_uint2(0xffffffffu, 0xffffffffu);
    PMax<float> pmax;
    auto load = [&](int w, int xb, int zb, unsigned char *st, uint64_t *bar) {
        if (w == 0) {
            mbar_expect_tx(bar, (unsigned)((L::XW * L::XH + L::ZW * L::ZH) * 4));
            tma_load_3d(st + L::o_vx, TS ? &M.vx_ring : &M.vx_halo, xb - 4, 0, TS ? zb - 1 : zb, bar);
            tma_load_3d(st + L::o_vz, TS ? &M.vz_ring : &M.vz_own, TS ? xb - 4 : xb, 0, zb - 4, bar);
        } else if (w == 1) {
            mbar_expect_tx(bar, (unsigned)(kTileN * 4 * (2 + (NL ? 1 : 0) + (TS ? 1 : 0))));
            tma_load_3d(st + L::o_p, &M.p_own, xb, 0, zb, bar);
            tma_load_3d(st + L::o_kd, &M.kdt, xb, 0, zb, bar);
            if (NL) tma_load_3d(st + L::o_bd, &M.b2dt, xb, 0, zb, bar);
            if (TS) tma_load_3d(st + L::o_rh, &M.rho_own, xb, 0, zb, bar);
        } else {
            mbar_expect_tx(bar, (unsigned)(kTileN * (2 + NM * sizeof(SP))));
            tma_load_3d(st + L::o_cls, &M.cls, xb, 0, zb, bar);
#pragma unroll
            for (int m = 0; m < NM; ++m) tma_load_3d(st + L::o_psi + m * kTileN * sizeof(SP), &M.psi[m], xb, 0, zb, bar);
        }
    };
    int io0 = 0, io1 = 0;                          // the tile's sources and receivers
    walk_tiles<NS, L::stage>(smem, gx, run, n_rows, A.mon, load, [&](int xb, int zb, unsigned char *st, auto wait) {
        PlanePos P;
        P.x0 = xb + 4 * tx;
        P.z = zb + ty;
        P.on = P.x0 < G.nx && P.z < G.nz;
        P.row = (long long)P.z * G.px + P.x0;
        const int x0 = P.x0, z = P.z;
        if (A.io.off) {
            const int *o = A.io.off + (long long)(zb / kTileH) * gx + xb / kTileW;
            io0 = __ldg(o);
            io1 = __ldg(o + 1);
        }
        const bool in[3] = {P.on && G.wabs > 0 && (x0 < G.wabs || x0 + 3 >= G.nx - G.wabs), false,
                            P.on && G.wabs > 0 && (z < G.wabs || z >= G.nz - G.wabs)};
        float pp[3][4];
#pragma unroll
        for (int ax = 0; ax < 3; ax += 2)
            if (in[ax]) Io<float>::ld(A.psip[ax] + P.row, pp[ax]);
        wait();
        if (!P.on) return;
        constexpr int xc = TS ? 4 : 0;     // column of x0 in the v_z tile at tx = 0
        const float *vx = reinterpret_cast<const float *>(st + L::o_vx) + (ty + (TS ? 1 : 0)) * L::XW + 4 * tx;
        const float *vz = reinterpret_cast<const float *>(st + L::o_vz) + ty * L::ZW + xc + 4 * tx;   // row z - 4
        const uint2 cl = *reinterpret_cast<const uint2 *>(reinterpret_cast<const uint16_t *>(st + L::o_cls) + e0);
        uint16_t cls4[4];
        quad_classes(cl, cls4);
        if (cl.x != key.x || cl.y != key.y) {
            C.load(A.lut, cls4, kLutA2, kLutB2, kLutIk2);
            key = cl;
        }
        float qz[8][4], w[12], kd[4], bd[4], pv[4], ps[NM][4], qd[3][4];
#pragma unroll
        for (int r = 0; r < 8; ++r) Sm<float>::ld(vz + r * L::ZW, qz[r]);
        Sm<float>::ld12(vx, w);
        Sm<float>::ld(reinterpret_cast<const float *>(st + L::o_kd) + e0, kd);
        if (NL) Sm<float>::ld(reinterpret_cast<const float *>(st + L::o_bd) + e0, bd);
        Sm<float>::ld(reinterpret_cast<const float *>(st + L::o_p) + e0, pv);
#pragma unroll
        for (int m = 0; m < NM; ++m) Sm<SP>::ld(reinterpret_cast<const SP *>(st + L::o_psi) + m * kTileN + e0, ps[m]);
        if (TS) {
            float rh[4], up[4], dn[4];
            Sm<float>::ld(reinterpret_cast<const float *>(st + L::o_rh) + e0, rh);
            Sm<float>::ld(vx - L::XW + 4, up);
            Sm<float>::ld(vx + L::XW + 4, dn);
            pres_divergence_ts_plane(G, kd, rh, qz, w, up, dn, vx[3 - L::XW], vx[3 + L::XW], vz[4 * L::ZW - 1],
                                     vz[3 * L::ZW - 1], vz[4 * L::ZW + 4], vz[3 * L::ZW + 4], x0, qd);
        } else {
            quad_diff_x(G, w, 4, qd[0]);
            quad_diff(G, qz, qd[2]);
        }
        float div[4], stp[4], rr[4] = {1.0f, 1.0f, 1.0f, 1.0f};
        pres_div_plane(G, x0, qd, div);
        if (in[0] || in[2]) plane_ramp(G, P, rr);
        quad_stretch<float, NM>(C, div, rr, G.hs2, ps, stp);
#pragma unroll
        for (int m = 0; m < NM; ++m) Io<SP>::st(A.psi[m] + P.row, ps[m]);
#pragma unroll
        for (int ax = 0; ax < 3; ax += 2) {
            if (!in[ax]) continue;
            plane_layer(A.pd, A.pa, C.ik, G.dt, ax, P, qd[ax], pp[ax], stp);
            Io<float>::st(A.psip[ax] + P.row, pp[ax]);
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const float fac = NL ? fmaf(bd[e], pv[e], kd[e]) : kd[e];
            pv[e] = fmaf(-fac, stp[e], pv[e]);
            pmax.see(pv[e]);
        }
        Io<float>::st(A.p + P.row, pv);
    }, [&] {
        if (io0 < io1) tile_io(A.io, A.p, io0, io1, ty * 32 + tx, 128, A.mon);
    });
    record_max(A.mon, pmax);
}

}  // namespace fwgb
