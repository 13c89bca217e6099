// Launch helpers: build kernel arguments from a medium and dispatch the
// template instance for (dimension, mechanisms, nonlinearity).  Included by
// one translation unit per storage type so that they compile in parallel.
#pragma once

#include "fw_plane.cuh"

#include <climits>

#include <cuda.h>

namespace fwgb {

// Launch with or without the programmatic attribute (pdl_wait in the kernels).
// Left out after an event of another stream and where events time each kernel.
template <typename... P, typename... A>
cudaError_t launch_kernel(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, bool pdl, A &&...args)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

// 3D CTA tiles: 64 x 8 points in FP32 (a quad per thread, 128 threads), two CTAs
// of the velocity sweep and three of the pressure sweep per SM; 64 x 4 in FP64.
// Against 128 x 4 the halo of p per plane is 15 x 72 instead of 11 x 136
// points and a row's last tile holds at most 63 idle columns; us per step,
// 128 x 4 / 64 x 8 / 32 x 16: 128^3 87.9 / 84.2 / 84.1, 231x187x301 383 / 354 /
// 360, 256^3 508 / 504 / 514, 256^3 binary16 391 / 374, 256^3 time-space 647 /
// 623, 512^3 3822 / 3826.
template <typename R> struct Tile3 {
    static constexpr int BX = kTile3W / 4, BYV = tile3_rows(sizeof(R)), BYP = BYV;
};

template <typename R> Geo<R> make_geo(const fw_medium *m)
{
    Geo<R> g{};
    g.nx = m->NX;
    g.ny = m->NY;
    g.nz = m->NZ;
    g.px = m->px;
    g.plane = (long long)m->plane;
    g.wabs = m->wabs;
    // 8th-order staggered weights (Taylor) divided by dx
    const double cm[4] = {1225.0 / 1024.0, -245.0 / 3072.0, 49.0 / 5120.0, -5.0 / 7168.0};
    g.c1 = R(cm[0] / m->dx);
    g.c2 = R(cm[1] / m->dx);
    g.c3 = R(cm[2] / m->dx);
    g.c4 = R(cm[3] / m->dx);
    g.dt = R(m->dt);
    g.hs1 = R(0.5 / psi_scale_of(m, 1));
    g.hs2 = R(0.5 / psi_scale_of(m, 2));
    g.lr = R(m->g.transition > 0 ? m->g.transition : 0.5 * m->g.pml);
    for (int i = 0; i < 4; ++i)
        for (int n = 0; n < 4; ++n) g.ta[i][n] = R(m->ts_a[i][n] / m->dx);
    g.tb = R(1.0 / (24.0 * m->dx));
    g.r2s = R(m->dt / (m->dx * m->dx));
    return g;
}

// Tensor maps of the streams that the sweeps stage by TMA: every array is
// addressed as a 3D tensor (px, NY, NZ) with the medium's pitches; boxes are
// the CTA tile (TW x BY along x and y, x and z in 2D) or its halo boxes (p:
// (TW+8) x (BY+7) from (xb-4, yb-3); rho: (TW+4) x (BY+1)).  Elements outside
// the tensor read as zero.  encode is the driver's tensor-map encoder.
using EncodeTiledFn = CUresult (*)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                   const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

template <typename T> constexpr CUtensorMapDataType map_type();
template <> constexpr CUtensorMapDataType map_type<float>() { return CU_TENSOR_MAP_DATA_TYPE_FLOAT32; }
template <> constexpr CUtensorMapDataType map_type<__nv_bfloat16>() { return CU_TENSOR_MAP_DATA_TYPE_BFLOAT16; }
template <> constexpr CUtensorMapDataType map_type<__half>() { return CU_TENSOR_MAP_DATA_TYPE_FLOAT16; }
template <> constexpr CUtensorMapDataType map_type<uint16_t>() { return CU_TENSOR_MAP_DATA_TYPE_UINT16; }

template <typename T>
bool encode_map(EncodeTiledFn encode, TensorMapBlob *out, const fw_medium *m, const void *base, unsigned bx,
                unsigned by)
{
    const cuuint64_t dims[3] = {(cuuint64_t)m->px, (cuuint64_t)m->NY, (cuuint64_t)m->NZ};
    const cuuint64_t strides[2] = {(cuuint64_t)m->px * sizeof(T), (cuuint64_t)m->plane * sizeof(T)};
    const cuuint32_t box[3] = {bx, m->ndim == 3 ? by : 1, m->ndim == 3 ? 1 : by}, estr[3] = {1, 1, 1};
    return encode(reinterpret_cast<CUtensorMap *>(out), map_type<T>(), 3, const_cast<void *>(base), dims, strides,
                  box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                  CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// 2D tiles (k_velocity_tiles, k_pressure_tiles)
template <typename SS, typename SP> bool build_plane_maps(EncodeTiledFn encode, fw_medium *m)
{
    constexpr unsigned W = kTileW, H = kTileH;
    const bool ts = m->time_order == 4;
    VelMaps &v = m->vel_maps;
    PresMaps &q = m->pres_maps;
    bool ok = encode_map<SS>(encode, &v.p_halo, m, m->p, W + 8, H + 7) &&
              encode_map<SS>(encode, &v.rho_halo, m, m->rho, W + 4, H + 1) &&
              encode_map<uint16_t>(encode, &v.cls, m, m->cls, W, H) && encode_map<SS>(encode, &v.kdt, m, m->kdt, W, H);
    q.cls = v.cls;
    q.kdt = v.kdt;
    for (int ax = 0; ax < 3; ax += 2) {
        ok = ok && encode_map<SS>(encode, &v.v[ax], m, m->v[ax], W, H);
        for (int n = 0; n < m->nmech; ++n) ok = ok && encode_map<SP>(encode, &v.psi[n][ax], m, m->psi1[n][ax], W, H);
    }
    for (int n = 0; n < m->nmech; ++n) ok = ok && encode_map<SP>(encode, &q.psi[n], m, m->psi2[n], W, H);
    ok = ok && encode_map<SS>(encode, &q.p_own, m, m->p, W, H) &&
         (!m->nonlinear || encode_map<SS>(encode, &q.b2dt, m, m->b2dt, W, H));
    if (ts)
        ok = ok && encode_map<SS>(encode, &q.vx_ring, m, m->v[0], W + 8, H + 2) &&
             encode_map<SS>(encode, &q.vz_ring, m, m->v[2], W + 8, H + 7) &&
             encode_map<SS>(encode, &q.rho_own, m, m->rho, W, H);
    else
        ok = ok && encode_map<SS>(encode, &q.vx_halo, m, m->v[0], W + 8, H) &&
             encode_map<SS>(encode, &q.vz_own, m, m->v[2], W, H + 7);
    return ok;
}

template <typename R, typename SS, typename SP>
bool build_vel_maps_t(EncodeTiledFn encode, fw_medium *m)
{
    if constexpr (sizeof(R) != 4) {
        return false;
    } else {
        if (m->ndim == 2) return build_plane_maps<SS, SP>(encode, m);
        constexpr int TW = 4 * Tile3<R>::BX, BY = Tile3<R>::BYV;
        VelMaps &v = m->vel_maps;
        bool ok = encode_map<SS>(encode, &v.p_halo, m, m->p, TW + 8, BY + 7) &&
                  encode_map<SS>(encode, &v.p_own, m, m->p, TW, BY) &&
                  encode_map<SS>(encode, &v.rho_halo, m, m->rho, TW + 4, BY + 1) &&
                  encode_map<SS>(encode, &v.rho_own, m, m->rho, TW, BY) &&
                  encode_map<uint16_t>(encode, &v.cls, m, m->cls, TW, BY) &&
                  encode_map<SS>(encode, &v.kdt, m, m->kdt, TW, BY);
        for (int ax = 0; ax < 3 && ok; ++ax) {
            ok = encode_map<SS>(encode, &v.v[ax], m, m->v[ax], TW, BY);
            for (int n = 0; n < m->nmech && ok; ++n) ok = encode_map<SP>(encode, &v.psi[n][ax], m, m->psi1[n][ax], TW, BY);
        }
        // pressure sweep: v_x box with 4 columns either side, v_y box with
        // 4 rows below and 3 above
        constexpr int BP = Tile3<R>::BYP;
        PresMaps &q = m->pres_maps;
        ok = ok && encode_map<SS>(encode, &q.vz_own, m, m->v[2], TW, BP) &&
             encode_map<SS>(encode, &q.vx_halo, m, m->v[0], TW + 8, BP) &&
             encode_map<SS>(encode, &q.vy_halo, m, m->v[1], TW, BP + 7) &&
             encode_map<SS>(encode, &q.p_own, m, m->p, TW, BP) && encode_map<SS>(encode, &q.kdt, m, m->kdt, TW, BP) &&
             encode_map<uint16_t>(encode, &q.cls, m, m->cls, TW, BP) &&
             encode_map<SS>(encode, &q.rho_own, m, m->rho, TW, BP) &&
             (!m->nonlinear || encode_map<SS>(encode, &q.b2dt, m, m->b2dt, TW, BP));
        for (int n = 0; n < m->nmech && ok; ++n) ok = encode_map<SP>(encode, &q.psi[n], m, m->psi2[n], TW, BP);
        if (m->time_order == 4)       // the time-space stencil's rings of v planes
            ok = ok && encode_map<SS>(encode, &q.vx_ring, m, m->v[0], TW + 8, BP + 2) &&
                 encode_map<SS>(encode, &q.vy_ring, m, m->v[1], TW + 8, BP + 7) &&
                 encode_map<SS>(encode, &q.vz_ring, m, m->v[2], TW + 8, BP + 2);
        return ok;
    }
}

// A state array of the medium, or the same array in the image read (rd) or
// written (nw) by an image step
struct StateAt {
    const char *slab;
    const StepImages *im;
    void *rd(void *a) const
    {
        return (a && im) ? const_cast<char *>(im->rd) + (static_cast<const char *>(a) - slab) : a;
    }
    void *nw(void *a) const { return (a && im) ? static_cast<char *>(rd(a)) + im->wofs : a; }
};

template <typename R, typename SS, typename SP, int NM>
VelArgs<R, SS, SP> vel_args(const fw_medium *m, const StepImages *im)
{
    const StateAt at{static_cast<const char *>(m->slab), im};
    VelArgs<R, SS, SP> va{};
    va.g = make_geo<R>(m);
    va.p = static_cast<const SS *>(at.rd(m->p));
    va.g.zseg = m->zseg[0];
    va.wofs = im ? im->wofs : 0;
    for (int ax = 0; ax < 3; ++ax) {
        va.v[ax] = static_cast<SS *>(at.rd(m->v[ax]));
        va.psip[ax] = static_cast<SS *>(at.rd(m->psi1p[ax]));
        va.pd[ax] = static_cast<const R *>(m->prof[ax][0]);
        va.pa[ax] = static_cast<const R *>(m->prof[ax][1]);
        for (int n = 0; n < NM; ++n) va.psi[n][ax] = static_cast<SP *>(at.rd(m->psi1[n][ax]));
    }
    va.rho = static_cast<const SS *>(m->rho);
    va.cls = m->cls;
    va.lut = static_cast<const R *>(m->lut);
    va.kdt = static_cast<const SS *>(m->kdt);
    va.mon = m->mon;
    return va;
}

// which step of the medium a pressure sweep injects and records: *d_it + j
// (its own counter); image steps give theirs
struct StepIo {
    const int *d_it;
    int j;
    bool record;
};

template <typename R, typename SS, typename SP, int NM>
PresArgs<R, SS, SP> pres_args(const fw_medium *m, const StepImages *im, const StepIo &io)
{
    const StateAt at{static_cast<const char *>(m->slab), im};
    PresArgs<R, SS, SP> pa{};
    pa.g = make_geo<R>(m);
    pa.p = static_cast<SS *>(at.rd(m->p));
    pa.g.zseg = m->zseg[1];
    pa.wofs = im ? im->wofs : 0;
    for (int ax = 0; ax < 3; ++ax) {
        pa.v[ax] = static_cast<const SS *>(at.nw(m->v[ax]));   // this step's velocity
        pa.psip[ax] = static_cast<SS *>(at.rd(m->psi2p[ax]));
        pa.pd[ax] = static_cast<const R *>(m->prof[ax][2]);
        pa.pa[ax] = static_cast<const R *>(m->prof[ax][3]);
    }
    for (int n = 0; n < NM; ++n) pa.psi[n] = static_cast<SP *>(at.rd(m->psi2[n]));
    pa.kdt = static_cast<const SS *>(m->kdt);
    pa.b2dt = static_cast<const SS *>(m->b2dt);
    pa.cls = m->cls;
    pa.lut = static_cast<const R *>(m->lut);
    pa.mon = m->mon;
    pa.rho = static_cast<const SS *>(m->rho);
    if (m->n_ent > 0) {
        IoArgs<R, SS> &a = pa.io;
        a.off = m->io_off;
        a.ent = static_cast<const IoEntry *>(m->ent_buf);
        a.gain = static_cast<const R *>(m->src_gain);
        a.waves = static_cast<const R *>(m->waves);
        a.wave_of = m->wave_of;
        a.wave_len = m->n_src > 0 ? m->wave_len : 0;
        a.traces = io.record && m->n_rcv > 0 ? static_cast<SS *>(m->traces) : nullptr;
        a.n_rec = m->n_rec;
        a.decim = m->decim;
        a.d_it = io.d_it;
        a.j = io.j;
        a.vol = (long long)m->vol;
    }
    return pa;
}

// Sweeps of one dimension, mechanism count and time scheme.  which: bit 0 =
// velocity sweep, bit 1 = pressure sweep, bit 2 = only opt the instances into
// their dynamic shared memory (done once at medium creation, outside any
// stream capture), bit 3 = launches without the programmatic attribute.  im (may be null): a step from one state image into another
// (StepImages) instead of the in-place step of the medium's own state.
// 2D FP32-state grids from kTileMin tiles on take the staged sweeps, in runs of
// two tiles per CTA, of four from kTileLong tiles on; smaller grids, FP64 media
// and image steps the unstaged ones.  Measured when the line was drawn, us per
// step (unstaged / staged in runs of 1, 2, 4, 8; N = 4, FP32): 512^2 (512 tiles)
// 10.7 / 13.1, 13.9, 20.1, 32.3; 1024^2 (2048) 28.3 / 30.7, 27.6, 31.5, 38.9;
// 2048^2 (8192) 116 / 114, 102, 104, 110; 4096^2 (32768) 431 / 415, 373, 363, 373.
// With sources inside the sweeps and programmatic launch (unstaged / staged;
// FP32 N = 2, N = 4, bfloat16 N = 4, time-space N = 4): 1024^2 19.8 / 21.7, 24.9 /
// 27.1, 20.8 / 23.4, 34.8 / 33.2; 1456^2 (4368) 38.7 / 38.3, 56.1 / 55.1, 41.8 /
// 41.9, 73.1 / 63.4; 2048^2 83.3 / 74.2, 112 / 102, 87.2 / 77.9, 142 / 115;
// 4096^2 316 / 253, 427 / 367, 330 / 262, 536 / 395: the leapfrog's two forms meet
// at about 4400 tiles now, the time-space stencil's at 2048.  A run hides
// the latency of a tile's copies behind the tile before it, a short one leaves
// the hardware more CTAs to balance: with one persistent CTA per slot and even
// shares the 4096^2 step took 439 us, its slowest SMs finishing last.
constexpr int kTileMin = 2048, kTileLong = 16384;

template <typename SP, int NM, bool TS>
cudaError_t launch_tiles(const fw_medium *m, cudaStream_t s, int which, int gx, int n_tiles, const StepIo &io)
{
    constexpr int NS = 2;   // stages: the tile computed and the one on its way
    using LV = VelTile<SP, NM, TS>;
    const size_t bv = NS * LV::stage + 8 * NS;
    const size_t bp = NS * (m->nonlinear ? PresTile<SP, NM, true, TS>::stage : PresTile<SP, NM, false, TS>::stage) + 8 * NS;
    const auto kv = k_velocity_tiles<SP, NM, TS, NS>;
    const auto kp = m->nonlinear ? k_pressure_tiles<SP, NM, true, TS, NS> : k_pressure_tiles<SP, NM, false, TS, NS>;
    if (which & 4) {
        const auto attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
        const cudaError_t e = cudaFuncSetAttribute(kv, attr, (int)bv);
        return e == cudaSuccess ? cudaFuncSetAttribute(kp, attr, (int)bp) : e;
    }
    const dim3 block(kTileW / 4, kTileH);
    const int run = n_tiles >= kTileLong ? 4 : 2;
    const int rows = n_tiles / gx, ctas = gx * ((rows + run - 1) / run);
    const bool pdl = !(which & 8);
    cudaError_t e = cudaSuccess;
    if (which & 1)
        e = launch_kernel(kv, dim3(ctas), block, bv, s, pdl, vel_args<float, float, SP, NM>(m, nullptr), m->vel_maps, gx, run, rows);
    if (e == cudaSuccess && (which & 2))
        e = launch_kernel(kp, dim3(ctas), block, bp, s, pdl, pres_args<float, float, SP, NM>(m, nullptr, io), m->pres_maps, gx, run, rows);
    return e;
}

template <typename R, typename SS, typename SP, int NM, bool TS>
cudaError_t launch_2d(const fw_medium *m, cudaStream_t s, int which, const StepImages *im, const StepIo &io)
{
    const int gx = (m->NX + kTileW - 1) / kTileW;
    if constexpr (sizeof(R) == 4) {
        const long long n_tiles = (long long)gx * ((m->NZ + kTileH - 1) / kTileH);
        if (which & 4) return launch_tiles<SP, NM, TS>(m, s, which, gx, 0, io);
        if (m->tma && !im && n_tiles >= kTileMin && n_tiles < INT_MAX) return launch_tiles<SP, NM, TS>(m, s, which, gx, (int)n_tiles, io);
    }
    if (which & 4) return cudaSuccess;
    const dim3 grid((unsigned)gx * (unsigned)((m->NZ + kTileH - 1) / kTileH)), block(kTileW / 4, kTileH);
    const bool pdl = !(which & 8);
    cudaError_t e = cudaSuccess;
    if (which & 1)
        e = launch_kernel(k_velocity_plane<R, SS, SP, NM, kTileH, TS>, grid, block, 0, s, pdl,
                          vel_args<R, SS, SP, NM>(m, im), gx);
    if (e == cudaSuccess && (which & 2))
        e = launch_kernel(m->nonlinear ? k_pressure_plane<R, SS, SP, NM, kTileH, true, TS>
                                       : k_pressure_plane<R, SS, SP, NM, kTileH, false, TS>,
                          grid, block, 0, s, pdl, pres_args<R, SS, SP, NM>(m, im, io), gx);
    return e;
}

template <typename R, typename SS, typename SP, int NM, bool TS, bool TMA>
cudaError_t launch_3d_as(const fw_medium *m, cudaStream_t s, int which, const StepImages *im, const StepIo &io)
{
    constexpr int BX = Tile3<R>::BX, BYV = Tile3<R>::BYV, BYP = Tile3<R>::BYP;
    using LV = VelSmem<R, SS, SP, NM, BX, BYV, TS, TMA>;
    using LP = PresSmem<R, SS, SP, NM, BX, BYP, TS, TMA>;
    const auto kv = k_velocity<R, SS, SP, NM, BX, BYV, TS, TMA>;
    const auto kp = k_pressure<R, SS, SP, NM, BX, BYP, false, TS, TMA>, kpn = k_pressure<R, SS, SP, NM, BX, BYP, true, TS, TMA>;
    if (which & 4) {
        const auto attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
        cudaError_t e = cudaFuncSetAttribute(kv, attr, (int)LV::bytes);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(kp, attr, (int)LP::bytes);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(kpn, attr, (int)LP::bytes);
        int per_sm[2] = {0, 0}, dev = 0, sms = 0;
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm[0], kv, BX * BYV, LV::bytes);
        if (e == cudaSuccess)
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm[1], m->nonlinear ? kpn : kp, BX * BYP, LP::bytes);
        if (e == cudaSuccess) e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        for (int i = 0; i < 2; ++i) m->slots[i] = per_sm[i] * sms;
        return e;
    }
    MapsArg<TMA, VelMaps> vm;
    MapsArg<TMA, PresMaps> pm;
    if constexpr (TMA) {
        vm = m->vel_maps;
        pm = m->pres_maps;
    }
    const int gx = (m->NX + 4 * BX - 1) / (4 * BX);
    auto segs = [m](int i) { return (m->NZ + m->zseg[i] - 1) / m->zseg[i]; };
    const bool pdl = !(which & 8);
    cudaError_t e = cudaSuccess;
    if (which & 1)
        e = launch_kernel(kv, dim3(gx, (m->NY + BYV - 1) / BYV, segs(0)), dim3(BX, BYV), LV::bytes, s, pdl,
                          vel_args<R, SS, SP, NM>(m, im), vm);
    if (e == cudaSuccess && (which & 2))
        e = launch_kernel(m->nonlinear ? kpn : kp, dim3(gx, (m->NY + BYP - 1) / BYP, segs(1)), dim3(BX, BYP), LP::bytes, s,
                          pdl, pres_args<R, SS, SP, NM>(m, im, io), pm);
    return e;
}

// The FP32-state sweeps stage their streams by TMA when the medium holds
// tensor maps for them (which address the medium's own arrays, so not for
// image steps), by cp.async otherwise.
template <typename R, typename SS, typename SP, int NM, bool TS>
cudaError_t launch_3d(const fw_medium *m, cudaStream_t s, int which, const StepImages *im, const StepIo &io)
{
    if constexpr (sizeof(R) == 4) {
        if (which & 4) {   // both forms: image steps take the second one
            const cudaError_t e = launch_3d_as<R, SS, SP, NM, TS, false>(m, s, which, im, io);
            return e == cudaSuccess && m->tma ? launch_3d_as<R, SS, SP, NM, TS, true>(m, s, which, im, io) : e;
        }
        if (m->tma && !im) return launch_3d_as<R, SS, SP, NM, TS, true>(m, s, which, im, io);
    }
    return launch_3d_as<R, SS, SP, NM, TS, false>(m, s, which, im, io);
}

template <typename R, typename SS, typename SP, bool TS>
cudaError_t launch_ts(const fw_medium *m, cudaStream_t s, int which, const StepImages *im, const StepIo &io)
{
    const bool d3 = m->ndim == 3;
    switch (m->nmech) {
    case 1: return d3 ? launch_3d<R, SS, SP, 1, TS>(m, s, which, im, io) : launch_2d<R, SS, SP, 1, TS>(m, s, which, im, io);
    case 2: return d3 ? launch_3d<R, SS, SP, 2, TS>(m, s, which, im, io) : launch_2d<R, SS, SP, 2, TS>(m, s, which, im, io);
    case 3: return d3 ? launch_3d<R, SS, SP, 3, TS>(m, s, which, im, io) : launch_2d<R, SS, SP, 3, TS>(m, s, which, im, io);
    case 4: return d3 ? launch_3d<R, SS, SP, 4, TS>(m, s, which, im, io) : launch_2d<R, SS, SP, 4, TS>(m, s, which, im, io);
    default: return cudaErrorInvalidValue;
    }
}

// leapfrog instances, or those of the time-space stencil (time_order 4); the
// pressure sweep of step *d_it + j of the medium's counter injects and records
template <typename R, typename SS, typename SP>
cudaError_t launch_sweeps(const fw_medium *m, cudaStream_t s, int which, const StepImages *im, const StepIo &io)
{
    return m->time_order == 4 ? launch_ts<R, SS, SP, true>(m, s, which, im, io)
                              : launch_ts<R, SS, SP, false>(m, s, which, im, io);
}

template <typename R, typename SS, typename SP>
cudaError_t launch_step_sweeps(const fw_medium *m, cudaStream_t s, int which, int j)
{
    return launch_sweeps<R, SS, SP>(m, s, which, nullptr, StepIo{m->d_it, j, true});
}

// One leapfrog step from the state image at im.rd into the one at
// im.rd + im.wofs (both laid out as the medium's state), sources included at
// step it (absolute), receivers with record; the images' step counters are not
// used (zero: a counter that holds 0).  For the adjoint: no copy of the state
// per step, the medium's own state untouched.
template <typename R, typename SS>
cudaError_t launch_image_step(const fw_medium *m, const StepImages &im, const int *zero, int it, bool record, bool pdl,
                              cudaStream_t s)
{
    const StepIo io{zero, it, record};
    if (pdl) return launch_sweeps<R, SS, SS>(m, s, 3, &im, io);
    // first kernel after an event of another stream
    const cudaError_t e = launch_sweeps<R, SS, SS>(m, s, 1 | 8, &im, io);
    return e == cudaSuccess ? launch_sweeps<R, SS, SS>(m, s, 2, &im, io) : e;
}

}  // namespace fwgb
