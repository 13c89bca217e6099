// Internal declarations shared by the library's translation units.
#pragma once

#include "../../include/fullwave_gb.h"

#include <atomic>
#include <functional>
#include <map>
#include <vector>

#include <cuda_runtime.h>

namespace fwgb {

// ---- calibration (fw_fit.cpp) ----------------------------------------------
struct FitJob {
    fw_relax_params p;
    double J, w, nrmse, disp;
    int n_iter, n_eval;
};
void default_opts(fw_fit_opts *o);
fw_relax_params lossless_params(int n);
FitJob run_weight(double alpha0, double y, int n_mech, const fw_fit_opts &o, int wi);
void select_fit(const std::vector<FitJob> &res, fw_relax_params *out, fw_fit_report *rep);
void parallel_for(int n_jobs, int n_threads, const std::function<void(int)> &fn);
int fit_check(double alpha0, double y, int n_mech, const fw_fit_opts &o);
int nelder_mead(int n, double *x, const double *lo, const double *hi,
                double (*f)(const double *, void *), void *ctx, int maxiter,
                double xatol, double fatol, double *fmin, int *n_iter, int *n_eval);

// ---- device layout ---------------------------------------------------------
constexpr int kLutStride = 20;   // values per class in the coefficient table
// table block offsets (in values): 0.. a1[4], 4.. b1[4], 8.. a2[4], 12.. b2[4],
// 16 1/kappa1, 17 what its rounding left off, 18, 19 the same of kappa2 (the
// remainders: FP32 media; both with the known rounding of the global factors
// taken back, see build_lut)
constexpr int kLutA1 = 0, kLutB1 = 4, kLutA2 = 8, kLutB2 = 12, kLutIk1 = 16, kLutIk2 = 18;

struct Monitor {
    unsigned int max_bits;   // bits of max |p| (non-negative float)
    int nonfinite;
    int bad_index;           // a source/receiver index or step counter out of range (skipped)
    int timeout;             // a bounded wait of a sweep on its staged copies gave up
};

// Tensor-map descriptors of the streams that a medium's velocity sweep stages
// (opaque 128-byte driver objects, built on the host at medium creation):
// p with its halo box and (3D) p own box, v_d, psi1[m][d], rho with its +1
// halo box and (3D) rho own box, the class index and K dt.
struct alignas(64) TensorMapBlob {
    unsigned char bytes[128];
};
struct VelMaps {
    TensorMapBlob p_halo, p_own, v[3], psi[FW_MAX_MECH][3], rho_halo, rho_own, cls, kdt;
};
// ... and its pressure sweep: v_z own box (3D: planes ahead; 2D: with its halo
// rows), v_x with its x halo, v_y with its y halo (3D), p, K dt, 2 beta dt,
// psi2[m], the class index, rho (time-space stencil)
struct PresMaps {
    TensorMapBlob vz_own, vx_halo, vy_halo, p_own, kdt, b2dt, psi[FW_MAX_MECH], cls, rho_own;
    TensorMapBlob vx_ring, vy_ring, vz_ring;   // time-space stencil: v boxes with x and y halos
};

// A step between two state images (buffers laid out as the medium's state):
// every state array is read at its offset in the image at rd and written at
// the same offset in the image wofs bytes further on; maps and tables stay
// the medium's.
struct StepImages {
    const char *rd;
    long long wofs;
};

// A cell that holds a source, a receiver or both: its index in the padded
// layout and the source's and receiver's numbers (-1: none)
struct IoEntry {
    long long cell;
    int src, rcv;
};

// CTA tiles: columns, and rows of depth (2D) or y (3D, by the bytes of a state
// element).  All sweeps and the reverse kernels take these: a cell's source or
// receiver is handled, without atomics, by the CTA that stores the cell, found by
// the tile it lies in.  A row of a 2D tile is a warp, a quad of columns per lane.
constexpr int kTileW = 128, kTileH = 4;
constexpr int kTile3W = 64;
constexpr int tile3_rows(size_t es) { return es == 8 ? 4 : 8; }

// Tiles of the pressure sweep's CTAs by kernel axes, in 3D one per depth plane,
// the planes of a tile following each other; the entries of a medium's cells
// are ordered by tile
struct IoTiling {
    int w, h;            // columns, and rows of y (3D) or depth (2D)
    int gx, gy;          // tiles along x, and along y (3D) or depth (2D)
    long long n;         // number of tiles
};

struct Graph {
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
};

}  // namespace fwgb

struct fw_medium;
namespace fwgb {
double psi_scale_of(const fw_medium *m, int side);   // stored memory variable = psi * scale (side 1 or 2)
}

struct fw_medium {
    fw_grid g{};
    int ndim = 0, nmech = 0, storage = 0;
    bool nonlinear = false;
    int NX = 0, NY = 0, NZ = 0;     // kernel axes: x, y (1 in 2D), depth
    int px = 0;                      // row pitch in elements
    size_t plane = 0, vol = 0;       // elements per plane / per array (padded)
    int es = 4, eps = 4;             // element bytes of state and of psi
    double dt = 0, dx = 0, c_max = 0, ceff_max = 0;
    int n_classes = 0;
    int wabs = 0;                    // transition + absorbing cells
    // device memory
    void *slab = nullptr;
    size_t slab_bytes = 0;
    void *p = nullptr, *v[3] = {}, *psi1[FW_MAX_MECH][3] = {}, *psi2[FW_MAX_MECH] = {};
    void *psi1p[3] = {}, *psi2p[3] = {};
    void *kdt = nullptr, *rho = nullptr, *b2dt = nullptr, *lut = nullptr;
    void *cdev = nullptr;            // c map (kept for the class coefficient rebuilds)
    uint16_t *cls = nullptr;
    void *prof[3][4] = {};           // per kernel axis: d, alpha at half points; d, alpha at integer points
    int *d_it = nullptr;
    fwgb::Monitor *mon = nullptr;
    std::vector<fw_relax_params> classes;
    // sources / receivers
    void *src_buf = nullptr, *rcv_buf = nullptr;
    long long *src_idx = nullptr;
    void *src_gain = nullptr, *waves = nullptr, *traces = nullptr;
    int *wave_of = nullptr;
    int n_src = 0, n_wave = 0, wave_len = 0;
    int n_rcv = 0, n_rec = 0, decim = 1;
    // the cells with a source or a receiver, ordered by tile, and where each
    // tile's entries begin (io_off: io_tiling(m).n + 1 values, in the slab)
    void *ent_buf = nullptr;
    size_t ent_cap = 0;
    int n_ent = 0;
    int *io_off = nullptr;
    std::vector<long long> h_src_idx, h_rcv_idx;   // the sources' and the receivers' cells, sorted
    // device buffers of the last gradient, kept for the next (workspace_take)
    void *ws = nullptr;
    size_t ws_bytes = 0;
    bool ws_busy = false;
    // bookkeeping
    long long step = 0;
    int sticky = 0;
    cudaStream_t last_stream = nullptr;
    cudaStream_t cap_stream = nullptr;
    std::map<int, fwgb::Graph> graphs;
    int zseg[2] = {16, 16};          // depth planes per CTA of the 3D velocity and pressure sweeps
    mutable int slots[2] = {0, 0};   // CTAs of either that the device holds at once, found at creation
    double psi_pref = 10.0;          // pressure reference [Pa] of binary16 memory variables
    int time_order = 2;              // 2: leapfrog; 4: time-space stencil (Sec. 3.3)
    double ts_a[4][4] = {};          // time-space weights a_m = sum_n ts_a[m][n] r^(2n)
    bool tma = false;                // the tensor maps below are there: sweeps staged by TMA copies
    fwgb::VelMaps vel_maps{};
    fwgb::PresMaps pres_maps{};
};
