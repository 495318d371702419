// Parameters and launchers of the TMA-staged 3-D step kernel (k_step3d.cu) and its
// host-side tensor-map helpers (tmap.cpp).  Internal to libfwi.
#pragma once

#include <cuda.h>
#include <cstdint>
#include <cuda_runtime.h>

#include "fwi_internal.h"

namespace fwi {

constexpr int kModeStep = 0;   // out = damped leapfrog update, written over prev
constexpr int kModeStepStore = 2;   // kModeStep that also writes a checkpoint of its input
                                    // pair (st_code); a separate instantiation, so the plain
                                    // step's code is unchanged
constexpr int kModeAdj = 1;    // the same update (no source) and g += aux * (L c), with the
                               // source-point term g -= dt^2 w[n] c / W

struct Step3dParams {
    int M;
    int nx, ny, nz, px;           // computed extents and row pitch (floats)
    int64_t plane, field;         // floats per z-plane and per shot
    int nshots;
    int rounds, round_ctas;       // whole-unit rounds and the CTAs each round uses
    int rem_ctas;                 // CTAs sharing the leftover units along z
    int zparts, zfirst;           // a unit is z-part h of a tile column: planes
                                  // [h zfirst, (h + 1) zfirst), the last part up to nz;
                                  // units are numbered part-major
    int rem_first, rem_ppu;       // leftover units go to CTAs rem_first ..
                                  // rem_first + rem_ctas - 1: cut into rem_ppu aligned
                                  // pieces each (rem_ppu > 0), or as one run cut into
                                  // equal pieces that may cross units (rem_ppu = 0)
    float cx[kMaxM + 1], cy[kMaxM + 1], cz[kMaxM + 1], c0;
    float2 cy2[kMaxM + 1], cz2[kMaxM + 1], c02;   // the same weights as packed pairs
    int iso;                      // hx = hy = hz: the isotropic instantiation may run
    float inv_h2;                 // 1 / h^2 of an isotropic grid
    const float *sig_x, *sig_y, *sig_z;
    const float *W;               // brick kernel: W and u^m are read without tensor maps
    const void *aux;
    int64_t aux_stride;           // elements per shot
    float *out;                   // the new state, over prev (in place)
    float *g;                     // kModeAdj: gradient accumulator
    const int64_t *src_off;       // may be null (kModeStep: injection; kModeAdj: g term)
    const PointTaps *src_pts;     // brick kernel, forward modes: off-grid sources, or null
    const float *wavelet;
    int nt, n;
    const int *n_dev;             // nullable: the step index is *n_dev + n
    float dt2;
    unsigned *err;                // status word: bit 1 (value 2) = a bounded wait gave up
    int aux_fmt;                  // kModeAdj: aux tile of FP32 (0) or BF16 (1) / FP16 (2)
                                  // checkpoint codes
    const float *aux_scale;       // kModeAdj with codes: per shot at [2 s] (u = code / scale)
    void *st_code;                // kModeStep, nullable: checkpoint of the input pair (c, prev)
    const unsigned *st_max;       //   written from the epilogue (see StepParams)
    float *st_scale;
    int st_dtype, st_comps;
    int64_t st_cstride;
    unsigned *maxbits;            // kModeStep, nullable: per shot, raise [2s] to the bits of
                                  // max|out| and [2s+1] to max|out - c| (the checkpoint
                                  // codec's scales of the new state pair)
    unsigned *max_clear;          // with maxbits: maxima cleared for the next step
    // receivers handled in the epilogue (rec_map nullable): every receiver is the node
    // (rec_z, y, x) with rec_map[shot][y][x] = its index (-1 elsewhere); forward modes
    // write rec_tr[shot][n][r] = out, the reverse mode adds
    // inj_scale[shot][r] * inj_q[shot][inj_n][r] to out (the same two roundings as the
    // separate injection kernel)
    const int *rec_map;
    int rec_z, nrec;
    float *rec_tr;
    const float *inj_q, *inj_scale;
    int inj_n;
};

// Kernel configurations of the 3-D step: tile height, points per thread along y,
// prefetch depth, planes between shifts of the register z-queue, and option bits
// (1: packed x-sums, 2: undamped fast path).  step3d_variant() picks the configuration
// used for radius M.
// Tile height, rows per thread, prefetch depth, queue shift interval, and the option bits
// (Cfg::F) of the plain forward step (opt) and of the store and reverse modes (opt_rev);
// tm = 1 selects the kernel whose z-stream lives in tensor memory (k_step3d_tm.cuh:
// 64 x 32 tiles, two CTAs per SM; ty is then 32 and the other fields do not apply);
// tile_g = 1 makes its reverse step read g as a TMA pointwise tile instead of staging it
// with per-thread asynchronous copies.
struct Step3dVariant {
    int ty, ry, pf, u, opt, opt_rev;
    int tm;
    int tile_g = 0;
    int half = 0;   // tensor-memory forward modes: 64 x 16 tiles, 4 warps, four CTAs per SM
};
// The tensor-memory reverse step takes g as a TMA tile when a launch has at least this
// many CTAs per 64 x 32 tile column less one, so that its columns are cut along z into as
// many short parts or pieces (23 to 72 planes on the 232^3 to 360^3 grids measured, 3-6 %
// faster there), and stages g per thread otherwise (424^3 and up, 4-15 % faster).
constexpr int kTileGParts = 5;
Step3dVariant step3d_variant(int M, int mode);
int step3d_smem_bytes(int M);
int step3d_threads(int M);
// Resident CTAs of the 3-D step kernel of `mode` on the current device (SMs x CTAs per
// SM), for the instantiation a launch on an isotropic (iso) or anisotropic grid uses;
// -e when a CUDA call of the query failed with error e.
int step3d_resident_ctas(int M, int mode, bool iso);

// map_c: 4-D [shot][z][y][x] map of the streamed field with the halo box;
// map_a, map_b, map_d, map_e: maps of the pointwise fields prev, W, aux, g with the
// 64 x TY tile box (map_d and map_e are read in kModeAdj only).  W's map has a shot
// extent of 1.
cudaError_t launch_step3d_tma(const Step3dParams &p, int mode, int ctas,
                              const CUtensorMap &map_c, const CUtensorMap &map_a,
                              const CUtensorMap &map_b, const CUtensorMap &map_d,
                              const CUtensorMap &map_e, cudaStream_t s);

// Per-radius pieces behind the dispatch (k_step3d_m4.cu, k_step3d_m8.cu).
typedef void (*Step3dKernel)(const Step3dParams, const CUtensorMap, const CUtensorMap,
                             const CUtensorMap, const CUtensorMap, const CUtensorMap);
struct Step3dKernelInfo {
    Step3dKernel fn;
    int threads, smem;
    int tmem_cols = 0;   // tensor-memory columns each CTA allocates
};
// iso: the grid is isotropic, so an instantiation with compile-time stencil weights
// (scaled by 1 / h^2 once per point) may be returned.
Step3dKernelInfo step3d_kernel_m4(const Step3dVariant &v, int mode, bool iso = false);
Step3dKernelInfo step3d_kernel_m8(const Step3dVariant &v, int mode, bool iso = false);
// The tensor-memory kernels (k_step3d_tm8.cu, k_step3d_tm4.cu).
Step3dKernelInfo step3d_kernel_tm8(int mode, bool iso, bool tile_g, bool half);
Step3dKernelInfo step3d_kernel_tm4(int mode, bool iso, bool tile_g, bool half);

// The brick kernel (k_step3d_brick.cu): extents (x, y, z) of its two halo boxes, and a launch
// with the streamed field's maps of those boxes.
void brick_boxes(int M, int (&mid)[3], int (&arm)[3]);
bool step3d_use_brick(const Step3dParams &p, int mode);
cudaError_t launch_step3d_brick(const Step3dParams &p, int mode, const CUtensorMap &mid,
                                const CUtensorMap &arm, cudaStream_t s);

// Encodes a 4-D tensor map over shots of a field laid out as in Geom (elements of
// `elem_bytes` = 4 or 2, shots `shot_stride` elements apart), with box (bx, by, bz, 1) and
// zero fill outside [0, nx) x [0, ny) x [0, nz) x [0, nshots).
int encode_field_map(CUtensorMap *map, const void *base, const Geom &g, int nshots, int bx,
                     int by, int bz, int elem_bytes, int64_t shot_stride);

// Segment idx (0, 1, ...) of CTA k in the persistent schedule of p over `columns` tile
// columns: tile column *col, output planes [*z0, *z1).  Returns false past its last
// segment.  The kernels walk it (k = blockIdx.x) and the planner evaluates it, so both
// read the same schedule.
__host__ __device__ inline bool schedule_segment(const Step3dParams &p, int columns, int k, int idx,
                                                 int *col, int *z0, int *z1)
{
    const int S = p.zparts;
    if (k < p.round_ctas) {
        if (idx < p.rounds) {
            const int u = idx * p.round_ctas + k;
            const int h = u / columns;
            *col = u - h * columns;
            *z0 = h * p.zfirst;
            *z1 = h == S - 1 ? p.nz : *z0 + p.zfirst;
            return true;
        }
        idx -= p.rounds;
    }
    const int first = p.rounds * p.round_ctas;   // first leftover unit
    const int rem = columns * S - first;
    const int kk = k - p.rem_first;
    if (rem <= 0 || kk < 0 || kk >= p.rem_ctas) return false;
    const int zb = (S - 1) * p.zfirst;            // the leftover units lie in the last part
    const int len_u = p.nz - zb;
    if (p.rem_ppu > 0) {                          // aligned pieces, one per CTA
        if (idx > 0) return false;
        const int u = first + kk / p.rem_ppu, piece = kk % p.rem_ppu;
        const int plen = (len_u + p.rem_ppu - 1) / p.rem_ppu;
        *col = u % columns;
        *z0 = zb + piece * plen;
        *z1 = *z0 + plen < p.nz ? *z0 + plen : p.nz;
        return *z0 < *z1;
    }
    const int64_t total = (int64_t)rem * len_u;
    const int64_t len = (total + p.rem_ctas - 1) / p.rem_ctas;
    const int64_t s0 = (int64_t)kk * len;
    const int64_t s1 = s0 + len < total ? s0 + len : total;
    const int64_t start = idx == 0 ? s0 : (s0 / len_u + idx) * len_u;
    if (start >= s1) return false;
    const int64_t end = (start / len_u + 1) * len_u < s1 ? (start / len_u + 1) * len_u : s1;
    const int u = first + (int)(start / len_u);
    *col = u % columns;
    *z0 = zb + (int)(start % len_u);
    *z1 = *z0 + (int)(end - start);
    return true;
}

// 3-D map [shot][z][x] of a 2-D field (elements of elem_bytes = 4 or 2, shots
// `shot_stride` elements apart) with box (bx, bz, 1) and zero fill outside the grid.
int encode_field_map2d(CUtensorMap *map, const void *base, const Geom &g, int nshots, int bx,
                       int bz, int elem_bytes, int64_t shot_stride);

// The 2-D step on halo tiles (k_step2d_tile.cu).  map: the streamed field with a box of the
// tile (step2d_tile_cols x step2d_tile_rows) and its halo.
int step2d_tile_cols();
int step2d_tile_rows(bool img);
cudaError_t launch_step2d_tile(const StepParams &p, int nshots, bool img, const CUtensorMap &map,
                               cudaStream_t s);

// Persistent schedule of one launch over `columns` tile columns of nz planes on
// `resident` CTAs: rounds of whole units, then the leftover units cut along z into pieces
// (each piece streams 2M warm-up planes).  A unit is a whole column, or, with `in_step`, one
// of several z-parts of a column that begin at the same z in every column: the CTAs of a
// round then stream z in step, so a tile's halo planes are still in L2 when its neighbours
// read them.  Units are numbered part-major, so that tiles next to one another in x run on
// CTAs next to one another.  With at least as many columns as CTAs, columns are cut into parts
// where whole rounds of them leave less to the last, partial round.  With fewer columns than
// CTAs the planner compares: the same number of parts of every column, at most one to a CTA
// and none left over; S = ceil(resident / columns) equal parts whose leftover last parts are
// cut over all CTAs; and S parts of which the first ones are longer and the leftover last parts
// go to the CTAs that ran a last part.  It keeps the one whose busiest CTA streams the fewest
// planes (warm-up planes included), the first one's weighed by (resident / CTAs used)^2 at
// radius 8: its steps are bound by the SMs' instruction issue, and idle CTAs cost more there.  Power
// 0 / 1 / 2 of that weight on 11 grids of 216^3 to 440^3 computed points, us a step, where they differ
// by more than 1 %: radius 8, 360^3 forward 162.4 / 157.6 / 157.8, store 182.5 / 175.7 / 175.6; two
// shots of 199 x 197 x 433 forward 123.6 / 123.9 / 121.5, store 137.6 / 138.1 / 135.9.  Radius 4 takes
// none: 296^3 reverse 109.0 / 112.5 / 112.4, 360^3 118.5 / 119.1 / 125.5 forward, 187.5 / 197.5 / 197.1
// reverse, 440^3 forward 221.7 / 220.4 / 229.0.
// Every launch of the step is planned in step.  Measured on GB300, us per step forward /
// store / reverse, against one run of the columns cut over all CTAs below 96 MB and no
// candidate without leftovers: radius 4, 216^3 39.0 / 44.9 / 65.8 -> 35.9 / 40.8 / 54.2, 280^3
// 99.9 / 117 / 159 -> 63.8 / 71.5 / 99.5, 296^3 74.9 / 84.6 / 112 -> 70.4 / 81.4 / 109; radius 8,
// 216^3 60.5 / 68.0 / 85.3 -> 51.3 / 57.2 / 59.5, 280^3 120 / 135 / 169 -> 86.2 / 95.9 / 102, 440^3
// 261 / 293 / 354 -> 255 / 287 / 344.  Parts numbered column by column (the reverse step then with
// two rows per thread): radius 4 360^3 122 / 152 / 214 against 119.6 / 137.8 / 212, 440^3 237 / 306 /
// 347 against 223 / 285 / 346.
// Fills the schedule fields of p and returns the grid size.
int plan_persistent(Step3dParams &p, int columns, int resident, bool in_step = false);

}  // namespace fwi
