// 2-D time stepping on chip (GB300, sm_103a): k steps of a small grid in one launch.
//
// A grid of some 10^4 to 10^5 points holds microseconds of work per step at most, so a step
// per launch costs its launch.  Here one thread-block cluster of C CTAs advances one shot by
// k steps: CTA r owns the rows [r nz / C, (r + 1) nz / C) and keeps them, with M halo rows on
// either side, in two shared-memory buffers used alternately (u^n read, u^{n+1} written).  A
// thread owns up to NU blocks of 4 columns x 2 rows for the whole launch and holds their W
// and, in the reverse sweep, gradient sums in registers.  It writes new values
// into its own CTA's next buffer and, near a band's edge, sends them into the neighbour's halo
// rows (st.async, which counts its bytes on an mbarrier of the neighbour), so every read is
// local.  A step waits for two things: a CTA barrier, and, for the threads whose rows read
// halo rows, the neighbours' bytes.  That is enough: the threads that read a halo row are
// those that send the rows next to it, so once a neighbour has a band's edge rows complete,
// nobody reads the halo rows that it overwrites next.  With checkpoints, the maxima that set
// a 16-bit code's scale travel the same way, each CTA's to every CTA; a step that stores the
// state waits for them after its z-sums, and the first thread waits for them in every step,
// so no CTA runs more than a step ahead of another there.
//
// Bound by latency: the messages and the dependent shared-memory reads and sums of a step.
// Measured on GB300 against single steps of the tile kernel (programmatic launches), us per
// step, forward / gradient (a forward step with store and a reverse step, and the call's fixed
// work), radius 4: 128^2 2.64 / 6.43 -> 1.00 / 3.74; 201^2 2.69 / 6.53 -> 1.28 / 4.64; 256^2
// 2.74 / 6.61 -> 1.75 / 5.70; 384^2 forward 3.44 -> 3.06, 440^2 3.58 -> 3.55 (computed grids of
// 168^2 to 480^2); radius 8: 256^2 forward 2.95 -> 2.41; four shots of 300^2 radius 4 3.56 /
// 9.19 -> 2.04 / 6.86, eight of 201^2 on clusters of 8 3.67 / 9.20 -> 2.20 / 7.14.  Not taken,
// since no faster: gradients with three blocks a thread at radius 4 (320^2 7.77 -> 7.95) or two
// at radius 8 (256^2 7.40 -> 7.57), forward steps with three at radius 8 (384^2 3.99 -> 4.21).
// With a cluster barrier per step instead of the messages: 201^2 1.52 / 5.75, 256^2 1.97 /
// 7.47.  Clusters of 8 and of 4 CTAs are slower wherever 16 run (201^2 forward 2.4 and 4.1 with
// the barrier) and still beat single steps where they fit, so they take the grids whose bands
// 16 CTAs would cut below M rows and the calls with more shots than clusters of 16.
#include <cooperative_groups.h>

#include "code16.cuh"
#include "fwi_internal.h"
#include "k_step3d.cuh"
#include "step2d_math.cuh"

namespace fwi {
namespace {

namespace cg = cooperative_groups;
using s2d::hi2;
using s2d::lap_x;
using s2d::lo2;
using s2d::update4;
using s2d::z_block;
using s3d::absmax_nan;
using s3d::mbar_expect_tx;
using s3d::mbar_init;
using s3d::smem_u32;

constexpr int kT = 512;        // threads per CTA
constexpr int kRZ = 2;         // rows per block
constexpr int kMaxC = 16;      // CTAs per cluster
constexpr int kSmemMax = 220 * 1024;
enum { kFwd = 0, kCkpt = 1, kRev = 2 };

// Shared-memory layout of one CTA, the same for every CTA of the cluster.
struct Layout {
    int G, SX, rows;           // groups of 4 columns, row stride, rows per buffer
    int floats;                // of both buffers and the sponge tables
};

__host__ __device__ inline Layout layout_of(int nz, int nx, int M, int C)
{
    Layout l;
    l.G = (nx + 3) / 4;
    l.SX = 4 * l.G + 2 * M;
    l.rows = ((nz + C - 1) / C + 1) / 2 * 2 + 2 * M;
    l.floats = 2 * l.rows * l.SX + 4 * l.G + l.rows;
    return l;
}

// The checkpoint codes of shot `shot` in the slot of a schedule entry d.
__device__ __forceinline__ char *slot_codes(const OnchipCkpt &a, int64_t field, int d, int shot)
{
    const int64_t cs = (d & kOnchipPairSlot ? 2 : 1) * field;
    return a.codes + __ldg(a.slot_off + (d & kOnchipSlot)) * a.half_slot + (int64_t)shot * cs * (a.dtype == 0 ? 4 : 2);
}

// Bounded wait (about 2^22 polls) for a phase that other CTAs of the cluster complete.
__device__ __forceinline__ bool wait_cluster(uint64_t *bar, uint32_t parity)
{
    for (int i = 0; i < (1 << 22); ++i) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(smem_u32(bar)), "r"(parity)
            : "memory");
        if (ok) return true;
    }
    return false;
}

__device__ __forceinline__ uint32_t in_cta(const void *p, int rank)   // p in CTA `rank` of the cluster
{
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_u32(p)), "r"(rank));
    return r;
}

// Sends 16 or 8 bytes to another CTA's shared memory and counts them on its barrier `bar`.
__device__ __forceinline__ void send(uint32_t addr, float4 v, uint32_t bar)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];"
                 ::"r"(addr), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w), "r"(bar)
                 : "memory");
}

__device__ __forceinline__ void send(uint32_t addr, uint2 v, uint32_t bar)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.u32 [%0], {%1, %2}, [%3];"
                 ::"r"(addr), "r"(v.x), "r"(v.y), "r"(bar)
                 : "memory");
}

template <int M, int MODE, int NU>
__device__ __forceinline__ void advance(const OnchipCkpt &a, const StepParams &p, float *u0, float *u1,
                                        int n0, int k, float *smem, int shot)
{
    cg::cluster_group cl = cg::this_cluster();
    const int C = (int)cl.num_blocks(), rank = (int)cl.block_rank(), tid = threadIdx.x;
    const int nz = p.g.nz, nx = p.g.nx, px = p.g.px;
    const Layout l = layout_of(nz, nx, M, C);
    const int r0 = (int)((int64_t)rank * nz / C), r1 = (int)((int64_t)(rank + 1) * nz / C), R = r1 - r0;
    const int Rup = rank > 0 ? r0 - (int)((int64_t)(rank - 1) * nz / C) : 0;
    const int SX = l.SX, G = l.G, U = G * ((R + kRZ - 1) / kRZ);
    float *buf0 = smem, *buf1 = smem + l.rows * SX;
    float *sxs = smem + 2 * l.rows * SX, *szs = sxs + 4 * G;
    __shared__ uint2 cmax[2][kMaxC];    // per parity, each CTA's maxima of the new state
    __shared__ uint2 wmax[2][kT / 32];
    // arrivals of state t: halo rows on halo_bar[t & 1], maxima on max_bar[t & 1]
    __shared__ __align__(8) uint64_t halo_bar[2], max_bar[2];
    bool dead = false;                  // a bounded wait of this thread gave up: it waits no more
    auto wait_for = [&](uint64_t *bar, int use) {
        if (dead || wait_cluster(bar, use & 1)) return;
        dead = true;
        atomicOr(p.err, 2u);
    };
    if (tid == 0) {
        for (int i = 0; i < 2; ++i) {
            mbar_init(halo_bar + i, 1);
            mbar_init(max_bar + i, 1);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        if (MODE == kCkpt) mbar_expect_tx(max_bar, 8 * C);   // state 0
    }
    const uint32_t halo_bytes = (uint32_t)((rank > 0) + (rank < C - 1)) * M * G * 16;
    const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);

    for (int i = tid; i < l.rows * SX / 2; i += kT) ((float4 *)smem)[i] = zero4;   // both buffers
    for (int i = tid; i < 4 * G; i += kT) sxs[i] = i < nx ? p.sig_x[i] : 0.0f;
    for (int i = tid; i < R; i += kT) szs[i] = p.sig_z[r0 + i];
    __syncthreads();
    {
        const int za = max(0, r0 - M), ze = min(nz, r1 + M);
        for (int i = tid; i < (ze - za) * G; i += kT) {
            const int z = za + i / G, g = i % G;
            const int at = (z - r0 + M) * SX + M + 4 * g;
            *(float4 *)(buf0 + at) = *(const float4 *)(u0 + (int64_t)z * px + 4 * g);
            if (z >= r0 && z < r1) *(float4 *)(buf1 + at) = *(const float4 *)(u1 + (int64_t)z * px + 4 * g);
        }
    }
    // this thread's blocks
    int soff[NU], goff[NU], lr0[NU];    // shared offset of the z-walk's first row, field offset
    float4 Wv[NU][kRZ], gv[MODE == kRev ? NU : 1][kRZ];
    uint4 ur[MODE == kRev ? NU : 1][kRZ];
    bool edge = false;                  // some of them read halo rows
    int src_u = -1, src_r = 0, src_e = 0, rec_u = -1, rec_r = 0;
    int4 ri = make_int4(-1, -1, -1, -1);
    const int64_t so = p.src_off ? p.src_off[shot] : -1;
#pragma unroll
    for (int u = 0; u < NU; ++u) {
        const int id = tid + u * kT;
        lr0[u] = id < U ? id / G * kRZ : R;          // R: no block
        const int g = id % G;
        soff[u] = lr0[u] * SX + M + 4 * g;
        goff[u] = (r0 + lr0[u]) * px + 4 * g;
        edge |= lr0[u] < R && (lr0[u] < M || lr0[u] + kRZ > R - M);
#pragma unroll
        for (int r = 0; r < kRZ; ++r) {
            const bool in = lr0[u] + r < R;
            Wv[u][r] = in ? __ldg((const float4 *)(p.W + goff[u] + r * px)) : zero4;
            if (MODE == kRev) gv[u][r] = in ? *(const float4 *)(p.gacc + (int64_t)shot * p.g.field + goff[u] + r * px) : zero4;
            const int64_t d = so - (goff[u] + r * px);
            if (in && so >= 0 && d >= 0 && d < 4) {
                src_u = u;
                src_r = r;
                src_e = (int)d;
            }
            if (in && p.rec_map && r0 + lr0[u] + r == p.rec_z) {
                rec_u = u;
                rec_r = r;
                ri = __ldg((const int4 *)(p.rec_map + (int64_t)shot * p.g.plane + 4 * g));
            }
        }
    }
    // The end of a step that made state t: a CTA barrier and, with checkpoints, this CTA's
    // maxima of the state into cmax[t & 1] of every CTA.
    auto end_step = [&](float mxa, float mxd, int t) {
        if (MODE == kCkpt) {
            const unsigned wa = __reduce_max_sync(0xffffffffu, __float_as_uint(mxa) & 0x7fffffffu);
            const unsigned wd = __reduce_max_sync(0xffffffffu, __float_as_uint(mxd) & 0x7fffffffu);
            if ((tid & 31) == 0) wmax[t & 1][tid >> 5] = make_uint2(wa, wd);
        }
        __syncthreads();
        if (MODE == kCkpt && tid < 32) {
            const uint2 w = tid < kT / 32 ? wmax[t & 1][tid] : make_uint2(0u, 0u);
            const uint2 c = make_uint2(__reduce_max_sync(0xffffffffu, w.x), __reduce_max_sync(0xffffffffu, w.y));
            if (tid < C) send(in_cta(&cmax[t & 1][rank], tid), c, in_cta(max_bar + (t & 1), tid));
        }
    };
    // The maxima of state t over the cluster, once they have arrived.
    auto state_max = [&](int t) {
        wait_for(max_bar + (t & 1), t >> 1);
        __syncwarp();
        const int i = tid & 31;
        const uint2 c = i < C ? cmax[t & 1][i] : make_uint2(0u, 0u);
        return make_uint2(__reduce_max_sync(0xffffffffu, c.x), __reduce_max_sync(0xffffffffu, c.y));
    };
    // operands of step s that come from global memory, one step ahead
    float srcv = 0.0f, ainv = 1.0f;
    float4 inj = zero4;
    // the schedule entry of the next step to fetch and its codes, found one step earlier still
    int nd = -1;
    char *ncodes = nullptr;
    auto look_up = [&](int s) {
        if (MODE == kFwd || s >= k) return;
        nd = __ldg(a.desc + s);
        if (nd >= 0) ncodes = slot_codes(a, p.g.field, nd, shot);
    };
    auto fetch = [&](int s) {
        if (s >= k) return;
        const int n = MODE == kRev ? n0 - s : n0 + s;
        if (src_u >= 0) srcv = p.dt2 * p.wavelet[(int64_t)shot * p.nt + n];
        if (MODE == kRev) {
            const int d = nd;
            const char *codes = ncodes;
            look_up(s + 1);
            ainv = a.dtype == 0 ? 1.0f : 1.0f / a.scales[((int64_t)(d & kOnchipSlot) * a.ns + shot) * 2];
#pragma unroll
            for (int u = 0; u < NU; ++u)
#pragma unroll
                for (int r = 0; r < kRZ; ++r) {
                    if (lr0[u] + r >= R) continue;
                    const int o = goff[u] + r * px;
                    if (a.dtype == 0) {
                        ur[u][r] = __ldg((const uint4 *)((const float *)codes + o));
                    } else {
                        const uint2 h = __ldg((const uint2 *)((const unsigned short *)codes + o));
                        ur[u][r].x = h.x;
                        ur[u][r].y = h.y;
                    }
                }
            if (rec_u >= 0) {
                const float *sc = p.inj_scale + (int64_t)shot * p.nrec;
                const float *q = p.inj_q + ((int64_t)shot * p.nt + n - 1) * p.nrec;
                // the products are rounded as the separate injection kernel rounds them
                if (ri.x >= 0) inj.x = __fmul_rn(sc[ri.x], q[ri.x]);
                if (ri.y >= 0) inj.y = __fmul_rn(sc[ri.y], q[ri.y]);
                if (ri.z >= 0) inj.z = __fmul_rn(sc[ri.z], q[ri.z]);
                if (ri.w >= 0) inj.w = __fmul_rn(sc[ri.w], q[ri.w]);
            }
        }
    };
    if (MODE == kRev) {
#pragma unroll
        for (int u = 0; u < NU; ++u)
#pragma unroll
            for (int r = 0; r < kRZ; ++r) ur[u][r] = make_uint4(0u, 0u, 0u, 0u);
    }
    look_up(0);
    fetch(0);
    if (MODE == kCkpt) {
        __syncthreads();   // the states are loaded
        float mxa = 0.0f, mxd = 0.0f;
        if (a.first_store) {
#pragma unroll
            for (int u = 0; u < NU; ++u)
#pragma unroll
                for (int r = 0; r < kRZ; ++r) {
                    if (lr0[u] + r >= R) continue;
                    const float4 c = *(const float4 *)(buf0 + soff[u] + (M + r) * SX);
                    const float4 v = *(const float4 *)(buf1 + soff[u] + (M + r) * SX);
                    mxa = absmax_nan(absmax_nan(absmax_nan(absmax_nan(mxa, c.x), c.y), c.z), c.w);
                    mxd = absmax_nan(absmax_nan(absmax_nan(absmax_nan(mxd, c.x - v.x), c.y - v.y), c.z - v.z), c.w - v.w);
                }
        }
        cl.sync();         // every CTA runs and its barriers are initialised
        end_step(mxa, mxd, 0);
    } else {
        cl.sync();
    }
    // the neighbours' copies of this CTA's edge rows, as offsets to a row's place in a buffer
    const uint32_t up_s = rank > 0 ? in_cta(smem, rank - 1) + (Rup + M) * SX * 4 : 0u;
    const uint32_t up_b = rank > 0 ? in_cta(halo_bar, rank - 1) : 0u;
    const uint32_t dn_s = rank < C - 1 ? in_cta(smem, rank + 1) - (R - M) * SX * 4 : 0u;
    const uint32_t dn_b = rank < C - 1 ? in_cta(halo_bar, rank + 1) : 0u;

    for (int s = 0; s < k; ++s) {
        const int n = MODE == kRev ? n0 - s : n0 + s;
        float *cur = (s & 1) ? buf1 : buf0, *nxt = (s & 1) ? buf0 : buf1;
        const int par = (s + 1) & 1;                       // of the state this step makes
        const uint32_t nxt_off = par ? l.rows * SX * 4 : 0;
        // state s's halo rows, and the counts of the messages this step's neighbours send
        if (s > 0 && (tid == 0 || edge)) wait_for(halo_bar + (s & 1), (s - 1) >> 1);
        if (tid == 0 && !dead) {
            mbar_expect_tx(halo_bar + par, halo_bytes);
            if (MODE == kCkpt) mbar_expect_tx(max_bar + par, 8 * C);
        }
        const int st = MODE == kCkpt && (s > 0 || a.first_store) ? nd : -1;
        char *codes = ncodes;
        float sca = 1.0f, scd = 1.0f;
        float mxa = 0.0f, mxd = 0.0f;
        float2 za[kRZ], zb[kRZ];
        float4 ctr[kRZ];
        if (lr0[0] < R) z_block<M, kRZ>(cur + soff[0], SX, p.c, ctr, za, zb);
        if (MODE == kCkpt) {
            look_up(s + 1);
            if (st >= 0) {
                const uint2 m = state_max(s);
                sca = snap_scale(m.x, a.dtype);
                scd = snap_scale(m.y, a.dtype);
                if (rank == 0 && tid == 0) {
                    float *sc = a.scales + ((int64_t)(st & kOnchipSlot) * a.ns + shot) * 2;
                    sc[0] = sca;
                    sc[1] = scd;
                    if (m.x >= 0x7f800000u) atomicOr(a.flag, 1u);
                }
            } else if (tid == 0) {
                wait_for(max_bar + (s & 1), s >> 1);
            }
        }
#pragma unroll
        for (int u = 0; u < NU; ++u) {
            if (lr0[u] >= R) continue;
            const float *col = cur + soff[u];
            if (u > 0) z_block<M, kRZ>(col, SX, p.c, ctr, za, zb);
            const int xg = (soff[u] - lr0[u] * SX - M);   // first column of the group
            const float4 sx = *(const float4 *)(sxs + xg);
#pragma unroll
            for (int r = 0; r < kRZ; ++r) {
                const int lr = lr0[u] + r;
                if (lr >= R) continue;
                float w[4 + 2 * M];
                const float *row = col + (r + M) * SX - M;
#pragma unroll
                for (int g4 = 0; g4 < (4 + 2 * M) / 4; ++g4) {
                    const float4 v = g4 == M / 4 ? ctr[r] : *(const float4 *)(row + 4 * g4);
                    w[4 * g4] = v.x, w[4 * g4 + 1] = v.y, w[4 * g4 + 2] = v.z, w[4 * g4 + 3] = v.w;
                }
                const float4 c = ctr[r];
                // u^{n-1} of this point lies where u^{n+1} goes
                float *own = nxt + soff[u] + (M + r) * SX;
                const float4 v = *(const float4 *)own;
                float2 l0, l1;
                lap_x<M>(w, c, p.c, za[r], zb[r], l0, l1);
                const bool at_src = u == src_u && r == src_r;
                float4 o = update4(c, l0, l1, v, Wv[u][r], sx, szs[lr],
                                   (MODE != kRev && at_src) ? src_e : -1, srcv);
                if (u == rec_u && r == rec_r) {
                    if (MODE == kRev) {
                        if (ri.x >= 0) o.x = __fadd_rn(o.x, inj.x);
                        if (ri.y >= 0) o.y = __fadd_rn(o.y, inj.y);
                        if (ri.z >= 0) o.z = __fadd_rn(o.z, inj.z);
                        if (ri.w >= 0) o.w = __fadd_rn(o.w, inj.w);
                    } else if (p.rec_tr && n >= a.rec_from) {
                        float *tr = p.rec_tr + ((int64_t)shot * p.nt + n) * p.nrec;
                        if (ri.x >= 0) tr[ri.x] = o.x;
                        if (ri.y >= 0) tr[ri.y] = o.y;
                        if (ri.z >= 0) tr[ri.z] = o.z;
                        if (ri.w >= 0) tr[ri.w] = o.w;
                    }
                }
                const int x = M + xg;
                *(float4 *)own = o;
                const uint32_t to = nxt_off + (uint32_t)(lr * SX + x) * 4;
                if (lr < M && rank > 0) send(up_s + to, o, up_b + 8 * par);
                if (lr >= R - M && rank < C - 1) send(dn_s + to, o, dn_b + 8 * par);
                if (MODE == kCkpt) {
                    mxa = absmax_nan(absmax_nan(absmax_nan(absmax_nan(mxa, o.x), o.y), o.z), o.w);
                    mxd = absmax_nan(absmax_nan(absmax_nan(absmax_nan(mxd, o.x - c.x), o.y - c.y), o.z - c.z), o.w - c.w);
                    if (st >= 0) {
                        const int ci = goff[u] + r * px;
                        if (a.dtype == 0) {
                            *(float4 *)((float *)codes + ci) = c;
                            if (st & kOnchipPair) *(float4 *)((float *)codes + ci + p.g.field) = v;
                        } else {
                            unsigned short *cc = (unsigned short *)codes + ci;
                            *(uint2 *)cc = pack_code4(c, a.dtype, sca);
                            if (st & kOnchipPair)
                                *(uint2 *)(cc + p.g.field) = pack_code4(
                                    make_float4(c.x - v.x, c.y - v.y, c.z - v.z, c.w - v.w), a.dtype, scd);
                        }
                    }
                }
                if (MODE == kRev) {
                    const uint4 q = ur[u][r];
                    const float4 um = a.dtype == 0
                                          ? make_float4(__uint_as_float(q.x), __uint_as_float(q.y),
                                                        __uint_as_float(q.z), __uint_as_float(q.w))
                                          : unpack_code4(make_uint2(q.x, q.y), a.dtype, ainv);
                    float2 g0 = __ffma2_rn(lo2(um), l0, lo2(gv[u][r]));
                    float2 g1 = __ffma2_rn(hi2(um), l1, hi2(gv[u][r]));
                    if (at_src) s3d::src_image(g0, g1, c, Wv[u][r], src_e, srcv);
                    gv[u][r] = make_float4(g0.x, g0.y, g1.x, g1.y);
                }
            }
        }
        fetch(s + 1);
        end_step(mxa, mxd, s + 1);
    }
    // no message may be on its way to a CTA that ends
    if (tid == 0) {
        wait_for(halo_bar + (k & 1), (k - 1) >> 1);
        if (MODE == kCkpt) wait_for(max_bar + (k & 1), k >> 1);
    }
    cl.sync();
    // back to global memory, in the buffers that k single steps would leave
    float *newest = (k & 1) ? u1 : u0, *older = (k & 1) ? u0 : u1;
    const float *cur = (k & 1) ? buf1 : buf0, *old = (k & 1) ? buf0 : buf1;
#pragma unroll
    for (int u = 0; u < NU; ++u)
#pragma unroll
        for (int r = 0; r < kRZ; ++r) {
            if (lr0[u] + r >= R) continue;
            const int o = goff[u] + r * px;
            *(float4 *)(newest + o) = *(const float4 *)(cur + soff[u] + (M + r) * SX);
            *(float4 *)(older + o) = *(const float4 *)(old + soff[u] + (M + r) * SX);
            if (MODE == kRev) *(float4 *)(p.gacc + (int64_t)shot * p.g.field + o) = gv[u][r];
        }
    if (MODE == kCkpt) {
        const uint2 m = state_max(k);
        if (rank == 0 && tid == 0) {
            a.maxbits[2 * shot] = m.x;
            a.maxbits[2 * shot + 1] = m.y;
            a.max_clear[2 * shot] = a.max_clear[2 * shot + 1] = 0u;
        }
    }
}

template <int M, int MODE, int NU>
__global__ void __launch_bounds__(kT, 1) k_step2d_onchip(const __grid_constant__ Onchip2d a)
{
    extern __shared__ __align__(16) float smem[];
    const int shot = blockIdx.x / a.C;
    const int64_t sb = (int64_t)shot * a.p.g.field;
    advance<M, MODE, NU>(a.ck, a.p, a.u0 + sb, a.u1 + sb, a.n0, a.k, smem, shot);
}

// The serving loop's form: one cluster per request of the table, at most k steps each.
template <int M>
__global__ void __launch_bounds__(kT, 1) k_step2d_cluster(const Batch2d *__restrict__ tab, int k)
{
    extern __shared__ __align__(16) float smem[];
    const int req = blockIdx.x / (int)cg::this_cluster().num_blocks();   // uniform per cluster
    if (req >= tab->count) return;
    const Batch2dEntry &E = tab->e[req];
    const OnchipCkpt none{};
    const int left = E.p.nt - E.n0;
    if (left > 0) advance<M, kFwd, onchip_units(M, kFwd)>(none, E.p, E.u0, E.u1, E.n0, left < k ? left : k, smem, 0);
}

typedef void (*OnchipKernel)(const Onchip2d);

template <int M, int MODE>
OnchipKernel onchip_kernel(int nu)
{
    constexpr int most = onchip_units(M, MODE);
    if (nu == 1) return k_step2d_onchip<M, MODE, 1>;
    if constexpr (most >= 2)
        if (nu == 2) return k_step2d_onchip<M, MODE, 2>;
    if constexpr (most >= 3)
        if (nu == 3) return k_step2d_onchip<M, MODE, 3>;
    if constexpr (most >= 4)
        if (nu == 4) return k_step2d_onchip<M, MODE, 4>;
    return nullptr;
}

OnchipKernel onchip_kernel(int M, int mode, int nu)
{
    if (M == 4)
        return mode == kFwd ? onchip_kernel<4, kFwd>(nu) : mode == kCkpt ? onchip_kernel<4, kCkpt>(nu)
                                                                          : onchip_kernel<4, kRev>(nu);
    if (M == 8)
        return mode == kFwd ? onchip_kernel<8, kFwd>(nu) : mode == kCkpt ? onchip_kernel<8, kCkpt>(nu)
                                                                          : onchip_kernel<8, kRev>(nu);
    return nullptr;
}

cudaError_t prepare(const void *fn)
{
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    return e;
}

struct ClusterConfig {
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute at[1];
    ClusterConfig(int C, int clusters, int smem, cudaStream_t s)
    {
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = C;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        cfg.gridDim = dim3(C * clusters, 1, 1);
        cfg.blockDim = dim3(kT, 1, 1);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = s;
        cfg.attrs = at;
        cfg.numAttrs = 1;
    }
};

// Clusters of C CTAs with full shared memory that run at once (0: none, or the query failed).
int active_clusters(int M, int C)
{
    const void *fn = M == 8 ? (const void *)k_step2d_cluster<8> : (const void *)k_step2d_cluster<4>;
    if (prepare(fn) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    ClusterConfig c(C, 1, kSmemMax, nullptr);
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, fn, &c.cfg) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return n;
}

// Blocks per thread of the fullest CTA.
int units_of(const Geom &g, int C)
{
    const Layout l = layout_of(g.nz, g.nx, g.M, C);
    const int rows = (g.nz + C - 1) / C;
    return (l.G * ((rows + kRZ - 1) / kRZ) + kT - 1) / kT;
}

}  // namespace

int onchip2d_smem(const Geom &g, int C)
{
    return (layout_of(g.nz, g.nx, g.M, C).floats * 4 + 1023) / 1024 * 1024;
}

bool onchip2d_fits(const Geom &g, int C, int mode)
{
    // bands of at least M rows (halos reach the next CTA only), no more than one row of
    // blocks per pass over the threads (a thread then meets the receiver row once)
    return C > 0 && g.ndim == 2 && g.nz / C >= g.M && (g.nx + 3) / 4 <= kT &&
           units_of(g, C) <= onchip_units(g.M, mode) && onchip2d_smem(g, C) <= kSmemMax;
}

int cluster2d_size(int M)
{
    for (int C : {kMaxC, 8})
        if (active_clusters(M, C) > 0) return C;
    return 0;
}

int onchip2d_clusters(int M, int C) { return C > 0 ? active_clusters(M, C) : 0; }

cudaError_t launch_step2d_onchip(const Onchip2d &a, int mode, cudaStream_t s)
{
    const OnchipKernel fn = onchip_kernel(a.p.g.M, mode, units_of(a.p.g, a.C));
    if (!fn) return cudaErrorInvalidValue;
    const cudaError_t e = prepare((const void *)fn);
    if (e != cudaSuccess) return e;
    ClusterConfig c(a.C, a.ck.ns, onchip2d_smem(a.p.g, a.C), s);
    return cudaLaunchKernelEx(&c.cfg, fn, a);
}

int cluster2d_max_smem() { return kSmemMax; }

cudaError_t launch_step2d_cluster(const Batch2d *tab, int M, int k, int C, int nreq, int smem, cudaStream_t s)
{
    ClusterConfig c(C, nreq > 0 ? nreq : 1, smem, s);
    if (M == 4) return cudaLaunchKernelEx(&c.cfg, k_step2d_cluster<4>, tab, k);
    if (M == 8) return cudaLaunchKernelEx(&c.cfg, k_step2d_cluster<8>, tab, k);
    return cudaErrorInvalidValue;
}

}  // namespace fwi
