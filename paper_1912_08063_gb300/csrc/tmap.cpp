// Host helpers of the TMA-staged 3-D step: tensor-map encoding (through the driver entry
// point, so the library needs no libcuda link) and the persistent schedule.
#include <cudaTypedefs.h>

#include <algorithm>

#include "step3d.h"

namespace fwi {

int encode_field_map(CUtensorMap *map, const void *base, const Geom &g, int nshots, int bx,
                     int by, int bz, int elem_bytes, int64_t shot_stride)
{
    if (elem_bytes != 4 && elem_bytes != 2) return -1;
    static PFN_cuTensorMapEncodeTiled_v12000 encode = nullptr;
    if (!encode) {
        void *f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000,
                                             cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess || !f) {
            cudaGetLastError();
            return -1;
        }
        encode = (PFN_cuTensorMapEncodeTiled_v12000)f;
    }
    const cuuint64_t dims[4] = {(cuuint64_t)g.nx, (cuuint64_t)g.ny, (cuuint64_t)g.nz,
                                (cuuint64_t)nshots};
    const cuuint64_t eb = (cuuint64_t)elem_bytes;
    const cuuint64_t strides[3] = {(cuuint64_t)g.px * eb, (cuuint64_t)g.plane * eb,
                                   (cuuint64_t)shot_stride * eb};
    const cuuint32_t box[4] = {(cuuint32_t)bx, (cuuint32_t)by, (cuuint32_t)bz, 1};
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    // 16-bit codes are moved as raw 16-bit words (zero fill = +0 in either format)
    const CUtensorMapDataType dt =
        elem_bytes == 4 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_UINT16;
    CUresult r = encode(map, dt, 4, const_cast<void *>(base), dims,
                        strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                        CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? 0 : -1;
}

int encode_field_map2d(CUtensorMap *map, const void *base, const Geom &g, int nshots, int bx,
                       int bz, int elem_bytes, int64_t shot_stride)
{
    if (elem_bytes != 4 && elem_bytes != 2) return -1;
    static PFN_cuTensorMapEncodeTiled_v12000 encode = nullptr;
    if (!encode) {
        void *f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000,
                                             cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess || !f) {
            cudaGetLastError();
            return -1;
        }
        encode = (PFN_cuTensorMapEncodeTiled_v12000)f;
    }
    const cuuint64_t eb = (cuuint64_t)elem_bytes;
    const cuuint64_t dims[3] = {(cuuint64_t)g.nx, (cuuint64_t)g.nz, (cuuint64_t)nshots};
    const cuuint64_t strides[2] = {(cuuint64_t)g.px * eb, (cuuint64_t)shot_stride * eb};
    const cuuint32_t box[3] = {(cuuint32_t)bx, (cuuint32_t)bz, 1};
    const cuuint32_t estr[3] = {1, 1, 1};
    const CUtensorMapDataType dt =
        elem_bytes == 4 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_UINT16;
    CUresult r = encode(map, dt, 3, const_cast<void *>(base), dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                        CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? 0 : -1;
}

// Planes (with warm-up) the busiest CTA streams under schedule p.
static int64_t schedule_cost(const Step3dParams &p, int columns, int grid)
{
    int64_t worst = 0;
    for (int k = 0; k < grid; ++k) {
        int64_t it = 0;
        int col, z0, z1;
        for (int i = 0; schedule_segment(p, columns, k, i, &col, &z0, &z1); ++i) it += z1 - z0 + 2 * p.M;
        if (it > worst) worst = it;
    }
    return worst;
}

int plan_persistent(Step3dParams &p, int columns, int resident, bool in_step)
{
    if (resident < 1) resident = 1;
    if (columns < 1) columns = 1;
    // whole columns: rounds, then the leftover columns cut into pieces of >= 4M planes
    p.zparts = 1;
    p.zfirst = p.nz;
    p.round_ctas = resident;
    p.rounds = columns / resident;
    p.rem_first = 0;
    p.rem_ppu = 0;
    {
        const long long rem_planes = (long long)(columns - p.rounds * resident) * p.nz;
        long long pieces = rem_planes / (4LL * p.M);
        if (pieces < 1) pieces = 1;
        if (pieces > resident) pieces = resident;
        p.rem_ctas = rem_planes > 0 ? (int)pieces : 0;
    }
    int grid = p.rounds > 0 ? resident : (p.rem_ctas > 0 ? p.rem_ctas : 1);
    if (!in_step) return grid;
    if (columns >= resident) {
        // Whole rounds of units and, for the leftover units, pieces of one length that begin
        // at the same z in every unit, so that the CTAs of a round stream z in step and a
        // tile's halo planes are still in L2 when its neighbours read them (one run cut over
        // all CTAs would put them at unrelated z).  S parts per column make the leftover a
        // smaller share at the price of S warm-ups; the S whose busiest CTA streams the
        // fewest planes is taken.  Measured on GB300, us per launch with one run / with
        // rounds and pieces in step: 140 x 1064 x 1064 radius 4 forward 531 / 447, store 635 /
        // 537, reverse 721 / 661; radius 8 626 / 477, 708 / 535, 858 / 714; 296 x 552 x 1064
        // radius 4 reverse 863 / 690; 1064^3 radius 4 forward 4218 / 3757.
        int64_t best = -1;
        Step3dParams b = p;
        for (int S = 1; S <= 16 && p.nz / S >= 4 * p.M; ++S) {
            const int len = p.nz / S, last = p.nz - (S - 1) * len;   // the last part is the longest
            const int64_t units = (int64_t)columns * S;
            const int rounds = (int)(units / resident), left = (int)(units - (int64_t)rounds * resident);
            int ppu = left > 0 ? resident / left : 0;
            while (ppu > 1 && last / ppu < 4 * p.M) --ppu;
            const int64_t cost = (int64_t)rounds * (last + 2 * p.M) +
                                 (left > 0 ? (last + ppu - 1) / ppu + 2 * p.M : 0);
            if (best >= 0 && cost >= best) continue;
            best = cost;
            b.zparts = S;
            b.zfirst = len;
            b.rounds = rounds;
            b.rem_ppu = ppu;
            b.rem_ctas = left * ppu;
        }
        if (best >= 0) {
            p.zparts = b.zparts;
            p.zfirst = b.zfirst;
            p.rounds = b.rounds;
            p.rem_ppu = b.rem_ppu;
            p.rem_ctas = b.rem_ctas;
        }
        return grid;
    }

    const int S = (resident + columns - 1) / columns;   // (S - 1) columns < resident
    Step3dParams best = p;
    int64_t best_cost = -1;
    int best_grid = grid;
    // (a) every column in the same number of pieces of at least M planes, one to a CTA
    {
        const int most = std::min(resident / columns, p.nz / p.M);
        if (most > 1) {
            best.zfirst = (p.nz + most - 1) / most;
            best.zparts = (p.nz + best.zfirst - 1) / best.zfirst;
            best.rounds = 1;
            best.round_ctas = best_grid = columns * best.zparts;
            best.rem_ctas = 0;
            best_cost = schedule_cost(best, columns, best_grid);
            if (p.M == 8) best_cost = best_cost * resident * resident / ((int64_t)best_grid * best_grid);
        }
    }
    if (p.nz / S >= 4 * p.M) {
        // (b) equal parts; the L leftover last parts in aligned pieces over all CTAs
        {
            const int L = columns * S - resident, ppu = L > 0 ? resident / L : 0;
            Step3dParams q = p;
            q.zparts = S;
            q.zfirst = p.nz / S;
            q.rounds = 1;
            q.rem_first = 0;
            q.rem_ppu = ppu;
            q.rem_ctas = L * ppu;
            const int64_t c = schedule_cost(q, columns, resident);
            if (best_cost < 0 || c < best_cost) {
                best = q;
                best_cost = c;
                best_grid = resident;
            }
        }
        // (c) longer first parts; the L leftover last parts go in ppu aligned pieces to the
        // qn CTAs that ran a last part, with lengths that balance both kinds of CTA:
        // first part + 2M = last part + 2M + last part / ppu + 2M
        {
            const int qn = resident - (S - 1) * columns, L = columns - qn;
            const int ppu = L > 0 ? qn / L : 0;
            if (L > 0 && ppu >= 1) {
                const double ll = (double)(p.nz - 2 * p.M * (S - 1)) / ((S - 1) * (1.0 + 1.0 / ppu) + 1.0);
                Step3dParams q = p;
                q.zparts = S;
                q.zfirst = (int)((p.nz - ll) / (S - 1) + 0.5);
                const int last = p.nz - (S - 1) * q.zfirst;
                if (last >= 2 * p.M && q.zfirst >= 4 * p.M) {
                    q.rounds = 1;
                    q.rem_first = (S - 1) * columns;
                    q.rem_ppu = ppu;
                    q.rem_ctas = L * ppu;
                    const int64_t c = schedule_cost(q, columns, resident);
                    if (best_cost < 0 || c < best_cost) {
                        best = q;
                        best_cost = c;
                        best_grid = resident;
                    }
                }
            }
        }
    }
    p.zparts = best.zparts;
    p.zfirst = best.zfirst;
    p.rounds = best.rounds;
    p.round_ctas = best.round_ctas;
    p.rem_first = best.rem_first;
    p.rem_ppu = best.rem_ppu;
    p.rem_ctas = best.rem_ctas;
    return best_grid;
}

}  // namespace fwi
