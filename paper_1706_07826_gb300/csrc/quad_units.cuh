// How the quad-group kernels (sweep_pm1q.cu, sweep_gq.cu) deal a work item's colour classes
// over the block: units (spin, every G-th group of the item's quads), listed once per item.
#pragma once
#include "sweep_common.cuh"

namespace spvar {

// How a colour class of nc spins is dealt over the block for np pairs of quads.
// Units (spin, group g of pairs g, g + G, ...) fill full rounds of B threads; the
// units left for a last partial round are each split into G2 sub-units (every
// G2-th pair of the unit's group), so that round uses the whole block.  G is the
// choice, within `most` rounds, that minimises the rounds' length, a unit's set-up
// counted as a fifth of a pair.  Returns (G, full units, remainder units, G2).
__device__ __forceinline__ int4 class_split(int nc, int np, int B, int most)
{
    int best = 0x7FFFFFFF;
    int4 pick = make_int4(1, 0, 0, 1);
    for (int G = 1; G <= np; ++G) {
        const int ppu = (np + G - 1) / G;
        const int U = nc * G, R = U / B, Ur = U - R * B;
        if (G > 1 && R + (Ur > 0) > most) break;
        int cost = R * (5 * ppu + 1), G2 = 1;
        if (Ur > 0) {
            G2 = max(1, min(ppu, B / Ur));
            cost += 5 * ((ppu + G2 - 1) / G2) + 1;
        }
        if (cost < best) {
            best = cost;
            pick = make_int4(G, R * B, Ur, G2);
        }
    }
    return pick;
}

// Per colour class (lo, spins, rounds of the block, first row of the unit list or -1), one
// thread.  A class's units are listed while its rounds fit its share of the list's rows;
// longer classes (and items of one group) are walked a spin per thread, every group at once.
template <int B>
__device__ __forceinline__ void unit_classes(const DevProb *P, int ncol, int ng, int unit_rows, int4 *cls)
{
    int row = 0;
    for (int c = 0; c < ncol; ++c) {
        const int lo = P->cptr[c], nc = P->cptr[c + 1] - lo, plain = (nc + B - 1) / B;
        int4 k = make_int4(lo, nc, plain, -1);
        const int most = (unit_rows - row) / (ncol - c);
        if (plain <= most && ng > 1) {
            const int4 sp = class_split(nc, ng, B, most);
            k.z = (sp.y + sp.z * sp.w + B - 1) / B;
            k.w = row;
            row += k.z;
        }
        cls[c] = k;
    }
}

// This thread's entries of the unit list ([unit_rows][B]): position | first group << 16 |
// group step << 24; a first group past the last means no unit.
template <int B>
__device__ __forceinline__ void unit_list(int ncol, int ng, int unit_rows, const int4 *cls, uint32_t *unit)
{
    for (int c = 0; c < ncol; ++c) {
        const int4 k = cls[c];
        if (k.w < 0) continue;
        const int4 sp = class_split(k.y, ng, B, (unit_rows - k.w) / (ncol - c));
        for (int r = 0; r < k.z; ++r) {
            const int u = r * B + (int)threadIdx.x;
            uint32_t d = 0xFF0000u;
            if (u < sp.y + sp.z * sp.w) {
                int uu = u, j = 0;
                if (u >= sp.y) {
                    j = (u - sp.y) / sp.z;
                    uu = u - j * sp.z;
                }
                const int g = uu / k.y, step = u < sp.y ? sp.x : sp.x * sp.w;
                d = (uint32_t)(k.x + uu - g * k.y) | (uint32_t)(g + j * sp.x) << 16 | (uint32_t)step << 24;
            }
            unit[(k.w + r) * B + (int)threadIdx.x] = d;
        }
    }
}

}  // namespace spvar
