// Parallel tempering with isoenergetic cluster moves (PTICM, Sec. III.D) as
// a sampler of Alg. 1, with the paper's sample: the K lowest-energy distinct
// states seen at each replica of the lower half of the temperatures.
//
// One CTA runs one PTICM run (start = start0 + blockIdx.x).  R inverse
// temperatures, two replicas (copies) each, replica r = 2k + c; a quad is four
// replicas (two temperatures) in one 32-bit word of shared memory per spin, by
// position: bit 0 of byte r & 3 of quad r >> 2 is the spin.  A sweep:
//   1. a Metropolis sweep of every replica at its temperature, a spin per lane: a
//      warp sets its 32 spins of a colour class up once and takes them through
//      every quad of its group (one Philox block per spin and quad, counter and
//      words of the SA sweep).  Up to degree 8 and dmax 254 the flip costs of four
//      replicas are formed byte-wise, one multiply-add per neighbour; other problems
//      use 16-bit lanes.  Energy changes are summed over the warp and reach the
//      replica energies once per quad;
//   2. Houdayer's cluster move at every temperature k >= icm_from whose
//      copies differ somewhere: the differing set D by
//      ballots in index order, the seed its element floor(u |D| / 2^32), then the
//      clusters of up to 32 temperatures by growth of one bit mask per spin; both
//      copies flip on their cluster, and their energies change by its boundary sum
//      (the couplers that leave it end outside D), so no energy pass follows;
//   3. replica exchange between temperatures k and k + 1 for k = t (mod 2):
//      the pairs are disjoint, so every decision is taken at once from the
//      replicas' energies and an integer threshold table, and accepted pairs
//      swap their bytes;
//   4. a warp per tracked replica offers its state, bit-packed in index
//      order, to the replica's list of the K lowest distinct states seen.
// Every wait is a CTA or warp barrier that all of its threads reach.
//
// Bound: the integer pipes (two 512-thread CTAs an SM, issue active 70 %).  3D L = 10,
// 304 runs x 32 temperatures, 500 sweeps: 92.5 ms with a byte per spin, byte-wise fields and
// a queue search per temperature, 28.9 ms now (3.4e11 Metropolis attempts/s).  Of a
// sweep's time the Metropolis part takes 25 us (150 instructions per four attempts of 32
// lanes, Philox 70 of them), the cluster moves 20 us (82 us with the queue search: 500
// instructions a step), the exchanges 4 us and the kept lists 7 us.  The byte-lane forms
// spill 52 to 92 bytes at the 64 registers of two CTAs an SM.
#include <climits>
#include <cstring>

#include "sweep_common.cuh"

namespace spvar {

namespace {

constexpr int kPtMaxR = 64;     // most temperatures
constexpr int kPtBlock = 512;   // threads per run: two runs (32 warps) per SM when shared memory allows
constexpr int kPtRowPad = 128;    // words after the rows: an index of a cost that is not positive reads up to 127 past its row
constexpr int kPtMaxN = 2048;     // most spins
constexpr int kPtWarpWords = kPtMaxN / 32;  // packed words of one state a warp keeps

struct PticmArgs {
    const DevProb *prob;
    const uint32_t *thr;   // [R][thr_stride]: Metropolis thresholds of each temperature
    const uint32_t *xthr;  // [R - 1][dx + 1]: exchange thresholds
    int32_t R, T, thr_stride, dx, icm_from, keep_from, K, flags;
    uint64_t seed;
    uint32_t start0, phase;
    uint32_t *kept;        // [runs][ntr][K][W] bit-packed, index order
    int64_t *kept_e;       // [runs][ntr][K] (with offset)
    int32_t *nkept;        // [runs][ntr]
    uint32_t *final_bits;  // [runs][2R][W]
    int64_t *final_e;      // [runs][2R] (with offset)
    // slot mode (the sampler of Alg. 2 in a plan): CTA b runs start b of the slot
    // table with that start's current problem, seed and phase; the kept lists go
    // to its sample rows and recorded energies and are compacted there
    Slot *slots;
    int32_t Smax;
};

__device__ __forceinline__ uint32_t word0(uint32_t w0, uint32_t y, uint32_t start, uint32_t k0, uint32_t k1)
{
    return philox4x32_10(make_uint4(w0, y, 0u, start), k0, k1).x;
}

// Energies (without offset) of every replica into E[r]: one warp per quad sums
// s_i (2 h_i + sum_j J_ij s_j) = 2E over its spins.  Contains __syncthreads.
template <int B>
__device__ void replica_energies(const DevProb *P, const uint32_t *sw, int NR, int *E)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n = P->n, cap_n = P->cap_n;
    for (int q = warp; 4 * q < NR; q += B / 32) {
        const uint32_t *s = sw + (size_t)q * n;
        int acc[4] = {0, 0, 0, 0};
        for (int p = lane; p < n; p += 32) {
            int c2[4];
            energy2<false>(s[p], P->meta[p], P->ell, cap_n, p, s, c2);
#pragma unroll
            for (int r = 0; r < 4; ++r) acc[r] += c2[r];
        }
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int t = __reduce_add_sync(0xFFFFFFFFu, acc[r]);
            if (lane == 0 && 4 * q + r < NR) E[4 * q + r] = t / 2;
        }
    }
    __syncthreads();
}

// One Metropolis sweep of every replica.  cls: per colour class, first position,
// spins, quad groups, rounds of the block's warps (a warp's unit is 32 spins of the
// class and every G-th quad).  qt: per quad (lo(M1 q) ^ key0 of round 2, the sweep's
// M0 (hi(M1 q) ^ y ^ key0), hi(M1 q) ^ key0).  rows: thresholds by temperature of the
// costs e = dE/2 = 1 .. bias.
// MAXD > 0: degree <= MAXD and dmax <= 254, byte lanes.  With b the spin bits the cost of
// a b_i = 0 replica is e = 2 sum_j J_ij b_j + h - sum_j J_ij and of b_i = 1 minus that;
// e + 127 of the four replicas is one multiply-add per neighbour (the sum is
// exact in each byte however the terms borrow) and its top bit says e > 0.  SMALL (dmax
// <= 62): 4e + 124 instead, the byte offset in the temperature's 256-byte row, which the
// byte permute merges with the row's address.
// MAXD = 0: any problem, the same in two words of 16-bit lanes with e + 32767.
template <int B, int MAXD, bool SMALL>
__device__ __forceinline__ void metropolis(const DevProb *P, uint32_t *sw, const uint32_t *rows, int n, int ncol, int nq,
                                           int R, int NR, int bias, const int4 *cls, const uint4 *qt, int *sE,
                                           uint32_t sk1, uint32_t k1w, const PhiloxKeys<2> &K)
{
    constexpr uint32_t M = 0x01010101u, H = 0x00FF00FFu;
    constexpr int D = MAXD > 0 ? MAXD : 1;
    constexpr uint32_t SC = SMALL ? 4u : 1u, ZERO = SMALL ? 124u : 127u;  // index of cost e: SC e + ZERO
    const int lane = threadIdx.x & 31, cap_n = P->cap_n;
    const int warp = __shfl_sync(0xFFFFFFFFu, (int)threadIdx.x >> 5, 0);  // uniform to the compiler
    const uint32_t *__restrict__ g_meta = P->meta;
    const uint32_t *__restrict__ g_ell = P->ell;
    const int32_t *__restrict__ g_idx = P->idx_of_pos;
    const uint32_t sw4 = shared_addr(sw), rows4 = shared_addr(rows), qt4 = shared_addr(qt), n4 = 4u * (uint32_t)n;
    for (int c = 0; c < ncol; ++c) {
        const int4 cl = cls[c];
        const int chunks = (cl.y + 31) >> 5;
        for (int r = 0; r < cl.w; ++r) {
            const int wu = r * (B / 32) + warp;
            if (wu >= chunks * cl.z) continue;
            const int g = cl.z > 1 ? wu / chunks : 0, k = 32 * (wu - g * chunks) + lane;
            const bool active = k < cl.y;
            const int p = cl.x + (active ? k : 0);
            const uint32_t meta = __ldg(g_meta + p);
            const int deg = (int)(meta & 0xFFFFu);
            uint32_t off[D];
            int J[D], sumJ = 0;
            if (MAXD > 0) {
#pragma unroll
                for (int d = 0; d < D; ++d) {
                    off[d] = 4u * (uint32_t)p;  // a missing neighbour: weight 0
                    J[d] = 0;
                    if (d < deg) {
                        const uint32_t e = __ldg(g_ell + (size_t)d * cap_n + p);
                        off[d] = 4u * (e & 0xFFFFu);
                        J[d] = (int)e >> 16;
                    }
                    sumJ += J[d];
                    if (SMALL) J[d] *= 8;  // 4 * 2
                }
            } else {
                for (int d = 0; d < deg; ++d) sumJ += (int)__ldg(g_ell + (size_t)d * cap_n + p) >> 16;
            }
            const int c0 = ((int)meta >> 16) - sumJ;
            const uint32_t cc = (ZERO + SC * (uint32_t)c0) * M, own4 = 4u * (uint32_t)p;
            uint32_t H0, L0, H2, L2;
            philox_mulhilo(kPhiloxM0, (uint32_t)__ldg(g_idx + p), H0, L0);
            philox_mulhilo(kPhiloxM1, H0 ^ sk1, H2, L2);
            const uint32_t L0k = L0 ^ k1w, mine = active ? M : 0u;
            uint32_t se = 0, so = 0, cnt = 0;  // lane v: the warp's sums for quad v
            for (int v = g; v < nq; v += cl.z) {
                const uint32_t base = sw4 + (uint32_t)v * n4;
                const uint32_t own = lds(base + own4);
                if (MAXD > 0) {
                    uint32_t w[D], a = cc;
#pragma unroll
                    for (int d = 0; d < D; ++d) w[d] = lds(base + off[d]);
                    const uint4 q = lds4(qt4 + 16u * (uint32_t)v);
                    if (SMALL) {
#pragma unroll
                        for (int d = 0; d < D; ++d) a += (uint32_t)J[d] * w[d];
                    } else {
                        uint32_t x = 0;
#pragma unroll
                        for (int d = 0; d < D; ++d) x += (uint32_t)J[d] * w[d];
                        a += 2u * x;
                    }
                    const uint32_t m = own * 255u;
                    const uint32_t idx = (a & ~m) | ((2u * ZERO * M - a) & m);
                    const uint4 u = philox_rounds<2>(make_uint4(H2 ^ q.x, L2, q.y ^ L0k, q.z), K);
                    const uint32_t ur[4] = {u.x, u.y, u.z, u.w};
                    const uint32_t row0 = rows4 + (SMALL ? 512u : 8u * (uint32_t)bias) * (uint32_t)v;
                    const uint32_t row1 = 2 * v + 1 < R ? row0 + (SMALL ? 256u : 4u * (uint32_t)bias) : row0;
                    uint32_t rej = 0;
#pragma unroll
                    for (int rr = 0; rr < 4; ++rr) {
                        const uint32_t row = rr < 2 ? row0 : row1;
                        const uint32_t thr = lds(SMALL ? __byte_perm(idx, row, 0x7650u | (uint32_t)rr)
                                                       : row + 4u * __byte_perm(idx & 0x7F7F7F7Fu, 0u, 0x4440u | (uint32_t)rr));
                        asm("{ .reg .pred p; setp.ge.u32 p, %1, %2; @p add.u32 %0, %0, %3; }"
                            : "+r"(rej)
                            : "r"(ur[rr]), "r"(thr), "r"(1u << (8 * rr)));
                    }
                    const uint32_t flips = mine & ~(rej & (idx >> 7));
                    // sums over the warp: the indices of the flipped replicas in 16-bit lanes, and their number
                    const uint32_t f = idx & (flips * 255u);
                    const uint32_t te = __reduce_add_sync(0xFFFFFFFFu, f & H), to = __reduce_add_sync(0xFFFFFFFFu, (f >> 8) & H);
                    const uint32_t tc = __reduce_add_sync(0xFFFFFFFFu, flips);
                    if (lane == v) {
                        se = te;
                        so = to;
                        cnt = tc;
                    }
                    if (active) sts(base + own4, own ^ flips);
                } else {
                    const uint4 q = qt[v];
                    const uint32_t *s = sw + v * n;
                    const uint32_t *row0 = rows + 2 * v * bias - 1, *row1 = rows + min(2 * v + 1, R - 1) * bias - 1;
                    uint32_t xe = 0, xo = 0;  // replicas 0, 2 and 1, 3
                    for (int d = 0; d < deg; ++d) {
                        const uint32_t e = __ldg(g_ell + (size_t)d * cap_n + p);
                        const uint32_t w = s[e & 0xFFFFu], j = (uint32_t)((int)e >> 16);
                        xe += j * (w & H);
                        xo += j * ((w >> 8) & H);
                    }
                    const uint32_t c16 = (uint32_t)(32767 + c0) * 0x00010001u;
                    const uint32_t ae = 2u * xe + c16, ao = 2u * xo + c16;
                    const uint4 u = philox_rounds<2>(make_uint4(H2 ^ q.x, L2, q.y ^ L0k, q.z), K);
                    const uint32_t ur[4] = {u.x, u.y, u.z, u.w};
                    uint32_t flips = 0;
                    int de[4];
#pragma unroll
                    for (int rr = 0; rr < 4; ++rr) {
                        const int t = (int)(((rr & 1 ? ao : ae) >> (16 * (rr >> 1))) & 0xFFFFu) - 32767;
                        const int e = ((own >> (8 * rr)) & 1u) ? -t : t;
                        const bool acc = active && (e <= 0 || ur[rr] < (rr < 2 ? row0 : row1)[max(e, 1)]);
                        flips |= (uint32_t)acc << (8 * rr);
                        de[rr] = acc ? 2 * e : 0;
                    }
#pragma unroll
                    for (int rr = 0; rr < 4; ++rr) {
                        const int t = __reduce_add_sync(0xFFFFFFFFu, de[rr]);
                        if (lane == rr && 4 * v + rr < NR && t != 0) atomicAdd(&sE[4 * v + rr], t);
                    }
                    if (active) sts(base + own4, own ^ flips);
                }
            }
            if (MAXD > 0 && cnt != 0)
#pragma unroll
                for (int rr = 0; rr < 4; ++rr) {
                    const int t = (int)(((rr & 1 ? so : se) >> (16 * (rr >> 1))) & 0xFFFFu);
                    const int de = 2 * (t - (int)ZERO * (int)((cnt >> (8 * rr)) & 0xFFu)) / (int)SC;
                    if (4 * lane + rr < NR && de != 0) atomicAdd(&sE[4 * lane + rr], de);
                }
        }
        __syncthreads();
    }
}

// Houdayer's moves at temperatures base .. end - 1, of at most 16 quads, all at once: bit
// q' + 16 (k & 1) of Dm[p] says that the copies differ at position p at temperature k of
// the q'-th of these quads, of Cm[p] that p is in that temperature's cluster.  The
// clusters grow by Cm[p] |= Dm[p] & (or of the neighbours' Cm) until nothing changes:
// a few instructions a spin serve every temperature (a search from a queue per
// temperature took 500 instructions for 32 spins of one).  Only spins of D couple
// the copies differently, so over the neighbours s^a_j + s^b_j is 0 in D and 2 s_j
// outside, and the boundary sum of a cluster, h_i s_i + s_i sum_{j outside} J_ij s_j,
// needs the copies' sum alone.  Contains __syncthreads, the last at its end.
template <int B, int MAXD>
__device__ __forceinline__ void cluster_moves(const DevProb *P, uint32_t *sw, uint32_t *Dm, uint32_t *Cm, int n, int base,
                                              int end, uint32_t y, uint32_t start, uint32_t k0, uint32_t k1, int *s_seed,
                                              int *s_sum, int *sE)
{
    constexpr uint32_t H = 0x00FF00FFu;
    constexpr int PER = kPtMaxN / B;  // spins of a thread
    constexpr int DD = MAXD > 0 ? MAXD : 1, DP = (DD + 1) / 2;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, cap_n = P->cap_n;
    constexpr uint32_t TWO = 0x00010001u;
    const int q0 = base >> 1, nqk = ((end + 1) >> 1) - q0;
    const uint32_t all = (1u << nqk) - 1u;
    const uint32_t valid = (all & ~(uint32_t)(base & 1)) | (all & ~((uint32_t)(end & 1) << (nqk - 1))) << 16;
    const uint32_t n4 = 4u * (uint32_t)n, sw4 = shared_addr(sw) + (uint32_t)q0 * n4;
    const uint32_t *__restrict__ g_meta = P->meta;
    const uint32_t *__restrict__ g_ell = P->ell;
    // D by position, and in index order (where the seeds are counted out)
    for (int p = tid; p < n; p += B) {
        uint32_t d = 0, a = sw4 + 4u * (uint32_t)p;
        for (int q = 0; q < nqk; ++q, a += n4) {
            const uint32_t w = lds(a);
            d |= ((w ^ (w >> 8)) & TWO) << q;
        }
        d &= valid;
        Dm[p] = d;
        Cm[__ldg(P->idx_of_pos + p)] = d;
    }
    if (tid < 32) {
        s_sum[tid] = 0;
        s_seed[tid] = -1;
    }
    __syncthreads();
    // seeds, a warp per temperature: element floor(u |D| / 2^32) of D in index order
    for (int k = base + warp; k < end; k += B / 32) {
        // lane l keeps the ballots of spins 32 l .. and 32 (l + 32) ..
        const int sh = 16 * (k & 1) + (k >> 1) - q0, words = (n + 31) >> 5;
        uint32_t d0 = 0, d1 = 0;
#pragma unroll 4
        for (int it = 0; it < words; ++it) {
            const int i = 32 * it + lane;
            const uint32_t bal = __ballot_sync(0xFFFFFFFFu, i < n && ((Cm[i] >> sh) & 1u));
            if (lane == (it & 31)) {
                if (it < 32) d0 = bal;
                else d1 = bal;
            }
        }
        const int c0 = __popc(d0), c1 = __popc(d1);
        const int n0 = __reduce_add_sync(0xFFFFFFFFu, c0), cnt = n0 + __reduce_add_sync(0xFFFFFFFFu, c1);
        if (cnt == 0) continue;
        const uint32_t u = word0(0xFFFF0000u | (uint32_t)k, y, start, k0, k1);
        int pick = (int)(((uint64_t)u * (uint64_t)cnt) >> 32);
        const bool second = pick >= n0;
        if (second) pick -= n0;
        const uint32_t mine = second ? d1 : d0;
        int before = second ? c1 : c0;
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xFFFFFFFFu, before, o);
            if (lane >= o) before += t;
        }
        before -= second ? c1 : c0;
        if (pick >= before && pick < before + __popc(mine)) {
            uint32_t m = mine;
            for (int j = pick - before; j > 0; --j) m &= m - 1u;
            s_seed[sh] = P->pos_of_idx[32 * (lane + (second ? 32 : 0)) + __ffs(m) - 1];
        }
    }
    __syncthreads();
    for (int p = tid; p < n; p += B) Cm[p] = 0u;
    __syncthreads();
    if (tid < 32 && s_seed[tid] >= 0) atomicOr(&Cm[s_seed[tid]], 1u << tid);
    // this thread's spins: D and (degree <= 8) the neighbours' byte offsets, two a register, kept over the rounds
    uint32_t dd[PER], nb[PER][DP];
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const int p = tid + i * B;
        dd[i] = p < n ? Dm[p] : 0u;
        if (MAXD > 0) {
#pragma unroll
            for (int j = 0; j < DP; ++j) nb[i][j] = 4u * (uint32_t)p * 0x00010001u;
            if (dd[i]) {
                const int deg = (int)(__ldg(g_meta + p) & 0xFFFFu);
#pragma unroll
                for (int d = 0; d < DD; ++d)
                    if (d < deg) {
                        const uint32_t e = 4u * (__ldg(g_ell + (size_t)d * cap_n + p) & 0xFFFFu);
                        nb[i][d / 2] = (d & 1) ? (nb[i][d / 2] & 0xFFFFu) | (e << 16) : (nb[i][d / 2] & 0xFFFF0000u) | e;
                    }
            }
        }
    }
    __syncthreads();
    // growth: values only gain bits, so a read that misses another thread's write is made good
    // in a later round; a round that changes nothing anywhere has read settled values
    const uint32_t c4 = shared_addr(Cm);
    for (;;) {
        bool changed = false;
#pragma unroll
        for (int rep = 0; rep < 2; ++rep)
#pragma unroll
            for (int i = 0; i < PER; ++i) {
                const int p = tid + i * B;
                if (dd[i]) {
                    const uint32_t c = lds(c4 + 4u * (uint32_t)p);
                    if (dd[i] & ~c) {
                        uint32_t any = 0;
                        if (MAXD > 0) {
#pragma unroll
                            for (int j = 0; j < DP; ++j) any |= lds(c4 + (nb[i][j] & 0xFFFFu)) | lds(c4 + (nb[i][j] >> 16));
                        } else {
                            const int deg = (int)(__ldg(g_meta + p) & 0xFFFFu);
                            for (int d = 0; d < deg; ++d) any |= lds(c4 + 4u * (__ldg(g_ell + (size_t)d * cap_n + p) & 0xFFFFu));
                        }
                        if (dd[i] & any & ~c) {
                            sts(c4 + 4u * (uint32_t)p, c | (dd[i] & any));
                            changed = true;
                        }
                    }
                }
            }
        if (!__syncthreads_or(changed)) break;
    }
    // boundary sums, 32 spins a warp: h_i - sum_j J_ij + sum_j J_ij (b^a_j + b^b_j), times s^a_i.
    // Byte lanes (dmax <= 254): sum_j J_ij b_j plus K = sum of |J_ij| over J_ij < 0 is in 0 .. 127 of each
    // copy's byte, so one multiply-add per neighbour serves both copies of both temperatures
    for (int p0 = 32 * warp; p0 < n; p0 += B) {
        const int p = p0 + lane;
        const uint32_t c = p < n ? Cm[p] : 0u;
        if (!__any_sync(0xFFFFFFFFu, c != 0u)) continue;
        int deg = 0, f0 = 0, K = 0, J[DD];
        uint32_t off[DD];
        if (c) {
            const uint32_t meta = __ldg(g_meta + p);
            deg = (int)(meta & 0xFFFFu);
            f0 = (int)meta >> 16;
        }
        const uint32_t own4 = sw4 + 4u * (uint32_t)(p < n ? p : 0);
#pragma unroll
        for (int d = 0; d < DD; ++d) {
            off[d] = own4;
            J[d] = 0;
            if (MAXD > 0 && d < deg) {
                const uint32_t e = __ldg(g_ell + (size_t)d * cap_n + p);
                off[d] = sw4 + 4u * (e & 0xFFFFu);
                J[d] = (int)e >> 16;
                f0 -= J[d];
                if (J[d] < 0) K -= J[d];
            }
        }
        if (MAXD == 0)
            for (int d = 0; d < deg; ++d) f0 -= (int)__ldg(g_ell + (size_t)d * cap_n + p) >> 16;
        f0 -= 2 * K;
        for (int q = 0; q < nqk; ++q) {
            const uint32_t two = (c >> q) & TWO, at = (uint32_t)q * n4;
            if (!__any_sync(0xFFFFFFFFu, two != 0u)) continue;
            int v0, v1;
            const uint32_t own = lds(own4 + at);
            if (MAXD > 0) {
                uint32_t x = (uint32_t)K * 0x01010101u;
#pragma unroll
                for (int d = 0; d < DD; ++d) x += (uint32_t)J[d] * lds(off[d] + at);
                x = (x & H) + ((x >> 8) & H);
                v0 = f0 + (int)(x & 0xFFFFu);
                v1 = f0 + (int)(x >> 16);
            } else {
                uint32_t x = (uint32_t)(32768 + f0) * 0x00010001u;
                if (two)
                    for (int d = 0; d < deg; ++d) {
                        const uint32_t e = __ldg(g_ell + (size_t)d * cap_n + p), w = lds(sw4 + at + 4u * (e & 0xFFFFu));
                        x += (uint32_t)((int)e >> 16) * ((w & H) + ((w >> 8) & H));
                    }
                v0 = (int)(x & 0xFFFFu) - 32768;
                v1 = (int)(x >> 16) - 32768;
            }
            v0 = (own & 1u) ? v0 : -v0;
            v1 = ((own >> 16) & 1u) ? v1 : -v1;
            v0 = __reduce_add_sync(0xFFFFFFFFu, (two & 1u) ? v0 : 0);
            v1 = __reduce_add_sync(0xFFFFFFFFu, (two >> 16) ? v1 : 0);
            if (lane < 2) atomicAdd(&s_sum[q + 16 * lane], lane ? v1 : v0);
        }
    }
    __syncthreads();
    // both copies flip on the cluster
    for (int p = tid; p < n; p += B) {
        const uint32_t c = Cm[p];
        uint32_t a = sw4 + 4u * (uint32_t)p;
        if (c)
            for (int q = 0; q < nqk; ++q, a += n4) sts(a, lds(a) ^ (((c >> q) & TWO) * 0x0101u));
    }
    if (tid < 32 && (valid >> tid) & 1u) {
        const int k = 2 * (q0 + (tid & 15)) + (tid >> 4);
        sE[2 * k] -= 2 * s_sum[tid];
        sE[2 * k + 1] += 2 * s_sum[tid];
    }
    __syncthreads();
}

template <int B, int MAXD, bool SMALL>
__global__ void __launch_bounds__(B, 2) k_pticm(const PticmArgs A)
{
    extern __shared__ __align__(256) unsigned char smem_pt[];
    __shared__ int sE[2 * kPtMaxR], sAcc[2 * kPtMaxR];
    __shared__ int4 s_cls[kMaxColours];
    __shared__ uint4 s_qt[kPtMaxR / 2];
    __shared__ uint32_t sPack[B / 32][kPtWarpWords];
    __shared__ int32_t s_nk[2 * kPtMaxR];  // slot mode: the kept lists' lengths
    __shared__ int s_seed[32], s_sum[32];  // cluster moves: seeds and boundary sums by temperature

    const int run = blockIdx.x;
    Slot *slot = A.slots ? A.slots + run : nullptr;
    if (slot && slot->mode == kDone) return;  // the whole CTA: a finished start
    const DevProb *P = slot ? slot->cur : A.prob;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n = P->n, ncol = P->ncol, bias = P->dmax >> 1;
    const int R = A.R, NR = 2 * R, T = A.T, nq = (NR + 3) >> 2;
    const int nic = R - A.icm_from;            // temperatures with cluster moves
    const int ntr = 2 * (R - A.keep_from);     // tracked replicas
    const int W = (n + 31) >> 5;
    const uint64_t seed = slot ? slot->seed : A.seed;
    const uint32_t start = slot ? slot->start : A.start0 + (uint32_t)run;
    const uint32_t phase = slot ? (uint32_t)slot->phase : A.phase;
    const uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32);
    const uint32_t k0w = k0 + kPhiloxW0, k1w = k1 + kPhiloxW1;
    const uint32_t phase_hi = phase << kSweepBits;
    // kept lists: list q, entry j at kept_rows + (q K + j) kstride words, energy kept_en[q K + j], length nk[q]
    const size_t kstride = slot ? (size_t)slot->W0 : (size_t)W;
    uint32_t *kept_rows = slot ? slot->spins : A.kept + (size_t)run * ntr * A.K * W;
    int64_t *kept_en = slot ? slot->rec_e + (size_t)slot->phase * A.Smax : A.kept_e + (size_t)run * ntr * A.K;
    int32_t *nk = slot ? s_nk : A.nkept + (size_t)run * ntr;
    if (slot)
        for (int q = tid; q < ntr; q += B) s_nk[q] = 0;
    constexpr int NW = B / 32;

    // acceptance rows, the cluster moves' masks, the quads' words
    constexpr int ROW = 64;                                      // SMALL: words of a row
    uint32_t *rows_s = reinterpret_cast<uint32_t *>(smem_pt);    // [R][ROW] or [R][bias]
    uint32_t *Cm = rows_s + (SMALL ? R * ROW : ((R * bias + 3) & ~3) + kPtRowPad), *Dm = Cm + n;  // [n] each
    uint32_t *sw = Dm + n;                                       // [nq][n]

    for (int c = tid; c < ncol; c += B) {
        // quad groups of a class: the choice that takes the block's warps the least, a unit's set-up counted
        // as half a quad
        const int lo = P->cptr[c], nc = P->cptr[c + 1] - lo, chunks = (nc + 31) >> 5;
        int best = 0x7FFFFFFF, G = 1, rounds = 0;
        for (int g = 1; g <= nq; ++g) {
            const int rr = (chunks * g + NW - 1) / NW, cost = rr * (2 * ((nq + g - 1) / g) + 1);
            if (cost < best) {
                best = cost;
                G = g;
                rounds = rr;
            }
        }
        s_cls[c] = make_int4(lo, nc, G, rounds);
    }
    // row k: the threshold of dE = 2e in word e - 1 (SMALL: word e + 31; the rest of the row is read and ignored)
    for (int x = tid; x < R * bias; x += B) {
        const int k = x / bias, e = x - k * bias + 1;
        rows_s[SMALL ? k * ROW + e + 31 : x] = A.thr[(size_t)k * A.thr_stride + 2 * e];
    }
    // initial states: the SA initial-state words of replica r
    for (int x = tid; x < nq * n; x += B) {
        const int q = x / n, p = x - q * n;
        const uint4 w = philox4x32_10(make_uint4((uint32_t)P->idx_of_pos[p], phase_hi | kInitSlot, (uint32_t)q, start),
                                      k0, k1);
        uint32_t b = (w.x >> 31) | (w.y >> 31) << 8;
        if (4 * q + 2 < NR) b |= (w.z >> 31) << 16 | (w.w >> 31) << 24;
        sw[x] = b;
    }
    for (int v = tid; v < nq; v += B) {
        uint32_t h1, l1;
        philox_mulhilo(kPhiloxM1, (uint32_t)v, h1, l1);
        uint4 q = make_uint4(l1 ^ k0w, 0u, 0u, h1 ^ k0);
        philox_mulhilo(kPhiloxM0, q.w ^ phase_hi, q.y, q.z);
        s_qt[v] = q;
    }
    __syncthreads();
    replica_energies<B>(P, sw, NR, sE);

    PhiloxKeys<2> K = philox_keys<2>(k0, k1);
    // opaque to the compiler, which would otherwise recompute them for every quad
#pragma unroll
    for (int i = 0; i < 8; ++i) asm("" : "+r"(K.k0[i]), "+r"(K.k1[i]));
    for (int t = 0; t < T; ++t) {
        const uint32_t y = phase_hi | (uint32_t)t;
        // 1. Metropolis sweep of every replica, colour class by colour class
        metropolis<B, MAXD, SMALL>(P, sw, rows_s, n, ncol, nq, R, NR, bias, s_cls, s_qt, sE, start ^ k1, k1w, K);
        // the next sweep's quad products (every later step of this sweep ends in a barrier)
        if (tid < nq) {
            uint4 q = s_qt[tid];
            philox_mulhilo(kPhiloxM0, q.w ^ (y + 1u), q.y, q.z);
            s_qt[tid] = q;
        }
        // 2. cluster moves at the lower temperatures, up to 32 at a time
        if ((A.flags & 2) && nic > 0) {
            for (int base = A.icm_from, end; base < R; base = end) {
                end = min(R, (base & ~1) + 32);
                cluster_moves<B, MAXD>(P, sw, Dm, Cm, n, base, end, y, start, k0, k1, s_seed, s_sum, sE);
            }
        }
        // 3. replica exchange between temperatures k and k + 1, k = t (mod 2)
        if (A.flags & 1) {
            const int odd = t & 1, npair = max((R - 1 - odd + 1) / 2, 0);  // k = odd, odd + 2, ... < R - 1
            bool any = false;
            for (int z = tid; z < 2 * npair; z += B) {
                const int k = odd + 2 * (z >> 1), c = z & 1;
                const int lo = 2 * k + c, hi = lo + 2;
                const int d = sE[lo] - sE[hi];
                const uint32_t u = word0(0xFFFE0000u | (uint32_t)lo, y, start, k0, k1);
                const bool acc = d <= 0 || u < A.xthr[(size_t)k * (A.dx + 1) + min(d, A.dx)];
                sAcc[z] = acc;
                if (acc) {
                    const int e = sE[lo];
                    sE[lo] = sE[hi];
                    sE[hi] = e;
                    any = true;
                }
            }
            if (__syncthreads_or(any)) {
                if (!odd) {
                    // pairs inside a quad: bytes c and c + 2
                    for (int q = 0; q < npair; ++q) {
                        const uint32_t sel = 0x3210u ^ (sAcc[2 * q] ? 0x0202u : 0u) ^ (sAcc[2 * q + 1] ? 0x2020u : 0u);
                        if (sel == 0x3210u) continue;
                        for (int p = tid; p < n; p += B) sw[q * n + p] = __byte_perm(sw[q * n + p], 0u, sel);
                    }
                } else {
                    // bytes 2, 3 of quad q and 0, 1 of quad q + 1: a thread takes a spin through every quad
                    for (int p = tid; p < n; p += B) {
                        uint32_t cur = sw[p], from = 0u, take = 0u;  // bytes 0, 1 of the next word and which of them
                        for (int q = 0; q < nq; ++q) {
                            const uint32_t nxt = q + 1 < nq ? sw[(size_t)(q + 1) * n + p] : 0u;
                            uint32_t m = 0u;
                            if (q < npair) m = (sAcc[2 * q] ? 0xFFu : 0u) | (sAcc[2 * q + 1] ? 0xFF00u : 0u);
                            uint32_t w = (cur & ~take) | (from & take);
                            w = (w & ~(m << 16)) | ((nxt & m) << 16);
                            sw[(size_t)q * n + p] = w;
                            from = cur >> 16;
                            take = m;
                            cur = nxt;
                        }
                    }
                }
                __syncthreads();
            }
        }
        // 4. each tracked replica's list of the K lowest distinct states seen
        for (int q = warp; q < ntr; q += NW) {
            const int r = 2 * (A.keep_from + q / 2) + (q & 1);
            const int64_t E = (int64_t)sE[r] + P->offset;
            int32_t *cntp = nk + q;
            int64_t *le = kept_en + (size_t)q * A.K;
            uint32_t *lst = kept_rows + (size_t)q * A.K * kstride;
            const int cnt = *cntp;
            if (cnt == A.K && E >= le[A.K - 1]) continue;
            // the list's energies, two a lane: entries not above E come before the state
            const int64_t l0 = lane < cnt ? le[lane] : LLONG_MAX, l1 = lane + 32 < cnt ? le[lane + 32] : LLONG_MAX;
            const uint32_t same0 = __ballot_sync(0xFFFFFFFFu, lane < cnt && l0 == E);
            const uint32_t same1 = __ballot_sync(0xFFFFFFFFu, lane + 32 < cnt && l1 == E);
            const int pos = __popc(__ballot_sync(0xFFFFFFFFu, lane < cnt && l0 <= E)) +
                            __popc(__ballot_sync(0xFFFFFFFFu, lane + 32 < cnt && l1 <= E));
            // the state, bit-packed in index order
            const uint32_t *s = sw + (size_t)(r >> 2) * n;
            const int sh = 8 * (r & 3);
#pragma unroll 4
            for (int w = 0; w < W; ++w) {
                const int i = 32 * w + lane;
                const bool b = i < n && ((s[__ldg(P->pos_of_idx + i)] >> sh) & 1u);
                const uint32_t bits = __ballot_sync(0xFFFFFFFFu, b);
                if (lane == 0) sPack[warp][w] = bits;
            }
            __syncwarp();
            bool dup = false;
            for (uint64_t m = (uint64_t)same1 << 32 | same0; m && !dup; m &= m - 1) {
                const int j = __ffsll((long long)m) - 1;
                bool diff = false;
                for (int w = lane; w < W; w += 32) diff |= lst[(size_t)j * kstride + w] != sPack[warp][w];
                dup = !__any_sync(0xFFFFFFFFu, diff);
            }
            if (dup) continue;
            const int last = cnt < A.K ? cnt : A.K - 1;
            // entries pos .. last - 1 move down one place: a lane moves its own words, four rows in flight
            for (int w = lane; w < W; w += 32) {
                int j = last;
                for (; j - 4 >= pos; j -= 4) {
                    uint32_t x[4];
#pragma unroll
                    for (int d = 0; d < 4; ++d) x[d] = lst[(size_t)(j - 1 - d) * kstride + w];
#pragma unroll
                    for (int d = 0; d < 4; ++d) lst[(size_t)(j - d) * kstride + w] = x[d];
                }
                for (; j > pos; --j) lst[(size_t)j * kstride + w] = lst[(size_t)(j - 1) * kstride + w];
                lst[(size_t)pos * kstride + w] = sPack[warp][w];
            }
            if (lane >= pos && lane < last) le[lane + 1] = l0;
            if (lane + 32 >= pos && lane + 32 < last) le[lane + 33] = l1;
            __syncwarp();
            if (lane == 0) {
                le[pos] = E;
                if (cnt < A.K) *cntp = cnt + 1;
            }
            __syncwarp();
        }
        __syncthreads();
    }
    if (slot) {
        // the phase's sample: the lists one after another.  List q moves down by
        // q K - (entries before it); rows are copied in waves of that distance, so
        // a wave never overwrites a row a later wave still reads
        int before = 0;
        for (int q = 0; q < ntr; ++q) {
            const int len = s_nk[q], shift = q * A.K - before;
            if (shift > 0)
                for (int j0 = 0; j0 < len; j0 += shift) {
                    const int jn = min(len, j0 + shift);
                    for (int x = tid; x < (jn - j0) * W; x += B) {
                        const int j = j0 + x / W, w = x - (x / W) * W;
                        kept_rows[(size_t)(before + j) * kstride + w] = kept_rows[(size_t)(q * A.K + j) * kstride + w];
                    }
                    for (int j = j0 + tid; j < jn; j += B) kept_en[before + j] = kept_en[q * A.K + j];
                    __syncthreads();
                }
            before += len;
        }
        if (tid == 0) slot->rec_count[slot->phase] = before;
        return;
    }
    // final states and energies of every replica
    for (int r = warp; r < NR; r += B / 32) {
        for (int w = 0; w < W; ++w) {
            const int i = 32 * w + lane;
            const bool b = i < n && ((sw[(size_t)(r >> 2) * n + P->pos_of_idx[i]] >> (8 * (r & 3))) & 1u);
            const uint32_t bits = __ballot_sync(0xFFFFFFFFu, b);
            if (lane == 0) A.final_bits[((size_t)run * NR + r) * W + w] = bits;
        }
        if (lane == 0) A.final_e[(size_t)run * NR + r] = (int64_t)sE[r] + P->offset;
    }
}

// Kernel of problems of at most maxdeg neighbours a spin and flip costs up to dmax.
bool pticm_small(int maxdeg, int dmax) { return dmax <= 62 && maxdeg <= 8; }
void *select_pticm(int maxdeg, int dmax)
{
    if (pticm_small(maxdeg, dmax))
        return maxdeg <= 6 ? reinterpret_cast<void *>(k_pticm<kPtBlock, 6, true>)
                           : reinterpret_cast<void *>(k_pticm<kPtBlock, 8, true>);
    if (dmax <= 254 && maxdeg <= 6) return reinterpret_cast<void *>(k_pticm<kPtBlock, 6, false>);
    if (dmax <= 254 && maxdeg <= 8) return reinterpret_cast<void *>(k_pticm<kPtBlock, 8, false>);
    return reinterpret_cast<void *>(k_pticm<kPtBlock, 0, false>);
}

}  // namespace

// The documented limit: 2Rn + 4R(dmax + 1) + 32n bytes fit a CTA.
size_t pticm_limit_bytes(int n, int R, int dmax)
{
    const size_t spins = (2 * (size_t)R * n + 15) & ~(size_t)15;
    return spins + 4 * (size_t)R * ((size_t)dmax + 1) + 2 * (size_t)(kPtBlock / 32) * n;
}

// What a launch takes: the rows, two masks per spin, the quads' words.
size_t pticm_smem_bytes(int n, int R, int maxdeg, int dmax)
{
    const size_t rows = pticm_small(maxdeg, dmax) ? 64 * (size_t)R : (((size_t)R * (dmax / 2) + 3) & ~(size_t)3) + kPtRowPad;
    return 4 * (rows + 2 * (size_t)n + (size_t)((2 * R + 3) / 4) * n);
}

int pticm_max_r() { return kPtMaxR; }
int pticm_max_n() { return 32 * kPtWarpWords; }

cudaError_t launch_pticm(const DevProb *prob, int maxdeg, int dmax, const uint32_t *thr, int thr_stride,
                         const uint32_t *xthr, int dx, int R, int T, int icm_from, int keep_from, int K, int flags, uint64_t seed,
                         uint32_t start0, uint32_t phase, int runs, size_t smem, uint32_t *kept, int64_t *kept_e,
                         int32_t *nkept, uint32_t *final_bits, int64_t *final_e, cudaStream_t st)
{
    PticmArgs A;
    A.prob = prob;
    A.thr = thr;
    A.xthr = xthr;
    A.R = R;
    A.T = T;
    A.thr_stride = thr_stride;
    A.dx = dx;
    A.icm_from = icm_from;
    A.keep_from = keep_from;
    A.K = K;
    A.flags = flags;
    A.seed = seed;
    A.start0 = start0;
    A.phase = phase;
    A.kept = kept;
    A.kept_e = kept_e;
    A.nkept = nkept;
    A.final_bits = final_bits;
    A.final_e = final_e;
    A.slots = nullptr;
    A.Smax = 0;
    void *k = select_pticm(maxdeg, dmax);
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    void *args[] = {&A};
    return cudaLaunchKernel(k, dim3(runs), dim3(kPtBlock), args, smem, st);
}

}  // namespace spvar

namespace spvar {

cudaError_t launch_pticm_slots(Slot *slots, int nslots, int Smax, int maxdeg, int dmax,
                               const uint32_t *thr, int thr_stride, const uint32_t *xthr, int dx, int R, int T, int K, size_t smem, cudaStream_t st)
{
    if (nslots <= 0) return cudaSuccess;
    PticmArgs A;
    std::memset(&A, 0, sizeof(A));
    A.thr = thr;
    A.xthr = xthr;
    A.R = R;
    A.T = T;
    A.thr_stride = thr_stride;
    A.dx = dx;
    A.icm_from = R / 2;
    A.keep_from = R / 2;
    A.K = K;
    A.flags = 3;
    A.slots = slots;
    A.Smax = Smax;
    void *k = select_pticm(maxdeg, dmax);
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    void *args[] = {&A};
    return cudaLaunchKernel(k, dim3(nslots), dim3(kPtBlock), args, smem, st);
}

}  // namespace spvar
