// Quad-group simulated-annealing sweep for +-1 couplers (the sampler of
// Sec. III.A): one work item is nq quads (4 nq replicas) of one start's
// problem, any n that fits shared memory.
//
// Same dynamics, random words and result as the other sweep kernels.  Two
// quads share a spin word ("pair"): replica r of the even quad is bit 8r, of the
// odd quad bit 8r + 4, so a neighbour sum of at most 8 couplers fits its nibble
// and one load, one add and one store serve eight replicas; a group is one or two
// pairs moved by one vector load.  Shared memory holds, per group, a plain copy
// and a copy with every replica bit inverted (word n of each is zero, the target
// of missing neighbours), and a record per spin (neighbour byte offsets with the
// inverted copy folded in for J < 0, index, flip-cost constant), so a thread has a
// spin set up in about 30 instructions and then sweeps it in every group of its
// unit; units left over for a last partial round of the block are split over more
// threads (class_split).  The Philox products that depend only on the quad and the
// sweep stand beside the group's words, refreshed once per sweep, so an item pays
// 16 wide multiplies.
//
// Bound: the integer pipes.  A pair takes about 145 instructions, 32 of them wide
// multiplies.  Timed in isolation (8 warps per scheduler), a wide multiply costs 2.5
// cycles beside three-input logic at 2 cycles each, not in its shadow, so the ALU's
// instructions and the multiplies add up: what helps is fewer instructions (round
// keys kept in registers, the row's address merged by the byte permute that extracts
// the index, one comparison per replica).  3D +-J batch, 64 problems of L = 6 .. 12,
// 2000 + 2000 samples, 1000 sweeps: 271 ms with one quad per word and no records,
// 175 ms now (1.2e12 attempts/s).  Two pairs a group need more than the 64 registers
// of two 512-thread blocks an SM: those forms spill 20 to 72 bytes (the batch's 32).
// Eligible when every |J| = 1, degree <= MAXD <= 8 and dmax <= 30.
#include "quad_units.cuh"

namespace spvar {

namespace {

constexpr int kQcap = 64;           // most quads per work item
constexpr int kPcap = kQcap / 2;    // most pairs
constexpr size_t kQuadRoom = 7 << 10;       // left beside a CTA's dynamic part where a default shape is chosen
constexpr size_t kQuadSmemMax = 218 << 10;  // dynamic shared memory records may bring a CTA to
constexpr uint32_t kM = 0x01010101u, kN = 0x11111111u, kOdd = 0x10101010u;

// NV words (one of every pair of a group) at once.
template <int NV>
__device__ __forceinline__ void lds_nv(uint32_t a, uint32_t (&v)[NV])
{
    if constexpr (NV == 1) {
        v[0] = lds(a);
    } else {
        const uint2 x = lds2(a);
        v[0] = x.x;
        v[1] = x.y;
    }
}
template <int NV>
__device__ __forceinline__ void sts_nv(uint32_t a, const uint32_t (&v)[NV])
{
    if constexpr (NV == 1) {
        sts(a, v[0]);
    } else {
        sts2(a, make_uint2(v[0], v[1]));
    }
}

// Degree <= 6: with z = x + 8 b_i (x < 8 the neighbour bits, b_i the spin's bit) and the
// spin's constant c8 = 15 + h - deg a second table gives the largest random word that is
// accepted, thr - 1, or 2^32 - 1 where the cost is not positive: word
// (c8 / 4) * 64 + 4 z + c8 % 4, so a nibble of z in the high half of a byte is already
// the entry's byte offset in its 256-byte block.  One comparison accepts; the table
// cannot hold thr = 0 (never accept), so sweeps whose row has one (large beta) use the
// first form.  So do launches without the table: degree 7 and 8, and a lone pair of a
// problem whose spin words leave no room for its 4 KB.
constexpr int kTabWords = 8 * 64;

// Acceptance rows of the current and the next sweep: the threshold of flip cost
// dE = 2e is the 32-bit word at byte 8e + 120, so the byte of a replica's index is
// the address and its top bit says dE > 0 (a cost that is not positive reads a word
// that is ignored).  Costs |e| <= 7, all a +-1 problem without large biases has, lie
// on different banks.  Rows are 256-byte aligned: the index byte replaces the low byte
// of the row's address.
template <bool TABS>
struct QuadSmem {
    uint32_t row[2][64];
    uint32_t tab[TABS ? 2 : 1][TABS ? kTabWords : 4];
    int zero[2];                 // the row holds a threshold of 0
    int c8lo, c8hi;              // range of the problem's flip-cost constants
    int e2[4 * kQcap];
    int4 cls[kMaxColours];  // per colour class, as unit_classes fills it
    int item;               // the queue's next work item
};
constexpr size_t quad_static(bool tabs) { return tabs ? sizeof(QuadSmem<true>) : sizeof(QuadSmem<false>); }
// a CTA takes 1 KB of the system's beside its own; an SM has 1 KB more than one CTA may take
static_assert(2 * (quad_static(true) + 1024) <= 2 * kQuadRoom + 1024, "two CTAs of a default shape share an SM");
static_assert(kQuadSmemMax + quad_static(true) <= kSmemOptin, "records and the static part fit a CTA");

// One quad's four acceptance tests: adds 1 << (8r + SH) to rej for every replica r whose
// word is not below its threshold.
template <int SH>
__device__ __forceinline__ void reject4(uint32_t &rej, uint32_t row, uint32_t idx, uint4 u)
{
    const uint32_t ur[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const uint32_t thr = lds(__byte_perm(idx, row, 0x7650u | (uint32_t)r));
        asm("{ .reg .pred p; setp.ge.u32 p, %1, %2; @p add.u32 %0, %0, %3; }"
            : "+r"(rej)
            : "r"(ur[r]), "r"(thr), "r"(1u << (8 * r + SH)));
    }
}

// The same from the second table: adds 1 << (8r + SH) to acc for every replica accepted.
template <int SH>
__device__ __forceinline__ void accept4(uint32_t &acc, uint32_t block, uint32_t idx, uint4 u)
{
    const uint32_t ur[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const uint32_t top = lds(__byte_perm(idx, block, 0x7650u | (uint32_t)r));
        asm("{ .reg .pred p; setp.le.u32 p, %1, %2; @p add.u32 %0, %0, %3; }"
            : "+r"(acc)
            : "r"(ur[r]), "r"(top), "r"(1u << (8 * r + SH)));
    }
}

// Entry (c8, z) of the second table for the threshold row thr (null entries of a
// problem's range are never read).
__device__ __forceinline__ uint32_t top_word(const uint32_t *__restrict__ thr, int c8, int z, int bias)
{
    int e = 2 * (z & 7) + c8 - 15;
    if (z & 8) e = -e;
    return (e <= 0 || e > bias) ? 0xFFFFFFFFu : thr[2 * e] - 1u;
}
__device__ __forceinline__ int tab_word(int c8, int z) { return (c8 >> 2) * 64 + 4 * z + (c8 & 3); }

// Final energies and bit-packed states of the item's replicas.
template <int NV>
__device__ __forceinline__ void finish_pairs(const DevProb *P, const SweepJob &job, int quad0, int nq,
                                             const uint32_t *sw, int *e2)
{
    const int tid = threadIdx.x, B = blockDim.x, lane = tid & 31, warp = tid >> 5;
    const int n = P->n, gw = group_words(n, NV), cap_n = P->cap_n;
    for (int x = tid; x < 4 * nq; x += B) e2[x] = 0;
    __syncthreads();
    for (int v = 0; 2 * v < nq; ++v) {
        const uint32_t *s = sw + (size_t)(v / NV) * gw + v % NV;
        int acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        for (int p = tid; p < n; p += B) {
            const uint32_t own = s[p * NV], meta = P->meta[p];
            const int deg = (int)(meta & 0xFFFFu), h2 = 2 * ((int)meta >> 16);
            uint32_t sat = 0;  // per nibble: satisfied bonds
            for (int d = 0; d < deg; ++d) {
                const uint32_t e = P->ell[(size_t)d * cap_n + p];
                sat += own ^ s[(e & 0xFFFFu) * NV] ^ ((e >> 31) ? kN : 0u);
            }
#pragma unroll
            for (int k = 0; k < 8; ++k)
                acc[k] += deg - 2 * (int)((sat >> (4 * k)) & 15u) + (((own >> (4 * k)) & 1u) ? h2 : -h2);
        }
        // nibble k: quad 2v + (k & 1), replica k >> 1
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int t = __reduce_add_sync(0xFFFFFFFFu, acc[k]);
            if (lane == 0 && 2 * v + (k & 1) < nq) atomicAdd(&e2[4 * (2 * v + (k & 1)) + (k >> 1)], t);
        }
    }
    __syncthreads();
    for (int x = tid; x < 4 * nq; x += B) {
        const int r = 4 * quad0 + x;
        if (r < job.S) job.energies[r] = (int64_t)(e2[x] / 2) + P->offset;
    }
    const int Wn = (n + 31) >> 5, np = (nq + 1) >> 1;
    for (int x = warp; x < np * Wn; x += B / 32) {
        const int v = x / Wn, w = x - v * Wn;
        const int i = 32 * w + lane;
        const uint32_t word = (i < n) ? sw[(size_t)(v / NV) * gw + P->pos_of_idx[i] * NV + v % NV] : 0u;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const uint32_t bits = __ballot_sync(0xFFFFFFFFu, (word >> (4 * k)) & 1u);
            const int q = 2 * v + (k & 1), r = 4 * (quad0 + q) + (k >> 1);
            if (lane == 0 && q < nq && r < job.S) job.spins[(size_t)r * job.W + w] = bits;
        }
    }
}

// What a sweep needs of its work item.  Bytes of shared memory: sw4 the address of the
// first pair's spin words, v4 from pair to pair, ns4 from a plain to its inverted copy.
struct QuadItem {
    uint32_t end4, v4, ns4, sw4;
    int np, n, ncol, bias, cap_n;
    bool both;  // false: an item of one quad, whose odd half is not swept
    uint32_t sk1, k1w;
    const uint32_t *meta, *ell;
    const int32_t *idx;
};

// One sweep, on acceptance row PAR (the sweep's parity: its row is at a compile-time
// address); y1 is the next sweep's counter word and next_thr its threshold row (null
// after the last sweep).
template <int B, int MAXD, int NV, bool STAGED, int PAR, bool TAB, bool TABS>
__device__ __forceinline__ void sweep_pairs(const QuadItem &I, QuadSmem<TABS> &sm, uint32_t *pairs, const uint4 *rec,
                                            const uint32_t *rec2, const uint32_t *unit, uint32_t y1,
                                            const uint32_t *__restrict__ next_thr, const PhiloxKeys<2> &K)
{
    const int tid = threadIdx.x;
    // next sweep's row and quad products (their buffers were last read in the previous sweep)
    const int tabs = 16 * (sm.c8hi - sm.c8lo + 1);  // entries of the second table in use
    uint32_t top = 0u;
    if (next_thr) {
        if (tid < 32) {
            const uint32_t v = tid < I.bias ? next_thr[2 * (tid + 1)] : 1u;
            if (tid < I.bias) sm.row[PAR ^ 1][2 * (tid + 1) + 30] = v;
            const bool zero = __any_sync(0xFFFFFFFFu, v == 0u);
            if (tid == 0) sm.zero[PAR ^ 1] = zero;
        }
        // loaded here, stored after the first class
        if (TABS && tid < tabs) top = top_word(next_thr, sm.c8lo + (tid >> 4), tid & 15, I.bias);
        if (tid < I.np) {
            uint4 *head = reinterpret_cast<uint4 *>(pairs + (size_t)(tid / NV) * (I.v4 / 4)) + tid % NV;
            const uint4 h = head[2 * NV];
            uint4 q;
            philox_mulhilo(kPhiloxM0, h.z ^ y1, q.x, q.y);
            philox_mulhilo(kPhiloxM0, h.w ^ y1, q.z, q.w);
            head[(PAR ^ 1) * NV] = q;
        }
    }
    const uint32_t row = shared_addr(TAB ? sm.tab[TABS ? PAR : 0] : sm.row[PAR]);
    const uint32_t first = I.sw4, last = I.sw4 + I.end4;
    for (int c = 0; c < I.ncol; ++c) {
        const int4 cl = sm.cls[c];
#pragma unroll 1
        for (int r = 0; r < cl.z; ++r) {
            uint32_t p, base, step4;
            if (STAGED && cl.w >= 0) {
                const uint32_t d = unit[(cl.w + r) * B + tid];
                p = d & 0xFFFFu;
                base = first + ((d >> 16) & 0xFFu) * I.v4;
                step4 = (d >> 24) * I.v4;
            } else {
                const int u = r * B + tid;
                p = (uint32_t)(cl.x + u);
                base = u < cl.y ? first : last;
                step4 = I.v4;
            }
            if (base < last) {
                uint32_t o4[MAXD], idx;
                int c8;
                if (STAGED) {
                    const uint4 k = rec[p];
                    o4[0] = k.x & 0xFFFFu;
                    o4[1] = k.x >> 16;
                    o4[2] = k.y & 0xFFFFu;
                    o4[3] = k.y >> 16;
                    o4[4] = k.z & 0xFFFFu;
                    o4[5] = k.z >> 16;
                    if constexpr (MAXD > 6) {
                        const uint32_t k2 = rec2[p];
                        o4[6] = k2 & 0xFFFFu;
                        o4[7] = k2 >> 16;
                    }
                    idx = k.w & 0xFFFFu;
                    c8 = (int)(k.w >> 16);
                } else {
                    const uint32_t meta = __ldg(I.meta + p);
                    const int deg = (int)(meta & 0xFFFFu);
#pragma unroll
                    for (int d = 0; d < MAXD; ++d) {
                        uint32_t o = 4u * NV * (uint32_t)I.n;  // missing neighbour: the pair's zero word
                        if (d < deg) {
                            const uint32_t e = __ldg(I.ell + (size_t)d * I.cap_n + p);
                            o = ((e >> 31) ? I.ns4 : 0u) + 4u * NV * (e & 0xFFFFu);
                        }
                        o4[d] = o;
                    }
                    idx = (uint32_t)__ldg(I.idx + p);
                    c8 = 15 + ((int)meta >> 16) - deg;
                }
                // a replica with x neighbour bits b_j ^ [J_ij < 0] set has e = dE/2 = 2x - deg + h for
                // b_i = 0 and minus that for b_i = 1.  With z = x ^ 15 b_i (that is x or 15 - x) the index
                // 8e + 120 is 16 z + c8 (8 - 16 b_i), c8 = 15 + h - deg, for both
                const uint32_t c0 = (uint32_t)(8 * c8) * kM, ce = (uint32_t)(-16 * c8), co = (uint32_t)(-c8);
                const uint32_t block = row + 256u * (uint32_t)(c8 >> 2), sub = 4u * (uint32_t)(c8 & 3) * kM;
                // Philox products of the spin and the start: rounds 1 (word 0) and 2 (word 2)
                uint32_t H0, L0, H2, L2;
                philox_mulhilo(kPhiloxM0, idx, H0, L0);
                philox_mulhilo(kPhiloxM1, H0 ^ I.sk1, H2, L2);
                const uint32_t L0k = L0 ^ I.k1w;
                const uint32_t own4 = 4u * NV * p;
#pragma unroll 1
                do {
                    const uint32_t oa = base + own4;
                    uint32_t own[NV], x[NV], w[NV];
                    lds_nv<NV>(oa, own);
                    lds_nv<NV>(base + o4[0], x);
#pragma unroll
                    for (int d = 1; d < MAXD; ++d) {
                        lds_nv<NV>(base + o4[d], w);
#pragma unroll
                        for (int k = 0; k < NV; ++k) x[k] += w[k];
                    }
                    uint32_t ie[NV], io[NV], inv[NV];
#pragma unroll
                    for (int k = 0; k < NV; ++k) {
                        if (TAB) {
                            const uint32_t z = own[k] * 8u + x[k];
                            ie[k] = ((z * 16u) & 0xF0F0F0F0u) | sub;
                            io[k] = (z & 0xF0F0F0F0u) | sub;
                        } else {
                            const uint32_t z = x[k] ^ (own[k] * 15u);
                            ie[k] = (z & 0x0F0F0F0Fu) * 16u + ((own[k] & kM) * ce + c0);
                            io[k] = (z & 0xF0F0F0F0u) + ((own[k] & kOdd) * co + c0);
                        }
                    }
#pragma unroll
                    for (int k = 0; k < NV; ++k) {
                        const uint4 qs = lds4(base + (16 * (PAR * NV + k) - 4 * kPairHead * NV));
                        const uint2 qk = lds2(base + (16 * (2 * NV + k) - 4 * kPairHead * NV));
                        const uint4 ue = philox_rounds<2>(make_uint4(H2 ^ qk.x, L2, qs.x ^ L0k, qs.y), K);
                        uint32_t hit = 0;
                        if (TAB) accept4<0>(hit, block, ie[k], ue);
                        else reject4<0>(hit, row, ie[k], ue);
                        if (NV > 1 || I.both) {
                            const uint4 uo = philox_rounds<2>(make_uint4(H2 ^ qk.y, L2, qs.z ^ L0k, qs.w), K);
                            if (TAB) accept4<4>(hit, block, io[k], uo);
                            else reject4<4>(hit, row, io[k], uo);
                        }
                        if (TAB) {
                            inv[k] = own[k] ^ hit ^ kN;
                        } else {
                            // flip where not rejected (a cost that is not positive never is)
                            const uint32_t up = ((ie[k] >> 7) & ~kOdd) | ((io[k] >> 3) & kOdd);
                            inv[k] = own[k] ^ (hit & up);  // = new word with every replica bit inverted
                        }
                    }
                    sts_nv<NV>(oa + I.ns4, inv);
#pragma unroll
                    for (int k = 0; k < NV; ++k) inv[k] ^= kN;
                    sts_nv<NV>(oa, inv);
                    base += step4;
                } while (base < last);
            }
        }
        if constexpr (TABS) {
            if (c == 0 && next_thr) {
                if (tid < tabs) sm.tab[PAR ^ 1][tab_word(sm.c8lo + (tid >> 4), tid & 15)] = top;
                for (int i = tid + B; i < tabs; i += B)
                    sm.tab[PAR ^ 1][tab_word(sm.c8lo + (i >> 4), i & 15)] =
                        top_word(next_thr, sm.c8lo + (i >> 4), i & 15, I.bias);
            }
        }
        __syncthreads();
    }
}

// The form the sweep's acceptance row allows.
template <int B, int MAXD, int NV, bool STAGED, int PAR, bool TABS>
__device__ __forceinline__ void sweep_pairs_par(const QuadItem &I, QuadSmem<TABS> &sm, uint32_t *pairs, const uint4 *rec,
                                                const uint32_t *rec2, const uint32_t *unit, uint32_t y1,
                                                const uint32_t *next_thr, const PhiloxKeys<2> &K)
{
    if (TABS && !sm.zero[PAR])
        sweep_pairs<B, MAXD, NV, STAGED, PAR, TABS>(I, sm, pairs, rec, rec2, unit, y1, next_thr, K);
    else
        sweep_pairs<B, MAXD, NV, STAGED, PAR, false>(I, sm, pairs, rec, rec2, unit, y1, next_thr, K);
}

template <int B, int MAXD, int NV, bool STAGED, bool TABS>
__device__ void run_item_pm1q(const SweepLaunch &L, const SweepJob &job, int quad0, int nq, QuadSmem<TABS> &sm,
                              uint32_t *smem)
{
    const int tid = threadIdx.x;
    const DevProb *P = job.prob;
    const int n = P->n, ncol = P->ncol, cap_n = P->cap_n;
    const uint32_t *__restrict__ g_meta = P->meta;
    const uint32_t *__restrict__ g_ell = P->ell;
    const int32_t *__restrict__ g_idx = P->idx_of_pos;
    const int bias = P->dmax >> 1;
    const int ns = n + 1, ng = (nq + 2 * NV - 1) / (2 * NV), np = ng * NV, gw = group_words(n, NV);
    const uint32_t ns4 = 4u * NV * (uint32_t)ns, v4 = 4u * (uint32_t)gw;  // bytes to the inverted copy / next group
    const int T = job_end(L, job), t0 = job.t0;
    // the seed's words from one lane: the compiler keeps the round keys in uniform registers
    const uint32_t k0 = __shfl_sync(0xFFFFFFFFu, (uint32_t)job.seed, 0);
    const uint32_t k1 = __shfl_sync(0xFFFFFFFFu, (uint32_t)(job.seed >> 32), 0), start = job.start;
    const uint32_t phase_hi = job.phase << kSweepBits;
    const uint32_t k0w = k0 + kPhiloxW0, k1w = k1 + kPhiloxW1;
    const uint32_t *__restrict__ thr = L.thr;
    const size_t ts = (size_t)L.thr_step;
    // staged: the units of every thread ([unit_rows][B]: position, first group, group step) and the spins'
    // records ([n] uint4, and [n] words for neighbours 6 and 7); then the pairs
    uint32_t *unit = smem;
    const int unit_rows = STAGED ? L.stage_ell : 0;
    uint4 *rec = reinterpret_cast<uint4 *>(smem + unit_rows * B);
    uint32_t *rec2 = smem + unit_rows * B + 4 * (size_t)n;
    uint32_t *pairs = STAGED ? smem + unit_rows * B + (((MAXD <= 6 ? 4 : 5) * n + 3) & ~3) : smem;
    uint32_t *sw = pairs + kPairHead * NV;

    if (tid < 32) {
        // range of the flip-cost constants
        int lo = 30, hi = 0;
        for (int p = tid; p < n; p += 32) {
            const uint32_t meta = g_meta[p];
            const int c8 = 15 + ((int)meta >> 16) - (int)(meta & 0xFFFFu);
            lo = min(lo, c8);
            hi = max(hi, c8);
        }
        lo = __reduce_min_sync(0xFFFFFFFFu, lo);
        hi = __reduce_max_sync(0xFFFFFFFFu, hi);
        if (tid == 0) {
            sm.c8lo = min(lo, hi);
            sm.c8hi = hi;
            sm.zero[t0 & 1] = 0;
        }
    }
    if (tid == B - 1) unit_classes<B>(P, ncol, ng, unit_rows, sm.cls);
    if (STAGED)
        for (int p = tid; p < n; p += B) {
            const uint32_t meta = g_meta[p];
            const int deg = (int)(meta & 0xFFFFu);
            uint32_t o[8];
#pragma unroll
            for (int d = 0; d < 8; ++d) {
                o[d] = 4u * NV * (uint32_t)n;
                if (d < MAXD && d < deg) {
                    const uint32_t e = g_ell[(size_t)d * cap_n + p];
                    o[d] = 4u * NV * (((e >> 31) ? (uint32_t)ns : 0u) + (e & 0xFFFFu));
                }
            }
            rec[p] = make_uint4(o[0] | o[1] << 16, o[2] | o[3] << 16, o[4] | o[5] << 16,
                                (uint32_t)g_idx[p] | (uint32_t)(15 + ((int)meta >> 16) - deg) << 16);
            if (MAXD > 6) rec2[p] = o[6] | o[7] << 16;
        }
    for (int x = tid; x < np * ns; x += B) {
        const int v = x / ns, p = x - v * ns;
        // quads past the item's end start at 0: a resumed sample reads the rows another block may be writing,
        // and only an item's own rows are safe to read
        uint32_t w = 0u;
        if (p < n && 2 * v < nq) {
            w = start_word(P, job, quad0 + 2 * v, p);
            if (2 * v + 1 < nq) w |= start_word(P, job, quad0 + 2 * v + 1, p) << 4;
        }
        uint32_t *d = sw + (size_t)(v / NV) * gw + p * NV + v % NV;
        d[0] = w;
        d[ns * NV] = p < n ? (w ^ kN) : 0u;
    }
    for (int v = tid; v < np; v += B) {
        uint4 h, q;
        philox_mulhilo(kPhiloxM1, (uint32_t)(quad0 + 2 * v), h.z, h.x);
        philox_mulhilo(kPhiloxM1, (uint32_t)(quad0 + 2 * v + 1), h.w, h.y);
        h.x ^= k0w;
        h.y ^= k0w;
        h.z ^= k0;
        h.w ^= k0;
        const uint32_t y = phase_hi | (uint32_t)t0;
        philox_mulhilo(kPhiloxM0, h.z ^ y, q.x, q.y);
        philox_mulhilo(kPhiloxM0, h.w ^ y, q.z, q.w);
        uint4 *head = reinterpret_cast<uint4 *>(pairs + (size_t)(v / NV) * gw) + v % NV;
        head[(t0 & 1) * NV] = q;
        head[2 * NV] = h;
    }
    for (int i = tid; i < 128; i += B) sm.row[i >> 6][i & 63] = 0u;
    __syncthreads();
    if (t0 < T) {
        const uint32_t *row = thr + (size_t)t0 * ts;
        if (tid < bias) {
            const uint32_t v = row[2 * (tid + 1)];
            sm.row[t0 & 1][2 * (tid + 1) + 30] = v;
            if (v == 0u) sm.zero[t0 & 1] = 1;
        }
        if constexpr (TABS)
            for (int i = tid; i < 16 * (sm.c8hi - sm.c8lo + 1); i += B)
                sm.tab[t0 & 1][tab_word(sm.c8lo + (i >> 4), i & 15)] = top_word(row, sm.c8lo + (i >> 4), i & 15, bias);
    }
    if (STAGED) unit_list<B>(ncol, ng, unit_rows, sm.cls, unit);
    __syncthreads();

    QuadItem I;
    I.end4 = (uint32_t)ng * v4;
    I.v4 = v4;
    I.ns4 = ns4;
    I.sw4 = shared_addr(sw);
    I.np = np;
    I.both = NV > 1 || nq > 1;
    I.n = n;
    I.ncol = ncol;
    I.bias = bias;
    I.cap_n = cap_n;
    I.sk1 = start ^ k1;
    I.k1w = k1w;
    I.meta = g_meta;
    I.ell = g_ell;
    I.idx = g_idx;
    PhiloxKeys<2> K = philox_keys<2>(k0, k1);
    // opaque to the compiler, which would otherwise recompute all sixteen for every pair
#pragma unroll
    for (int i = 0; i < 8; ++i) asm("" : "+r"(K.k0[i]), "+r"(K.k1[i]));
    auto next = [&](int t) { return t + 1 < T ? thr + (size_t)(t + 1) * ts : nullptr; };
    int t = t0;
    if (t < T && (t & 1)) {
        sweep_pairs_par<B, MAXD, NV, STAGED, 1>(I, sm, pairs, rec, rec2, unit, phase_hi | (uint32_t)(t + 1), next(t), K);
        ++t;
    }
    for (; t + 1 < T; t += 2) {
        sweep_pairs_par<B, MAXD, NV, STAGED, 0>(I, sm, pairs, rec, rec2, unit, phase_hi | (uint32_t)(t + 1), next(t), K);
        sweep_pairs_par<B, MAXD, NV, STAGED, 1>(I, sm, pairs, rec, rec2, unit, phase_hi | (uint32_t)(t + 2), next(t + 1), K);
    }
    if (t < T) sweep_pairs_par<B, MAXD, NV, STAGED, 0>(I, sm, pairs, rec, rec2, unit, phase_hi | (uint32_t)(t + 1), nullptr, K);
    finish_pairs<NV>(P, job, quad0, nq, sw, sm.e2);
}

template <int B, int MAXD, int NV, bool STAGED, bool TABS>
__global__ void __launch_bounds__(B, 1024 / B) k_sweep_pm1q(const SweepLaunch L)
{
    __shared__ __align__(256) QuadSmem<TABS> sm;
    extern __shared__ __align__(16) uint32_t smem_pm1q[];
    for (int iter = 0;; ++iter) {
        SweepJob job;
        int quad0, nq;
        if (!next_item(L, iter, &sm.item, job, quad0, nq)) break;
        run_item_pm1q<B, MAXD, NV, STAGED, TABS>(L, job, quad0, nq, sm, smem_pm1q);
        __syncthreads();
    }
}

void *select_q(int block, int maxd, int nv, bool staged, bool tabs)
{
#define SPVAR_PM1Q_CASE(BB, MD, NVV, ST, TB)                              \
    if (block == BB && maxd == MD && nv == NVV && staged == ST && tabs == TB) \
        return reinterpret_cast<void *>(k_sweep_pm1q<BB, MD, NVV, ST, TB>);
#define SPVAR_PM1Q_BLOCK(BB)                                                                              \
    SPVAR_PM1Q_CASE(BB, 6, 1, true, true) SPVAR_PM1Q_CASE(BB, 6, 2, true, true)                           \
    SPVAR_PM1Q_CASE(BB, 6, 1, false, true) SPVAR_PM1Q_CASE(BB, 6, 2, false, true)                         \
    SPVAR_PM1Q_CASE(BB, 6, 1, false, false)                                                               \
    SPVAR_PM1Q_CASE(BB, 8, 1, true, false) SPVAR_PM1Q_CASE(BB, 8, 2, true, false)                         \
    SPVAR_PM1Q_CASE(BB, 8, 1, false, false) SPVAR_PM1Q_CASE(BB, 8, 2, false, false)
    SPVAR_PM1Q_BLOCK(128) SPVAR_PM1Q_BLOCK(256) SPVAR_PM1Q_BLOCK(512) SPVAR_PM1Q_BLOCK(1024)
#undef SPVAR_PM1Q_BLOCK
#undef SPVAR_PM1Q_CASE
    return nullptr;
}

}  // namespace

// Q quads of a problem of at most max_n spins per work item.
bool pm1q_shape_ok(int block, int maxd, int max_n, int Q)
{
    return select_q(block, maxd, 1, false, false) != nullptr && Q >= 1 && Q <= kQcap && max_n < 0xFFFF;
}

// Pairs of quads per group (one vector load).
static int pm1q_group(int max_n, int Q)
{
    return Q >= 4 && 16LL * (max_n + 1) <= 0x10000LL ? 2 : 1;
}

// Shared memory of a launch whose largest problem has max_n spins, Q quads an item.  A
// spin's record is four words (six neighbour byte offsets as 16-bit halves, index and
// flip-cost constant), five for degree 7 and 8; without records (0 words) the kernel
// reads the problem's own arrays, where a byte offset does not fit 16 bits or the
// records do not fit beside the spin words.  The units of up to 8 rounds of the block
// are listed where there is room (without the list a class is swept a spin per thread,
// every group at once).
QuadLayout pm1q_layout(int block, int max_n, int Q, int maxd)
{
    QuadLayout l;
    l.nv = pm1q_group(max_n, Q);
    const size_t groups = (size_t)((Q + 2 * l.nv - 1) / (2 * l.nv)) * group_words(max_n, l.nv);
    const int w = maxd <= 6 ? 4 : 5;
    const size_t recs = ((size_t)w * max_n + 3) & ~(size_t)3, units = (size_t)kUnitRows * block;
    l.rec = l.unit_rows = 0;
    if (8LL * l.nv * (max_n + 1) <= 0x10000LL && 4 * (recs + groups) <= kQuadSmemMax) {
        l.rec = w;
        if (4 * (units + recs + groups) <= kQuadSmemMax) l.unit_rows = kUnitRows;
    }
    l.fit_words = (int)((l.rec ? recs : 0) + groups);
    l.bytes = 4 * ((size_t)l.fit_words + (size_t)l.unit_rows * block);
    // the second table everywhere but in a lone pair's last 4 KB (28276 .. 28787 spins), the one place where a
    // problem that ran without it would not fit a CTA with it
    l.tabs = maxd <= 6 && (l.rec > 0 || l.nv > 1 || l.bytes + quad_static(true) <= kSmemOptin);
    l.stat = quad_static(l.tabs);
    return l;
}

bool pm1q_fits(int block, int max_n, int Q, int maxd, size_t optin)
{
    const QuadLayout l = pm1q_layout(block, max_n, Q, maxd);
    return pm1q_shape_ok(block, maxd, max_n, Q) && l.bytes + l.stat <= optin;
}

// Block and quads per item for problems of at most max_n spins where nothing is tuned:
// the most quads, up to 8, with which two 512-thread CTAs share an SM, else one of 1024
// threads and a pair (or what fits).  Measured on 3D +-J, 20 starts x (250 + 250):
// L = 12 10.8 ms with 512 threads and 4 quads, 11.2 ms with 2 quads, 12.5 ms with 1024
// threads; L = 20 18.7 ms with 1024 threads, 20.3 ms with 512 (one CTA either way).
// block 0: no shape fits.
SweepShape pm1q_default(int max_n, int maxd, size_t optin)
{
    for (int Q : {8, 4, 2})
        if (2 * (pm1q_layout(512, max_n, Q, maxd).bytes + kQuadRoom) <= optin) return SweepShape{6, 512, Q, 0, 0, maxd};
    for (int Q : {2, 1})
        if (pm1q_layout(1024, max_n, Q, maxd).bytes + kQuadRoom <= optin) return SweepShape{6, 1024, Q, 0, 0, maxd};
    return SweepShape{6, 0, 1, 0, 0, maxd};
}

cudaError_t launch_sweep_pm1q(const SweepLaunch &L, int block, int maxd, int Q, int grid, size_t smem, cudaStream_t st)
{
    const QuadLayout l = pm1q_layout(block, L.max_n, Q, maxd);
    void *k = select_q(block, maxd, l.nv, l.rec > 0, l.tabs);
    if (!k) return cudaErrorInvalidValue;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    SweepLaunch A = L;
    A.stage_ell = l.unit_rows;
    void *args[] = {&A};
    return cudaLaunchKernel(k, dim3(grid), dim3(block), args, smem, st);
}

int pm1q_max_active_blocks(int block, int maxd, int max_n, int Q, size_t smem)
{
    const QuadLayout l = pm1q_layout(block, max_n, Q, maxd);
    void *k = select_q(block, maxd, l.nv, l.rec > 0, l.tabs);
    if (!k) return 0;
    cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    int nb = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k, block, smem);
    return nb;
}

}  // namespace spvar
