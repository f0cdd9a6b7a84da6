// Quad-group simulated-annealing sweep for integer couplers (the sampler of
// Sec. III.A on real-valued problems scaled to integers, and on couplers of
// several magnitudes): one work item is nq quads (4 nq replicas) of one start's
// problem.
//
// Same dynamics, random words and result as the other sweep kernels.  Replica
// bits stand in lanes wide enough for the flip cost e = dE/2, so one
// multiply-add per neighbour adds J_ij b_j for every replica of a word, however
// the terms borrow from lane to lane: the sum over all neighbours plus the
// spin's constant is exact in each lane.
//   BYTE (dmax <= 254): four replicas a word, lanes hold e + 127, whose top bit
//   says e > 0.
//   else (dmax <= 16382): two words of 16-bit lanes (replicas 0, 2 and 1, 3) with
//   4 (e - 1) + 32768: the top bit says e > 0, the rest is the byte offset in the
//   acceptance row.
// A thread sets a spin up once (neighbour byte offsets and couplers from its record in
// shared memory, the Philox products of spin and start) and sweeps it in every quad
// of its unit (quad_units.cuh).  The next sweep's acceptance row, thresholds of dE =
// 2 .. dmax, is copied asynchronously while the current sweep runs.
//
// Bound: the integer pipes, about 125 instructions (BYTE) or 150 per quad and spin, 66 of
// them Philox.  Gaussian couplers x 100 on 3D L = 9 (dmax 2050), 1000 samples x 1000 sweeps:
// 5.1 ms with one multiply-add per replica and neighbour and a row in 32-bit words read through
// the L1 cache, 2.8 ms now (fewer quads than two an SM: barriers first).
#include "quad_units.cuh"

namespace spvar {

namespace {

constexpr int kGqHead = 8;          // words of Philox products before a quad's spin words
constexpr int kGqCap = 64;          // most quads per work item
constexpr int kGqPad = 128;         // BYTE: words after the rows (an index of a cost that is not positive reads up to 127)
constexpr size_t kGqStatic = 3 << 10;  // static shared memory and the system's 1 KB, rounded up

struct GqSmem {
    int e2[4 * kGqCap];
    int4 cls[kMaxColours];
};

// Words of a spin's record: neighbour byte offsets (16 bits), couplers (16 bits), index
// and constant.
__host__ __device__ constexpr int gq_rec_words(int maxd) { return maxd <= 6 ? 8 : 12; }

__device__ __forceinline__ void cp_async4(uint32_t dst, const void *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
}

// One sweep; rows: shared addresses of this sweep's and the next one's acceptance row.
template <int B, int MAXD, bool BYTE>
__device__ __forceinline__ void sweep_quads(GqSmem &sm, const uint4 *rec, const uint32_t *unit, uint32_t *quads, int ncol,
                                            int nq, int bias, int gw, int par, uint32_t y1,
                                            const uint32_t *__restrict__ next_thr, uint32_t row, uint32_t next_row,
                                            uint32_t sk1, uint32_t k1w, const PhiloxKeys<2> &K)
{
    constexpr uint32_t M = 0x01010101u, T = 0x00010001u;
    constexpr int NW = BYTE ? 1 : 2, RW = gq_rec_words(MAXD) / 4;
    const int tid = threadIdx.x;
    if (next_thr) {
        for (int e = tid; e < bias; e += B) cp_async4(next_row + 4u * (uint32_t)e, next_thr + 2 * (e + 1));
        for (int v = tid; v < nq; v += B) {
            uint32_t *head = quads + (size_t)v * gw;
            philox_mulhilo(kPhiloxM0, head[5] ^ y1, head[2 * (par ^ 1)], head[2 * (par ^ 1) + 1]);
        }
    }
    const uint32_t v4 = 4u * (uint32_t)gw, first = shared_addr(quads) + 4u * kGqHead, last = first + (uint32_t)nq * v4;
    const uint32_t par8 = 8u * (uint32_t)par;
    for (int c = 0; c < ncol; ++c) {
        const int4 cl = sm.cls[c];
#pragma unroll 1
        for (int r = 0; r < cl.z; ++r) {
            uint32_t p, base, step4;
            if (cl.w >= 0) {
                const uint32_t d = unit[(cl.w + r) * B + tid];
                p = d & 0xFFFFu;
                base = first + ((d >> 16) & 0xFFu) * v4;
                step4 = (d >> 24) * v4;
            } else {
                const int u = r * B + tid;
                p = (uint32_t)(cl.x + u);
                base = u < cl.y ? first : last;
                step4 = v4;
            }
            if (base < last) {
                uint32_t off[8];
                int J[8], f0;
                uint32_t idx;
                const uint4 k0 = rec[RW * p], k1 = rec[RW * p + 1];
                if (MAXD <= 6) {
                    const uint32_t o[3] = {k0.x, k0.y, k0.z}, j[3] = {k0.w, k1.x, k1.y};
#pragma unroll
                    for (int d = 0; d < 3; ++d) {
                        off[2 * d] = o[d] & 0xFFFFu;
                        off[2 * d + 1] = o[d] >> 16;
                        J[2 * d] = (int)(short)(j[d] & 0xFFFFu);
                        J[2 * d + 1] = (int)j[d] >> 16;
                    }
                    idx = k1.z;
                    f0 = (int)k1.w;
                } else {
                    const uint4 k2 = rec[RW * p + 2];
                    const uint32_t o[4] = {k0.x, k0.y, k0.z, k0.w}, j[4] = {k1.x, k1.y, k1.z, k1.w};
#pragma unroll
                    for (int d = 0; d < 4; ++d) {
                        off[2 * d] = o[d] & 0xFFFFu;
                        off[2 * d + 1] = o[d] >> 16;
                        J[2 * d] = (int)(short)(j[d] & 0xFFFFu);
                        J[2 * d + 1] = (int)j[d] >> 16;
                    }
                    idx = k2.x;
                    f0 = (int)k2.y;
                }
                if (!BYTE)
#pragma unroll
                    for (int d = 0; d < 8; ++d) J[d] *= 8;  // 4 (2 J b)
                // the lane of a b_i = 0 replica, f = f0 + 2 sum_j J_ij b_j, f0 = h - sum_j J_ij; b_i = 1: -f
                const uint32_t cc = BYTE ? (uint32_t)(f0 + 127) * M : (uint32_t)(4 * (f0 - 1) + 32768) * T;
                uint32_t H0, L0, H2, L2;
                philox_mulhilo(kPhiloxM0, idx, H0, L0);
                philox_mulhilo(kPhiloxM1, H0 ^ sk1, H2, L2);
                const uint32_t L0k = L0 ^ k1w, own4 = 4u * NW * p;
#pragma unroll 1
                do {
                    const uint32_t oa = base + own4;
                    const uint2 qs = lds2(base + par8 - 4u * kGqHead);
                    const uint32_t L1k = lds(base + 16u - 4u * kGqHead);
                    if (BYTE) {
                        const uint32_t own = lds(oa);
                        uint32_t x = 0;
#pragma unroll
                        for (int d = 0; d < MAXD; ++d) x += (uint32_t)J[d] * lds(base + off[d]);
                        const uint32_t a = 2u * x + cc, m = own * 255u;
                        const uint32_t ix = (a & ~m) | ((254u * M - a) & m), low = ix & 0x7F7F7F7Fu;
                        const uint4 u = philox_rounds<2>(make_uint4(H2 ^ L1k, L2, qs.x ^ L0k, qs.y), K);
                        const uint32_t ur[4] = {u.x, u.y, u.z, u.w};
                        uint32_t rej = 0;
#pragma unroll
                        for (int rr = 0; rr < 4; ++rr) {
                            const uint32_t thr = lds(row + 4u * __byte_perm(low, 0u, 0x4440u | (uint32_t)rr));
                            asm("{ .reg .pred p; setp.ge.u32 p, %1, %2; @p add.u32 %0, %0, %3; }"
                                : "+r"(rej)
                                : "r"(ur[rr]), "r"(thr), "r"(1u << (8 * rr)));
                        }
                        sts(oa, own ^ M ^ (rej & (ix >> 7) & M));
                    } else {
                        const uint2 own = lds2(oa);
                        uint32_t ae = cc, ao = cc;
#pragma unroll
                        for (int d = 0; d < MAXD; ++d) {
                            const uint2 w = lds2(base + off[d]);
                            ae += (uint32_t)J[d] * w.x;
                            ao += (uint32_t)J[d] * w.y;
                        }
                        const uint32_t me = own.x * 0xFFFFu, mo = own.y * 0xFFFFu;
                        const uint32_t xe = (ae & ~me) | ((65528u * T - ae) & me), xo = (ao & ~mo) | ((65528u * T - ao) & mo);
                        const uint32_t ue = (xe >> 15) & T, uo = (xo >> 15) & T;
                        const uint32_t be = xe & (ue * 0x7FFFu), bo = xo & (uo * 0x7FFFu);
                        const uint4 u = philox_rounds<2>(make_uint4(H2 ^ L1k, L2, qs.x ^ L0k, qs.y), K);
                        const uint32_t ur[4] = {u.x, u.y, u.z, u.w};
                        const uint32_t at[4] = {be & 0xFFFFu, bo & 0xFFFFu, be >> 16, bo >> 16};
                        uint32_t rej[2] = {0u, 0u};
#pragma unroll
                        for (int rr = 0; rr < 4; ++rr) {
                            const uint32_t thr = lds(row + at[rr]);
                            asm("{ .reg .pred p; setp.ge.u32 p, %1, %2; @p add.u32 %0, %0, %3; }"
                                : "+r"(rej[rr & 1])
                                : "r"(ur[rr]), "r"(thr), "r"(1u << (16 * (rr >> 1))));
                        }
                        sts2(oa, make_uint2(own.x ^ T ^ (rej[0] & ue), own.y ^ T ^ (rej[1] & uo)));
                    }
                    base += step4;
                } while (base < last);
            }
        }
        if (c == ncol - 1) asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
    }
}

template <int B, int MAXD, bool BYTE>
__device__ void run_item_gq(const SweepLaunch &L, const SweepJob &job, int quad0, int nq, GqSmem &sm, uint32_t *smem)
{
    constexpr uint32_t T = 0x00010001u;
    constexpr int NW = BYTE ? 1 : 2, RW = gq_rec_words(MAXD);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const DevProb *P = job.prob;
    const int n = P->n, ncol = P->ncol, cap_n = P->cap_n, bias = P->dmax >> 1;
    const uint32_t *__restrict__ g_meta = P->meta;
    const uint32_t *__restrict__ g_ell = P->ell;
    const int gw = gq_quad_words(n, NW), Tend = job_end(L, job), t0 = job.t0;
    const uint32_t k0 = (uint32_t)job.seed, k1 = (uint32_t)(job.seed >> 32), phase_hi = job.phase << kSweepBits;
    const uint32_t *__restrict__ thr = L.thr;
    const size_t ts = (size_t)L.thr_step;
    // records, acceptance rows, units, quads
    const int row_words = (L.thr_stride / 2 + 3) & ~3;
    uint4 *rec = reinterpret_cast<uint4 *>(smem);
    uint32_t *rows = smem + (size_t)RW * n;
    uint32_t *unit = rows + 2 * row_words + kGqPad;
    uint32_t *quads = unit + L.stage_ell * B;

    if (tid == B - 1) unit_classes<B>(P, ncol, nq, L.stage_ell, sm.cls);
    for (int p = tid; p < n; p += B) {
        const uint32_t meta = g_meta[p];
        const int deg = (int)(meta & 0xFFFFu);
        uint32_t o[8], j[8];
        int f0 = (int)meta >> 16;
#pragma unroll
        for (int d = 0; d < 8; ++d) {
            o[d] = 4u * NW * (uint32_t)p;  // a missing neighbour: coupler 0
            j[d] = 0u;
            if (d < MAXD && d < deg) {
                const uint32_t e = g_ell[(size_t)d * cap_n + p];
                o[d] = 4u * NW * (e & 0xFFFFu);
                j[d] = e >> 16;
                f0 -= (int)e >> 16;
            }
        }
        const uint32_t idx = (uint32_t)P->idx_of_pos[p];
        uint4 *k = rec + RW / 4 * p;
        if (MAXD <= 6) {
            k[0] = make_uint4(o[0] | o[1] << 16, o[2] | o[3] << 16, o[4] | o[5] << 16, j[0] | j[1] << 16);
            k[1] = make_uint4(j[2] | j[3] << 16, j[4] | j[5] << 16, idx, (uint32_t)f0);
        } else {
            k[0] = make_uint4(o[0] | o[1] << 16, o[2] | o[3] << 16, o[4] | o[5] << 16, o[6] | o[7] << 16);
            k[1] = make_uint4(j[0] | j[1] << 16, j[2] | j[3] << 16, j[4] | j[5] << 16, j[6] | j[7] << 16);
            k[2] = make_uint4(idx, (uint32_t)f0, 0u, 0u);
        }
    }
    for (int x = tid; x < nq * n; x += B) {
        const int v = x / n, p = x - v * n;
        const uint32_t w = start_word(P, job, quad0 + v, p);
        uint32_t *d = quads + (size_t)v * gw + kGqHead + NW * p;
        d[0] = BYTE ? w : w & T;
        if (!BYTE) d[1] = (w >> 8) & T;
    }
    for (int v = tid; v < nq; v += B) {
        uint32_t h1, l1, *head = quads + (size_t)v * gw;
        philox_mulhilo(kPhiloxM1, (uint32_t)(quad0 + v), h1, l1);
        head[4] = l1 ^ (k0 + kPhiloxW0);
        head[5] = h1 ^ k0;
        philox_mulhilo(kPhiloxM0, h1 ^ k0 ^ (phase_hi | (uint32_t)t0), head[2 * (t0 & 1)], head[2 * (t0 & 1) + 1]);
    }
    for (int x = tid; x < 4 * nq; x += B) sm.e2[x] = 0;
    if (BYTE)
        for (int x = tid; x < kGqPad; x += B) rows[2 * row_words + x] = 0u;
    if (t0 < Tend)
        for (int e = tid; e < bias; e += B) rows[(t0 & 1) * row_words + e] = thr[(size_t)t0 * ts + 2 * (e + 1)];
    __syncthreads();
    unit_list<B>(ncol, nq, L.stage_ell, sm.cls, unit);
    __syncthreads();

    PhiloxKeys<2> K = philox_keys<2>(k0, k1);
    // opaque to the compiler, which would otherwise recompute them for every quad
#pragma unroll
    for (int i = 0; i < 8; ++i) asm("" : "+r"(K.k0[i]), "+r"(K.k1[i]));
    const uint32_t row0 = shared_addr(rows), row1 = row0 + 4u * (uint32_t)row_words;
    for (int t = t0; t < Tend; ++t) {
        const int par = t & 1;
        sweep_quads<B, MAXD, BYTE>(sm, rec, unit, quads, ncol, nq, bias, gw, par, phase_hi | (uint32_t)(t + 1),
                                   t + 1 < Tend ? thr + (size_t)(t + 1) * ts : nullptr, par ? row1 : row0,
                                   par ? row0 : row1, job.start ^ k1, k1 + kPhiloxW1, K);
    }

    // final energies and bit-packed states
    for (int v = 0; v < nq; ++v) {
        const uint32_t *s = quads + (size_t)v * gw + kGqHead;
        int acc[4] = {0, 0, 0, 0};
        for (int p = tid; p < n; p += B) {
            const uint32_t meta = g_meta[p];
            const int deg = (int)(meta & 0xFFFFu), h2 = 2 * ((int)meta >> 16);
            int f[4] = {h2, h2, h2, h2};
            for (int d = 0; d < deg; ++d) {
                const uint32_t e = g_ell[(size_t)d * cap_n + p];
                const uint32_t *w = s + NW * (e & 0xFFFFu);
                const int Jv = (int)e >> 16;
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const uint32_t b = BYTE ? (w[0] >> (8 * r)) & 1u : (w[r & 1] >> (16 * (r >> 1))) & 1u;
                    f[r] += b ? Jv : -Jv;
                }
            }
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const uint32_t b = BYTE ? (s[p] >> (8 * r)) & 1u : (s[2 * p + (r & 1)] >> (16 * (r >> 1))) & 1u;
                acc[r] += b ? f[r] : -f[r];
            }
        }
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int t = __reduce_add_sync(0xFFFFFFFFu, acc[r]);
            if (lane == 0) atomicAdd(&sm.e2[4 * v + r], t);
        }
    }
    __syncthreads();
    for (int x = tid; x < 4 * nq; x += B) {
        const int r = 4 * quad0 + x;
        if (r < job.S) job.energies[r] = (int64_t)(sm.e2[x] / 2) + P->offset;
    }
    const int Wn = (n + 31) >> 5;
    for (int x = warp; x < nq * Wn; x += B / 32) {
        const int v = x / Wn, w = x - v * Wn, i = 32 * w + lane;
        const uint32_t *s = quads + (size_t)v * gw + kGqHead + (i < n ? NW * P->pos_of_idx[i] : 0);
#pragma unroll
        for (int rr = 0; rr < 4; ++rr) {
            const uint32_t b = BYTE ? s[0] >> (8 * rr) : s[rr & 1] >> (16 * (rr >> 1));
            const uint32_t bits = __ballot_sync(0xFFFFFFFFu, i < n && (b & 1u));
            const int r = 4 * (quad0 + v) + rr;
            if (lane == 0 && r < job.S) job.spins[(size_t)r * job.W + w] = bits;
        }
    }
}

template <int B, int MAXD, bool BYTE>
__global__ void __launch_bounds__(B, 1024 / B) k_sweep_gq(const SweepLaunch L)
{
    __shared__ GqSmem sm;
    extern __shared__ __align__(16) uint32_t smem_gq[];
    __shared__ int s_item;
    for (int iter = 0;; ++iter) {
        SweepJob job;
        int quad0, nq;
        if (!next_item(L, iter, &s_item, job, quad0, nq)) break;
        run_item_gq<B, MAXD, BYTE>(L, job, quad0, nq, sm, smem_gq);
        __syncthreads();
    }
}

void *select_gq(int block, int maxd, bool byte)
{
#define SPVAR_GQ_CASE(BB, MD)                                                           \
    if (block == BB && maxd == MD)                                                      \
        return byte ? reinterpret_cast<void *>(k_sweep_gq<BB, MD, true>)                \
                    : reinterpret_cast<void *>(k_sweep_gq<BB, MD, false>);
    SPVAR_GQ_CASE(256, 6) SPVAR_GQ_CASE(512, 6) SPVAR_GQ_CASE(1024, 6)
    SPVAR_GQ_CASE(256, 8) SPVAR_GQ_CASE(512, 8) SPVAR_GQ_CASE(1024, 8)
#undef SPVAR_GQ_CASE
    return nullptr;
}

bool gq_byte(int thr_stride) { return thr_stride - 1 <= 254; }

}  // namespace

// Launches whose acceptance rows are thr_stride wide (flip costs up to thr_stride - 1), Q
// quads of a problem of at most max_n spins an item.  0 quad words: the kernel does not
// apply or its records, rows and quads do not fit.
GqLayout gq_layout(int block, int max_n, int Q, int maxd, int thr_stride, size_t optin)
{
    GqLayout l{0, 0, 0, 0, 0};
    const bool byte = gq_byte(thr_stride);
    const int nw = byte ? 1 : 2;
    if (!select_gq(block, maxd, byte) || Q < 1 || Q > kGqCap || thr_stride > 16383 || 4LL * nw * max_n > 0xFFFFLL) return l;
    const size_t recs = (size_t)gq_rec_words(maxd) * max_n, rows = 2 * (size_t)((thr_stride / 2 + 3) & ~3) + kGqPad;
    const size_t quads = (size_t)Q * gq_quad_words(max_n, nw), units = (size_t)kUnitRows * block;
    if (4 * (recs + rows + quads) + kGqStatic > optin) return l;
    l.unit_rows = 4 * (recs + rows + quads + units) + kGqStatic <= optin ? kUnitRows : 0;
    l.nw = nw;
    l.rec = gq_rec_words(maxd);
    l.fit_words = (int)(recs + quads);
    l.bytes = 4 * (recs + rows + quads + (size_t)l.unit_rows * block);
    return l;
}

// Block and quads per item where nothing is tuned: the most quads, up to 8, with which
// two 512-thread CTAs share an SM, else one of 1024 threads.  block 0: none fits.
SweepShape gq_default(int max_n, int maxd, int thr_stride, size_t optin)
{
    for (int Q : {8, 4, 2}) {
        const GqLayout l = gq_layout(512, max_n, Q, maxd, thr_stride, optin);
        if (l.nw > 0 && 2 * (l.bytes + kGqStatic) <= optin) return SweepShape{7, 512, Q, 0, 0, maxd};
    }
    for (int Q : {4, 2, 1})
        if (gq_layout(1024, max_n, Q, maxd, thr_stride, optin).nw > 0) return SweepShape{7, 1024, Q, 0, 0, maxd};
    return SweepShape{7, 0, 1, 0, 0, maxd};
}

cudaError_t launch_sweep_gq(const SweepLaunch &L, int block, int maxd, int Q, int grid, size_t smem, cudaStream_t st)
{
    void *k = select_gq(block, maxd, gq_byte(L.thr_stride));
    if (!k) return cudaErrorInvalidValue;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    SweepLaunch A = L;
    A.stage_ell = gq_layout(block, L.max_n, Q, maxd, L.thr_stride, (size_t)1 << 30).bytes <= smem ? kUnitRows : 0;
    void *args[] = {&A};
    return cudaLaunchKernel(k, dim3(grid), dim3(block), args, smem, st);
}

int gq_max_active_blocks(int block, int maxd, int thr_stride, size_t smem)
{
    void *k = select_gq(block, maxd, gq_byte(thr_stride));
    if (!k) return 0;
    cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    int nb = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k, block, smem);
    return nb;
}

}  // namespace spvar
