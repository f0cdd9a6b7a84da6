// Allocation-free fold/compact: spvar_reduce_noalloc.
//
// For callers that must not allocate device memory while they run -- for
// example code that executes inside a memory-pool budget that is already
// fully committed, or an embedding runtime that owns every allocation and
// forbids cudaMalloc/cudaFree (and allocating library routines) after
// start-up.  It computes the same reduced problem as spvar_reduce, but writes
// it as plain CSR arrays into buffers the caller provides, and keeps its
// working arrays in one statically sized device array of this file instead
// of allocating them.
//
// The static array exists once per device that loads the library and lives
// until the process exits.  Its device address is looked up with
// cudaGetSymbolAddress on the first call made on each device (with that
// device current); make that first call before any stream capture.  Every
// call shares the array: calls that can overlap on the GPU (different
// streams, or concurrent host threads) race on it and must be serialised by
// the caller.  Nothing in the array needs to start at zero: each call writes
// every entry it later reads.
#include <cooperative_groups.h>

#include <mutex>

#include "persist.cuh"

namespace cg = cooperative_groups;

namespace spvar {
namespace {

// new index of every old spin (-1: fixed)
__device__ __align__(256) int32_t g_reduce_scratch[SPVAR_NOALLOC_MAX_N];

std::mutex g_addr_mu;
int32_t *g_addr[64] = {nullptr};

int scratch_address(int32_t **out)
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return SPVAR_ECUDA;
    std::lock_guard<std::mutex> g(g_addr_mu);
    if (!g_addr[dev]) {
        void *p = nullptr;
        if (cudaGetSymbolAddress(&p, g_reduce_scratch) != cudaSuccess) {
            cudaGetLastError();
            return SPVAR_ECUDA;
        }
        g_addr[dev] = static_cast<int32_t *>(p);
    }
    *out = g_addr[dev];
    return SPVAR_OK;
}

constexpr int kCsrCluster = 8;  // blocks, each with a contiguous range of the spins
constexpr int kCsrSpins = (SPVAR_NOALLOC_MAX_N + kCsrCluster * kBigBlock - 1) / (kCsrCluster * kBigBlock);
constexpr int kCsrOneBlock = kCsrSpins * kBigBlock;  // the most spins one block takes
constexpr int kCsrGather = 4;   // CSR entries of a row loaded at once

struct CsrTotals {
    int32_t nfree, nnz;
    unsigned long long off;
};

// Fold the fixed spins into h and the offset and write the CSR of the free
// spins (renumbered in increasing old index) to the caller's arrays.
// Bound by the latency of the dependent gathers (spin, row, neighbour), so the
// spins are dealt to the blocks of one cluster and a thread holds its own
// (at most kCsrSpins) in registers; the blocks exchange their totals through
// shared memory, and only the new indices go through the scratch array.
// 8000 spins of a cubic lattice: 61.7 us a call on one block, 14.6 here.  Up
// to kCsrOneBlock spins one block takes the same two spins a thread, and its
// launch is 2 to 3 us cheaper for the host (elite, counts and this reduction
// of Chimera C16, n = 2048: 64.4 us a call by the cluster, 57.5 by the block;
// C19, n = 2888: 80.7 us by one block to the end on the device, 68.8 here).
template <int NB>  // blocks
__device__ __forceinline__ void reduce_csr(const DevProb *S, const int8_t *fixed, int32_t *row_ptr, int32_t *col,
                                           int32_t *val, int32_t *h_out, int64_t *offset_out, int32_t *old_of_new,
                                           int32_t *n_out, int32_t *scratch)
{
    __shared__ int s_warp[32];
    __shared__ CsrTotals s_tot;
    auto sync = [] {
        if (NB > 1) cg::this_cluster().sync();
        else __syncthreads();
    };
    const int tid = threadIdx.x, rank = NB > 1 ? blockIdx.x : 0;
    const int n = S->n, len = (n + NB - 1) / NB;
    const int first = rank * len, last = min(n, first + len);
    const int32_t *srow = S->row_ptr, *scol = S->col, *sval = S->val;
    if (tid == 0) s_tot.off = 0ull;
    __syncthreads();

    // folded biases, free-free row lengths, and their sums over the spins before, by block
    int32_t hf[kCsrSpins], a[kCsrSpins], q[kCsrSpins];
    bool fr[kCsrSpins];
    long long off = 0;
    int nfree = 0, nnz = 0;
#pragma unroll
    for (int u = 0; u < kCsrSpins; ++u) {
        const int i = first + u * kBigBlock + tid;
        const bool ok = i < last;
        const int vi = ok ? fixed[i] : 0, h = ok ? S->h[i] : 0;
        const int p0 = ok ? srow[i] : 0, p1 = ok ? srow[i + 1] : 0;
        long long hs = h;
        int cnt = 0;
        for (int p = p0; p < p1; p += kCsrGather) {
            int j[kCsrGather], v[kCsrGather], f[kCsrGather];
#pragma unroll
            for (int d = 0; d < kCsrGather; ++d) {
                j[d] = p + d < p1 ? scol[p + d] : -1;
                v[d] = p + d < p1 ? sval[p + d] : 0;
            }
#pragma unroll
            for (int d = 0; d < kCsrGather; ++d) f[d] = j[d] >= 0 ? fixed[j[d]] : 0;
#pragma unroll
            for (int d = 0; d < kCsrGather; ++d) {
                if (j[d] < 0) continue;
                if (vi) {
                    if (f[d] && j[d] > i) off += (long long)v[d] * vi * f[d];
                } else if (f[d]) {
                    hs += (long long)v[d] * f[d];
                } else {
                    ++cnt;
                }
            }
        }
        if (vi) off += (long long)h * vi;
        fr[u] = ok && !vi;
        hf[u] = (int32_t)hs;
        int tot;
        a[u] = nfree + block_scan_excl(fr[u] ? 1 : 0, s_warp, &tot);
        nfree += tot;
        q[u] = nnz + block_scan_excl(fr[u] ? cnt : 0, s_warp, &tot);
        nnz += tot;
    }
#pragma unroll
    for (int sh = 16; sh > 0; sh >>= 1) off += __shfl_xor_sync(0xFFFFFFFFu, off, sh);
    if ((tid & 31) == 0) atomicAdd(&s_tot.off, (unsigned long long)off);
    if (tid == 0) {
        s_tot.nfree = nfree;
        s_tot.nnz = nnz;
    }
    sync();  // every block's totals

    int base_n = 0, base_z = 0, m = 0, z = 0;
    unsigned long long osum = 0ull;
    for (int r = 0; r < NB; ++r) {
        const CsrTotals *t = NB > 1 ? cg::this_cluster().map_shared_rank(&s_tot, r) : &s_tot;
        if (r < rank) {
            base_n += t->nfree;
            base_z += t->nnz;
        }
        m += t->nfree;
        z += t->nnz;
        osum += t->off;
    }
    if (rank == 0 && tid == 0) {
        row_ptr[m] = z;
        *n_out = m;
        *offset_out = S->offset + (long long)osum;
    }
#pragma unroll
    for (int u = 0; u < kCsrSpins; ++u) {
        const int i = first + u * kBigBlock + tid;
        a[u] += base_n;
        q[u] += base_z;
        if (i < last) scratch[i] = fr[u] ? a[u] : -1;
        if (fr[u]) {
            old_of_new[a[u]] = i;
            h_out[a[u]] = hf[u];
            row_ptr[a[u]] = q[u];
        }
    }
    sync();  // the new indices, and no block leaves while its totals are read

#pragma unroll
    for (int u = 0; u < kCsrSpins; ++u) {
        const int i = first + u * kBigBlock + tid;
        const int p0 = fr[u] ? srow[i] : 0, p1 = fr[u] ? srow[i + 1] : 0;
        int w = q[u];
        for (int p = p0; p < p1; p += kCsrGather) {
            int j[kCsrGather], v[kCsrGather];
#pragma unroll
            for (int d = 0; d < kCsrGather; ++d) {
                j[d] = p + d < p1 ? scol[p + d] : -1;
                v[d] = p + d < p1 ? sval[p + d] : 0;
            }
#pragma unroll
            for (int d = 0; d < kCsrGather; ++d) j[d] = j[d] >= 0 ? scratch[j[d]] : -1;
#pragma unroll
            for (int d = 0; d < kCsrGather; ++d)
                if (j[d] >= 0) {
                    col[w] = j[d];
                    val[w] = v[d];
                    ++w;
                }
        }
    }
}

__global__ void __cluster_dims__(kCsrCluster, 1, 1) __launch_bounds__(kBigBlock)
    k_reduce_csr(const DevProb *S, const int8_t *fixed, int32_t *row_ptr, int32_t *col, int32_t *val,
                 int32_t *h_out, int64_t *offset_out, int32_t *old_of_new, int32_t *n_out, int32_t *scratch)
{
    reduce_csr<kCsrCluster>(S, fixed, row_ptr, col, val, h_out, offset_out, old_of_new, n_out, scratch);
}

__global__ void __launch_bounds__(kBigBlock)
    k_reduce_csr_block(const DevProb *S, const int8_t *fixed, int32_t *row_ptr, int32_t *col, int32_t *val,
                       int32_t *h_out, int64_t *offset_out, int32_t *old_of_new, int32_t *n_out, int32_t *scratch)
{
    reduce_csr<1>(S, fixed, row_ptr, col, val, h_out, offset_out, old_of_new, n_out, scratch);
}

}  // namespace
}  // namespace spvar

using namespace spvar;

extern "C" int spvar_reduce_noalloc(const spvar_problem *p, const int8_t *fixed, int32_t *row_ptr,
                                    int32_t *col, int32_t *val, int32_t *h, int64_t *offset,
                                    int32_t *old_of_new, int32_t *n_out, void *stream)
{
    if (!p) return SPVAR_EINVAL;
    const Problem *S = reinterpret_cast<const Problem *>(p);
    const DevProb &H = S->hdr;
    if (H.n > SPVAR_NOALLOC_MAX_N) return SPVAR_ELIMIT;
    if (!row_ptr || !offset || !n_out || (H.n > 0 && (!fixed || !h || !old_of_new)) ||
        (H.nnz > 0 && (!col || !val)))
        return SPVAR_EINVAL;
    int32_t *scratch = nullptr;
    const int rc = scratch_address(&scratch);
    if (rc != SPVAR_OK) return rc;
    // launched through cudaLaunchKernel so that its own status is checked, not an
    // earlier error left pending on this thread by unrelated work
    const DevProb *src = S->dev;
    void *args[] = {(void *)&src, (void *)&fixed, (void *)&row_ptr, (void *)&col, (void *)&val, (void *)&h,
                    (void *)&offset, (void *)&old_of_new, (void *)&n_out, (void *)&scratch};
    const bool one = H.n <= kCsrOneBlock;
    const cudaError_t e = cudaLaunchKernel(reinterpret_cast<const void *>(one ? k_reduce_csr_block : k_reduce_csr),
                                           dim3(one ? 1 : kCsrCluster), dim3(kBigBlock), args, 0,
                                           reinterpret_cast<cudaStream_t>(stream));
    return e == cudaSuccess ? SPVAR_OK : SPVAR_ECUDA;
}
