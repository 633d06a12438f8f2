// Counting sort of the grain store by zone key: exclusive scan of the key
// counts, scatter of (id, source) pairs, an id sort inside every key and a
// gather of the store columns (keys are computed by the geometry-specific
// sort_keys kernel).  The live grains' order is deterministic: by key, then
// id.  Removed grains (the last key) come after them in the scatter's order:
// nothing is computed from them, and sorting that segment, which grows with
// every removal, would make the sort's cost grow with the run's length.
#include "dust_sort.cuh"

namespace dust {

// chunk sums for chunks of at least 256 threads x kScanItems counts
int64_t scan_block_sums_size(int64_t n) { return (n + 256 * kScanItems - 1) / (256 * kScanItems) + 1; }

// Buffers the scan's kernels clear on their way, so that the clears need no
// launches of their own: the next counts (zero, as many as are scanned) and the
// deposit of the coming step (words of 16 bytes).
struct ScanClears {
    int32_t *zero;
    uint4 *dep;
    int64_t dep_words;
};

__device__ __forceinline__ void clear_deposit(const ScanClears &C)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < C.dep_words;
         i += (int64_t)gridDim.x * blockDim.x)
        C.dep[i] = make_uint4(0u, 0u, 0u, 0u);
}

__global__ void scan_reduce_kernel(const int32_t *data, int64_t n, int32_t *block_sums, const ScanClears C)
{
    __shared__ int32_t ws[32];
    scan_reduce_block(data, n, block_sums, blockIdx.x, ws, C.zero);
    clear_deposit(C);
}

__global__ void scan_sums_kernel(int32_t *block_sums, int64_t nb)
{
    __shared__ int32_t ws[32];
    scan_sums_block(block_sums, nb, ws);
}

// sums_scanned: the chunk sums are already an exclusive scan.
__global__ void scan_finish_kernel(int32_t *data, int64_t n, const int32_t *block_sums, int sums_scanned, int32_t *copy,
                                   int32_t *big)
{
    __shared__ int32_t ws[32];
    if (sums_scanned) scan_apply_block(data, n, block_sums, blockIdx.x, ws, copy);
    else scan_finish_block(data, n, block_sums, blockIdx.x, ws, copy);
    if (blockIdx.x == 0 && threadIdx.x == 0) big[0] = 0;
}

// A few chunks: block 0 scans them in turn; the other blocks only clear.
__global__ void scan_small_kernel(int32_t *data, int64_t n, int32_t *copy, int32_t *big, const ScanClears C)
{
    __shared__ int32_t ws[32];
    clear_deposit(C);
    if (blockIdx.x > 0) return;
    int32_t from = 0;
    for (int64_t vb = 0; vb * kScanTile < n; ++vb) from += scan_chunk(data, n, from, vb, ws, copy, C.zero);
    if (threadIdx.x == 0) big[0] = 0;
}

// Up to kScanDirect chunks, each block of the second kernel sums the chunk sums
// before it; beyond (a grid of more than 4M keys) that costs more than a
// kernel between the two that scans them.  Up to kScanSmall chunks take one
// launch.  The copy to the cursors and the clears are part of these kernels: they
// were a copy and three clears of their own (64^2 box: sort and clears 35.7 ->
// 27.3 us with two launches).
constexpr int64_t kScanDirect = 1024, kScanSmall = 4;

int64_t scan_direct_counts() { return kScanDirect * kScanTile; }
int64_t scan_small_counts() { return kScanSmall * kScanTile; }

cudaError_t launch_exclusive_scan(int32_t *data, int64_t n, int32_t *block_sums, int32_t *copy, int32_t *big,
                                  int32_t *zero, void *dep, int64_t dep_bytes, cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    const int64_t nb = (n + kScanTile - 1) / kScanTile;
    const ScanClears C{zero, static_cast<uint4 *>(dep), dep_bytes / (int64_t)sizeof(uint4)};
    // enough blocks to clear the deposit at the memory's rate
    if (nb <= kScanSmall) {
        const int64_t clears = (C.dep_words + kScanTile - 1) / kScanTile;
        scan_small_kernel<<<(unsigned)(1 + (clears < 304 ? clears : 304)), kScanThreads, 0, s>>>(data, n, copy, big, C);
        return cudaGetLastError();
    }
    scan_reduce_kernel<<<(unsigned)nb, kScanThreads, 0, s>>>(data, n, block_sums, C);
    if (nb > kScanDirect) scan_sums_kernel<<<1, kScanThreads, 0, s>>>(block_sums, nb);
    scan_finish_kernel<<<(unsigned)nb, kScanThreads, 0, s>>>(data, n, block_sums, nb > kScanDirect, copy, big);
    return cudaGetLastError();
}

template <typename Real>
__global__ void sort_scatter_pairs_kernel(const SortArgs<Real> A)
{
    scatter_pairs_block(A, blockIdx.x);
}

template <typename Real>
__global__ void __launch_bounds__(kSegThreads) sort_segments_kernel(const SortArgs<Real> A)
{
    __shared__ int32_t sid[kSegThreads / 32][kSegStage];
    __shared__ int32_t ssrc[kSegThreads / 32][kSegStage];
    segments_block(A, blockIdx.x, sid, ssrc);
}

template <typename Real>
__global__ void __launch_bounds__(kBigThreads) sort_big_segments_kernel(const SortArgs<Real> A)
{
    __shared__ int32_t sid[kBigChunk];
    __shared__ int32_t ssrc[kBigChunk];
    big_segments_block(A, blockIdx.x, gridDim.x, sid, ssrc);
}

// Gather every store column into sorted order (coalesced writes; the
// sources are nearly in order because grains move little between sorts).
template <typename Real>
__global__ void sort_gather_kernel(const SortArgs<Real> A)
{
    const int64_t pos = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (pos >= A.src.n) return;
    const int32_t src = A.pair_src[pos];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        A.dst.q[d][pos] = A.src.q[d][src];
        A.dst.p[d][pos] = A.src.p[d][src];
    }
    A.dst.id[pos] = A.pair_id[pos];
    if (A.src.species) A.dst.species[pos] = A.src.species[src];
    if (A.src.param) A.dst.param[pos] = A.src.param[src];
}

template <typename Real>
cudaError_t launch_sort_scatter(const SortArgs<Real> &a, cudaStream_t s, bool gather)
{
    if (a.src.n == 0) return cudaSuccess;
    const unsigned nb = (unsigned)((a.src.n + 255) / 256);
    const unsigned nbs = (unsigned)((a.src.n + 256 * kScatterItems - 1) / (256 * kScatterItems));
    sort_scatter_pairs_kernel<Real><<<nbs, 256, 0, s>>>(a);
    sort_segments_kernel<Real><<<(unsigned)((a.nkeys1 + kSegThreads - 1) / kSegThreads), kSegThreads, 0, s>>>(a);
    // long segments, if any (the kernel reads their count on the device)
    sort_big_segments_kernel<Real><<<kBigSortBlocks, kBigThreads, 0, s>>>(a);
    if (gather) sort_gather_kernel<Real><<<nb, 256, 0, s>>>(a);
    return cudaGetLastError();
}

template cudaError_t launch_sort_scatter<float>(const SortArgs<float> &, cudaStream_t, bool);
template cudaError_t launch_sort_scatter<double>(const SortArgs<double> &, cudaStream_t, bool);

}  // namespace dust
