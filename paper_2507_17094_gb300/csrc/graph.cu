// Graph pruning on the GPU (the build the paper times in Section 5.7,
// Fig. 16; the graph itself is an input of the search, Section 2.1;
// the kNN lists are knn.cu's):
//
//   ann_graph_prune the detour-count pruning with reverse edges: one warp per
//                   node counts detours with a sorted (id, rank) table of its
//                   list in shared memory and orders the list by (detours,
//                   rank); the kept edges' reverse offers are bucketed by
//                   target (count, scan, scatter) and each target takes its
//                   smallest (position, source) offers; one warp per node
//                   assembles the row (kept, reverse, rest; repeats and the
//                   node itself dropped).
#include <algorithm>
#include <vector>

#include "ann_internal.cuh"

using namespace ann;

namespace {

// ------------------------------------------------------------ pruning
// Detour counts and the (detours, rank) order of node u's list: warp per
// node, dynamic shared memory per warp: ids sorted by (id, rank) with their
// ranks (K x 8 bytes) and the counts (K x 4).
__global__ void detour_order_kernel(const uint32_t *__restrict__ knn, uint32_t n, uint32_t K,
                                    uint32_t *__restrict__ ordered)
{
    extern __shared__ __align__(16) uint8_t sm[];
    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t u = blockIdx.x * (blockDim.x >> 5) + warp;
    uint32_t *sid = reinterpret_cast<uint32_t *>(sm) + warp * 3 * K;   // sorted ids
    uint32_t *srk = sid + K;                                            // their ranks
    uint32_t *det = srk + K;
    if (u >= n) return;
    const uint32_t *N = knn + (size_t)u * K;
    // sort (id, rank) by rank counting (K <= ANN_MAX_DEGREE * 2)
    for (uint32_t r = lane; r < K; r += 32) {
        const uint32_t v = N[r];
        uint32_t pos = 0;
        for (uint32_t r2 = 0; r2 < K; ++r2) {
            const uint32_t w = N[r2];
            pos += (w < v || (w == v && r2 < r)) ? 1u : 0u;
        }
        sid[pos] = v;
        srk[pos] = r;
        det[r] = 0;
    }
    __syncwarp();
    for (uint32_t a = 0; a < K; ++a) {
        const uint32_t w = N[a];
        if (w == ANN_INVALID_ID || w >= n) continue;
        for (uint32_t c = lane; c < K; c += 32) {
            const uint32_t x = knn[(size_t)w * K + c];
            // lower bound of x among the sorted ids: its smallest rank
            uint32_t lo = 0, hi = K;
            while (lo < hi) {
                const uint32_t mid = (lo + hi) >> 1;
                if (sid[mid] < x) lo = mid + 1;
                else hi = mid;
            }
            if (lo < K && sid[lo] == x && x != ANN_INVALID_ID) {
                const uint32_t r = srk[lo];
                if (a < r && c < r) atomicAdd(&det[r], 1u);
            }
        }
    }
    __syncwarp();
    for (uint32_t r = lane; r < K; r += 32) {
        const uint32_t dr = det[r];
        uint32_t pos = 0;
        for (uint32_t r2 = 0; r2 < K; ++r2) {
            const uint32_t d2 = det[r2];
            pos += (d2 < dr || (d2 == dr && r2 < r)) ? 1u : 0u;
        }
        ordered[(size_t)u * K + pos] = N[r];
    }
}

// Reverse offers of the kept edges: count per target.
__global__ void offer_count_kernel(const uint32_t *__restrict__ ordered, uint32_t n, uint32_t K, uint32_t half,
                                   uint32_t *__restrict__ cnt)
{
    const uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
    if (i >= (uint64_t)n * half) return;
    const uint32_t w = (uint32_t)(i / half), p = (uint32_t)(i % half);
    const uint32_t v = ordered[(size_t)w * K + p];
    if (v < n) atomicAdd(&cnt[v], 1u);
}

// Exclusive scan of `cnt` (n) into off (n + 1): per-block scans, then a scan
// of the block sums (one block, looping), then the block offsets added.
__global__ void scan_block_kernel(const uint32_t *__restrict__ in, uint32_t n, uint32_t *__restrict__ out,
                                  uint32_t *__restrict__ block_sums)
{
    __shared__ uint32_t wsum[32];
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t v = i < n ? in[i] : 0u;
    uint32_t x = v;
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= (uint32_t)o) x += y;
    }
    if (lane == 31) wsum[warp] = x;
    __syncthreads();
    if (warp == 0) {
        uint32_t s = lane < (blockDim.x >> 5) ? wsum[lane] : 0u;
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= (uint32_t)o) s += y;
        }
        wsum[lane] = s;
    }
    __syncthreads();
    const uint32_t incl = x + (warp ? wsum[warp - 1] : 0u);
    if (i < n) out[i] = incl - v;
    if (threadIdx.x == blockDim.x - 1) block_sums[blockIdx.x] = incl;
}

__global__ void scan_sums_kernel(uint32_t *__restrict__ sums, uint32_t nb, uint32_t *__restrict__ total)
{
    if (threadIdx.x == 0) {
        uint32_t s = 0;
        for (uint32_t b = 0; b < nb; ++b) {
            const uint32_t v = sums[b];
            sums[b] = s;
            s += v;
        }
        *total = s;
    }
}

__global__ void scan_add_kernel(uint32_t *__restrict__ out, uint32_t n, const uint32_t *__restrict__ sums)
{
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] += sums[blockIdx.x];
}

// Offers bucketed by target: key (position p in the source's kept list,
// source w) as one 64-bit word (p high), at an atomically claimed slot.
__global__ void offer_scatter_kernel(const uint32_t *__restrict__ ordered, uint32_t n, uint32_t K, uint32_t half,
                                     const uint32_t *__restrict__ off, uint32_t *__restrict__ cursor,
                                     uint64_t *__restrict__ keys)
{
    const uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
    if (i >= (uint64_t)n * half) return;
    const uint32_t w = (uint32_t)(i / half), p = (uint32_t)(i % half);
    const uint32_t v = ordered[(size_t)w * K + p];
    if (v < n) keys[off[v] + atomicAdd(&cursor[v], 1u)] = ((uint64_t)p << 32) | w;
}

// Row assembly, warp per node v: its nr smallest offers (repeated warp
// minima over its bucket), then kept ++ reverse ++ rest with repeats and v
// dropped, first `degree` entries (INVALID-padded).
__global__ void assemble_kernel(const uint32_t *__restrict__ ordered, uint32_t n, uint32_t K, uint32_t half,
                                uint32_t degree, const uint32_t *__restrict__ off, const uint64_t *__restrict__ keys,
                                uint32_t *__restrict__ graph)
{
    extern __shared__ __align__(16) uint8_t sm[];
    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t v = blockIdx.x * (blockDim.x >> 5) + warp;
    const uint32_t L = K + (degree - half);
    uint32_t *cand = reinterpret_cast<uint32_t *>(sm) + warp * L;
    if (v >= n) return;
    const uint32_t nr = degree - half;
    for (uint32_t j = lane; j < half; j += 32) cand[j] = ordered[(size_t)v * K + j];
    const uint64_t *kv = keys + off[v];
    const uint32_t nk = off[v + 1] - off[v];
    uint64_t last = 0;
    bool have_last = false;
    uint32_t taken = 0;
    for (; taken < nr; ++taken) {
        uint64_t best = ~0ull;
        for (uint32_t j = lane; j < nk; j += 32) {
            const uint64_t k = kv[j];
            if ((!have_last || k > last) && k < best) best = k;
        }
        for (int o = 16; o; o >>= 1) {
            const uint64_t other = __shfl_xor_sync(0xffffffffu, best, o);
            best = other < best ? other : best;
        }
        if (best == ~0ull) break;
        if (lane == 0) cand[half + taken] = (uint32_t)best;
        last = best;
        have_last = true;
    }
    const uint32_t nrev = taken;
    for (uint32_t j = lane; j < K - half; j += 32) cand[half + nrev + j] = ordered[(size_t)v * K + half + j];
    __syncwarp();
    const uint32_t total = half + nrev + (K - half);
    uint32_t written = 0;
    for (uint32_t b = 0; b < total && written < degree; b += 32) {
        const uint32_t j = b + lane;
        bool keep = false;
        uint32_t x = ANN_INVALID_ID;
        if (j < total) {
            x = cand[j];
            keep = x < n && x != v;
            for (uint32_t t = 0; t < j && keep; ++t) keep = cand[t] != x;
        }
        const uint32_t m = __ballot_sync(0xffffffffu, keep);
        const uint32_t at = written + __popc(m & ((1u << lane) - 1u));
        if (keep && at < degree) graph[(size_t)v * degree + at] = x;
        written += __popc(m);
    }
    for (uint32_t j = written + lane; j < degree; j += 32) graph[(size_t)v * degree + j] = ANN_INVALID_ID;
}

int grid_for(uint64_t n, int threads) { return (int)std::max<uint64_t>(1, (n + threads - 1) / threads); }

}  // namespace

extern "C" {

ann_status ann_graph_prune(const uint32_t *knn, uint64_t n, uint32_t K, uint32_t degree, uint32_t *graph,
                           void *stream)
{
    if (!knn || !graph || n == 0 || n > 0xFFFFFFFEull || K == 0 || K > 2 * ANN_MAX_DEGREE || degree == 0 ||
        degree > K || degree > ANN_MAX_DEGREE) {
        set_error("ann_graph_prune: need n >= 1, 1 <= degree <= min(K, %u), K <= %u", ANN_MAX_DEGREE,
                  2 * ANN_MAX_DEGREE);
        return ANN_EINVAL;
    }
    cudaStream_t st = (cudaStream_t)stream;
    const uint32_t nn = (uint32_t)n, half = degree / 2;
    const uint32_t nb = (nn + 1023) / 1024;
    uint32_t *ordered = nullptr, *cnt = nullptr, *off = nullptr, *sums = nullptr, *cursor = nullptr;
    uint64_t *keys = nullptr;
    cudaError_t e = cudaMalloc(&ordered, (size_t)n * K * 4);
    if (e == cudaSuccess) e = cudaMalloc(&cnt, (size_t)n * 4);
    if (e == cudaSuccess) e = cudaMalloc(&off, (size_t)(n + 1) * 4);
    if (e == cudaSuccess) e = cudaMalloc(&sums, (size_t)nb * 4);
    if (e == cudaSuccess) e = cudaMalloc(&cursor, (size_t)n * 4);
    if (e == cudaSuccess) e = cudaMalloc(&keys, (size_t)n * std::max(1u, half) * 8);
    if (e == cudaSuccess) e = cudaMemsetAsync(cnt, 0, (size_t)n * 4, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(cursor, 0, (size_t)n * 4, st);
    if (e == cudaSuccess) {
        const int wpb = 8;
        detour_order_kernel<<<grid_for(n, wpb), wpb * 32, (size_t)wpb * 3 * K * 4, st>>>(knn, nn, K, ordered);
        offer_count_kernel<<<grid_for((uint64_t)n * half, 256), 256, 0, st>>>(ordered, nn, K, half, cnt);
        scan_block_kernel<<<nb, 1024, 0, st>>>(cnt, nn, off, sums);
        scan_sums_kernel<<<1, 32, 0, st>>>(sums, nb, off + nn);
        scan_add_kernel<<<nb, 1024, 0, st>>>(off, nn, sums);
        offer_scatter_kernel<<<grid_for((uint64_t)n * half, 256), 256, 0, st>>>(ordered, nn, K, half, off, cursor,
                                                                                keys);
        const uint32_t L = K + (degree - half);
        assemble_kernel<<<grid_for(n, wpb), wpb * 32, (size_t)wpb * L * 4, st>>>(ordered, nn, K, half, degree, off,
                                                                               keys, graph);
        e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    }
    cudaFree(ordered);
    cudaFree(cnt);
    cudaFree(off);
    cudaFree(sums);
    cudaFree(cursor);
    cudaFree(keys);
    return e == cudaSuccess ? ANN_OK : cuda_fail(e, "ann_graph_prune");
}

}  // extern "C"
