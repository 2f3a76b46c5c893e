// Graph pruning on the GPU (the build the paper times in Section 5.7,
// Fig. 16; the graph itself is an input of the search, Section 2.1;
// the kNN lists are knn.cu's):
//
//   ann_graph_prune the detour-count pruning with reverse edges: one warp per
//                   node counts detours with a hash table of its list in
//                   shared memory and orders the list by (detours,
//                   rank); the kept edges' reverse offers are bucketed by
//                   target (count, scan, scatter) and each target takes its
//                   smallest (position, source) offers; one warp per node
//                   assembles the row (kept, reverse, rest; repeats and the
//                   node itself dropped).
#include <algorithm>

#include "ann_internal.cuh"

using namespace ann;

namespace {

// ------------------------------------------------------------ pruning
constexpr uint32_t kEmptySlot = ANN_INVALID_ID;   // never inserted

__device__ __forceinline__ uint32_t table_home(uint32_t x, uint32_t slots)
{
    return (x * 2654435761u) >> (32 - (31 - __clz(slots)));
}

// The (detours, rank) order of a node's list, a warp per node: det holds the
// counts (and is overwritten), mine the lane's entries. Each entry's place is
// the number of smaller keys (detours are below 2^16, so the keys are exact and
// distinct).
template <uint32_t NW>
__device__ __forceinline__ void write_order(uint32_t *det, const uint32_t (&mine)[NW], uint32_t K, uint32_t lane,
                                            uint32_t *__restrict__ out)
{
    __syncwarp();
    uint32_t key[NW], pos[NW];
#pragma unroll
    for (uint32_t i = 0; i < NW; ++i) {
        const uint32_t r = lane + 32 * i;
        key[i] = r < K ? (det[r] << 8) | r : 0xFFFFFFFFu;
        pos[i] = 0;
    }
    __syncwarp();
#pragma unroll
    for (uint32_t i = 0; i < NW; ++i) det[lane + 32 * i] = key[i];
    __syncwarp();
#pragma unroll 2
    for (uint32_t j = 0; j < NW * 32; j += 4) {
        const uint4 k4 = *reinterpret_cast<const uint4 *>(det + j);
#pragma unroll
        for (uint32_t i = 0; i < NW; ++i)
            pos[i] += (k4.x < key[i]) + (k4.y < key[i]) + (k4.z < key[i]) + (k4.w < key[i]);
    }
#pragma unroll
    for (uint32_t i = 0; i < NW; ++i)
        if (lane + 32 * i < K) out[pos[i]] = mine[i];
}

// Detour counts of lists of up to 128 entries. Every entry of every listed
// node's list is looked up in u's own list (K x K lookups a node). The lookup
// is a table of 4,096 ranks in shared memory under a multiplicative hash chosen
// per node so that the list's ids fall into different slots (a random multiplier
// does for 96 ids in one try of three), and a comparison with the id of that
// rank: no probing, so the lanes of a warp never diverge. Eight second-hop
// lists are gathered at once (K x K x 4 bytes a node, half of them from DRAM at
// 500,000 x 96) by one loop over the ranks: unrolled over the lane's NW words as
// well, its code left the instruction cache (128 entries: 8.7 ms against 6.0
// for 300,000 nodes). Measured at 500,000 x 96: a binary search of a sorted copy
// of the list 16.0 ms, linear probing 9.3 ms (40 instructions a lookup: some
// lane always probes on), this 3.9 ms (2, 4, 8 lists at once 5.9, 5.6, 5.5 ms for
// the whole pruning).
constexpr uint32_t kRankSlots = 4096, kNoRank = 128;
constexpr uint32_t kLists = 8;          // second-hop lists gathered at once
constexpr uint32_t kHashTries = 64;   // multipliers tried; a list none of them keeps apart is searched in order

template <uint32_t NW>
__global__ void __launch_bounds__(256) detour_rank_kernel(const uint32_t *__restrict__ knn, uint32_t n, uint32_t K,
                                                          uint32_t *__restrict__ ordered)
{
    static_assert(32 * NW <= kNoRank, "ranks fit below the marker");
    extern __shared__ __align__(16) uint8_t sm[];
    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t u = blockIdx.x * (blockDim.x >> 5) + warp;
    uint8_t *tab = sm + warp * (kRankSlots + 2 * (kNoRank + 4) * 4);   // rank of the id in each slot
    uint32_t *ids = reinterpret_cast<uint32_t *>(tab + kRankSlots);    // by rank; [kNoRank] matches nothing
    uint32_t *det = ids + kNoRank + 4;                                 // counts, [kNoRank] unused
    if (u >= n) return;
    uint4 *t4 = reinterpret_cast<uint4 *>(tab);
    constexpr uint32_t kEmpty4 = kNoRank * 0x01010101u;
    for (uint32_t i = lane; i < kRankSlots / 16; i += 32) t4[i] = make_uint4(kEmpty4, kEmpty4, kEmpty4, kEmpty4);
    uint32_t mine[NW], last[NW];   // last: the largest of the lane's ranks that a lookup must exceed
#pragma unroll
    for (uint32_t i = 0; i < NW; ++i) {
        const uint32_t r = lane + 32 * i;
        mine[i] = r < K ? knn[(size_t)u * K + r] : ANN_INVALID_ID;
        last[i] = r < K ? r : kNoRank;
        det[r] = 0;
        ids[r] = mine[i];
    }
    if (lane == 0) ids[kNoRank] = ANN_INVALID_ID;
    // a multiplier under which no two of the ids share a slot: every id writes
    // its rank and finds it (or an equal id's) again
    uint32_t mul = 2654435761u;
    bool apart = false;
    for (uint32_t attempt = 0; attempt < kHashTries && !apart; ++attempt) {
        uint32_t slot[NW];
#pragma unroll
        for (uint32_t i = 0; i < NW; ++i) {
            slot[i] = (mine[i] * mul) >> 20;
            if (mine[i] != ANN_INVALID_ID) tab[slot[i]] = (uint8_t)(lane + 32 * i);
        }
        __syncwarp();
        bool good = true, repeat = false;
#pragma unroll
        for (uint32_t i = 0; i < NW; ++i)
            if (mine[i] != ANN_INVALID_ID) {
                const uint32_t r = tab[slot[i]];
                good = good && ids[r] == mine[i];
                repeat = repeat || (ids[r] == mine[i] && r != lane + 32 * i);
            }
        __syncwarp();
        apart = __all_sync(0xffffffffu, good);
        if (apart) {
            // repeated ids count at their smallest rank
            if (__any_sync(0xffffffffu, repeat))
                for (uint32_t r = 32 * NW; r-- > 0;) {
                    if (lane == (r & 31u) && ids[r] != ANN_INVALID_ID) tab[(ids[r] * mul) >> 20] = (uint8_t)r;
                    __syncwarp();
                }
        } else {
#pragma unroll
            for (uint32_t i = 0; i < NW; ++i) tab[slot[i]] = kNoRank;
            mul = (mul * 1664525u + 1013904223u) | 1u;
        }
        __syncwarp();
    }
    __syncwarp();
    // entry c of the list of the node ranked p
    auto entry = [&](uint32_t p, uint32_t c) {
        const uint32_t w = ids[p];
        return w < n && lane + 32 * c < K ? __ldg(knn + (size_t)w * K + lane + 32 * c) : ANN_INVALID_ID;
    };
    // an unused slot's rank is the marker: its id matches only an invalid
    // entry, counted where nothing reads
    auto count = [&](uint32_t p, uint32_t c, uint32_t x, uint32_t r) {
        if (ids[r] == x && max(p, last[c]) < r) atomicAdd(&det[r], 1u);
    };
    if (apart) {
        #pragma unroll 1
        for (uint32_t p = 0; p < K; p += kLists) {   // past K the ids are invalid
            uint32_t x[kLists][NW];
#pragma unroll
            for (uint32_t j = 0; j < kLists; ++j)
#pragma unroll
                for (uint32_t c = 0; c < NW; ++c) x[j][c] = entry(p + j, c);
#pragma unroll
            for (uint32_t j = 0; j < kLists; ++j)
#pragma unroll
                for (uint32_t c = 0; c < NW; ++c) count(p + j, c, x[j][c], tab[(x[j][c] * mul) >> 20]);
        }
    } else {
        #pragma unroll 1
        for (uint32_t p = 0; p < K; ++p)
#pragma unroll
            for (uint32_t c = 0; c < NW; ++c) {
                const uint32_t x = entry(p, c);
                uint32_t r = kNoRank;
                #pragma unroll 1
                for (uint32_t k = K; k-- > 0;) r = ids[k] == x && x != ANN_INVALID_ID ? k : r;   // invalid: no edge
                count(p, c, x, r);
            }
    }
    write_order<NW>(det, mine, K, lane, ordered + (size_t)u * K);
}

// The same for longer lists, which a table of ranks cannot keep apart: id ->
// smallest rank by a hash table with linear probing.
template <uint32_t NW>
__global__ void __launch_bounds__(256) detour_order_kernel(const uint32_t *__restrict__ knn, uint32_t n, uint32_t K,
                                                           uint32_t *__restrict__ ordered)
{
    constexpr uint32_t SLOTS = 1024, ROWS = 2;
    extern __shared__ __align__(16) uint8_t sm[];
    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t u = blockIdx.x * (blockDim.x >> 5) + warp;
    uint8_t *base = sm + warp * (SLOTS * 5 + NW * 32 * 4);
    uint32_t *tab = reinterpret_cast<uint32_t *>(base);
    uint32_t *det = tab + SLOTS;                                   // NW x 32: counts, then order keys
    uint8_t *rank = reinterpret_cast<uint8_t *>(det + NW * 32);    // of the slot's entry
    if (u >= n) return;
    for (uint32_t i = lane; i < SLOTS; i += 32) tab[i] = kEmptySlot;
    uint32_t mine[NW];
#pragma unroll
    for (uint32_t i = 0; i < NW; ++i) {
        const uint32_t r = lane + 32 * i;
        mine[i] = r < K ? knn[(size_t)u * K + r] : ANN_INVALID_ID;
        det[r] = 0;
    }
    __syncwarp();
    // entries in rank order; of equal ids the smallest rank is kept
#pragma unroll
    for (uint32_t i = 0; i < NW; ++i) {
        const uint32_t v = mine[i];
        const uint32_t same = __match_any_sync(0xffffffffu, v);
        if (v != ANN_INVALID_ID && (uint32_t)(__ffs(same) - 1) == lane) {
            uint32_t s = table_home(v, SLOTS);
            for (;;) {
                const uint32_t old = atomicCAS(tab + s, kEmptySlot, v);
                if (old == kEmptySlot) { rank[s] = (uint8_t)(lane + 32 * i); break; }
                if (old == v) break;
                s = (s + 1) & (SLOTS - 1);
            }
        }
        __syncwarp();
    }
#pragma unroll
    for (uint32_t i = 0; i < NW; ++i) {
#pragma unroll 1
        for (uint32_t l0 = 0; l0 < 32 && 32 * i + l0 < K; l0 += ROWS) {
            uint32_t x[ROWS][NW];
#pragma unroll
            for (uint32_t j = 0; j < ROWS; ++j) {
                const uint32_t w = __shfl_sync(0xffffffffu, mine[i], l0 + j);   // past K: invalid
#pragma unroll
                for (uint32_t c = 0; c < NW; ++c)
                    x[j][c] = w < n && lane + 32 * c < K ? __ldg(knn + (size_t)w * K + lane + 32 * c) : ANN_INVALID_ID;
            }
#pragma unroll
            for (uint32_t j = 0; j < ROWS; ++j)
#pragma unroll
                for (uint32_t c = 0; c < NW; ++c) {
                    const uint32_t v = x[j][c];
                    uint32_t s = table_home(v, SLOTS), got = tab[s];
                    while (got != v && got != kEmptySlot) {
                        s = (s + 1) & (SLOTS - 1);
                        got = tab[s];
                    }
                    if (got == v && v != ANN_INVALID_ID) {
                        const uint32_t r = rank[s];
                        if (32 * i + l0 + j < r && lane + 32 * c < r) atomicAdd(&det[r], 1u);
                    }
                }
        }
    }
    write_order<NW>(det, mine, K, lane, ordered + (size_t)u * K);
}

cudaError_t launch_detours(const uint32_t *knn, uint32_t n, uint32_t K, uint32_t *ordered, cudaStream_t st)
{
    // blocks of four warps pack 44 of the rank tables on an SM, of eight 40
    auto go = [&](auto kernel, size_t per_warp, uint32_t warps) {
        const uint32_t grid = (n + warps - 1) / warps;
        const size_t smem = warps * per_warp;
        cudaError_t e = raise_shared_limit(kernel, smem);   // each kernel's own constant
        if (e != cudaSuccess) return e;
        kernel<<<grid, warps * 32, smem, st>>>(knn, n, K, ordered);
        return cudaGetLastError();
    };
    constexpr size_t ranks = kRankSlots + 2 * (kNoRank + 4) * 4;
    auto probing = [](uint32_t nw) { return (size_t)1024 * 5 + nw * 32 * 4; };
    switch ((K + 31) / 32) {
    case 1: return go(detour_rank_kernel<1>, ranks, 4);
    case 2: return go(detour_rank_kernel<2>, ranks, 4);
    case 3: return go(detour_rank_kernel<3>, ranks, 4);
    case 4: return go(detour_rank_kernel<4>, ranks, 4);
    case 5: case 6: return go(detour_order_kernel<6>, probing(6), 8);
    default: return go(detour_order_kernel<8>, probing(8), 8);
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

// Row assembly, warp per node v: its nr smallest offers, then kept ++ reverse
// ++ rest with repeats and v dropped, first `degree` entries
// (INVALID-padded). Up to kOfferMax offers (a kept list holds `half` of them on
// average) are ranked by counting in shared memory; a hub's larger bucket by
// repeated warp minima. Repeats are found through a hash table id -> first
// position. (Minima for all and a scan of the earlier entries for each: 1.9 ms
// on 500,000 x 96 lists of degree 64; this 0.74 ms.)
constexpr uint32_t kOfferMax = 96;

__host__ __device__ constexpr uint32_t assemble_slots(uint32_t L) { return L <= 128 ? 512 : 1024; }

__global__ void __launch_bounds__(256) assemble_kernel(const uint32_t *__restrict__ ordered, uint32_t n, uint32_t K,
                                                       uint32_t half, uint32_t degree,
                                                       const uint32_t *__restrict__ off,
                                                       const uint64_t *__restrict__ keys, uint32_t *__restrict__ graph)
{
    extern __shared__ __align__(16) uint8_t sm[];
    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31, warps = blockDim.x >> 5;
    const uint32_t v = blockIdx.x * warps + warp;
    const uint32_t L = K + (degree - half), slots = assemble_slots(L);
    uint64_t *ok = reinterpret_cast<uint64_t *>(sm) + warp * kOfferMax;
    uint2 *tab = reinterpret_cast<uint2 *>(sm + warps * kOfferMax * 8) + warp * slots;   // (id, first position)
    uint32_t *cand = reinterpret_cast<uint32_t *>(sm + warps * (kOfferMax + slots) * 8) + warp * L;
    if (v >= n) return;
    const uint32_t nr = degree - half;
    const uint64_t *kv = keys + off[v];
    const uint32_t nk = off[v + 1] - off[v];
    for (uint32_t i = lane; i < slots; i += 32) tab[i] = make_uint2(kEmptySlot, 0xFFFFFFFFu);
    for (uint32_t j = lane; j < half; j += 32) cand[j] = ordered[(size_t)v * K + j];
    const uint32_t nrev = min(nk, nr);
    for (uint32_t j = lane; j < K - half; j += 32) cand[half + nrev + j] = ordered[(size_t)v * K + half + j];
    if (nk <= kOfferMax) {
        for (uint32_t j = lane; j < nk; j += 32) ok[j] = kv[j];
        __syncwarp();
        for (uint32_t j = lane; j < nk; j += 32) {
            const uint64_t k = ok[j];
            uint32_t r = 0;
#pragma unroll 4
            for (uint32_t i = 0; i < nk; ++i) r += ok[i] < k ? 1u : 0u;   // keys are distinct
            if (r < nr) cand[half + r] = (uint32_t)k;
        }
    } else {
        uint64_t last = 0;
        for (uint32_t taken = 0; taken < nr; ++taken) {
            uint64_t best = ~0ull;
            for (uint32_t j = lane; j < nk; j += 32) {
                const uint64_t k = kv[j];
                if ((taken == 0 || k > last) && k < best) best = k;
            }
            for (int o = 16; o; o >>= 1) {
                const uint64_t other = __shfl_xor_sync(0xffffffffu, best, o);
                best = other < best ? other : best;
            }
            if (lane == 0) cand[half + taken] = (uint32_t)best;
            last = best;
        }
    }
    __syncwarp();
    const uint32_t total = half + nrev + (K - half);
    for (uint32_t j = lane; j < total; j += 32) {
        const uint32_t x = cand[j];
        if (x >= n || x == v) continue;
        uint32_t s = table_home(x, slots);
        for (;;) {
            const uint32_t old = atomicCAS(&tab[s].x, kEmptySlot, x);
            if (old == kEmptySlot || old == x) break;
            s = (s + 1) & (slots - 1);
        }
        atomicMin(&tab[s].y, j);
    }
    __syncwarp();
    uint32_t written = 0;
    for (uint32_t b = 0; b < total && written < degree; b += 32) {
        const uint32_t j = b + lane;
        bool keep = false;
        uint32_t x = ANN_INVALID_ID;
        if (j < total) {
            x = cand[j];
            if (x < n && x != v) {
                uint32_t s = table_home(x, slots);
                while (tab[s].x != x) s = (s + 1) & (slots - 1);
                keep = tab[s].y == j;
            }
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
    // one allocation: the ordered lists, the offer buckets and their offsets
    size_t bytes = 0;
    auto take = [&](size_t b) {
        const size_t at = bytes;
        bytes += (b + 255) & ~(size_t)255;
        return at;
    };
    const size_t o_cnt = take((size_t)n * 4), o_cur = take((size_t)n * 4), zeroed = bytes;
    const size_t o_ord = take((size_t)n * K * 4), o_off = take((size_t)(n + 1) * 4), o_sums = take((size_t)nb * 4);
    const size_t o_keys = take((size_t)n * std::max(1u, half) * 8);
    uint8_t *ws = nullptr;
    cudaError_t e = cudaMalloc((void **)&ws, bytes);
    uint32_t *ordered = reinterpret_cast<uint32_t *>(ws + o_ord), *cnt = reinterpret_cast<uint32_t *>(ws + o_cnt);
    uint32_t *off = reinterpret_cast<uint32_t *>(ws + o_off), *sums = reinterpret_cast<uint32_t *>(ws + o_sums);
    uint32_t *cursor = reinterpret_cast<uint32_t *>(ws + o_cur);
    uint64_t *keys = reinterpret_cast<uint64_t *>(ws + o_keys);
    if (e == cudaSuccess) e = cudaMemsetAsync(ws, 0, zeroed, st);
    const uint32_t L = K + (degree - half);
    constexpr int wpb = 8;
    constexpr auto asm_bytes = [](uint32_t len) { return wpb * ((kOfferMax + assemble_slots(len)) * 8 + (size_t)len * 4); };
    const size_t asm_smem = asm_bytes(L);
    if (e == cudaSuccess)
        e = raise_shared_limit(assemble_kernel, asm_bytes(2 * ANN_MAX_DEGREE + (ANN_MAX_DEGREE + 1) / 2));
    if (e == cudaSuccess) e = launch_detours(knn, nn, K, ordered, st);
    if (e == cudaSuccess) {
        offer_count_kernel<<<grid_for((uint64_t)n * half, 256), 256, 0, st>>>(ordered, nn, K, half, cnt);
        scan_block_kernel<<<nb, 1024, 0, st>>>(cnt, nn, off, sums);
        scan_sums_kernel<<<1, 32, 0, st>>>(sums, nb, off + nn);
        scan_add_kernel<<<nb, 1024, 0, st>>>(off, nn, sums);
        offer_scatter_kernel<<<grid_for((uint64_t)n * half, 256), 256, 0, st>>>(ordered, nn, K, half, off, cursor,
                                                                                keys);
        assemble_kernel<<<grid_for(n, wpb), wpb * 32, asm_smem, st>>>(ordered, nn, K, half, degree, off, keys, graph);
        e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    }
    cudaFree(ws);
    return e == cudaSuccess ? ANN_OK : cuda_fail(e, "ann_graph_prune");
}

}  // extern "C"
