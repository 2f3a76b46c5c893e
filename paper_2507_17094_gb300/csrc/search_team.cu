// The search of small batches: a thread block (a team) per query, where the
// warp kernel of search.cu gives a query one warp.
//
// A query is a chain of dependent iterations, each two rounds of gathers (the
// parents' lists, the neighbours' rows) and the work between them. With
// thousands of queries in flight other warps fill the time a gather takes;
// with a few hundred or fewer the length of the chain is the call's time (one
// query, 300,000 x 96 FP16, itopk 64: 13,100 clocks an iteration in the warp
// kernel, of which the two gathers need some 1,500). Here the work between the
// gathers is spread over a block and its latencies are cut:
//   - the visited set is the warp kernel's table (same size, hash and reset
//     rule), but in shared memory: two global atomics in a row cost 3,500
//     clocks an iteration;
//   - a thread per neighbour loads its id and direction words straight into
//     registers; the rows come by 16-byte asynchronous copies of all threads (a
//     bulk copy per row is issued one lane after the other: 1,450 clocks for
//     an iteration's rows, measured);
//   - four lanes rank a neighbour or compute a row's distance, all rows of an
//     iteration at once where they fit, and a thread per candidate and per
//     queue entry merges;
//   - queue and candidates are 64-bit keys (distance bits, id), which compare
//     as integers; every warp selects the parents for itself.
// The operations on each distance, the order of the queue, the seeds, the
// termination and the counters are those of the warp kernel, so results and
// counters are the same. Measured, us a call, warps / teams: one query of FP16
// 96-d rows with rerank, itopk 64: 477 / 228; 61 queries of E4M3 128-d rows:
// 586 / 304; 152 queries of FP32 256-d rows, itopk 256: 3,294 / 1,239. Nothing
// here waits on a barrier that a copy completes, so there is no time-out to
// report.
#include <algorithm>

#include "search_common.cuh"

using namespace ann;

namespace {

constexpr uint32_t kTableBits = kVisitedBits;
constexpr uint32_t kDirWords = 8;   // direction words of a neighbour held in registers

struct TeamLayout {  // byte offsets in the team's shared memory
    uint32_t q, qk, bs, ck, ci, pos, adj, score, sign, misc, table, bits, stage, total;
};

struct TeamArgs {
    TeamSearch t;
    TeamLayout lay;
    uint32_t rows, stride, rr_rows, rr_stride;   // rows per gather round and their stride: stored rows, FP32 rerank
    uint32_t q_part;                             // floats between the parts of the query
    uint32_t row_magic, row32_magic;             // ceil(2^32 / 16-byte chunks of a row): chunk index -> row
};

// Shared counters: the candidates found and the survivors of a loop pass,
// double-buffered (a pass resets the other pass's pair).
struct Misc {
    uint32_t nc[2], ns[2];
};

__device__ __forceinline__ void copy16(void *dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}

__device__ __forceinline__ void copies_done()
{
    asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
}

template <int ST, int NT>
struct Team {
    static constexpr uint32_t kWarps = NT / 32, kQuads = NT / 4, kEntries = ANN_MAX_ITOPK / NT;
    const TeamArgs &g;
    const TeamSearch &a;
    uint8_t *base;
    uint32_t tid, lane, warp;
    uint32_t cnt = 0, hash_count = 0, par = 0;
    bool gbm = false;
    uint64_t qid = 0;
    ann_query_stats st;

    __device__ Team(const TeamArgs &args, uint8_t *b)
        : g(args), a(args.t), base(b), tid(threadIdx.x), lane(threadIdx.x & 31), warp(threadIdx.x >> 5)
    {
    }

    // the query, in the layout of query_pos for four lanes per row
    __device__ __forceinline__ float *q() const { return reinterpret_cast<float *>(base + g.lay.q); }
    __device__ __forceinline__ uint64_t *qk() const { return reinterpret_cast<uint64_t *>(base + g.lay.qk); }
    __device__ __forceinline__ uint8_t *bs() const { return base + g.lay.bs; }
    __device__ __forceinline__ uint64_t *ck() const { return reinterpret_cast<uint64_t *>(base + g.lay.ck); }
    __device__ __forceinline__ uint32_t *ci() const { return reinterpret_cast<uint32_t *>(base + g.lay.ci); }
    __device__ __forceinline__ uint32_t *pos() const { return reinterpret_cast<uint32_t *>(base + g.lay.pos); }
    __device__ __forceinline__ uint32_t *adj() const { return reinterpret_cast<uint32_t *>(base + g.lay.adj); }
    __device__ __forceinline__ uint32_t *score() const { return reinterpret_cast<uint32_t *>(base + g.lay.score); }
    __device__ __forceinline__ uint32_t *sign() const { return reinterpret_cast<uint32_t *>(base + g.lay.sign); }
    __device__ __forceinline__ Misc &misc() const { return *reinterpret_cast<Misc *>(base + g.lay.misc); }
    __device__ __forceinline__ uint32_t *table() const { return reinterpret_cast<uint32_t *>(base + g.lay.table); }
    __device__ __forceinline__ uint32_t *gbits() const { return reinterpret_cast<uint32_t *>(base + g.lay.bits); }
    __device__ __forceinline__ uint8_t *stage() const { return base + g.lay.stage; }

    static __device__ __forceinline__ uint64_t make_key(float d, uint32_t id)
    {
        return ((uint64_t)__float_as_uint(d) << 32) | id;
    }
    static __device__ __forceinline__ float key_dist(uint64_t k) { return __uint_as_float((uint32_t)(k >> 32)); }

    // ---------------------------------------------------------- visited set
    __device__ __forceinline__ bool hash_insert(uint32_t v)
    {
        if (gbm) {
            const uint32_t bit = 1u << (v & 31);
            return (atomicOr(gbits() + (v >> 5), bit) & bit) == 0;
        }
        uint32_t s = (v * 2654435761u) >> (32 - kTableBits);
        #pragma unroll 1
        for (uint32_t probe = 0; probe < (1u << kTableBits); ++probe) {   // never more than half full
            const uint32_t old = atomicCAS(table() + s, 0u, v + 1);
            if (old == 0) return true;
            if (old == v + 1) return false;
            s = (s + 1) & ((1u << kTableBits) - 1);
        }
        return true;
    }

    // An empty set; the caller's next barrier makes it visible.
    __device__ void hash_clear()
    {
        if (gbm) {
            for (uint32_t i = tid; i < a.gbm_words; i += NT) gbits()[i] = 0;
        } else {
            uint4 *t4 = reinterpret_cast<uint4 *>(table());
            for (uint32_t i = tid; i < (1u << kTableBits) / 4; i += NT) t4[i] = make_uint4(0, 0, 0, 0);
        }
        hash_count = 0;
    }

    // Clear the table and insert the queue's ids (no other use of the table
    // may be pending; ends with a barrier).
    __device__ void hash_refill()
    {
        hash_clear();
        __syncthreads();
        for (uint32_t i = tid; i < cnt; i += NT) hash_insert((uint32_t)qk()[i]);
        __syncthreads();
        hash_count = cnt;
    }

    __device__ __forceinline__ void hash_make_room(uint32_t incoming)
    {
        if (!gbm && hash_count + incoming > (1u << (kTableBits - 1))) {
            hash_refill();
            st.hash_resets++;
        }
    }

    // Append the warp's new ids to the candidate list.
    __device__ __forceinline__ void collect(bool valid, uint32_t v)
    {
        const bool isnew = valid && hash_insert(v);
        const uint32_t m = __ballot_sync(0xffffffffu, isnew);
        if (!m) return;
        uint32_t at = 0;
        if (lane == 0) at = atomicAdd(&misc().nc[par], __popc(m));
        at = __shfl_sync(0xffffffffu, at, 0) + __popc(m & lanemask_lt());
        if (isnew) ci()[at] = v;
    }

    // ----------------------------------------------------- evaluate rows
    // Distances of rows id(0 .. n) of `codes`, R (<= 2 kQuads) per gather
    // round, handed to out(i, distance) by one lane each. The caller's
    // barrier precedes (ids visible, staging area free).
    template <int RST, typename Id, typename Out>
    __device__ __forceinline__ void evaluate(const uint8_t *codes, const float *scales, uint32_t row_bytes,
                                             uint32_t magic, uint32_t n, uint32_t R, uint32_t stride, Id id, Out out)
    {
        const uint32_t quad = tid >> 2, chunks = row_bytes >> 4;
        const float *qj = q() + (lane & 3) * g.q_part;
        #pragma unroll 1
        for (uint32_t b0 = 0; b0 < n; b0 += R) {
            const uint32_t rows = min(R, n - b0);
            if (b0) __syncthreads();
            #pragma unroll 2
            for (uint32_t c = tid; c < rows * chunks; c += NT) {
                const uint32_t r = chunks > 1 ? __umulhi(c, magic) : c, off = (c - r * chunks) * 16;
                copy16(stage() + r * stride + off, codes + (uint64_t)id(b0 + r) * row_bytes + off);
            }
            float s0 = 1.0f, s1 = 1.0f;
            if (RST != ANN_F32) {
                if (quad < rows) s0 = __ldg(scales + id(b0 + quad));
                if (quad + kQuads < rows) s1 = __ldg(scales + id(b0 + quad + kQuads));
            }
            copies_done();
            __syncthreads();
            #pragma unroll 1
            for (uint32_t r = quad; r - quad < rows; r += kQuads, s0 = s1) {
                float part = 0.0f;
                if (r < rows) part = row_dist_quarter<RST>(stage() + r * stride, qj, s0, a.d, lane & 3);
                part = __fadd_rn(part, __shfl_xor_sync(0xffffffffu, part, 1));
                part = __fadd_rn(part, __shfl_xor_sync(0xffffffffu, part, 2));
                if (r < rows && (lane & 3) == 0) out(b0 + r, part);
            }
        }
    }

    // --------------------------------------------------------------- merge
    // Merge the ns candidate keys into the queue, keeping the first lcap. A
    // candidate's slot is its rank among the candidates plus its insertion
    // point, an entry moves by the candidates before it; everything is read
    // before the barrier and written after it. The last warps take the
    // candidates, the first ones the entries.
    __device__ __forceinline__ void merge(uint32_t ns, uint32_t lcap)
    {
        uint64_t key[kEntries];
        uint32_t to[kEntries], state[kEntries];
#pragma unroll
        for (uint32_t e = 0; e < kEntries; ++e) {
            const uint32_t i = tid + e * NT;
            key[e] = 0;
            to[e] = i;
            state[e] = 0;
            if (i < cnt) {
                key[e] = qk()[i];
                state[e] = bs()[i];
#pragma unroll 4
                for (uint32_t c = 0; c < ns; ++c) to[e] += ck()[c] < key[e] ? 1u : 0u;
            }
        }
        for (uint32_t c = NT - 1 - tid; c < ns; c += NT) {
            const uint64_t k = ck()[c];
            uint32_t r = 0;
#pragma unroll 4
            for (uint32_t c2 = 0; c2 < ns; ++c2) r += ck()[c2] < k ? 1u : 0u;
            uint32_t lo = 0, hi = cnt;
            while (lo < hi) {
                const uint32_t mid = (lo + hi) >> 1;
                if (qk()[mid] < k) lo = mid + 1;
                else hi = mid;
            }
            pos()[c] = lo + r;
        }
        __syncthreads();
#pragma unroll
        for (uint32_t e = 0; e < kEntries; ++e) {
            const uint32_t i = tid + e * NT;
            if (i < cnt && to[e] != i && to[e] < lcap) {
                qk()[to[e]] = key[e];
                bs()[to[e]] = (uint8_t)state[e];
            }
        }
        for (uint32_t c = NT - 1 - tid; c < ns; c += NT) {
            const uint32_t p = pos()[c];
            if (p < lcap) {
                qk()[p] = ck()[c];
                bs()[p] = kUnexpanded;
            }
        }
        cnt = min(lcap, cnt + ns);
        __syncthreads();
    }

    // ---------------------------------------------------------- iterations
    // The first W eligible queue entries in queue order, by every warp for
    // itself; lane i holds parent i's queue slot.
    __device__ __forceinline__ uint32_t select_parents(uint32_t W, bool cool, uint32_t &slot)
    {
        uint32_t np = 0;
        if (W == 1) {   // four entries' states a lane
            #pragma unroll 1
            for (uint32_t b = 0; b < cnt; b += 128) {
                const uint32_t i = b + 4 * lane;
                uint32_t e = 0;
                if (i < cnt) {
                    const uint32_t s = *reinterpret_cast<const uint32_t *>(bs() + i);
                    e = __vcmpeq4(s, kUnexpanded * 0x01010101u);
                    if (cool) e |= __vcmpeq4(s, kPartial * 0x01010101u);
                    if (cnt - i < 4) e &= (1u << (8 * (cnt - i))) - 1u;
                }
                const uint32_t m = __ballot_sync(0xffffffffu, e != 0);
                if (m) {
                    const uint32_t src = __ffs(m) - 1;
                    slot = b + 4 * src + ((__ffs(__shfl_sync(0xffffffffu, e, src)) - 1) >> 3);
                    return 1;
                }
            }
            return 0;
        }
        #pragma unroll 1
        for (uint32_t b = 0; b < cnt && np < W; b += 32) {
            const uint32_t i = b + lane;
            bool e = false;
            if (i < cnt) {
                const uint32_t s = bs()[i];
                e = s == kUnexpanded || (cool && s == kPartial);
            }
            uint32_t m = __ballot_sync(0xffffffffu, e);
            while (m && np < W) {
                const uint32_t bit = __ffs(m) - 1;
                m &= m - 1;
                if (lane == np) slot = b + bit;
                ++np;
            }
        }
        return np;
    }

    __device__ bool any_partial()
    {
        bool p = false;
        for (uint32_t i = lane; i < cnt; i += 32) p |= bs()[i] == kPartial;
        return __any_sync(0xffffffffu, p);
    }

    // Direction-guided selection of np parents' neighbours (lane i of every
    // warp holds parent i's id) and the visited test of the kept ones. Scores
    // are keys (score + 2) << 8 | (255 - slot), which order by (score, earlier
    // slot): score + 2 is 1 for an empty slot, 0 past the degree (never kept).
    __device__ __forceinline__ void guided(const View &v, uint32_t np, uint32_t pid, uint32_t n_keep,
                                           uint32_t min_match)
    {
        const uint32_t deg = v.deg, dp = v.deg_pad, w = a.w, slots = np * dp;
        // a thread's neighbour: its id and first direction words, in flight
        // while the signs are formed
        uint32_t x = tid, nb = ANN_INVALID_ID, p = 0, j = 0;
        const uint32_t *dw = v.dir;
        uint32_t word[kDirWords];
        auto load = [&]() {
            p = __umulhi(x, v.deg_magic);
            j = x - p * dp;
            const uint64_t parent = __shfl_sync(0xffffffffu, pid, min(p, np - 1));
            if (x < slots) {
                const uint64_t at = parent * dp + j;
                nb = __ldg(v.graph + at);
                dw = v.dir + at * w;
                if (w % 4 == 0) {
#pragma unroll
                    for (uint32_t t = 0; t < kDirWords; t += 4)
                        if (t < w) {
                            const uint4 d4 = __ldg(reinterpret_cast<const uint4 *>(dw + t));
                            word[t] = d4.x; word[t + 1] = d4.y; word[t + 2] = d4.z; word[t + 3] = d4.w;
                        }
                } else {
#pragma unroll
                    for (uint32_t t = 0; t < kDirWords; ++t)
                        if (t < w) word[t] = __ldg(dw + t);
                }
            }
        };
        load();
        // the query's sign bits relative to each parent, a warp per 32 dimensions
        #pragma unroll 2
        for (uint32_t y = warp; y < np * w; y += kWarps) {
            const uint32_t pp = np == 1 ? 0 : y / w, i = 32 * (y - pp * w) + lane;
            const uint32_t parent = __shfl_sync(0xffffffffu, pid, pp);
            const float ps = ST != ANN_F32 ? __ldg(v.scales + parent) : 1.0f;
            bool b = false;
            if (i < a.d)
                b = q()[query_pos<4>(i, g.q_part)] > stored_elem<ST>(v.codes + (uint64_t)parent * v.row_bytes, i, ps);
            const uint32_t bits = __ballot_sync(0xffffffffu, b);
            if (lane == 0) sign()[y] = bits;
        }
        __syncthreads();
        for (;;) {
            if (x < slots) {
                const uint32_t *sw = sign() + p * w;
                uint32_t diff = 0;
#pragma unroll
                for (uint32_t t = 0; t < kDirWords; ++t)
                    if (t < w) diff += __popc(word[t] ^ sw[t]);
                if (w % 4 == 0) {
                    #pragma unroll 2
                    for (uint32_t t = kDirWords; t < w; t += 4) {
                        const uint4 d4 = __ldg(reinterpret_cast<const uint4 *>(dw + t));
                        diff += __popc(d4.x ^ sw[t]) + __popc(d4.y ^ sw[t + 1]) + __popc(d4.z ^ sw[t + 2]) +
                                __popc(d4.w ^ sw[t + 3]);
                    }
                } else {
                    #pragma unroll 4
                    for (uint32_t t = kDirWords; t < w; ++t) diff += __popc(__ldg(dw + t) ^ sw[t]);
                }
                const uint32_t u = j >= deg ? 0u : nb != ANN_INVALID_ID ? a.d + 2 - diff : 1u;
                score()[x] = (u << 8) | (255u - j);
                adj()[x] = nb;
            }
            if (x - tid + NT >= slots) break;
            x += NT;
            load();
        }
        __syncthreads();
        if (min_match > 0) {
            #pragma unroll 1
            for (uint32_t b = warp * 32; b < slots; b += NT) {
                const uint32_t y = b + lane;
                const uint32_t n = y < slots ? adj()[y] : ANN_INVALID_ID;
                collect(n != ANN_INVALID_ID && (score()[min(y, slots - 1)] >> 8) >= min_match + 2, n);
            }
            return;
        }
        // kept: fewer than n_keep of the parent's scores are larger; four lanes count
        #pragma unroll 1
        for (uint32_t b = warp * 8; b < slots; b += kQuads) {
            const uint32_t y = b + (lane >> 2);
            uint32_t n = ANN_INVALID_ID, better = 0;
            if (y < slots) {
                const uint32_t pp = __umulhi(y, v.deg_magic), mine = score()[y];
                n = adj()[y];
                const uint4 *s4 = reinterpret_cast<const uint4 *>(score() + pp * dp);
#pragma unroll 4
                for (uint32_t t = lane & 3; t < dp / 4; t += 4) {
                    const uint4 o = s4[t];
                    better += (o.x > mine) + (o.y > mine) + (o.z > mine) + (o.w > mine);
                }
            }
            better += __shfl_xor_sync(0xffffffffu, better, 1);
            better += __shfl_xor_sync(0xffffffffu, better, 2);
            // past the degree the list holds no ids
            collect((lane & 3) == 0 && n != ANN_INVALID_ID && better < n_keep, n);
        }
    }

    // Seeds, then iterations of parents, adjacency, direction-guided
    // selection, visited test, distances and merge (the warp kernel's
    // iterate, whose comments give the passages).
    __device__ __forceinline__ void iterate(const View &v, const uint32_t *seed_ids, uint32_t m,
                                            uint64_t seed_key, uint32_t lcap, uint32_t W, uint32_t T, uint32_t T_ext,
                                            float judge, uint32_t n_keep, uint32_t min_match, uint32_t it_cool,
                                            uint32_t reexpand, uint32_t &c_iters, uint32_t &c_parents,
                                            uint32_t &c_dgs, uint32_t &c_rows)
    {
        const uint32_t deg = v.deg;
        const bool dgs_on = v.dir != nullptr && (min_match > 0 || n_keep < deg);
        bool cool = false;
        uint32_t j0 = 0, it = 0;
        for (;;) {
            uint32_t np = 0, slot = 0, mark = kExpanded;
            if (j0 < m) {
                const uint32_t chunk = min(a.cap_cand, m - j0);
                hash_make_room(chunk);
                #pragma unroll 1
                for (uint32_t b = warp * 32; b < chunk; b += NT) {
                    const uint32_t j = j0 + b + lane;
                    uint32_t id = kEmpty;
                    if (b + lane < chunk)
                        id = seed_ids ? __ldcg(seed_ids + j)
                                      : (uint32_t)(splitmix64(seed_key ^ (qid << 32) ^ (uint64_t)j) % v.n);
                    collect(id < v.n, id);
                }
                j0 += chunk;
            } else {
                if (it == T) {
                    if (T_ext <= T || cnt == 0 || !(key_dist(qk()[0]) > judge)) break;
                    T = T_ext;   // judged too far: the rest of the ghost iterations
                }
                if (dgs_on && it >= it_cool) cool = true;
                np = select_parents(W, cool, slot);
                if (np == 0 && dgs_on && reexpand && !cool && any_partial()) {
                    cool = true;
                    np = select_parents(W, cool, slot);
                }
                if (np == 0) break;
                ++it;
                ++c_iters;
                c_parents += np;
                const bool dgs_now = dgs_on && !cool;
                if (dgs_now && reexpand) mark = kPartial;
                const uint32_t pid = lane < np ? (uint32_t)qk()[slot] : 0u;
                hash_make_room(np * deg);
                if (dgs_now) {
                    c_dgs += np;
                    guided(v, np, pid, n_keep, min_match);
                } else {
                    const uint32_t dp = v.deg_pad;
                    #pragma unroll 1
                    for (uint32_t b = warp * 32; b < np * dp; b += NT) {
                        const uint32_t x = b + lane, p = __umulhi(x, v.deg_magic);
                        const uint64_t parent = __shfl_sync(0xffffffffu, pid, min(p, np - 1));
                        const uint32_t nb = x < np * dp ? __ldg(v.graph + parent * dp + (x - p * dp)) : ANN_INVALID_ID;
                        collect(nb != ANN_INVALID_ID, nb);   // past the degree the list holds no ids
                    }
                }
            }
            __syncthreads();
            // every warp has selected: the parents can be marked
            if (warp == 0 && lane < np) bs()[slot] = (uint8_t)mark;
            const uint32_t nc = misc().nc[par];
            if (tid == 0) misc().nc[par ^ 1] = misc().ns[par ^ 1] = 0;
            hash_count += nc;
            c_rows += nc;
            // candidates no better than the last entry of a full queue are dropped
            const uint64_t worst = cnt == lcap ? qk()[cnt - 1] : ~0ull;
            evaluate<ST>(
                v.codes, v.scales, v.row_bytes, g.row_magic, nc, g.rows, g.stride, [&](uint32_t i) { return ci()[i]; },
                [&](uint32_t i, float d) {
                    const uint64_t k = make_key(d, ci()[i]);
                    if (k < worst) ck()[atomicAdd(&misc().ns[par], 1u)] = k;
                });
            __syncthreads();
            const uint32_t ns = misc().ns[par];
            par ^= 1;
            if (ns) merge(ns, lcap);
        }
    }

    // ------------------------------------------------------------- a query
    __device__ void run(const QParams &qp, uint64_t qidx, const float *qg, const uint32_t *given_row, uint32_t *oid,
                        float *odist, ann_query_stats *stats_out)
    {
        qid = qp.qid_base + qidx;
        st = ann_query_stats{};
        cnt = 0;
        const uint32_t dpad = (a.d + 31) & ~31u;
        for (uint32_t i = tid; i < dpad; i += NT)
            q()[query_pos<4>(i, g.q_part)] = i < a.d ? __ldcg(qg + i) : 0.0f;
        const bool ghost = ghost_entry(qp.entry);
        gbm = ghost && a.gbm_words > 0;
        hash_clear();
        if (tid == 0) misc() = Misc{};
        par = 0;
        const uint32_t *given = nullptr;
        if (given_entry(qp.entry) && given_row && given_row[0] != ANN_INVALID_ID) given = given_row;
        __syncthreads();
        #pragma unroll 1
        for (uint32_t stage = ghost ? 0u : 1u; stage < 2; ++stage) {
            const View &v = stage ? a.base : a.ghost;
            uint32_t rows = 0, iters = 0, parents = 0, dgs_parents = 0;
            if (stage == 1 && ghost) {
                // the top g ghost results become the base queue (ghost ids
                // ascend, so the order carries over); a new visited set
                __syncthreads();
                cnt = min(min(qp.g, cnt), qp.L);
                for (uint32_t i = tid; i < cnt; i += NT) {
                    const uint64_t k = qk()[i];
                    qk()[i] = (k & 0xFFFFFFFF00000000ull) | __ldg(a.ghost_ids + (uint32_t)k);
                    bs()[i] = kUnexpanded;
                }
                gbm = false;
                hash_refill();
            }
            const bool seeded = !(stage == 1 && ghost);
            const bool judged = stage == 0 && given && qp.judge > 0.0f && qp.Tg > qp.Tg_given;
            iterate(v, given,
                    seeded ? (given ? qp.n_given : (stage ? qp.m : v.deg)) : 0,
                    splitmix64(qp.seed ^ (stage ? 0 : kGhostTag)), stage ? qp.L : qp.Lg, stage ? qp.W : qp.Wg,
                    stage ? qp.T : (given ? qp.Tg_given : qp.Tg), judged ? qp.Tg : 0u, judged ? qp.judge : 0.0f,
                    stage ? qp.n_keep : v.deg, stage ? qp.min_match : 0, stage ? qp.it_cool : 0,
                    stage ? qp.reexpand : 0, iters, parents, dgs_parents, rows);
            given = nullptr;
            if (stage) {
                st.iters = iters;
                st.parents = parents;
                st.dgs_parents = dgs_parents;
                st.vec_rows = rows;
            } else {
                st.ghost_iters = iters;
                st.ghost_parents = parents;
                st.ghost_vec_rows = rows;
            }
        }
        if (qp.rerank) {
            // FP32 distances of the whole queue on the originals, then the top k
            evaluate<ANN_F32>(
                a.x32, nullptr, a.row32_bytes, g.row32_magic, cnt, g.rr_rows, g.rr_stride,
                [&](uint32_t i) { return (uint32_t)qk()[i]; },
                [&](uint32_t i, float d) { qk()[i] = make_key(d, (uint32_t)qk()[i]); });
            st.rerank_rows += cnt;
            __syncthreads();
            for (uint32_t e = tid; e < cnt; e += NT) {
                const uint64_t k = qk()[e];
                uint32_t r = 0;
#pragma unroll 4
                for (uint32_t e2 = 0; e2 < cnt; ++e2) r += qk()[e2] < k ? 1u : 0u;
                if (r < qp.k) {
                    oid[r] = (uint32_t)k;
                    odist[r] = key_dist(k);
                }
            }
        } else {
            for (uint32_t j = tid; j < min(qp.k, cnt); j += NT) {
                oid[j] = (uint32_t)qk()[j];
                odist[j] = key_dist(qk()[j]);
            }
        }
        for (uint32_t j = cnt + tid; j < qp.k; j += NT) {
            oid[j] = ANN_INVALID_ID;
            odist[j] = INFINITY;
        }
        if (stats_out && tid == 0) *stats_out = st;
    }
};

constexpr uint32_t kMostPerSm = 7;   // resident teams of 128 threads by their registers

template <int ST, int NT>
__global__ void __launch_bounds__(NT, NT == 256 ? 4 : kMostPerSm) team_kernel(const __grid_constant__ TeamArgs g)
{
    extern __shared__ __align__(128) uint8_t smem[];
    Team<ST, NT> t(g, smem);
    const TeamSearch &a = g.t;
    const uint32_t qi = blockIdx.x;
    t.run(a.qp, qi, a.queries + (uint64_t)qi * a.d,
          (given_entry(a.qp.entry) && a.given) ? a.given + (uint64_t)qi * a.qp.n_given : nullptr,
          a.out_ids + (uint64_t)qi * a.qp.k, a.out_dists + (uint64_t)qi * a.qp.k, a.stats ? a.stats + qi : nullptr);
}

TeamArgs plan(const TeamSearch &t, uint32_t rows, uint32_t max_rows)
{
    TeamArgs g{};
    g.t = t;
    const uint32_t W = t.qp.W;
    uint32_t o = 0;
    auto take = [&](uint32_t bytes) {
        const uint32_t at = o;
        o = round_up(o + bytes, 16);
        return at;
    };
    TeamLayout &L = g.lay;
    g.q_part = query_part(t.d, 4);
    L.q = take(g.q_part * 16);
    L.qk = take(t.cap_buf * 8);
    L.bs = take(t.cap_buf);
    L.ck = take(t.cap_cand * 8);
    L.ci = take(t.cap_cand * 4);
    L.pos = take(t.cap_cand * 4);
    L.adj = take(t.dgs ? W * t.base.deg_pad * 4 : 0);
    L.score = take(t.dgs ? W * t.base.deg_pad * 4 : 0);
    L.sign = take(t.dgs ? W * t.w * 4 : 0);
    L.misc = take(sizeof(Misc));
    L.table = take(4u << kTableBits);
    L.bits = take(t.gbm_words * 4);
    g.rows = rows;
    g.stride = smem_row_stride(t.base.row_bytes);
    g.rr_stride = t.qp.rerank ? smem_row_stride(t.row32_bytes) : 0u;
    const uint32_t bytes = std::max(rows * g.stride, g.rr_stride);
    g.rr_rows = g.rr_stride ? std::min(max_rows, bytes / g.rr_stride) : 0u;
    L.stage = take(bytes);
    L.total = o;
    g.row_magic = magic32(t.base.row_bytes / 16);
    g.row32_magic = magic32(std::max(16u, t.row32_bytes) / 16);
    return g;
}

// One launch of NT-thread teams if all queries get one at once, with as many
// rows per gather round as allow that. The line lies there because a second
// wave of teams doubles the time while the warp kernel has room: us a call,
// warps / teams, FP16 96-d: 608 queries 550 / 321, 1,064 queries (the last that
// fit) 578 / 385, then 587 (warps) at 1,216; FP16 128-d, itopk 128: 1,064
// queries 1,266 / 846, two waves of which exceed the 1,414 of 2,432 queries in
// warps. 256 threads are faster while they fit (one query 228 us against 315
// with 128 threads).
template <int ST, int NT>
bool try_teams(const TeamSearch &t, uint32_t least_rows, cudaStream_t stream, cudaError_t *e)
{
    for (uint32_t rows = NT / 2; rows >= least_rows; rows /= 2) {
        const TeamArgs g = plan(t, std::min(rows, round_up(t.cap_cand, 4)), NT / 2);
        if (g.lay.total > t.smem_optin) continue;
        int nb = 0;
        *e = raise_shared_limit(team_kernel<ST, NT>, t.smem_optin);
        if (*e == cudaSuccess)
            *e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, team_kernel<ST, NT>, NT, g.lay.total);
        if (*e != cudaSuccess) return true;
        if ((uint64_t)nb * t.num_sms < t.nq) continue;
        team_kernel<ST, NT><<<t.nq, NT, g.lay.total, stream>>>(g);
        *e = cudaGetLastError();
        return true;
    }
    return false;
}

template <int ST>
bool run_teams(const TeamSearch &t, cudaStream_t stream, cudaError_t *e)
{
    if (t.nq > kMostPerSm * (uint64_t)t.num_sms) return false;
    return try_teams<ST, 256>(t, 16, stream, e) || try_teams<ST, 128>(t, 8, stream, e);
}

}  // namespace

namespace ann {

bool team_search(const TeamSearch &t, cudaStream_t stream, cudaError_t *e)
{
    switch (t.storage) {
    case ANN_F32: return run_teams<ANN_F32>(t, stream, e);
    case ANN_F16: return run_teams<ANN_F16>(t, stream, e);
    default: return run_teams<ANN_E4M3>(t, stream, e);
    }
}

}  // namespace ann
