// What the search kernels share: the graph view, the order of queue entries,
// the random seeds, and the distance of a staged row.
#pragma once

#include "ann_internal.cuh"

namespace ann {

constexpr uint32_t kUnexpanded = 0, kPartial = 1, kExpanded = 2;
constexpr uint64_t kGhostTag = 0x67686F7374ull;
constexpr uint32_t kEmpty = 0xFFFFFFFFu;

// Entries that run the ghost stage first.
__host__ __device__ __forceinline__ bool ghost_entry(uint32_t e)
{
    return e == ANN_ENTRY_GHOST || e == ANN_ENTRY_GIVEN_GHOST;
}
// Entries that read a row of caller-given seeds.
__host__ __device__ __forceinline__ bool given_entry(uint32_t e)
{
    return e == ANN_ENTRY_GIVEN_GHOST || e == ANN_ENTRY_GIVEN_BASE;
}

// ceil(2^32 / d): __umulhi(x, magic32(d)) = x / d for x d < 2^32 and d > 1.
inline uint32_t magic32(uint32_t d) { return d > 1 ? (uint32_t)(((1ull << 32) + d - 1) / d) : 0u; }

struct View {
    const uint8_t *codes;
    const float *scales;   // nullptr for FP32
    uint32_t row_bytes;
    const uint32_t *graph;
    uint32_t deg, deg_pad, deg_magic;   // deg_magic = magic32(deg_pad)
    const uint32_t *dir;   // nullptr: no DGS on this graph
    uint32_t n;
};

// Ghost sets up to this many nodes get an exact shared-memory bitmap as the
// ghost stage's visited set (2 KB per warp at most).
constexpr uint32_t kGhostBitmapMax = 16384;

__device__ __forceinline__ uint64_t splitmix64(uint64_t x)
{
    uint64_t z = x + 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// (da, ia) < (db, ib) in (distance, id) order. Distances are squared L2,
// never negative nor NaN, and non-negative floats order as their bit
// patterns do, so the key compares as one 64-bit integer (bits, id): two
// integer compares instead of three float and integer ones.
__device__ __forceinline__ bool key_less(float da, uint32_t ia, float db, uint32_t ib)
{
    return (((uint64_t)__float_as_uint(da) << 32) | ia) < (((uint64_t)__float_as_uint(db) << 32) | ib);
}

__device__ __forceinline__ uint32_t lanemask_lt()
{
    uint32_t m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

// One element: df = q - x, acc += df * df with a single rounding.
__device__ __forceinline__ void step(float qv, float xv, float &acc)
{
    const float df = __fsub_rn(qv, xv);
    acc = __fmaf_rn(df, df, acc);
}

// Element i of a stored row as the number that the scale multiplies.
template <int ST>
__device__ __forceinline__ float code_value(const uint8_t *row, uint32_t i)
{
    if (ST == ANN_F32) return reinterpret_cast<const float *>(row)[i];
    if (ST == ANN_F16) return __half2float(reinterpret_cast<const __half *>(row)[i]);
    return __half2float(__half(__nv_cvt_fp8_to_halfraw((__nv_fp8_storage_t)row[i], __NV_E4M3)));
}

// Stored value of element i (decoded to FP32).
template <int ST>
__device__ __forceinline__ float stored_elem(const uint8_t *row, uint32_t i, float scale)
{
    const float c = code_value<ST>(row, i);
    return ST == ANN_F32 ? c : __fmul_rn(scale, c);
}

// One element of the distance: acc += (q - stored)^2, the difference
// rounded once. An FP16 row's scale is a power of two, so its stored value
// s * h is exact in FP32 (for every row whose largest |x| is at least 2^-88,
// where s * h stays a normal number) and q - s * h is one fused multiply-add,
// equal to the rounded difference of q and the stored value; E4M3 scales are
// not powers of two, so that stored value is rounded first.
template <int ST>
__device__ __forceinline__ void elem_step(float qv, const uint8_t *row, uint32_t i, float scale, float &acc)
{
    if (ST == ANN_F16) {
        const float df = __fmaf_rn(-scale, __half2float(reinterpret_cast<const __half *>(row)[i]), qv);
        acc = __fmaf_rn(df, df, acc);
    } else {
        step(qv, stored_elem<ST>(row, i, scale), acc);
    }
}

// The query in shared memory is laid out for the lanes that read it: part p
// of LPR holds, in order, the elements that lane p of a row's LPR lanes
// works on (LPR 2: elements 4 g + 2 p and the next; LPR 4: elements 4 g + p),
// so that a lane reads four of its elements with one 16-byte load where index
// order gave it one or two. The elements from d on are zero. Parts whose
// length would put the lanes of a row on the same banks are 16 bytes apart.
constexpr uint32_t query_part(uint32_t d, uint32_t lpr)
{
    const uint32_t part = ((d + 31) & ~31u) / lpr;
    return part + (part & 32 / lpr ? 0 : 4);
}

template <int LPR>
__device__ __forceinline__ uint32_t query_pos(uint32_t i, uint32_t part)
{
    return LPR == 2 ? ((i >> 1) & 1) * part + (i >> 2) * 2 + (i & 1) : (i & 3) * part + (i >> 2);
}

// One of the four partial sums of the squared L2 between a staged row and
// the query (q: part j): lane j of a row's four lanes runs sum j (elements
// i = j, j + 4, ... in index order, one fused multiply-add each), so the four
// lanes together do the work of one row with the same operations as the
// definition; the differences are rounded two at a time. Used by the teams
// and by the warp kernel's rounds of at most 8 rows. Bound by its
// instructions: for 4 elements 11 (FP32) or 15 (FP16), against 16 or 20 with
// the query in index order (3,001 queries of FP16 768-d 2,390 -> 2,175 us, one
// query of FP16 768-d by a team 494 -> 436).
template <int ST>
__device__ __forceinline__ float row_dist_quarter(const uint8_t *row, const float *q, float scale, uint32_t d,
                                                  uint32_t j)
{
    float s = 0.0f;
    const float2 sc = make_float2(scale, scale), nsc = make_float2(-scale, -scale);
    const float4 *yp = reinterpret_cast<const float4 *>(q);
    const uint32_t units = d / 16;
#pragma unroll 2
    for (uint32_t u = 0; u < units; ++u) {
        const float4 y = yp[u];
        const uint32_t i = 16 * u;
        float2 x[2];   // elements i + j, i + j + 4 and i + j + 8, i + j + 12
        if (ST == ANN_E4M3) {
            // 16 codes at once, byte j of each word (code by code: one query of
            // E4M3 128-d by a team 346 us instead of 304)
            const uint4 w = *reinterpret_cast<const uint4 *>(row + i);
            const uint32_t sel = j | (j + 4) << 4;
            x[0] = __half22float2(__half2(
                __nv_cvt_fp8x2_to_halfraw2((__nv_fp8x2_storage_t)__byte_perm(w.x, w.y, sel), __NV_E4M3)));
            x[1] = __half22float2(__half2(
                __nv_cvt_fp8x2_to_halfraw2((__nv_fp8x2_storage_t)__byte_perm(w.z, w.w, sel), __NV_E4M3)));
        } else {
            x[0] = make_float2(code_value<ST>(row, i + j), code_value<ST>(row, i + j + 4));
            x[1] = make_float2(code_value<ST>(row, i + j + 8), code_value<ST>(row, i + j + 12));
        }
#pragma unroll
        for (uint32_t g = 0; g < 2; ++g) {
            const float2 yg = g ? make_float2(y.z, y.w) : make_float2(y.x, y.y);
            float2 df;
            if (ST == ANN_F32) df = __ffma2_rn(x[g], make_float2(-1.0f, -1.0f), yg);
            else if (ST == ANN_F16) df = __ffma2_rn(nsc, x[g], yg);
            else df = __ffma2_rn(__fmul2_rn(sc, x[g]), make_float2(-1.0f, -1.0f), yg);
            s = __fmaf_rn(df.x, df.x, s);
            s = __fmaf_rn(df.y, df.y, s);
        }
    }
    #pragma unroll 1
    for (uint32_t i = 16 * units; i + j < d; i += 4) elem_step<ST>(q[i / 4], row, i + j, scale, s);
    return s;
}

// ------------------------------------------------------------- small batches
// A search by teams (a thread block per query, search_team.cu): what plan_args
// has derived for the warp kernel, less the launch shape.
struct TeamSearch {
    View base, ghost;
    const uint32_t *ghost_ids;
    const uint8_t *x32;
    uint32_t row32_bytes, d, w, cap_buf, cap_cand, gbm_words;
    bool dgs;
    QParams qp;
    const float *queries;
    uint32_t nq;
    const uint32_t *given;
    uint32_t *out_ids;
    float *out_dists;
    ann_query_stats *stats;
    int *err;
    int storage, num_sms;
    size_t smem_optin;
};

// Launches the search by teams if every query of the batch gets a team at
// once; false (and nothing launched) if not, and the warp kernel then runs.
// *e receives the launch's status.
bool team_search(const TeamSearch &t, cudaStream_t stream, cudaError_t *e);

}  // namespace ann
