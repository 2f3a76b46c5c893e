// Exact kNN lists (the lists a proximity graph is pruned from; the paper
// times its graph build in Section 5.7, Fig. 16).
//
// The lists rank by (distance, id), the distance being the squared L2 in FP32,
// one fused multiply-add per element in index order. Computing every one of
// the n^2 distances that way is bound by the FP32 pipe and by the
// shared-memory operand of each step (120,000 x 128: 265 ms). Almost all of
// them only have to be shown to be too large, which an approximate distance
// with a proven error bound does as well, and that is a matrix product:
//
//   1. the rows, centred and scaled by a power of two, become FP16 operands in
//      a pseudo-random order (so that any prefix of the columns is a sample),
//      with their FP32 norms and the largest relative rounding error of a row;
//   2. knn_filter_kernel multiplies row blocks with column tiles on the tensor
//      cores (tcgen05, FP32 accumulation in tensor memory) and keeps, per row,
//      the columns whose lower bound does not exceed the row's threshold;
//   3. knn_select_kernel finds the K-th smallest upper bound a row has kept:
//      no entry whose lower bound is larger can be among the K nearest. It is
//      the threshold for the next, several times wider, range of columns, and
//      what it does not exclude is carried;
//   4. knn_rescore_kernel computes the exact distances of the few columns left
//      (K and those too close to call) and writes the K first.
//
// Measured: 120,000 x 128, K 64: 265 -> 7.1 ms (filter 4.5, selection 1.8,
// rescoring 0.8; the product alone at the measured BF16 rate would take 1.9);
// 10,000 x 96, K 32: 2,504 -> 269 us.
//
// Steps 2 and 3 repeat over growing column ranges (4 tiles, then 2 to 6 times
// more each time), so a row sees about K (growth - 1) survivors per range
// whatever n is. Survivor buffers have a fixed size: a row that overflows one
// (many equal distances), and every row if the input holds a value the FP16
// operands cannot bound (infinities, NaN, magnitudes near either end of FP32's
// range), is done by knn_exact_kernel, the plain computation, which also serves
// small inputs.
//
// Bounds. With x' the centred rows, |x' - fp16(x')| <= delta |x'| + eta
// measured over all rows (eta: FP16 subnormals), the product's error is at
// most delta (2 + delta) (N_u + N_v) / 2 + ..., N the squared norms, using
// |x'_u| |x'_v| <= (N_u + N_v) / 2; FP32 accumulation, the centring, the norms
// and the exact distance's own rounding each add a multiple of (N_u + N_v) of
// the order of d 2^-24. So |approx - exact| <= c (N_u + N_v) + kappa, and the
// test of column v against row u needs one number per column and one per row:
// (1 - c) N_v - 2 dot(u, v) <= T_u.
//
// That holds while the exact distance neither overflows nor loses bits among
// the subnormal numbers. With the largest |x'| below 2^(e + 1), a distance is
// below d 2^(2 e + 4), and its subnormal roundings add at most d 2^-150, which
// is d 2^(-122 - 2 e) in the operands' units and has to vanish in kappa. Both
// hold with room for -50 <= e <= 50 (kExponent) and any d that is taken.
#include <algorithm>
#include <cfloat>
#include <cmath>

#include <cuda_fp16.h>

#include "tcgen05.cuh"

using namespace ann;

namespace {

// Device state of one call's filter (zeroed at its start).
struct KnnState {
    uint32_t sample_max;   // largest |x| of the sample rows (FP32 bits)
    uint32_t max;          // largest |x - mean| of all rows (FP32 bits; infinities and NaN sort above)
    uint32_t delta;        // largest relative FP16 rounding error of a row (FP32 bits)
    uint32_t listed;       // rows left to the plain kernel
    uint32_t all;          // 1: every row is (the operands cannot bound the input)
    int err;               // a bounded wait ran out: every row is, too
};

constexpr int KQ = 32;          // query rows per block
constexpr int KC = 64;          // candidate rows per shared-memory tile
constexpr int KW = 8;           // warps per block (4 queries each)

__device__ __forceinline__ bool kless(float da, uint32_t ia, float db, uint32_t ib)
{
    return da < db || (da == db && ia < ib);
}

// Insert (d, id) into a warp's sorted list lst_d/lst_i of K entries if it
// beats the last one (all lanes call it with the same arguments).
__device__ __forceinline__ void list_insert(float *lst_d, uint32_t *lst_i, uint32_t K, float d, uint32_t id,
                                            uint32_t lane)
{
    if (!kless(d, id, lst_d[K - 1], lst_i[K - 1])) return;
    uint32_t pos = 0;
    for (uint32_t j = lane; j < K; j += 32) pos += kless(lst_d[j], lst_i[j], d, id) ? 1u : 0u;
    pos = __reduce_add_sync(0xffffffffu, pos);
    // shift [pos, K - 1) right by one, from the top (each lane one entry
    // per pass, read before any write of the pass)
    for (int32_t top = (int32_t)K - 2; top >= (int32_t)pos; top -= 32) {
        const int32_t j = top - (int32_t)lane;
        float vd = 0.0f;
        uint32_t vi = 0;
        const bool mine = j >= (int32_t)pos;
        if (mine) { vd = lst_d[j]; vi = lst_i[j]; }
        __syncwarp();
        if (mine) { lst_d[j + 1] = vd; lst_i[j + 1] = vi; }
        __syncwarp();
    }
    if (lane == 0) { lst_d[pos] = d; lst_i[pos] = id; }
    __syncwarp();
}

// The plain computation: block b handles query rows [32 b, 32 b + 32), or,
// LISTED, those of the rows that the filter has left over (all, or a list; none,
// the usual case, ends the block at once). Dynamic shared memory holds the 32
// query rows, one tile of KC candidate rows (row stride d + 1 floats: lanes
// reading one element of 32 different rows hit 32 banks; a query row's last word
// is its number) and the 32 lists of K entries. Bound by the latency of its tile
// loop, so a listed row is looked up before it: looked up in it, from global
// memory by one kernel for both forms, 1,000 x 96 rows took 374 us instead of 350,
// and 30,000 x 64 equal ones, all left over, 10,930 instead of 9,165.
template <bool LISTED>
__global__ void __launch_bounds__(KW * 32) knn_exact_kernel(const float *__restrict__ X, uint32_t n, uint32_t d,
                                                            uint32_t K, uint32_t *__restrict__ out,
                                                            const KnnState *__restrict__ todo,
                                                            const uint32_t *__restrict__ list)
{
    extern __shared__ __align__(16) uint8_t sm[];
    const bool all = !LISTED || todo->all || todo->err;
    const uint32_t rows = all ? n : todo->listed;
    const uint32_t ds = d + 1;
    float *sq = reinterpret_cast<float *>(sm);                 // KQ x ds
    float *sc = sq + KQ * ds;                                  // KC x ds
    float *ld = sc + KC * ds;                                  // KQ x K
    uint32_t *li = reinterpret_cast<uint32_t *>(ld + KQ * K);  // KQ x K
    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t q0 = blockIdx.x * KQ;
    if (LISTED && q0 >= rows) return;
    // query r's row, n past the last
    auto row_of = [&](uint32_t r) { return LISTED ? __float_as_uint(sq[r * ds + d]) : q0 + r; };
    if (LISTED) {
        if (threadIdx.x < KQ) {
            const uint32_t r = q0 + threadIdx.x;
            sq[threadIdx.x * ds + d] = __uint_as_float(r >= rows ? n : all ? r : list[r]);
        }
        __syncthreads();
    }
    for (uint32_t i = threadIdx.x; i < KQ * d; i += blockDim.x) {
        const uint32_t r = i / d, c = i % d, u = row_of(r);
        sq[r * ds + c] = u < n ? X[(size_t)u * d + c] : 0.0f;
    }
    for (uint32_t i = threadIdx.x; i < KQ * K; i += blockDim.x) {
        ld[i] = INFINITY;
        li[i] = ANN_INVALID_ID;
    }
    uint32_t mine[4];   // this warp's queries
#pragma unroll
    for (int a = 0; a < 4; ++a) mine[a] = row_of(warp * 4 + a);
    for (uint32_t c0 = 0; c0 < n; c0 += KC) {
        __syncthreads();
        for (uint32_t i = threadIdx.x; i < KC * d; i += blockDim.x) {
            const uint32_t r = i / d, c = i % d;
            sc[r * ds + c] = c0 + r < n ? X[(size_t)(c0 + r) * d + c] : 0.0f;
        }
        __syncthreads();
        // this warp's 4 queries x the tile's 64 candidates: lane owns
        // candidates lane and lane + 32
        float acc[4][2];
#pragma unroll
        for (int a = 0; a < 4; ++a) acc[a][0] = acc[a][1] = 0.0f;
        const float *x0 = sc + lane * ds, *x1 = sc + (lane + 32) * ds;
        const float *qw = sq + (warp * 4) * ds;
#pragma unroll 2
        for (uint32_t i = 0; i < d; ++i) {
            const float xa = x0[i], xb = x1[i];
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                const float qv = qw[a * ds + i];
                const float da = __fsub_rn(qv, xa), db = __fsub_rn(qv, xb);
                acc[a][0] = __fmaf_rn(da, da, acc[a][0]);
                acc[a][1] = __fmaf_rn(db, db, acc[a][1]);
            }
        }
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            const uint32_t qi = LISTED ? mine[a] : q0 + warp * 4 + a;
            float *lda = ld + (warp * 4 + a) * K;
            uint32_t *lia = li + (warp * 4 + a) * K;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const uint32_t cid = c0 + lane + 32 * h;
                const bool cand = qi < n && cid < n && cid != qi;
                const float dv = acc[a][h];
                uint32_t m = __ballot_sync(0xffffffffu, cand && kless(dv, cid, lda[K - 1], lia[K - 1]));
                while (m) {
                    const uint32_t src = __ffs(m) - 1;
                    m &= m - 1;
                    list_insert(lda, lia, K, __shfl_sync(0xffffffffu, dv, src), __shfl_sync(0xffffffffu, cid, src),
                                lane);
                }
            }
        }
    }
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < KQ * K; i += blockDim.x) {
        const uint32_t u = row_of(i / K);
        if (u < n) out[(size_t)u * K + (i % K)] = li[i];
    }
}


// ------------------------------------------------------------ operands
constexpr uint32_t kTileRows = 128;      // rows of a tensor-core tile (and columns of a column tile)
constexpr uint32_t kBK = 64;             // FP16 elements of a 128-byte swizzled tile row
constexpr uint32_t kTileBytes = kTileRows * kBK * 2;
constexpr uint32_t kMinStages = 4, kMaxStages = 12;   // column tiles (64 elements deep) in flight
constexpr uint32_t kSample = 4096;       // rows the centre is estimated from
constexpr uint32_t kCarry = 512;         // columns a row carries from range to range
constexpr uint32_t kEntries = 768, kFewEntries = 576;   // carried and new columns one selection can hold
constexpr uint32_t kFirstTiles = 4;      // column tiles of the first range: kept whole
constexpr uint32_t kMaxS = kFirstTiles;  // column segments of a range (one CTA each)
constexpr uint32_t kParts = 4;           // parts of the columns: one half of every second tile, an epilogue warp each
constexpr uint32_t kSelectWarps = 4, kRescoreWarps = 8;
constexpr uint32_t kChunk = 32;          // elements of a row staged at a time by the rescoring
constexpr uint32_t kChunkStride = kChunk + 4;   // floats: 8 lanes' 16-byte reads hit 8 bank groups
static_assert(2 * ANN_MAX_DEGREE <= kCarry && 2 * ANN_MAX_DEGREE < kFirstTiles * kTileRows, "K entries are carried");

// Row of X behind operand row j: a fixed stride coprime to n spreads every
// prefix of the operand rows evenly over X.
__device__ __forceinline__ uint32_t source_row(uint32_t j, uint32_t stride, uint32_t n)
{
    return (uint32_t)((uint64_t)j * stride % n);
}

// Column sums and the largest magnitude of the sample rows.
__global__ void knn_sample_kernel(const float *__restrict__ X, uint32_t n, uint32_t d, uint32_t samples,
                                  float *__restrict__ sum, KnnState *st)
{
    const uint32_t per = (samples + gridDim.x - 1) / gridDim.x;
    const uint32_t s0 = blockIdx.x * per, s1 = min(samples, s0 + per);
    uint32_t mx = 0;
    for (uint32_t c = threadIdx.x; c < d; c += blockDim.x) {
        float t = 0.0f;
        for (uint32_t i = s0; i < s1; ++i) {
            const float x = X[(uint64_t)i * n / samples * d + c];
            t += x;
            mx = max(mx, __float_as_uint(fabsf(x)));
        }
        if (s0 < s1) atomicAdd(sum + c, t);
    }
    mx = __reduce_max_sync(0xffffffffu, mx);
    if ((threadIdx.x & 31) == 0) atomicMax(&st->sample_max, mx);
}

// The sample mean of column c, rounded to 2^-8 of the largest magnitude's
// binade: integers stay exact in FP16 after the centring. Any value is
// valid, the rows only have to be centred alike.
__device__ __forceinline__ float centre(float sum, uint32_t samples, uint32_t sample_max)
{
    const int e = (int)(sample_max >> 23) - 127 - 8;
    if (e < -100 || e > 60) return 0.0f;
    const float q = exp2f((float)e);
    return rintf(sum / (float)samples / q) * q;
}

__global__ void knn_centre_kernel(const float *__restrict__ X, size_t total, uint32_t d, uint32_t samples,
                                  const float *__restrict__ sum, KnnState *st)
{
    extern __shared__ float mu[];
    for (uint32_t c = threadIdx.x; c < d; c += blockDim.x) mu[c] = centre(sum[c], samples, st->sample_max);
    __syncthreads();
    uint32_t mx = 0;
    // whole rows per block, so the column index needs no division per element
    const uint32_t rows = (uint32_t)(total / d);
    for (uint32_t r = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); r < rows; r += gridDim.x * (blockDim.x >> 5))
        for (uint32_t c = threadIdx.x & 31; c < d; c += 32)
            mx = max(mx, __float_as_uint(fabsf(X[(size_t)r * d + c] - mu[c])));
    mx = __reduce_max_sync(0xffffffffu, mx);
    if ((threadIdx.x & 31) == 0) atomicMax(&st->max, mx);
}

// Whether the bounds hold for rows whose largest |x'| has the bits mb.
constexpr int kExponent = 50;
__device__ __forceinline__ bool in_range(uint32_t mb)
{
    const int e = (int)(mb >> 23) - 127;
    return mb == 0 || (e >= -kExponent && e <= kExponent);
}

// The FP16 operand row j (row stride ld >= d elements, zero past d), scaled
// so that the largest magnitude lies in [2^14, 2^15), its squared norm in
// those units, and the relative rounding error. One warp per row.
__global__ void knn_operand_kernel(const float *__restrict__ X, uint32_t n, uint32_t d, uint32_t ld, uint32_t stride,
                                   uint32_t samples, const float *__restrict__ sum, __half *__restrict__ H,
                                   float *__restrict__ norm, KnnState *st)
{
    extern __shared__ float mu[];
    for (uint32_t c = threadIdx.x; c < d; c += blockDim.x) mu[c] = centre(sum[c], samples, st->sample_max);
    __syncthreads();
    const uint32_t mb = st->max;
    if (!in_range(mb)) return;   // knn_bound_kernel leaves every row to the plain kernel
    const int e = (int)(mb >> 23) - 127;
    const float s = mb ? exp2f((float)(14 - e)) : 1.0f;
    const uint32_t lane = threadIdx.x & 31;
    const float eta = sqrtf((float)d) * 2.98023224e-8f;   // 2^-25 per element: half an FP16 subnormal step
    float worst = 0.0f;
    for (uint32_t j = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); j < n; j += gridDim.x * (blockDim.x >> 5)) {
        const float *x = X + (size_t)source_row(j, stride, n) * d;
        float nn = 0.0f, ee = 0.0f;
        for (uint32_t c = lane; c < ld; c += 32) {
            const float v = c < d ? s * (x[c] - mu[c]) : 0.0f;
            const __half h = __float2half_rn(v);
            H[(size_t)j * ld + c] = h;
            const float r = v - __half2float(h);
            nn = fmaf(v, v, nn);
            ee = fmaf(r, r, ee);
        }
        for (int o = 16; o; o >>= 1) {
            nn += __shfl_xor_sync(0xffffffffu, nn, o);
            ee += __shfl_xor_sync(0xffffffffu, ee, o);
        }
        if (lane == 0) norm[j] = nn;
        const float excess = sqrtf(ee) * 1.00002f - eta;
        if (nn > 0.0f && excess > 0.0f) worst = fmaxf(worst, excess / sqrtf(nn));
    }
    if (lane == 0 && worst > 0.0f) atomicMax(&st->delta, __float_as_uint(worst * 1.00002f));
}

// The bound's coefficients: c of (N_u + N_v), and the constant kappa.
__device__ __forceinline__ float bound_c(const KnnState *st, uint32_t d)
{
    const float delta = __uint_as_float(st->delta);
    // the operands' rounding; accumulation in tensor memory (2 d + 256 units
    // of 2^-24), the exact distance's rounding (2 d + 4), centring and norms
    return delta * (2.0f + delta) * 1.001f + (4.0f * (float)d + 352.0f) * 5.96046448e-8f;
}

__device__ __forceinline__ float bound_kappa(uint32_t d) { return (float)d * 0.0045f; }   // 4.1 eta max|x'|, 2 eta^2

// lower[j] = (1 - c) N_j, +infinity past n; and whether the operands bound
// the input at all.
__global__ void knn_bound_kernel(const float *__restrict__ norm, uint32_t n, uint32_t n_pad, uint32_t d,
                                 float *__restrict__ lower, KnnState *st)
{
    const float c = bound_c(st, d);
    const bool bad = !in_range(st->max) || !(c < 0.25f);
    for (uint32_t j = blockIdx.x * blockDim.x + threadIdx.x; j < n_pad; j += gridDim.x * blockDim.x)
        lower[j] = j < n ? (1.0f - c) * norm[j] : INFINITY;
    if (bad && blockIdx.x == 0 && threadIdx.x == 0) st->all = 1;
}

// ------------------------------------------------------------ filter
struct KnnWork {
    const float *lower;      // per operand row: (1 - c) N
    float *T;                // per row of the chunk: threshold
    uint2 *carry;            // chunk rows x kCarry: (upper value bits, column)
    uint32_t *n_carry;       // chunk rows
    uint2 *kept;             // chunk rows x kParts S x cap: (lower value bits, column)
    uint32_t *n_kept;        // chunk rows x kParts S
    KnnState *st;
    uint32_t S, cap;         // column segments; entries per row, segment and part
    uint32_t stages;         // slots of the column-tile ring
    uint32_t low_slots;      // slots of lower[] in shared memory (a power of two)
    uint32_t entries;        // columns that a selection can hold
};

// One CTA: NSUB x 128 operand rows against the column tiles of one segment
// of [t0, t1). The rows stay in shared memory; the column tiles (and their
// lower[]) stream through rings by TMA (warp 0), warp 1 issues the MMAs, each
// stage serving all NSUB row tiles, into one of two accumulator sets; eight of
// the sixteen epilogue warps test a set's values while the next is computed.
// Survivors of a thread (one row, one part of the columns) go to a segment of
// its own in the row's buffer, so appending needs no atomics.
// What bounds it (120,000 x 128, the last range, per 128 columns and two row
// tiles: 2,350 clocks): the test of every value, 6 instructions per 4 columns
// when none survives (packed multiply-adds and a minimum) and some 20 more when
// one does; with next to no tests left in, the MMAs alone take 1,900 (102 a
// 128 x 128 x 16, where both operands' shared-memory reads allow 64). Two row
// tiles per CTA, where their operands fit, halve the L2 -> shared memory stream
// of the column tiles.
__device__ __forceinline__ float fmin3(float a, float b, float c)
{
    float r;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// Entries of columns nb .. nb + 3 at p (32-byte aligned).
__device__ __forceinline__ void store_four(uint2 *p, float2 x, float2 y, uint32_t nb)
{
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(__float_as_uint(x.x)),
                 "r"(nb), "r"(__float_as_uint(x.y)), "r"(nb + 1), "r"(__float_as_uint(y.x)), "r"(nb + 2),
                 "r"(__float_as_uint(y.y)), "r"(nb + 3)
                 : "memory");
}

// Append (v, col) to a list at p if v <= T, without a branch: the lanes that
// append differ from value to value.
__device__ __forceinline__ void append_if(uint2 *&p, float v, float T, uint32_t col)
{
    asm volatile(
        "{\n\t.reg .pred a;\n\tsetp.le.f32 a, %1, %2;\n\t"
        "@a st.global.v2.b32 [%0], {%3, %4};\n\t"
        "@a add.u64 %0, %0, 8;\n\t}"
        : "+l"(p)
        : "f"(v), "f"(T), "r"(__float_as_uint(v)), "r"(col)
        : "memory");
}

constexpr int kFilterEpiWarps = 4 * kParts;
constexpr int kFilterThreads = 64 + 32 * kFilterEpiWarps;
constexpr uint32_t kLowSlots = 8;        // column tiles whose lower[] is in shared memory, at most
constexpr uint32_t kFilterBars = 384;    // bytes for the barriers

template <int NSUB, bool FIRST>
__global__ void __launch_bounds__(kFilterThreads, 1)
    knn_filter_kernel(const __grid_constant__ CUtensorMap map, uint32_t n, uint32_t nkb, uint32_t row0, uint32_t t0,
                      uint32_t t1, KnnWork w)
{
    extern __shared__ uint8_t smem_raw[];
    if (w.st->all) return;
    const uint32_t pad = (1024u - (smem_addr(smem_raw) & 1023u)) & 1023u;
    uint8_t *sA = smem_raw + pad;                       // NSUB x nkb tiles
    uint8_t *sB = sA + NSUB * nkb * kTileBytes;         // w.stages tiles
    float *sLow = reinterpret_cast<float *>(sB + w.stages * kTileBytes);   // kLowSlots x 128
    uint64_t *full = reinterpret_cast<uint64_t *>(sLow + w.low_slots * kTileRows);
    const uint32_t low_mask = w.low_slots - 1, low_shift = __popc(low_mask);
    uint64_t *empty = full + kMaxStages;
    uint64_t *acc_full = empty + kMaxStages;               // [2]
    uint64_t *acc_empty = acc_full + 2;                 // [2]
    uint64_t *low_full = acc_empty + 2;                 // [kLowSlots]
    uint64_t *low_empty = low_full + kLowSlots;         // [kLowSlots]
    uint64_t *a_full = low_empty + kLowSlots;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(a_full + 1);
    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rb = blockIdx.x / w.S, seg = blockIdx.x % w.S;
    const uint32_t arow = row0 + rb * NSUB * kTileRows;
    const uint32_t b0 = t0 + (uint32_t)((uint64_t)(t1 - t0) * seg / w.S);
    const uint32_t b1 = t0 + (uint32_t)((uint64_t)(t1 - t0) * (seg + 1) / w.S);
    constexpr uint32_t kCols = 2 * NSUB * kTileRows;    // tensor-memory columns: two sets of NSUB accumulators
    if (threadIdx.x == 0) {
        for (uint32_t s = 0; s < w.stages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&acc_full[b], 1);
            mbar_init(&acc_empty[b], kFilterEpiWarps / 2);
        }
        for (uint32_t s = 0; s < kLowSlots; ++s) {
            mbar_init(&low_full[s], 1);
            mbar_init(&low_empty[s], kFilterEpiWarps / 2);
        }
        mbar_init(a_full, 1);
        fence_mbar_init();
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(tmem_slot)),
                     "r"(kCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    int *err = &w.st->err;
    bool ok = true;                         // false: a wait of this thread ran out
    uint32_t it = 0, tc = 0, issued = 0;    // stages and lower[] slots it has loaded, stages it issued MMAs on

    if (warp == 0) {
        if (lane == 0) {
            mbar_arrive_expect_tx(a_full, NSUB * nkb * kTileBytes);
            for (uint32_t sub = 0; sub < NSUB; ++sub)
                for (uint32_t kb = 0; kb < nkb; ++kb)
                    tma_load_2d(sA + (sub * nkb + kb) * kTileBytes, &map, (int)(kb * kBK),
                                (int)(arow + sub * kTileRows), a_full);
            uint32_t s = 0, ph = 0;
            for (uint32_t t = b0; t < b1 && ok; ++t, ++tc) {
                const uint32_t ls = tc & low_mask;
                if (!(ok = mbar_wait_bounded(&low_empty[ls], ((tc >> low_shift) & 1) ^ 1, err))) break;
                mbar_arrive_expect_tx(&low_full[ls], kTileRows * 4);
                bulk_g2s(sLow + ls * kTileRows, w.lower + (size_t)t * kTileRows, kTileRows * 4, &low_full[ls]);
                for (uint32_t kb = 0; kb < nkb; ++kb) {
                    if (!(ok = mbar_wait_bounded(&empty[s], ph ^ 1, err))) break;
                    mbar_arrive_expect_tx(&full[s], kTileBytes);
                    tma_load_2d(sB + s * kTileBytes, &map, (int)(kb * kBK), (int)(t * kTileRows), &full[s]);
                    ++it;
                    if (++s == w.stages) { s = 0; ph ^= 1; }
                }
            }
            if (b0 == b1) ok = mbar_wait_bounded(a_full, 0, err);
        }
    } else if (warp == 1) {
        constexpr uint32_t idesc = idesc_fp16(kTileRows, kTileRows);
        const uint32_t a_lo = desc_lo(smem_addr(sA)), b_lo = desc_lo(smem_addr(sB));
        auto wait = [&](uint64_t *bar, uint32_t parity) {
            return __all_sync(0xffffffffu, mbar_wait_bounded(bar, parity, err));
        };
        uint32_t s = 0, ph = 0;
        ok = b0 == b1 || wait(a_full, 0);
        for (uint32_t t = b0; t < b1 && ok; ++t, ++tc) {
            const uint32_t buf = tc & 1, use = tc >> 1;
            if (!(ok = wait(&acc_empty[buf], (use & 1) ^ 1))) break;
            for (uint32_t kb = 0; kb < nkb; ++kb) {
                if (!(ok = wait(&full[s], ph))) {
                    issued = kb;
                    break;
                }
                tc_fence_after();
                const uint32_t bb = b_lo + s * (kTileBytes >> 4);
                if (elect_one()) {
#pragma unroll
                    for (uint32_t sub = 0; sub < NSUB; ++sub) {
                        const uint32_t aa = a_lo + (sub * nkb + kb) * (kTileBytes >> 4);
                        const uint32_t acc = tmem + (buf * NSUB + sub) * kTileRows;
                        if (kb == 0) mma_f16kind_lo<false>(acc, aa, bb, idesc);
                        else mma_f16kind_lo<true>(acc, aa, bb, idesc);
#pragma unroll
                        for (uint32_t k = 1; k < kBK / 16; ++k)
                            mma_f16kind_lo<true>(acc, aa + 2 * k, bb + 2 * k, idesc);
                    }
                    mma_commit(&empty[s]);
                    if (kb + 1 == nkb) mma_commit(&acc_full[buf]);
                }
                __syncwarp();
                if (++s == w.stages) { s = 0; ph ^= 1; }
            }
            if (!ok) break;
        }
        issued += tc * nkb;
    } else {
        // warp's rows: 32 (warp % 4) .. + 31 of each row tile; its part: one
        // half of the columns of every second tile. The two groups of eight
        // warps take turns, so one's accumulator loads overlap the other's
        // tests.
        const uint32_t q = warp & 3, h = (warp - 2) >> 2, buf = h >> 1, half = (h & 1) * 64;
        const uint32_t cap = w.cap, lists = kParts * w.S;
        float T[NSUB];
        uint2 *list[NSUB], *next[NSUB];
#pragma unroll
        for (int sub = 0; sub < NSUB; ++sub) {
            const uint32_t lr = rb * NSUB * kTileRows + sub * kTileRows + q * 32 + lane;
            T[sub] = row0 + lr >= n ? -FLT_MAX : FIRST ? FLT_MAX : w.T[lr];
            list[sub] = next[sub] = w.kept + ((size_t)lr * lists + seg * kParts + h) * cap;
        }
        for (uint32_t t = b0 + buf; t < b1; t += 2) {
            const uint32_t at = t - b0, ls = at & low_mask;
            ok = __all_sync(0xffffffffu, mbar_wait_bounded(&low_full[ls], (at >> low_shift) & 1, err) &&
                                             mbar_wait_bounded(&acc_full[buf], (at >> 1) & 1, err));
            if (!ok) break;
            tc_fence_after();
            // a list without room for the whole part is marked overfull
#pragma unroll
            for (int sub = 0; sub < NSUB; ++sub)
                if (next[sub] - list[sub] + 64 > (ptrdiff_t)cap) {
                    next[sub] = list[sub] + cap + 1;
                    T[sub] = -FLT_MAX;
                }
#pragma unroll
            for (uint32_t c = half; c < half + 64; c += 32) {
                float v[NSUB][32];
                __syncwarp();
                const uint32_t ta = tmem + buf * NSUB * kTileRows + ((q * 32u) << 16) + c;
                if constexpr (NSUB == 2) tmem_ld32x2(ta, ta + kTileRows, v[0], v[1]);
                else tmem_ld32(ta, v[0]);
                if (c != half) {
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&acc_empty[buf]);
                }
                const float *low = sLow + ls * kTileRows + c;
                const uint32_t nb = t * kTileRows + c;
                auto values = [&](int sub, int g, const float4 &l, float2 &x, float2 &y) {
                    x = __ffma2_rn(make_float2(v[sub][g], v[sub][g + 1]), make_float2(-2.0f, -2.0f),
                                   make_float2(l.x, l.y));
                    y = __ffma2_rn(make_float2(v[sub][g + 2], v[sub][g + 3]), make_float2(-2.0f, -2.0f),
                                   make_float2(l.z, l.w));
                };
                if (FIRST) {
                    // every column of every row is kept (none lies past n): four
                    // entries to a store (one by one, the lanes' lists being
                    // apart: 190 us instead of 38 for 38,912 rows)
#pragma unroll
                    for (int g = 0; g < 32; g += 4) {
                        const float4 l = *reinterpret_cast<const float4 *>(low + g);
#pragma unroll
                        for (int sub = 0; sub < NSUB; ++sub) {
                            float2 x, y;
                            values(sub, g, l, x, y);
                            if (T[sub] > 0.0f) {
                                store_four(next[sub], x, y, nb + g);
                                next[sub] += 4;
                            }
                        }
                    }
                } else {
#pragma unroll
                    for (int g = 0; g < 32; g += 4) {
                        const float4 l = *reinterpret_cast<const float4 *>(low + g);
#pragma unroll
                        for (int sub = 0; sub < NSUB; ++sub) {
                            float2 x, y;
                            values(sub, g, l, x, y);
                            // the row itself is dropped by the selection
                            if (fmin3(fminf(x.x, x.y), y.x, y.y) <= T[sub]) {
                                append_if(next[sub], x.x, T[sub], nb + g);
                                append_if(next[sub], x.y, T[sub], nb + g + 1);
                                append_if(next[sub], y.x, T[sub], nb + g + 2);
                                append_if(next[sub], y.y, T[sub], nb + g + 3);
                            }
                        }
                    }
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&low_empty[ls]);
        }
#pragma unroll
        for (int sub = 0; sub < NSUB; ++sub) {
            const uint32_t lr = rb * NSUB * kTileRows + sub * kTileRows + q * 32 + lane;
            w.n_kept[(size_t)lr * lists + seg * kParts + h] = (uint32_t)(next[sub] - list[sub]);
        }
    }
    tc_fence_before();
    if (__syncthreads_or(!ok)) {
        // a role gave up: what the others have in flight ends before the CTA does
        auto wait = [&](uint64_t *bar, uint32_t parity) { mbar_wait_bounded(bar, parity, err); };
        if (warp == 0) {
            wait_last_uses(it, w.stages, [&](uint32_t i, uint32_t parity) { wait(&full[i], parity); });
            wait_last_uses(tc, w.low_slots, [&](uint32_t i, uint32_t parity) { wait(&low_full[i], parity); });
            wait(a_full, 0);
        }
        if (warp == 1) wait_last_use(issued, w.stages, [&](uint32_t i, uint32_t parity) { wait(&empty[i], parity); });
        __syncthreads();
    }
    if (warp == 1)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kCols) : "memory");
}

// ------------------------------------------------------------ selection
// One warp per row of the chunk: the new threshold from an upper bound of the
// K-th smallest upper value among the carried and newly kept columns (two
// rounds of a 256-bin histogram, linear between the smallest and the largest
// value left: bins by leading bits would put most values, which share an
// exponent, into a few), then the columns it does not exclude are carried.
// A row that overflowed a buffer gets the threshold -FLT_MAX: it keeps
// nothing any more and is left to the plain kernel. Bound by the latency of
// its short dependent steps and of its gathers, which 36 warps per SM and four
// loads a lane in flight hide.
__global__ void __launch_bounds__(kSelectWarps * 32)
    knn_select_kernel(uint32_t n, uint32_t d, uint32_t K, uint32_t row0, uint32_t rows, uint32_t first, KnnWork w)
{
    extern __shared__ __align__(16) uint8_t sm[];
    if (w.st->all) return;
    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t lr = blockIdx.x * kSelectWarps + warp;
    if (lr >= rows) return;
    uint2 *e = reinterpret_cast<uint2 *>(sm) + warp * w.entries;   // (upper value bits, column)
    uint32_t *hist = reinterpret_cast<uint32_t *>(sm + kSelectWarps * w.entries * 8) + warp * 256;
    const float c = bound_c(w.st, d), up = 2.0f * c / (1.0f - c);   // upper - lower value = 2 c N = up * lower[]
    const uint32_t lists = kParts * w.S;   // at most 16
    uint2 *carry = w.carry + (size_t)lr * kCarry;
    uint32_t m = 0;
    bool over = !first && w.T[lr] == -FLT_MAX;
    float lo = INFINITY, hi = -INFINITY;
    // four entries a lane at a time, so that their loads are in flight together
    if (!first && !over) {
        m = w.n_carry[lr];
        for (uint32_t b = 0; b < m; b += 128) {
            uint2 x[4];
#pragma unroll
            for (uint32_t u = 0; u < 4; ++u)
                if (b + 32 * u + lane < m) x[u] = carry[b + 32 * u + lane];
#pragma unroll
            for (uint32_t u = 0; u < 4; ++u)
                if (b + 32 * u + lane < m) {
                    lo = fminf(lo, __uint_as_float(x[u].x));
                    hi = fmaxf(hi, __uint_as_float(x[u].x));
                    e[b + 32 * u + lane] = x[u];
                }
        }
    }
    const uint32_t counts = lane < lists ? w.n_kept[(size_t)lr * lists + lane] : 0u;
    uint32_t ends = counts;   // of this lane's list among the new entries
    for (int o = 1; o < 16; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, ends, o);
        if (lane >= (uint32_t)o) ends += y;
    }
    const uint32_t fresh = __shfl_sync(0xffffffffu, ends, 15);
    over = over || __any_sync(0xffffffffu, counts > w.cap) || m + fresh > w.entries;
    bool self = false;
    if (!over) {
        // the lists as one sequence
        const uint2 *src = w.kept + (size_t)lr * lists * w.cap;
        for (uint32_t b = 0; b < fresh; b += 128) {
            uint2 x[4];
            float nv[4];
#pragma unroll
            for (uint32_t u = 0; u < 4; ++u) {
                const uint32_t i = b + 32 * u + lane;
                uint32_t s = 0;   // the list that holds entry i
#pragma unroll
                for (uint32_t step = 8; step; step >>= 1)
                    if (__shfl_sync(0xffffffffu, ends, s + step - 1) <= i) s += step;
                const uint32_t begin = __shfl_sync(0xffffffffu, ends, s ? s - 1 : 0);
                if (i < fresh) x[u] = src[s * w.cap + i - (s ? begin : 0u)];
            }
#pragma unroll
            for (uint32_t u = 0; u < 4; ++u)
                if (b + 32 * u + lane < fresh) nv[u] = __ldg(w.lower + x[u].y);
#pragma unroll
            for (uint32_t u = 0; u < 4; ++u) {
                const uint32_t i = b + 32 * u + lane;
                if (i >= fresh) continue;
                float v = fmaf(up, nv[u], __uint_as_float(x[u].x));
                if (x[u].y == row0 + lr) { v = INFINITY; self = true; }   // the row itself
                lo = fminf(lo, v);
                if (v < INFINITY) hi = fmaxf(hi, v);
                e[m + i] = make_uint2(__float_as_uint(v), x[u].y);
            }
        }
        m += fresh;
        __syncwarp();
        self = __any_sync(0xffffffffu, self);
    }
    if (!over && m - (self ? 1u : 0u) >= K) {
        const uint32_t slack = 4 + K / 16;
        uint32_t need = K;
        float tau = INFINITY;
        for (int o = 16; o; o >>= 1) {
            lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
            hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
        }
#pragma unroll 1
        for (int round = 0; round < 2; ++round) {
            // values in [lo, hi], `need` of them to be covered; bin() is
            // monotone, so the bins up to the one that reaches `need` hold the
            // `need` smallest values and tau is the largest value in them
            const float scale = hi > lo ? 255.0f / (hi - lo) : 0.0f;
            auto bin = [&](float v) { return min(255, (int)((v - lo) * scale)); };
            for (uint32_t i = lane; i < 256; i += 32) hist[i] = 0;
            __syncwarp();
            for (uint32_t i = lane; i < m; i += 32) {
                const float v = __uint_as_float(e[i].x);
                if (v >= lo && v <= hi) atomicAdd(&hist[bin(v)], 1u);
            }
            __syncwarp();
            uint32_t mine[8], sum = 0;
#pragma unroll
            for (int b = 0; b < 8; ++b) { mine[b] = hist[lane * 8 + b]; sum += mine[b]; }
            uint32_t incl = sum;
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= (uint32_t)o) incl += y;
            }
            const uint32_t before = incl - sum;
            const bool here = before < need && need <= incl;
            uint32_t at = 0, left = need - before, in_bin = 0;
            if (here) {
                bool found = false;
#pragma unroll
                for (int b = 0; b < 8; ++b)
                    if (!found) {
                        if (left <= mine[b]) { at = lane * 8 + b; in_bin = mine[b]; found = true; }
                        else left -= mine[b];
                    }
            }
            const uint32_t src = __ffs(__ballot_sync(0xffffffffu, here)) - 1;
            at = __shfl_sync(0xffffffffu, at, src);
            need = __shfl_sync(0xffffffffu, left, src);
            in_bin = __shfl_sync(0xffffffffu, in_bin, src);
            float blo = INFINITY, bhi = -INFINITY;   // the values of that bin
            for (uint32_t i = lane; i < m; i += 32) {
                const float v = __uint_as_float(e[i].x);
                if (v >= lo && v <= hi && (uint32_t)bin(v) == at) {
                    blo = fminf(blo, v);
                    bhi = fmaxf(bhi, v);
                }
            }
            for (int o = 16; o; o >>= 1) {
                blo = fminf(blo, __shfl_xor_sync(0xffffffffu, blo, o));
                bhi = fmaxf(bhi, __shfl_xor_sync(0xffffffffu, bhi, o));
            }
            lo = blo;
            hi = bhi;
            tau = bhi;
            __syncwarp();
            if (in_bin - need <= slack) break;   // so few more than K: not worth a second round
        }
        const float nu = __ldg(w.lower + row0 + lr) / (1.0f - c);
        // the row's own share of both bounds, and the rounding of the few
        // operations on these values
        const float T = tau + 2.0f * c * nu + 2.0f * bound_kappa(d) + (fabsf(tau) + nu) * 3.8146973e-6f;
        uint32_t kept = 0;
        for (uint32_t b = 0; b < m; b += 128) {
            uint2 x[4];
            float low[4];
#pragma unroll
            for (uint32_t u = 0; u < 4; ++u) {
                const uint32_t i = b + 32 * u + lane;
                x[u] = i < m ? e[i] : make_uint2(__float_as_uint(INFINITY), 0u);
                // the lower value is no larger than the upper one: needed only
                // of what that alone does not keep
                low[u] = __uint_as_float(x[u].x);
                if (low[u] > T && low[u] < INFINITY) low[u] = fmaf(-up, __ldg(w.lower + x[u].y), low[u]);
            }
#pragma unroll
            for (uint32_t u = 0; u < 4; ++u) {
                const bool keep = low[u] <= T && low[u] < INFINITY;
                const uint32_t mask = __ballot_sync(0xffffffffu, keep);
                const uint32_t at = kept + __popc(mask & ((1u << lane) - 1u));
                if (keep && at < kCarry) carry[at] = x[u];
                kept += __popc(mask);
            }
        }
        over = kept > kCarry;
        if (!over && lane == 0) {
            w.T[lr] = T;
            w.n_carry[lr] = kept;
        }
    } else {
        over = true;
    }
    if (over && lane == 0) {
        w.T[lr] = -FLT_MAX;
        w.n_carry[lr] = 0;
    }
}

template <int N>
__device__ __forceinline__ void copy_async(void *dst, const void *src)
{
    if (N == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(smem_addr(dst)), "l"(src), "n"(N) : "memory");
}

// One warp per row of the chunk: the exact distances of the carried columns
// (a lane each, one fused multiply-add per element in index order), ranked by
// (distance, id); rows without a valid carried list are listed for the plain
// kernel. Bound by the gathers: a column's row is read in pieces of kChunk
// elements by asynchronous copies, neighbouring lanes copying neighbouring
// units, one piece ahead of the arithmetic (120,000 x 128, K 64, us per 38,912
// rows: 268; one bulk copy per lane and no overlap 295; read by the lanes
// directly, every load touching 32 lines, 544).
__global__ void __launch_bounds__(kRescoreWarps * 32)
    knn_rescore_kernel(const float *__restrict__ X, uint32_t n, uint32_t d, uint32_t K, uint32_t stride, uint32_t row0,
                       uint32_t rows, bool wide, KnnWork w, uint32_t *__restrict__ list,
                       uint32_t *__restrict__ out)
{
    extern __shared__ __align__(16) uint8_t sm[];
    if (w.st->all) return;
    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t lr = blockIdx.x * kRescoreWarps + warp;
    if (lr >= rows) return;
    float *stage = reinterpret_cast<float *>(sm) + warp * 2 * 32 * kChunkStride;
    uint64_t *keys = reinterpret_cast<uint64_t *>(sm + kRescoreWarps * 2 * 32 * kChunkStride * 4) + warp * kCarry;
    float *q = reinterpret_cast<float *>(sm + kRescoreWarps * (2 * 32 * kChunkStride * 4 + kCarry * 8)) +
               warp * ((d + 3) & ~3u);
    const uint32_t u = source_row(row0 + lr, stride, n);
    const uint32_t m = w.n_carry[lr];
    if (m < K) {
        if (lane == 0) list[atomicAdd(&w.st->listed, 1u)] = u;
        return;
    }
    for (uint32_t i = lane; i < d; i += 32) q[i] = X[(size_t)u * d + i];
    const uint2 *carry = w.carry + (size_t)lr * kCarry;
    // steps of 32 columns by kChunk elements, the next one's copies in flight
    // while one is computed
    const uint32_t steps = (m + 31) / 32 * ((d + kChunk - 1) / kChunk);
    uint32_t ib = 0, ic = 0, iv = 0;   // the step being copied: first column, first element, this lane's row
    auto issue = [&](uint32_t buf) {
        if (ic == 0) iv = source_row(carry[min(ib + lane, m - 1)].y, stride, n);
        const uint32_t rows = min(32u, m - ib), len = min(kChunk, d - ic);
        float *dst = stage + buf * 32 * kChunkStride;
        if (wide) {   // 16-byte units: 8 lanes a row
#pragma unroll
            for (uint32_t r0 = 0; r0 < 32; r0 += 4) {
                const uint32_t r = r0 + (lane >> 3), c = (lane & 7) * 4;
                const uint32_t v = __shfl_sync(0xffffffffu, iv, r);
                if (r < rows && c < len) copy_async<16>(dst + r * kChunkStride + c, X + (size_t)v * d + ic + c);
            }
        } else {
#pragma unroll 4
            for (uint32_t r = 0; r < rows; ++r) {
                const uint32_t v = __shfl_sync(0xffffffffu, iv, r);
                if (lane < len) copy_async<4>(dst + r * kChunkStride + lane, X + (size_t)v * d + ic + lane);
            }
        }
        ic += kChunk;
        if (ic >= d) { ic = 0; ib += 32; }
    };
    issue(0);
    asm volatile("cp.async.commit_group;" ::: "memory");
    float acc = 0.0f;
    uint32_t b = 0, c0 = 0;   // the step being computed
    for (uint32_t t = 0; t < steps; ++t) {
        const uint32_t mine = iv;   // (the next batch's after the issue)
        if (t + 1 < steps) issue((t + 1) & 1);
        asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 1;" ::: "memory");
        __syncwarp();
        const float *row = stage + ((t & 1) * 32 + lane) * kChunkStride;
        const uint32_t len = min(kChunk, d - c0);
        auto step = [&](float a, float y) {
            const float df = __fsub_rn(a, y);
            acc = __fmaf_rn(df, df, acc);
        };
        uint32_t c = 0;
#pragma unroll 4
        for (; c + 4 <= len; c += 4) {
            const float4 xv = *reinterpret_cast<const float4 *>(row + c);
            const float4 qv = *reinterpret_cast<const float4 *>(q + c0 + c);
            step(qv.x, xv.x);
            step(qv.y, xv.y);
            step(qv.z, xv.z);
            step(qv.w, xv.w);
        }
        for (; c < len; ++c) step(q[c0 + c], row[c]);
        c0 += kChunk;
        if (c0 >= d) {
            if (b + lane < m)   // non-negative: the bits order as the values
                keys[b + lane] = ((uint64_t)__float_as_uint(acc) << 32) | mine;
            acc = 0.0f;
            c0 = 0;
            b += 32;
        }
        __syncwarp();   // the step's buffer has been read
    }
    for (uint32_t i = lane; i < m; i += 32) {
        const uint64_t k = keys[i];
        uint32_t r = 0;
#pragma unroll 4
        for (uint32_t j = 0; j < m; ++j) r += keys[j] < k ? 1u : 0u;
        if (r < K) out[(size_t)u * K + r] = (uint32_t)k;
    }
}

// ------------------------------------------------------------ host
// Rows from which the filter runs. Measured plain / filtered, us a call: 1,024
// rows 194 / 85 (32 dimensions, K 16), 357 / 96 (96, 32), 1,274 / 142 (64,
// 256); 4,096 rows 425 / 129, 877 / 151, 2,301 / 300. After a synchronisation,
// with the workspace kept (temporary_alloc), 1,024 x 8, K 8: 134 / 86; 2,000 x 32,
// K 16: 293 / 95; 10,000 x 96, K 32: 2,550 / 275 (280, 360 and 700 with a workspace
// mapped anew).
constexpr uint64_t kFilterMin = 1024;

uint32_t gcd(uint32_t a, uint32_t b)
{
    while (b) {
        const uint32_t t = a % b;
        a = b;
        b = t;
    }
    return a;
}

template <int NSUB, bool FIRST>
cudaError_t launch_filter(const CUtensorMap &map, uint32_t blocks, size_t smem, int optin, uint32_t n, uint32_t nkb,
                          uint32_t row0, uint32_t t0, uint32_t t1, const KnnWork &w, cudaStream_t st)
{
    cudaError_t e = raise_shared_limit(knn_filter_kernel<NSUB, FIRST>, optin);
    if (e != cudaSuccess) return e;
    knn_filter_kernel<NSUB, FIRST><<<blocks, kFilterThreads, smem, st>>>(map, n, nkb, row0, t0, t1, w);
    return cudaGetLastError();
}

int grid_for(uint64_t n, int threads) { return (int)std::max<uint64_t>(1, (n + threads - 1) / threads); }

// The filtered computation. ANN_ENOMEM (nothing launched) if its workspace
// cannot be had: the caller then runs the plain kernel, which needs none.
ann_status knn_filtered(const float *X, uint32_t n, uint32_t d, uint32_t K, uint32_t *ids, size_t plain_smem, int dev,
                        int optin, cudaStream_t st)
{
    int sms = 0;
    ANN_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const uint32_t ld = round_up(d, 8), nkb = (d + kBK - 1) / kBK;
    const uint32_t n_tiles = (n + kTileRows - 1) / kTileRows, n_pad = n_tiles * kTileRows;
    // two row tiles per CTA where both operands fit beside the stages
    auto smem_of = [&](uint32_t nsub, uint32_t slots) {
        return (size_t)(nsub * nkb + kMinStages) * kTileBytes + slots * kTileRows * 4 + kFilterBars + 1024;
    };
    const uint32_t nsub = smem_of(2, kLowSlots) <= (size_t)optin && n_tiles >= 2u * (uint32_t)sms ? 2 : 1;
    const uint32_t slots = smem_of(nsub, kLowSlots) <= (size_t)optin ? kLowSlots : 2;
    const uint32_t stages =
        kMinStages + (uint32_t)std::min<size_t>(kMaxStages - kMinStages, (optin - smem_of(nsub, slots)) / kTileBytes);
    const size_t filter_smem = smem_of(nsub, slots) + (stages - kMinStages) * kTileBytes;
    const uint32_t block_rows = nsub * kTileRows;
    const uint32_t chunk_rows = std::min<uint32_t>((uint32_t)sms * block_rows, round_up(n, block_rows));
    // About K (growth - 1) columns of a range survive the threshold of the
    // ranges before it; larger growth means fewer ranges but more survivors.
    // A row's list per segment and part holds half as many again as expected
    // and eight standard deviations (and its share of the first range), and
    // the 64 columns of a tile that have to fit before it is tested.
    const uint32_t growth = K <= 32 ? 6 : K <= 128 ? 4 : 2;
    // A selection's entries, carried (about K) and new: the first range's 512,
    // and with K up to 64 at most 260 expected, eight standard deviations below
    // 576; their shared memory decides how many warps are resident (36 an SM
    // against 28).
    const uint32_t entries = K <= 64 ? kFewEntries : kEntries;
    auto segments = [&](uint32_t blocks) {   // a power of two: the first range divides evenly
        uint32_t S = 1;
        while (2 * S <= kMaxS && blocks * 2 * S <= (uint32_t)sms) S *= 2;
        return S;
    };
    auto list_cap = [&](uint32_t S) {
        const double mean = (double)K * (growth - 1) / (kParts * S);
        return round_up(std::max((uint32_t)(1.5 * mean + 8.0 * std::sqrt(mean) + 72.0), 64 * ((kFirstTiles / S + 1) / 2)), 8);
    };
    // rows x lists of a chunk of `rows` rows
    auto kept_bytes = [&](uint32_t rows) {
        const uint32_t S = segments((rows + block_rows - 1) / block_rows);
        return (size_t)round_up(rows, block_rows) * kParts * S * list_cap(S) * 8;
    };
    const uint32_t samples = std::min(n, kSample);

    size_t bytes = 0;
    auto take = [&](size_t b) {
        const size_t at = bytes;
        bytes += (b + 255) & ~(size_t)255;
        return at;
    };
    const size_t o_state = take(sizeof(KnnState)), o_sum = take((size_t)d * 4), zeroed = bytes;
    const size_t o_h = take((size_t)n * ld * 2), o_norm = take((size_t)n * 4), o_low = take((size_t)n_pad * 4);
    const size_t o_list = take((size_t)n * 4), o_t = take((size_t)chunk_rows * 4);
    const size_t o_carry = take((size_t)chunk_rows * kCarry * 8), o_nc = take((size_t)chunk_rows * 4);
    const uint32_t last_rows = (n - 1) % chunk_rows + 1;
    const size_t o_kept = take(std::max(kept_bytes(chunk_rows), kept_bytes(last_rows)));
    const size_t o_nk = take((size_t)chunk_rows * kParts * kMaxS * 4);
    uint8_t *ws = nullptr;
    if (temporary_alloc((void **)&ws, bytes, st) != cudaSuccess) {
        cudaGetLastError();
        set_error("ann_knn_exact: no room for a workspace of %zu bytes", bytes);
        return ANN_ENOMEM;
    }
    KnnState *state = reinterpret_cast<KnnState *>(ws + o_state);
    float *sum = reinterpret_cast<float *>(ws + o_sum), *norm = reinterpret_cast<float *>(ws + o_norm);
    float *lower = reinterpret_cast<float *>(ws + o_low);
    __half *H = reinterpret_cast<__half *>(ws + o_h);
    uint32_t *list = reinterpret_cast<uint32_t *>(ws + o_list);
    KnnWork w{lower,
                    reinterpret_cast<float *>(ws + o_t),
                    reinterpret_cast<uint2 *>(ws + o_carry),
                    reinterpret_cast<uint32_t *>(ws + o_nc),
                    reinterpret_cast<uint2 *>(ws + o_kept),
                    reinterpret_cast<uint32_t *>(ws + o_nk),
                    state, 1, 0, stages, slots, entries};
    uint32_t stride = std::max(1u, (uint32_t)(0.6180339887 * n));
    while (gcd(stride, n) != 1) ++stride;
    CUtensorMap map;
    ann_status s = make_map16(&map, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, H, n, d, ld, kTileRows);
    cudaError_t e = cudaSuccess;
    auto run = [&](cudaError_t r) {
        if (e == cudaSuccess) e = r;
        return e == cudaSuccess;
    };
    if (s == ANN_OK && run(cudaMemsetAsync(ws, 0, zeroed, st))) {
        knn_sample_kernel<<<256, 128, 0, st>>>(X, n, d, samples, sum, state);
        knn_centre_kernel<<<std::min(grid_for(n, 8), sms * 8), 256, d * 4, st>>>(X, (size_t)n * d, d, samples, sum, state);
        knn_operand_kernel<<<std::min(grid_for(n, 8), sms * 8), 256, d * 4, st>>>(X, n, d, ld, stride, samples, sum, H,
                                                                                norm, state);
        knn_bound_kernel<<<std::min(grid_for(n_pad, 256), sms * 8), 256, 0, st>>>(norm, n, n_pad, d, lower, state);
        run(cudaGetLastError());
        const size_t sel_smem = kSelectWarps * (w.entries * 8 + 1024);
        const size_t res_smem =
            kRescoreWarps * (2 * 32 * kChunkStride * 4 + kCarry * 8 + (size_t)((d + 3) & ~3u) * 4);
        // rows of whole 16-byte units
        const bool wide = d % 4 == 0 && (reinterpret_cast<uintptr_t>(X) & 15u) == 0;
        run(raise_shared_limit(knn_select_kernel, optin));
        run(raise_shared_limit(knn_rescore_kernel, optin));
        for (uint32_t row0 = 0; row0 < n && e == cudaSuccess; row0 += chunk_rows) {
            const uint32_t rows = std::min(chunk_rows, n - row0);
            const uint32_t blocks = (rows + block_rows - 1) / block_rows;
            w.S = segments(blocks);
            w.cap = list_cap(w.S);
            uint32_t t0 = 0, t1 = std::min(kFirstTiles, n_tiles);
            while (t0 < n_tiles && e == cudaSuccess) {
                const uint32_t first = t0 == 0;
                const auto launch = nsub == 2 ? (first ? launch_filter<2, true> : launch_filter<2, false>)
                                              : (first ? launch_filter<1, true> : launch_filter<1, false>);
                run(launch(map, blocks * w.S, filter_smem, optin, n, nkb, row0, t0, t1, w, st));
                knn_select_kernel<<<grid_for(rows, kSelectWarps), kSelectWarps * 32, sel_smem, st>>>(
                    n, d, K, row0, rows, first, w);
                t0 = t1;
                t1 = (uint32_t)std::min<uint64_t>(n_tiles, (uint64_t)t1 * growth);
            }
            knn_rescore_kernel<<<grid_for(rows, kRescoreWarps), kRescoreWarps * 32, res_smem, st>>>(
                X, n, d, K, stride, row0, rows, wide, w, list, ids);
            run(cudaGetLastError());
        }
        run(raise_shared_limit(knn_exact_kernel<true>, optin));
        knn_exact_kernel<true><<<grid_for(n, KQ), KW * 32, plain_smem, st>>>(X, n, d, K, ids, state, list);
        run(cudaGetLastError());
    }
    run(cudaFreeAsync(ws, st));
    if (s == ANN_OK && e != cudaSuccess) s = cuda_fail(e, "ann_knn_exact");
    return s;
}

}  // namespace

extern "C" {

ann_status ann_knn_exact(const float *X, uint64_t n, uint32_t dim, uint32_t K, uint32_t *ids, void *stream)
{
    if (!X || !ids || n < 2 || n > 0xFFFFFFFEull || dim == 0 || dim > ANN_MAX_DIM || K == 0 || K >= n ||
        K > 2 * ANN_MAX_DEGREE) {
        set_error("ann_knn_exact: need 2 <= n < 2^32 - 1, 1 <= dim <= %u, 1 <= K < n, K <= %u", ANN_MAX_DIM,
                  2 * ANN_MAX_DEGREE);
        return ANN_EINVAL;
    }
    const size_t smem = (size_t)(KQ + KC) * (dim + 1) * 4 + (size_t)KQ * K * 8;
    int dev = 0, optin = 0;
    ANN_CUDA(cudaGetDevice(&dev));
    ANN_CUDA(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    if (smem > (size_t)optin) {
        set_error("ann_knn_exact: %zu bytes of shared memory needed (dim %u, K %u), %d available", smem, dim, K, optin);
        return ANN_EINVAL;
    }
    if (n >= kFilterMin && n < (1ull << 31)) {
        const ann_status s = knn_filtered(X, (uint32_t)n, dim, K, ids, smem, dev, optin, (cudaStream_t)stream);
        if (s != ANN_ENOMEM) return s;
    }
    ANN_CUDA(raise_shared_limit(knn_exact_kernel<false>, optin));
    knn_exact_kernel<false><<<grid_for(n, KQ), KW * 32, smem, (cudaStream_t)stream>>>(X, (uint32_t)n, dim, K, ids,
                                                                                      nullptr, nullptr);
    ANN_CUDA(cudaGetLastError());
    return ANN_OK;
}

}  // extern "C"
