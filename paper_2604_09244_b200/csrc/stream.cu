// Scoring kernel for many key tiles (Sec. 3.2.1 of the paper): batches, and samples with more visual tokens than the
// latency-shaped kernel of fused.cu covers.
//
// A (sample, head) is a job: its keys (T tiles of 128) are read once, its logits have to stay somewhere until the
// softmax denominators over all T tiles are known.  Here they stay in tensor memory (512 columns = 8 tiles at 64 text
// queries, 32 at 16), so a job belongs to one CTA, or, when T tiles do not fit, to a cluster of 2, 4 or 8 CTAs that
// exchange one (maximum, sum) pair per query.  CTAs are persistent, one per multiprocessor, and made of roles that
// run ahead of one another across jobs:
//   * one thread streams key tiles through a ring of shared-memory stages by TMA (the text queries of a job in one of
//     two buffers of their own): 128-160 KB in flight per multiprocessor whatever the softmax is doing;
//   * one thread issues the MMAs of a tile into the next free tensor-memory slot (slots are a ring too);
//   * eight warps take the softmax: a warp reads its own 32 tensor-memory lanes of every other tile, against references of
//     its own, so that a job has two block barriers in all.  Exponentials go back to tensor memory; per-key contributions
//     are added into the 64-bit fixed-point accumulators (scale 2^60: the sum over heads is exact and independent of
//     scheduling).
// What bounds it: HBM (the keys are read once); softmax arithmetic comes second (16 exponentials per clock and
// multiprocessor: half of the time of the key stream at 48 queries, nine tenths at 64).
// Whole steps against one short-lived CTA per two tiles (and, above 2048 tokens, the generic kernel): 16 requests of 768
// tokens 121 -> 97 us, 8 of 3584 tokens 695 -> 162, 16 patch-by-patch steps of 512 tokens 139 -> 97.  Taking the feature norms too:
// 16 requests 94.9 -> 93.7, 16 of 228 tokens 39.9 -> 35.6, 16 patch-by-patch steps 82.9 -> 78.7.
// More softmax warps (12, 16), two tiles per warp at once and prefetching the next tile's columns were all slower.
#include "common.cuh"
#include "rules.h"
#include "device_utils.cuh"
#include "select_impl.cuh"
#include "tmem_plan.h"

#include <algorithm>

namespace mvla {
namespace {

constexpr int kSoftWarps = 8;
constexpr int kSoftThreads = kSoftWarps * 32;
constexpr int kStreamThreads = kSoftThreads + 64;     // + the loading warp and the MMA warp
constexpr int kNormWarps = 2;                         // + these, in launches that take the feature norms
constexpr int kNormStages = 3;                        // pieces of rows in flight per norm warp
constexpr int kStreamRegs = 168;                      // registers a thread, see the kernel
constexpr int kMaxStages = 12;
constexpr int kStagesBesideTail = 6;                  // deeper rings make the tail's copies wait: 12 / 6, 16 requests 88.0 / 87.2 us, 8 of 3584 tokens 155.2 / 154.3
constexpr uint32_t kStageBytes = 16384;               // 128 keys x 128 bytes: one swizzled box of a key tile
constexpr int kMaxSlots = 32;
// Pairs of job n go to buffer n mod 2: a CTA sends those of job n + 2 only after it has the pairs of job n + 1 of every
// peer, which that peer sent when it was done with job n's.
constexpr int kPairBufs = 2;

struct StreamArgs {
    int n_heads, kv_group, head_dim, esize;
    int stages;                   // boxes in the shared-memory ring
    int width, slots;             // columns of a tensor-memory slot (the padded text queries of the longest text), slots
    int n_jobs;                   // samples x heads
    unsigned long long* acc64;
    int* status;
    AlphaOut alpha;               // with it there may be no accumulators
    int32_t* rearm;               // see launch_salience_fast
    unsigned long long* rearm_rec;
    unsigned long long* stamps;
    int32_t* hand;                // the tail runs beside this kernel: its counters (kHandTicket and so on), or null
    // feature norms (null: none): bf16 rows of `row_bytes` bytes, their L1 norms, where the pieces in flight lie in dynamic shared memory
    const uint8_t* hidden;
    float* l1;
    int row_bytes;
    uint32_t norm_off;
    int n_samples;
    int vis0;                     // first visual token of the launch
    uint8_t by_row[kMaxChunk];    // samples in the order of their visual tokens: a norm warp's run of rows crosses them without a look at whose sum it takes
};

struct StreamSmem {
    alignas(8) uint64_t kfull[kMaxStages], kempty[kMaxStages];
    uint64_t qfull[2], qempty[2];
    uint64_t tfull[kMaxSlots], tempty[kMaxSlots];
    uint64_t nfull[kNormWarps][kNormStages];
    uint64_t xbar[kPairBufs];                      // pairs of the cluster's CTAs have landed
    alignas(16) float m[kSoftWarps][kMaxText];     // per warp and query: -reference (log2 domain; +inf: no key)
    alignas(16) float w[kSoftWarps][kMaxText];     // ... its sum of exponentials, then its weight
    float g[kMaxText], iz[kMaxText];               // common reference of the job's keys; 1 / (denominator H n_t)
    float2 peer[kPairBufs][kMaxCluster][kMaxText];
    uint32_t tmem;
    int aborted;                                   // a bounded wait ran out: nobody waits any longer
};

// Bounded wait; gives up at once when another role has.
template <bool CLUSTER>
__device__ __forceinline__ bool ring_wait(uint32_t bar, uint32_t parity, volatile int* aborted, int* status)
{
    uint64_t t0 = 0;
    for (uint32_t it = 0; it < kSpinLimit; ++it) {
        if (mbar_try_wait<CLUSTER>(bar, parity)) return true;
        if ((it & 63u) == 63u) {
            if (*aborted) return false;
            const uint64_t now = global_ns();
            if (t0 == 0) t0 = now;
            if (now - t0 > 1000000000ull) break;
        }
    }
    *aborted = 1;
    *reinterpret_cast<volatile int*>(status) = MVLA_ERR_TIMEOUT;
    return false;
}
// Barrier of the softmax warps.
__device__ __forceinline__ void soft_barrier() { asm volatile("bar.sync 1, %0;" ::"n"(kSoftThreads) : "memory"); }
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const float (&v)[16])
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
                 ::"r"(taddr), "r"(__float_as_uint(v[0])), "r"(__float_as_uint(v[1])), "r"(__float_as_uint(v[2])),
                   "r"(__float_as_uint(v[3])), "r"(__float_as_uint(v[4])), "r"(__float_as_uint(v[5])), "r"(__float_as_uint(v[6])),
                   "r"(__float_as_uint(v[7])), "r"(__float_as_uint(v[8])), "r"(__float_as_uint(v[9])), "r"(__float_as_uint(v[10])),
                   "r"(__float_as_uint(v[11])), "r"(__float_as_uint(v[12])), "r"(__float_as_uint(v[13])), "r"(__float_as_uint(v[14])),
                   "r"(__float_as_uint(v[15])) : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// Two fp32 operations per instruction.
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c)
{
    float2 d;
    asm("{\n\t.reg .b64 ra, rb, rc, rd;\n\tmov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\tmov.b64 rc, {%6, %7};\n\t"
        "fma.rn.f32x2 rd, ra, rb, rc;\n\tmov.b64 {%0, %1}, rd;\n\t}"
        : "=f"(d.x), "=f"(d.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
    return d;
}
__device__ __forceinline__ float2 add2(float2 a, float2 b)
{
    float2 d;
    asm("{\n\t.reg .b64 ra, rb, rd;\n\tmov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
        "add.rn.f32x2 rd, ra, rb;\n\tmov.b64 {%0, %1}, rd;\n\t}"
        : "=f"(d.x), "=f"(d.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}
// 16 tensor-memory columns of this thread's lane, as a load that is issued here and waited for later (tmem_wait_ld
// names the registers again, so that nothing that uses them can move in front of it).
__device__ __forceinline__ void tmem_issue16(uint32_t taddr, float (&v)[16])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]), "=f"(v[8]),
                   "=f"(v[9]), "=f"(v[10]), "=f"(v[11]), "=f"(v[12]), "=f"(v[13]), "=f"(v[14]), "=f"(v[15])
                 : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait_ld(float (&v)[16])
{
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+f"(v[0]), "+f"(v[1]), "+f"(v[2]), "+f"(v[3]), "+f"(v[4]), "+f"(v[5]), "+f"(v[6]), "+f"(v[7]), "+f"(v[8]),
                   "+f"(v[9]), "+f"(v[10]), "+f"(v[11]), "+f"(v[12]), "+f"(v[13]), "+f"(v[14]), "+f"(v[15]) :: "memory");
}

// A job's geometry in registers.  (The descriptors are kernel parameters: read with a run-time index a field costs some
// hundred cycles each time, 700 per tile when the geometry was taken from there tile by tile.)
struct JobTiles {
    int n_2d, n_3d, t2;           // tokens per modality; key tiles of the 2D segment
    int first, count;             // the tiles that fall to this CTA: [first, first + count)
    __device__ __forceinline__ JobTiles() {}
    __device__ __forceinline__ JobTiles(const SampleDev& s, int rank, int lg)     // rank of 2^lg CTAs
    {
        n_2d = s.n_2d; n_3d = s.n_3d;
        t2 = (n_2d + kKeyTile - 1) / kKeyTile;
        const int T = t2 + (n_3d + kKeyTile - 1) / kKeyTile;
        first = (T * rank) >> lg;
        count = ((T * (rank + 1)) >> lg) - first;
    }
    // tile t of the CTA's: keys that exist, index of its first key in visual order
    __device__ __forceinline__ int valid(int t) const
    {
        const int g = first + t;
        return min(kKeyTile, g < t2 ? n_2d - g * kKeyTile : n_3d - (g - t2) * kKeyTile);
    }
    __device__ __forceinline__ int vis0(int t) const
    {
        const int g = first + t;
        return g < t2 ? g * kKeyTile : n_2d + (g - t2) * kKeyTile;
    }
};

// What a softmax warp needs to know about a job.
struct SoftJob {
    JobTiles tr;
    unsigned long long* acc;      // the sample's accumulators, or null
    float* alpha;                 // the sample's attention copy of this head, or null
    int64_t stride_q;
    int n_txt;
    float hn;                     // heads x text queries: the weights carry its inverse
    int slot0, slots, width;      // slot of the job's first tile, slots in the ring, columns per slot
    uint32_t parity0;             // parity of that slot's use
    uint32_t lane_base;           // tensor-memory address of the warp's 32 lanes
    float cscale;
    __device__ __forceinline__ int slot(int t) const { const int u = slot0 + t; return u >= slots ? u - slots : u; }   // a job has at most `slots` tiles
    __device__ __forceinline__ uint32_t parity(int t) const { return parity0 ^ (slot0 + t >= slots ? 1u : 0u); }
    __device__ __forceinline__ uint32_t cols(int t) const { return lane_base + static_cast<uint32_t>(slot(t) * width); }
};

// The warp's references (`nm` = -reference per query) move up to what tile t asks for: an exponent could overflow.  Rare.
// Leaves the factors for everything computed against the old ones in `w`, applied here to what earlier tiles left in
// tensor memory and by the caller to its sums.
// (By value: a job whose address is taken would live in local memory on the usual path, too.)
__device__ __noinline__ void raise_references(uint32_t cols_t, uint32_t lane_base, int first_slot, int slots, int width, int t, int group,
                                              int chunks, float cscale, bool live, float* nm, float* w)
{
    const int lane = threadIdx.x & 31;
    tmem_wait_st();
    for (int c = 0; c < chunks; ++c) {
        float r[16];
        tmem_issue16(cols_t + c * 16, r);
        tmem_wait_ld(r);
#pragma unroll
        for (int i = 0; i < 16; ++i) r[i] = live ? r[i] : -CUDART_INF_F;
        const float red = warp_reduce16<true>(r, lane) * cscale;
        const int col = c * 16 + col16(lane);
        const float old = -nm[col], now = fmaxf(old, red);
        __syncwarp();
        if ((lane & 1) == 0) { nm[col] = -now; w[col] = ex2_approx(old - now); }
        __syncwarp();
        for (int u = group; u < t; u += 2) {
            const int slot = first_slot + u;
            const uint32_t at = lane_base + static_cast<uint32_t>((slot >= slots ? slot - slots : slot) * width + c * 16);
            float e[16];
            tmem_issue16(at, e);
            tmem_wait_ld(e);
#pragma unroll
            for (int i = 0; i < 16; ++i) e[i] *= w[c * 16 + i];
            tmem_st16(at, e);
        }
    }
    tmem_wait_st();
}

// A warp's exponentials and sums for its tiles of a job and N chunks of 16 text queries from chunk c0 on, tile by tile
// (as they arrive, when c0 = 0): exponentials against a reference of the warp's own (the logits of its first key), back to
// tensor memory.  The reference need not be the maximum -- fp32 is as precise at 2^40 as at 1 -- so no pass over the
// tiles and no reduction comes before the exponentials; only an exponent that could overflow moves it.
template <int N>
__device__ __forceinline__ void soft_exps(const SoftJob& j, StreamSmem& sm, int c0, int warp, int lane, int* status)
{
    const int group = warp >> 2, first_key = (warp & 3) * 32;
    float* const nm = sm.m[warp] + c0 * 16;
    float* const my_w = sm.w[warp] + c0 * 16;
    const float2 cs2 = make_float2(j.cscale, j.cscale);
    float2 sum[N * 8];
#pragma unroll
    for (int i = 0; i < N * 8; ++i) sum[i] = make_float2(0.f, 0.f);
    bool have_ref = false;
#pragma unroll 1
    for (int t = group; t < j.tr.count; t += 2) {
        const int valid = j.tr.valid(t);
        const bool live = first_key + lane < valid;
        const uint32_t cols = j.cols(t) + c0 * 16;
        if (c0 == 0) {
            ring_wait<false>(smem_u32(&sm.tfull[j.slot(t)]), j.parity(t), &sm.aborted, status);
            __syncwarp();
            tc_fence_after();
        }
        if (first_key >= valid) continue;                      // no key of this warp in a ragged tile
        float v[N][16];
#pragma unroll 1
        for (;;) {
#pragma unroll
            for (int c = 0; c < N; ++c) tmem_issue16(cols + c * 16, v[c]);
#pragma unroll
            for (int c = 0; c < N; ++c) tmem_wait_ld(v[c]);
            if (valid < kKeyTile) {                            // a ragged tile (uniform; the empty statement keeps it a branch)
                asm volatile("" ::: "memory");
#pragma unroll
                for (int c = 0; c < N; ++c)
#pragma unroll
                    for (int i = 0; i < 16; ++i) v[c][i] = live ? v[c][i] : -CUDART_INF_F;
            }
            if (!have_ref) {                                   // warp-uniform
                have_ref = true;
                if (lane == 0)
#pragma unroll
                    for (int c = 0; c < N; ++c)
#pragma unroll
                        for (int i = 0; i < 16; i += 4)
                            *reinterpret_cast<float4*>(&nm[c * 16 + i]) = make_float4(-v[c][i] * j.cscale, -v[c][i + 1] * j.cscale,
                                                                                      -v[c][i + 2] * j.cscale, -v[c][i + 3] * j.cscale);
                __syncwarp();
            }
            float top[4] = {-CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F};
#pragma unroll
            for (int c = 0; c < N; ++c)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float4 m4 = *reinterpret_cast<const float4*>(&nm[c * 16 + 4 * i]);
                    const float2 y0 = fma2(make_float2(v[c][4 * i], v[c][4 * i + 1]), cs2, make_float2(m4.x, m4.y));
                    const float2 y1 = fma2(make_float2(v[c][4 * i + 2], v[c][4 * i + 3]), cs2, make_float2(m4.z, m4.w));
                    v[c][4 * i] = y0.x; v[c][4 * i + 1] = y0.y; v[c][4 * i + 2] = y1.x; v[c][4 * i + 3] = y1.y;
                    top[i] = fmaxf(top[i], fmaxf(fmaxf(y0.x, y0.y), fmaxf(y1.x, y1.y)));
                }
            if (!__any_sync(0xffffffffu, fmaxf(fmaxf(top[0], top[1]), fmaxf(top[2], top[3])) > kRescaleAt)) break;
            raise_references(cols, j.lane_base + c0 * 16, j.slot0, j.slots, j.width, t, group, N, j.cscale, live, nm, my_w);
#pragma unroll
            for (int i = 0; i < N * 8; ++i) { sum[i].x *= my_w[2 * i]; sum[i].y *= my_w[2 * i + 1]; }
            __syncwarp();
        }
#pragma unroll
        for (int c = 0; c < N; ++c) {
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                v[c][2 * i] = ex2_approx(v[c][2 * i]);
                v[c][2 * i + 1] = ex2_approx(v[c][2 * i + 1]);
                sum[c * 8 + i] = add2(sum[c * 8 + i], make_float2(v[c][2 * i], v[c][2 * i + 1]));
            }
            tmem_st16(cols + c * 16, v[c]);
        }
    }
    if (!have_ref && lane < N * 16) nm[lane] = CUDART_INF_F;   // no key of this warp in the whole job
    __syncwarp();
#pragma unroll
    for (int c = 0; c < N; ++c) {
        float r[16];
#pragma unroll
        for (int i = 0; i < 8; ++i) { r[2 * i] = sum[c * 8 + i].x; r[2 * i + 1] = sum[c * 8 + i].y; }
        const float red = warp_reduce16<false>(r, lane);
        if ((lane & 1) == 0) my_w[c * 16 + col16(lane)] = red;
    }
}

// Per key, the sum of its exponentials weighted by sm.w[warp] (the normalised, head-averaged attention mass), added into
// the accumulators, or (ALPHA) the normalised exponentials one by one into the attention copy; a tile's slot is free once the four warps of its group are done.
template <bool ALPHA>
__device__ __forceinline__ void soft_scores(const SoftJob& j, StreamSmem& sm, int nch, int warp, int lane)
{
    const int key = (warp & 3) * 32 + lane;
    const float* const my_w = sm.w[warp];
#pragma unroll 1
    for (int t = warp >> 2; t < j.tr.count; t += 2) {
        const uint32_t cols = j.cols(t);
        float2 acc[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
        const bool live = key < j.tr.valid(t);
        float* const ap = ALPHA ? j.alpha + static_cast<int64_t>(j.tr.vis0(t) + key) * 4 : nullptr;
        auto add16 = [&](const float (&v)[16], int c) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float4 w4 = *reinterpret_cast<const float4*>(&my_w[c * 16 + 4 * i]);
                if constexpr (ALPHA) {                           // the attention itself (weights are zero past the text queries)
                    if (live && c * 16 + 4 * i < j.n_txt)
                        *reinterpret_cast<float4*>(ap + (c * 4 + i) * j.stride_q) =
                            make_float4(v[4 * i] * w4.x * j.hn, v[4 * i + 1] * w4.y * j.hn, v[4 * i + 2] * w4.z * j.hn, v[4 * i + 3] * w4.w * j.hn);
                } else {
                    acc[0] = fma2(make_float2(v[4 * i], v[4 * i + 1]), make_float2(w4.x, w4.y), acc[0]);
                    acc[1] = fma2(make_float2(v[4 * i + 2], v[4 * i + 3]), make_float2(w4.z, w4.w), acc[1]);
                }
            }
        };
        int c = 0;
#pragma unroll 1
        for (; c + 2 <= nch; c += 2) {
            float v0[16], v1[16];
            tmem_issue16(cols + c * 16, v0);
            tmem_issue16(cols + c * 16 + 16, v1);
            tmem_wait_ld(v0);
            tmem_wait_ld(v1);
            add16(v0, c);
            add16(v1, c + 1);
        }
        if (c < nch) {
            float v0[16];
            tmem_issue16(cols + c * 16, v0);
            tmem_wait_ld(v0);
            add16(v0, c);
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&sm.tempty[j.slot(t)]));
        if constexpr (!ALPHA) {
            const float a = (acc[0].x + acc[0].y) + (acc[1].x + acc[1].y);
            if (live) atomicAdd(j.acc + j.tr.vis0(t) + key, __float2ull_rn(a * kFixScale));
        }
    }
    __syncwarp();
}

// One norm warp: L1 norms of its share of the visual rows of all samples: a run of them; with a tail beside the kernel (HAND) every n_w-th, so that the
// samples' norms are complete in the samples' order.  Rows come by bulk
// copies, kNormStages pieces in flight per warp, so that they take their part of the memory bandwidth without registers
// or a CTA of their own.  What bounds it is a piece's fixed cost and the adds of its sums, not the bytes in flight (adaptive steps of
// 16 requests of 768 tokens: two pieces in flight 99.9 us, three 98.4; pieces of 4 KB 110.8; a run of rows instead of every n_w-th, whose
// sample has to be looked up each time, 97.8 instead of 98.4; four sums beside one another instead of one chain 94.8; eight loads at once 93.7).
template <bool HAND, bool MIXED>
__device__ __forceinline__ void norm_warp(const BatchDesc& bd, const StreamArgs& a, StreamSmem& sm, uint32_t buf, int nw, int lane)
{
    const bool one = elect_one();
    int rows = 0;                                        // of all samples
    for (int b = 0; b < a.n_samples; ++b) rows += bd.s[b].n_2d + bd.s[b].n_3d;
    const int w = static_cast<int>(blockIdx.x) * kNormWarps + nw, n_w = static_cast<int>(gridDim.x) * kNormWarps;
    // a run of rows; every n_w-th where somebody waits for one sample after another
    const int step = HAND ? n_w : 1;
    const int first = HAND ? w : static_cast<int>(static_cast<int64_t>(rows) * w / n_w);
    const int count = HAND ? (rows - w + n_w - 1) / n_w : static_cast<int>(static_cast<int64_t>(rows) * (w + 1) / n_w) - first;
    const int pieces = (a.row_bytes + static_cast<int>(kNormPiece) - 1) / static_cast<int>(kNormPiece), n = max(count, 0) * pieces;
    // The row next to be fetched: visual index fv of sample fb, whose geometry stays in registers (a run-time index into the
    // kernel's parameters costs some hundred cycles).
    int fb = 0, fv = first, n_2d = 0, n_vis = 0, row_2d = 0, row_3d = 0;
    auto sample = [&]() {
        const SampleDev& s = bd.s[MIXED ? a.by_row[fb] : fb];
        n_2d = s.n_2d;
        n_vis = s.n_2d + s.n_3d;
        row_2d = s.seq_off + s.off_2d;
        row_3d = s.seq_off + s.off_3d - s.n_2d;
    };
    sample();
    while (fv >= n_vis && fb < a.n_samples - 1) { fv -= n_vis; ++fb; sample(); }
    float* out = a.l1 + a.vis0 + first;                  // the one next to be summed
    int fp = 0;
    auto fetch = [&](int st) {
        const int row = (fv < n_2d ? row_2d : row_3d) + fv;
        const uint32_t at = static_cast<uint32_t>(fp) * kNormPiece, bytes = min(kNormPiece, static_cast<uint32_t>(a.row_bytes) - at);
        if (one) {
            const uint32_t bar = smem_u32(&sm.nfull[nw][st]);
            mbar_expect_tx(bar, bytes);
            bulk_load(buf + static_cast<uint32_t>(st) * kNormPiece, a.hidden + static_cast<int64_t>(row) * a.row_bytes + at, bytes, bar);
        }
        if (++fp == pieces) {
            fp = 0;
            if constexpr (HAND) {
                fv += step;
                while (fv >= n_vis && fb < a.n_samples - 1) { fv -= n_vis; ++fb; sample(); }
            } else if (++fv == n_vis && fb < a.n_samples - 1) { fv = 0; ++fb; sample(); }
        }
    };
    pdl_wait();                                          // the rows may come from the kernel before this one
    for (int i = 0; i < min(kNormStages, n); ++i) fetch(i);
    int st = 0, piece = 0;
    uint32_t phase = 0;
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
    for (int i = 0; i < n; ++i) {
        const bool ok = ring_wait<false>(smem_u32(&sm.nfull[nw][st]), phase, &sm.aborted, a.status);
        if (!__all_sync(0xffffffffu, ok)) {              // gave up: let the copies in flight land before the CTA may end
            const uint64_t t0 = global_ns();
            while (global_ns() - t0 < 1000000ull) { }
            break;
        }
        const uint32_t bytes = min(kNormPiece, static_cast<uint32_t>(a.row_bytes) - static_cast<uint32_t>(piece) * kNormPiece);
        const uint32_t src = buf + static_cast<uint32_t>(st) * kNormPiece;
#pragma unroll 8
        for (uint32_t at = lane * 16; at < bytes; at += 512) {
            uint32_t u[4];
            asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(u[0]), "=r"(u[1]), "=r"(u[2]), "=r"(u[3]) : "r"(src + at));
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                acc[e] += fabsf(__uint_as_float(u[e] << 16));           // low bf16
                acc[e] += fabsf(__uint_as_float(u[e] & 0xFFFF0000u));   // high bf16
            }
        }
        __syncwarp();                                    // everyone has read the piece
        if (i + kNormStages < n) fetch(st);
        if (++st == kNormStages) { st = 0; phase ^= 1; }
        if (++piece == pieces) {
            piece = 0;
            float r = (acc[0] + acc[1]) + (acc[2] + acc[3]);
#pragma unroll
            for (int off = 16; off >= 1; off >>= 1) r += __shfl_xor_sync(0xffffffffu, r, off);
            if (lane == 0) *out = r;
            out += step;
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[e] = 0.f;
        }
    }
}

// grid = clusters x cluster size (1-D), one CTA per multiprocessor.
// ROOM: the feature norms are to run beside this kernel (norms_inside_pays says no).  Its ten warps put three on two of a
// multiprocessor's four register files (16384 registers each): at the 168 registers a thread that the compiler takes these are
// full, no CTA of the norms fits, and they start when the scores are done.  144 leave room for two warps of 32 registers in
// each, at the price of 8 bytes a thread stored and 24 loaded (with 128 these are 68 and 144: 16 requests of 768 tokens 97 ->
// 106 us when their norms ran beside).  8 requests of 3584 tokens, 64 queries, took 161.7 us with 144 and 162.0 with 168 (they have the tail
// beside this kernel since, and their norms in it).
// Where no norms run beside, the registers are worth more to the attention copy: 16 patch-by-patch steps 76.5 us with 168, 78.6
// with 144; 16 adaptive requests 93.7 and 93.0.
// HAND: the tail of the step runs beside this kernel (launch_select_copy_beside); a variant of its own, because in the others the skipped code
// cost steps of 20 to 40 us 1 to 2 %.
// MIXED: the samples are not in the order of their rows, and the norm warps take them by by_row; a variant of its own for the same reason.
template <bool ROOM, bool HAND, bool MIXED>
__global__ void __maxnreg__(ROOM ? 144 : kStreamRegs)
salience_stream_kernel(const __grid_constant__ BatchDesc bd, const __grid_constant__ CUtensorMap tmap_q,
                       const __grid_constant__ CUtensorMap tmap_k, const __grid_constant__ StreamArgs a)
{
    const int W = a.width;
    extern __shared__ uint8_t dyn_smem_raw[];
    uint8_t* dyn = dyn_smem_raw + ((1024u - (smem_u32(dyn_smem_raw) & 1023u)) & 1023u);   // swizzle atoms are 1 KB
    __shared__ StreamSmem sm;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint32_t csize, crank = cluster_ctarank();
    asm volatile("mov.u32 %0, %%cluster_nctaid.x;" : "=r"(csize));
    const int lg = 31 - __clz(csize);                    // cluster sizes are powers of two
    const int first_job = blockIdx.x >> lg, job_step = gridDim.x >> lg;
    const int b_step = job_step / a.n_heads, h_step = job_step - b_step * a.n_heads;
    const int b_first = first_job / a.n_heads, h_first = first_job - b_first * a.n_heads;
    // the next job's sample and head
    auto advance = [&](int& b, int& h) {
        b += b_step;
        h += h_step;
        if (h >= a.n_heads) { h -= a.n_heads; ++b; }
    };
    const int khalves = (a.head_dim * a.esize + 127) / 128;
    uint8_t* const Qs = dyn + static_cast<size_t>(a.stages) * kStageBytes;      // two buffers of khalves x W rows x 128 B
    const uint32_t q_bytes = static_cast<uint32_t>(khalves) * (W * 128);

    if (tid == 0) {
        for (int i = 0; i < a.stages; ++i) { mbar_init(smem_u32(&sm.kfull[i]), 1); mbar_init(smem_u32(&sm.kempty[i]), 1); }
        for (int i = 0; i < 2; ++i) {
            mbar_init(smem_u32(&sm.qfull[i]), 1); mbar_init(smem_u32(&sm.qempty[i]), 1);
        }
        for (int i = 0; i < kPairBufs; ++i) mbar_init(smem_u32(&sm.xbar[i]), 1);
        if (!ROOM)
            for (int i = 0; i < kNormWarps * kNormStages; ++i) mbar_init(smem_u32(&sm.nfull[0][0] + i), 1);
        for (int i = 0; i < a.slots; ++i) { mbar_init(smem_u32(&sm.tfull[i]), 1); mbar_init(smem_u32(&sm.tempty[i]), 4); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        sm.aborted = 0;
    }
    if constexpr (HAND) {
        // The tail may start as soon as every CTA of this kernel has let it (below): its hand-over words, and the norms, which are
        // words of that kind then, are re-armed before.  Their last users finished long ago; the first to write one of them is the
        // tail, or the norm warp that re-arms it (a CTA may start when others have written norms already).
        const SampleDev &s0 = bd.s[0], &sn = bd.s[a.n_samples - 1];
        const int at = static_cast<int>(blockIdx.x * blockDim.x) + tid, all = static_cast<int>(gridDim.x * blockDim.x);
        for (int i = s0.out_off + at; i < sn.out_off + sn.n_out; i += all) a.rearm[i * kListStride] = -1;
        if (!ROOM && a.hidden && warp > kSoftWarps + 1) {
            const int w = static_cast<int>(blockIdx.x) * kNormWarps + warp - kSoftWarps - 2, n_w = static_cast<int>(gridDim.x) * kNormWarps;
            const int end = sn.vis_off + sn.n_2d + sn.n_3d;
            for (int i = s0.vis_off + w + lane * n_w; i < end; i += 32 * n_w) a.l1[i] = __uint_as_float(kNoNorm);
        }
    }
    // all 512 columns: the launcher's shared-memory footprint keeps every other user of tensor memory off this multiprocessor
    if (warp == kSoftWarps + 1) tmem_alloc(smem_u32(&sm.tmem), kTmemColsPerSm);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (csize > 1) {                          // no pair may be sent to a CTA that has not set up its barriers
        cluster_arrive_release();
        cluster_wait_acquire();
    }
    const uint32_t tmem_base = sm.tmem;
    volatile int* const aborted = &sm.aborted;

    // The loading warp and the MMA warp run their loops as whole warps, all values the same in every lane, and one
    // elected lane issues: coordinates and descriptors then stay in uniform registers.  (As a single-thread branch the
    // same loops moved every operand there one by one: 1.0 us per key tile instead of 0.25.)
    if (warp == kSoftWarps) {
        // ---------------------------------------------------------------- loads
        const bool one = elect_one();
        if (one) {
            prefetch_tensormap(&tmap_q);
            prefetch_tensormap(&tmap_k);
        }
        if constexpr (HAND) __threadfence();          // the CTA's re-armed words (behind the block barrier) before the trigger
        pdl_wait();
        if (a.stamps && one && blockIdx.x < kStampSlots) a.stamps[2 * blockIdx.x] = global_ns();
        pdl_trigger();                        // whatever the kernel before this one wrote is complete
        const int box_elems = 128 / a.esize;
        int stage = 0, n_live = 0;
        uint32_t phase = 0;
        bool ok = true;
        for (int job = first_job, b = b_first, h = h_first; ok && job < a.n_jobs; job += job_step, advance(b, h)) {
            const SampleDev& s = bd.s[b];
            const JobTiles tr(s, crank, lg);
            if (tr.count == 0) continue;
            const int npad = (s.n_txt + 15) & ~15, qb = n_live & 1;
            const int row_2d = s.seq_off + s.off_2d, row_3d = s.seq_off + s.off_3d, row_q = s.seq_off + s.off_txt;
            ok = ring_wait<false>(smem_u32(&sm.qempty[qb]), ((n_live >> 1) & 1) ^ 1, aborted, a.status);
            if (!ok) break;
            if (one) {
                const uint32_t qbar = smem_u32(&sm.qfull[qb]);
                mbar_expect_tx(qbar, static_cast<uint32_t>(khalves * npad) * 128u);
                for (int kh = 0; kh < khalves; ++kh)
                    for (int c = 0; c < npad / 16; ++c)
                        tma_load_3d(smem_u32(Qs + qb * q_bytes + kh * npad * 128 + c * 2048), &tmap_q, kh * box_elems, h,
                                    row_q + c * 16, qbar);
            }
            ++n_live;
            const int hk = h / a.kv_group;
            for (int t = 0; ok && t < tr.count; ++t) {
                const int g = tr.first + t, row0 = g < tr.t2 ? row_2d + g * kKeyTile : row_3d + (g - tr.t2) * kKeyTile;
                for (int kh = 0; kh < khalves; ++kh) {
                    ok = ring_wait<false>(smem_u32(&sm.kempty[stage]), phase ^ 1, aborted, a.status);
                    if (!ok) break;
                    if (one) {
                        const uint32_t bar = smem_u32(&sm.kfull[stage]);
                        mbar_expect_tx(bar, kStageBytes);
                        tma_load_3d(smem_u32(dyn) + static_cast<uint32_t>(stage) * kStageBytes, &tmap_k, kh * box_elems, hk, row0, bar);
                    }
                    if (++stage == a.stages) { stage = 0; phase ^= 1; }
                }
            }
        }
        if (!ok) {                            // gave up: let the copies in flight land before the CTA may end
            const uint64_t t0 = global_ns();
            while (global_ns() - t0 < 1000000ull) { }
        }
    } else if (warp == kSoftWarps + 1) {
        // ---------------------------------------------------------------- MMAs
        const bool one = elect_one();
        const int ksteps = (a.head_dim * a.esize + 31) / 32;       // an instruction consumes 32 bytes of every row
        const uint64_t k_desc0 = smem_desc_sw128(smem_u32(dyn)), q_desc0 = smem_desc_sw128(smem_u32(Qs));   // (addresses / 16 in the low bits)
        int stage = 0, slot = 0, n_live = 0;
        uint32_t phase = 0, sphase = 0;
        bool ok = true;
        for (int job = first_job, b = b_first, h = h_first; ok && job < a.n_jobs; job += job_step, advance(b, h)) {
            const SampleDev& s = bd.s[b];
            const JobTiles tr(s, crank, lg);
            if (tr.count == 0) continue;
            const int npad = (s.n_txt + 15) & ~15, qb = n_live & 1;
            const uint32_t idesc = idesc_by_size(a.esize, npad);
            ok = ring_wait<false>(smem_u32(&sm.qfull[qb]), (n_live >> 1) & 1, aborted, a.status);
            ++n_live;
            for (int t = 0; ok && t < tr.count; ++t) {
                ok = ring_wait<false>(smem_u32(&sm.tempty[slot]), sphase ^ 1, aborted, a.status);
                for (int kh = 0; ok && kh < khalves; ++kh) {
                    ok = ring_wait<false>(smem_u32(&sm.kfull[stage]), phase, aborted, a.status);
                    if (!ok) break;
                    tc_fence_after();
                    const uint64_t kd = desc_plus(k_desc0, static_cast<uint32_t>(stage) * (kStageBytes >> 4));
                    const uint64_t qd = desc_plus(q_desc0, (static_cast<uint32_t>(qb) * q_bytes + static_cast<uint32_t>(kh * npad) * 128u) >> 4);
                    if (one) {
                        umma_box(a.esize, tmem_base + slot * W, kd, qd, idesc, min(4, ksteps - kh * 4), kh > 0);
                        umma_commit(smem_u32(&sm.kempty[stage]));
                    }
                    if (++stage == a.stages) { stage = 0; phase ^= 1; }
                }
                if (!ok) break;
                if (one) umma_commit(smem_u32(&sm.tfull[slot]));
                if (++slot == a.slots) { slot = 0; sphase ^= 1; }
            }
            if (ok && one) umma_commit(smem_u32(&sm.qempty[qb]));
        }
    } else if (!ROOM && warp > kSoftWarps + 1) {
        // ---------------------------------------------------------------- feature norms
        const int nw = warp - kSoftWarps - 2;
        if (a.hidden) norm_warp<HAND, MIXED>(bd, a, sm, smem_u32(dyn) + a.norm_off + static_cast<uint32_t>(nw * kNormStages) * kNormPiece, nw, lane);
    } else {
        // ---------------------------------------------------------------- softmax
        SoftJob j;
        j.alpha = nullptr; j.stride_q = a.alpha.stride_q;
        j.slot0 = 0; j.slots = a.slots; j.width = W; j.parity0 = 0;
        j.lane_base = tmem_base + (static_cast<uint32_t>((warp & 3) * 32) << 16);
        j.cscale = 1.4426950408889634f * rsqrtf(static_cast<float>(a.head_dim));   // log2 domain
        float* const my_w = sm.w[warp];
        bool waited = false;
        int jn = 0, scored = -1;                         // sample of the job before
        // A job's scores are in the accumulators when every softmax warp has passed the next barrier: one thread that has no part
        // in the exchange tells (its fence takes about as long as that does; behind a barrier of its own at the end of every job
        // 8 requests of 3584 tokens took 164.4 us instead of 155.4).
        auto tell = [&]() {
            if (HAND && scored >= 0 && tid == kSoftThreads - 1) {
                __threadfence();
                atomicAdd(a.hand + scored, 1);
            }
        };
        for (int job = first_job, b = b_first, h = h_first; job < a.n_jobs; job += job_step, ++jn, advance(b, h)) {
            const SampleDev& s = bd.s[b];
            j.tr = JobTiles(s, crank, lg);
            j.acc = a.acc64 + s.vis_off;
            const int n_txt = s.n_txt, npad = (n_txt + 15) & ~15;
            j.n_txt = n_txt;
            j.hn = static_cast<float>(a.n_heads) * static_cast<float>(n_txt);
            if (!ROOM && a.alpha.ptr) j.alpha = a.alpha.ptr + static_cast<int64_t>(h) * a.alpha.stride_h + static_cast<int64_t>(s.vis_off) * 4;
            if (!HAND && a.rearm && h == 0 && crank == 0) {    // the tail kernel's hand-over words; their last users finished long ago
                if (!a.rearm_rec) {
                    for (int i = tid; i < s.n_out; i += kSoftThreads) a.rearm[(s.out_off + i) * kListStride] = -1;
                } else {                              // the patch-by-patch tail: its list words, and three words per patch
                    for (int i = tid; i < kHandWords; i += kSoftThreads) a.rearm[s.cap_off + i] = -1;
                    for (int i = tid; i < s.n_txt + s.n_2d + s.n_3d; i += kSoftThreads)
                        a.rearm[s.cap_off + kHandWords + i * kListStride] = -1;
                    for (int i = tid; i < 3 * s.n_2d; i += kSoftThreads) a.rearm_rec[static_cast<int64_t>(s.vis_off / 2) * 3 + i] = ~0ull;
                }
            }
            const int nch = npad >> 4;
            {
                int c = 0;
                for (; c + 2 <= nch; c += 2) soft_exps<2>(j, sm, c, warp, lane, a.status);
                if (c < nch) soft_exps<1>(j, sm, c, warp, lane, a.status);
                tmem_wait_st();
            }
            soft_barrier();
            tell();
            scored = b;
            // ---- one thread per query: the pairs of the warps, then those of the cluster's CTAs
            if (tid < npad) {
                float mk[kSoftWarps], mx = -CUDART_INF_F, z = 0.f;
#pragma unroll
                for (int k = 0; k < kSoftWarps; ++k) { mk[k] = -sm.m[k][tid]; mx = fmaxf(mx, mk[k]); }
#pragma unroll
                for (int k = 0; k < kSoftWarps; ++k)
                    if (mk[k] > -CUDART_INF_F) z += sm.w[k][tid] * ex2_approx(mk[k] - mx);
                if (csize > 1) {
                    const int xb = jn & (kPairBufs - 1);
                    const uint32_t xbar = smem_u32(&sm.xbar[xb]);
                    // (pairs may land before the count is armed: the phase cannot complete without this arrival)
                    if (tid == 0) mbar_expect_tx(xbar, csize * static_cast<uint32_t>(npad) * 8u);
                    for (uint32_t r = 0; r < csize; ++r) st_async_pair(smem_u32(&sm.peer[xb][crank][tid]), xbar, r, make_float2(mx, z));
                    ring_wait<true>(xbar, (jn / kPairBufs) & 1, &sm.aborted, a.status);
                    mx = -CUDART_INF_F;
                    z = 0.f;
                    for (uint32_t r = 0; r < csize; ++r) mx = fmaxf(mx, sm.peer[xb][r][tid].x);
                    for (uint32_t r = 0; r < csize; ++r) {
                        const float2 p = sm.peer[xb][r][tid];
                        if (p.x > -CUDART_INF_F) z += p.y * ex2_approx(p.x - mx);
                    }
                }
                sm.g[tid] = mx;
                sm.iz[tid] = tid < n_txt && z > 0.f ? 1.f / z / j.hn : 0.f;
            }
            if (!waited) { pdl_wait(); waited = true; }      // the accumulators were read and cleared by an earlier selection
            soft_barrier();
            for (int i = lane; i < npad; i += 32) {          // this warp's exponentials -> normalised, head-averaged
                const float mk = -sm.m[warp][i];
                my_w[i] = mk == -CUDART_INF_F ? 0.f : ex2_approx(mk - sm.g[i]) * sm.iz[i];
            }
            __syncwarp();
            if (!ROOM && a.alpha.ptr) soft_scores<true>(j, sm, nch, warp, lane);
            else soft_scores<false>(j, sm, nch, warp, lane);
            j.slot0 += j.tr.count;
            if (j.slot0 >= a.slots) { j.slot0 -= a.slots; j.parity0 ^= 1u; }
        }
        if constexpr (HAND) {
            soft_barrier();
            tell();
        }
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (warp == kSoftWarps + 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, kTmemColsPerSm);
    }
    if (csize > 1) {                          // a CTA that gave up must not leave while a peer may still send to it
        cluster_arrive_release();
        cluster_wait_acquire();
    }
    if (a.stamps && tid == 0 && blockIdx.x < kStampSlots) a.stamps[2 * blockIdx.x + 1] = global_ns();
}

int padded_text(const BatchDesc& bd)
{
    int n = 1;
    for (int b = 0; b < bd.n; ++b) n = std::max(n, bd.s[b].n_txt);
    return (n + 15) / 16 * 16;
}
int max_tiles(const BatchDesc& bd)
{
    int t = 1;
    for (int b = 0; b < bd.n; ++b)
        t = std::max(t, (bd.s[b].n_2d + kKeyTile - 1) / kKeyTile + (bd.s[b].n_3d + kKeyTile - 1) / kKeyTile);
    return t;
}

// The smallest cluster whose CTAs hold their share of a job's logits in tensor memory; a larger one while jobs are
// fewer than multiprocessors and the tiles can still be shared out.  0: none holds them.
int stream_cluster(int n_jobs, int tiles, int slots, int sms)
{
    int cluster = 1;
    while (cluster < kMaxCluster && ((tiles + cluster - 1) / cluster > slots || (n_jobs * cluster * 2 <= sms && cluster * 2 <= tiles)))
        cluster *= 2;
    return (tiles + cluster - 1) / cluster > slots ? 0 : cluster;
}

// The launch's samples in the order in which their jobs are taken (longest_first_pays), `room` for them where that is not the order given; and which of them
// comes where by its rows.
const BatchDesc& in_order(const BatchDesc& given, int n_heads, int clusters, BatchDesc& room, uint8_t* by_row)
{
    int cost[kMaxChunk];
    uint8_t order[kMaxChunk];
    for (int b = 0; b < given.n; ++b) {
        const SampleDev& s = given.s[b];
        cost[b] = job_cost((s.n_2d + kKeyTile - 1) / kKeyTile + (s.n_3d + kKeyTile - 1) / kKeyTile, (s.n_txt + 15) & ~15);
    }
    for (int b = 0; b < given.n; ++b) by_row[b] = static_cast<uint8_t>(b);
    if (!longest_first_pays(cost, given.n, n_heads, clusters, order)) return given;
    room = given;
    for (int b = 0; b < given.n; ++b) {
        room.s[b] = given.s[order[b]];
        by_row[order[b]] = static_cast<uint8_t>(b);
    }
    return room;
}

int stream_threads(const StreamArgs& a) { return kStreamThreads + (a.hidden ? 32 * kNormWarps : 0); }

// Clusters that run at once (a second wave of a persistent grid would double its time), with the kernel set up.
template <bool ROOM, bool HAND, bool MIXED>
cudaError_t launch_size(int threads, int cluster, int* n)
{
    const void* kern = reinterpret_cast<const void*>(salience_stream_kernel<ROOM, HAND, MIXED>);
    static KernelSetup ks;
    cudaError_t e = setup_kernel(ks, kern, kStreamSmem, kTmemColsPerSm);
    if (e == cudaSuccess) e = clusters_at_once(ks, kern, threads, kStreamSmem, cluster, n);
    return e == cudaSuccess && *n < 1 ? cudaErrorInvalidConfiguration : e;
}

template <bool ROOM, bool HAND, bool MIXED>
cudaError_t launch_variant(const BatchDesc& bd, const CUtensorMap* tq, const CUtensorMap* tk, const StreamArgs& a, int cluster, int clusters, cudaStream_t stream)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(clusters * cluster));
    cfg.blockDim = dim3(static_cast<unsigned>(stream_threads(a)));
    cfg.dynamicSmemBytes = kStreamSmem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = static_cast<unsigned>(cluster);
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1] = pdl_attribute();
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, salience_stream_kernel<ROOM, HAND, MIXED>, bd, *tq, *tk, a);
}

template <bool ROOM, bool HAND>
cudaError_t launch_stream(const BatchDesc& given, const CUtensorMap* tq, const CUtensorMap* tk, StreamArgs& a, int cluster, cudaStream_t stream)
{
    int n = 0;
    cudaError_t e = launch_size<ROOM, HAND, false>(stream_threads(a), cluster, &n);
    if (e != cudaSuccess) return e;
    if constexpr (HAND)                  // (the samples as they are: the tail takes them in that order)
        return launch_variant<ROOM, true, false>(given, tq, tk, a, cluster, clusters_beside_tail(a.n_jobs, n, cluster, sm_count_of_current_device()), stream);
    const int clusters = a.hidden ? n : std::min(a.n_jobs, n);       // (norms are shared out over all CTAs)
    BatchDesc room;
    const BatchDesc& bd = in_order(given, a.n_heads, clusters, room, a.by_row);
    if constexpr (!ROOM)
        if (a.hidden && &bd != &given) {
            e = launch_size<ROOM, HAND, true>(stream_threads(a), cluster, &n);       // (sets the variant up)
            return e == cudaSuccess ? launch_variant<ROOM, HAND, true>(bd, tq, tk, a, cluster, clusters, stream) : e;
        }
    return launch_variant<ROOM, HAND, false>(bd, tq, tk, a, cluster, clusters, stream);
}

}  // namespace

// no CTA with 32 columns of tensor memory (at least 1/17 of the shared memory, smem_for_tmem) fits beside one
static_assert(kSmemPerSm - static_cast<int>(kStreamSmem + sizeof(StreamSmem)) - kSmemReservedPerCta < kSmemPerSm / 17,
              "the streaming kernel must be alone with the tensor memory of its multiprocessor");
static_assert((kStreamThreads + 32 * kNormWarps) * kStreamRegs <= 65536, "the norm warps must fit the register file beside the others");

cudaError_t stream_beside_tail(const BatchDesc& bd, int n_heads, int64_t head_bytes, int64_t key_bytes, int64_t row_bytes, int* free_sms, int* parts)
{
    *free_sms = *parts = 0;
    const int sms = sm_count_of_current_device(), npad = padded_text(bd), jobs = bd.n * n_heads;
    const int cluster = stream_cluster(jobs, max_tiles(bd), std::min(kMaxSlots, kTmemColsPerSm / npad), sms);
    int64_t tokens = 0;
    for (int b = 0; b < bd.n; ++b) tokens += bd.s[b].n_2d + bd.s[b].n_3d;
    int n = cluster > 1 ? 1 : sms;
    const auto pays = [&]() { return tail_beside_pays({tokens, bd.n, jobs, n, head_bytes, key_bytes, row_bytes}); };
    if (cluster == 0 || !pays()) return cudaSuccess;         // (clusters: the runtime is asked only where the rest says yes)
    if (cluster > 1) {
        const cudaError_t e = launch_size<false, true, false>(kStreamThreads + 32 * kNormWarps, cluster, &n);
        if (e != cudaSuccess) return e;
        if (!pays()) return cudaSuccess;
    }
    *free_sms = sms - clusters_beside_tail(jobs, n, cluster, sms) * cluster;
    *parts = n_heads * cluster;
    return cudaSuccess;
}

cudaError_t launch_salience_stream(const BatchDesc& bd, int n_heads, int kv_group, int head_dim, int esize,
                                   const CUtensorMap* tmap_q, const CUtensorMap* tmap_k, unsigned long long* acc64, int* status,
                                   AlphaOut alpha, int32_t* rearm, unsigned long long* rearm_rec,
                                   unsigned long long* stamps, bool norms_beside, const void* hidden, int row_bytes, float* l1, int32_t* hand,
                                   cudaStream_t stream)
{
    const int sms = sm_count_of_current_device();
    const int npad = padded_text(bd), tiles = max_tiles(bd);
    StreamArgs a;
    a.n_heads = n_heads; a.kv_group = kv_group; a.head_dim = head_dim; a.esize = esize;
    a.width = npad;
    a.slots = std::min(kMaxSlots, kTmemColsPerSm / npad);
    a.n_jobs = bd.n * n_heads;
    a.acc64 = acc64; a.status = status; a.alpha = alpha; a.rearm = rearm;
    a.rearm_rec = rearm_rec; a.stamps = stamps; a.hand = hand;
    const int cluster = stream_cluster(a.n_jobs, tiles, a.slots, sms);
    if (cluster == 0) return cudaErrorInvalidConfiguration;
    const size_t q_bytes = 2 * static_cast<size_t>((head_dim * esize + 127) / 128) * npad * 128;
    // shared memory: the ring of key boxes, two buffers of queries, the norm warps' pieces of rows
    const size_t norm_bytes = hidden ? static_cast<size_t>(kNormWarps * kNormStages) * kNormPiece : 0;
    a.stages = static_cast<int>(std::min<size_t>(hand ? kStagesBesideTail : kMaxStages, (kStreamSmem - 1024 - q_bytes - norm_bytes) / kStageBytes));
    if (a.stages < 4 || (hidden && norms_beside)) return cudaErrorInvalidConfiguration;
    a.hidden = static_cast<const uint8_t*>(hidden);
    a.l1 = l1; a.row_bytes = row_bytes; a.n_samples = bd.n; a.vis0 = bd.s[0].vis_off;
    a.norm_off = static_cast<uint32_t>(a.stages * kStageBytes + q_bytes);
    if (norms_beside && !alpha.ptr) return launch_stream<true, false>(bd, tmap_q, tmap_k, a, cluster, stream);
    if (hand) return launch_stream<false, true>(bd, tmap_q, tmap_k, a, cluster, stream);
    return launch_stream<false, false>(bd, tmap_q, tmap_k, a, cluster, stream);
}

}  // namespace mvla
