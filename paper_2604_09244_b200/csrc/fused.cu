// Latency-shaped scoring kernels (Sec. 3.2.1 of the paper): bf16 and e4m3 on the tensor cores, fp32 by FMAs; for
// launches whose CTAs all run at once (batches and larger samples: stream.cu).
//
// Same decomposition as the generic salience kernel (one cluster per (sample, head), one CTA per one or
// two tiles of 128 keys; TMA -> shared memory -> tcgen05.mma -> tensor memory), but built as one short
// dependency chain, because at ~40 KB of input per CTA the kernel is latency bound.  Of the 5 us that one sample of
// 768 tokens and 32 heads of 128 takes (2.6 us would be its share of the key stream at full bandwidth), 1.5 are the
// tiles' flight, 0.6 the MMAs, 1.7 the softmax with the exchange, the rest launch and drain.  So:
//   * everything that reads nothing of the kernel before comes before the wait for it (barriers, cluster arrive,
//     tensor-memory allocation, hand-over words, load operands): a release issued behind the loads waits as long as
//     they do.  A step of one frame 12.8 -> 12.0 us, eight action steps 161.8 -> 153.4;
//   * a variant per use (scores, with the logit cache, with the attention copy): the code runs once per launch from
//     a cold instruction cache, and what a step does not use cost eight action steps 4 us;
//   * exponents are taken against the logits of each warp's first key, not a maximum: two block barriers less;
//   * each thread reads ALL its logits from tensor memory once (one wide tcgen05.ld) and keeps them in
//     registers through exp2 -> sum -> weighted sum;
//   * the per-query (max, sum) pairs travel between the CTAs of a cluster as asynchronous remote
//     shared-memory stores that credit the receiver's mbarrier when they land (st.async with
//     complete_tx): one one-way trip, no cluster-wide hardware barrier and no fence on the critical path;
//   * per-head contributions are added into one 64-bit fixed-point accumulator per token (scale 2^60):
//     integer adds commute, so the sum over heads is exact and independent of scheduling.
#include "common.cuh"
#include "device_utils.cuh"
#include "select_impl.cuh"
#include "tmem_ld.cuh"
#include "tmem_plan.h"

#include <algorithm>
#include <cstring>

namespace mvla {
namespace {

constexpr int kFastThreads = 128;

// Shared memory of the softmax part, per warp of the four that cover a tile's 128 keys, and per query.
struct FastSmem {
    alignas(16) float m[4][kMaxText];        // -reference of the exponents (log2 domain)
    alignas(16) float w[4][kMaxText];        // sum of the exponentials, then their weight in the scores
    float2 peer[kMaxCluster][kMaxText];      // (reference, sum) of every CTA of the cluster
};
constexpr size_t kFastStaticSmem = sizeof(FastSmem) + 32;   // of salience_fast_kernel: + its barriers and a tensor-memory address
// What the softmax part writes.
struct FastOut {
    unsigned long long* acc64;               // null: the attention copy only
    int* status;
    int n_heads;
    AlphaOut alpha;
    bool early;                              // the accumulators need no wait
};

// From the raw dot products of this thread's key(s) -- L[t * TC + i]: tile t, text query c0 + i -- to the outputs.
// vis0[t], valid[t]: the tiles' first visual index and number of keys.
//
// A warp takes its exponentials against a reference of its own, the logits of its first key, not against a maximum
// over the CTA's keys: fp32 is as precise at 2^40 as at 1, so a reference only has to keep the exponents from
// overflowing, and the two shared-memory round trips, two block barriers and the butterfly that found the maximum leave
// the chain (a warp whose exponents exceed kRescaleAt takes its true maxima after all).  The pairs (reference, sum) of
// the four warps are combined per query, then those of the cluster's CTAs.
//
// `before_exchange` runs when every warp has its logits in registers and before anything waits for another CTA.
template <int TCOL, int NTILE, int SPLIT, bool ALPHA, class Hook>
__device__ __forceinline__ void softmax_scores(float (&L)[NTILE * TCOL / SPLIT], const SampleDev& s, const int (&valid)[NTILE],
                                               const int (&vis0)[NTILE], bool ok, int npad, int h, float cscale, uint32_t bar_x,
                                               FastSmem& sm, const FastOut& o, Hook before_exchange)
{
    constexpr int TC = TCOL / SPLIT;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int key = tid & (kFastThreads - 1), kwarp = warp & 3, c0 = (tid / kFastThreads) * TC;
    const uint32_t crank = cluster_ctarank(), csize = gridDim.x;
    float* const nm = sm.m[kwarp] + c0;
    // The registers keep the raw dot products; the scale enters with the exponent below (one FFMA).  Keys
    // past the end of a ragged tile are masked; a full tile needs no pass over the registers at all, and
    // columns past the padded query count are never looked at.
#pragma unroll
    for (int t = 0; t < NTILE; ++t) {
        if (ok && valid[t] == kKeyTile) continue;         // block-uniform
        const bool live = ok && key < valid[t];
#pragma unroll
        for (int i = 0; i < TC; ++i) L[t * TC + i] = live ? L[t * TC + i] : -CUDART_INF_F;
    }

    // ---- references: the warp's first key (zero for a warp without one: its exponentials are all zero)
    if (lane == 0) {
#pragma unroll
        for (int i = 0; i < TC; i += 4) {
            if ((i & 15) == 0 && c0 + i >= npad) break;
            float r[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                r[k] = L[i + k];
#pragma unroll
                for (int t = 1; t < NTILE; ++t) r[k] = valid[0] > kwarp * 32 ? r[k] : L[t * TC + i + k];
                r[k] = r[k] == -CUDART_INF_F ? 0.f : -r[k] * cscale;
            }
            *reinterpret_cast<float4*>(nm + i) = make_float4(r[0], r[1], r[2], r[3]);
        }
    }
    __syncwarp();
    {
        float top = -CUDART_INF_F;
#pragma unroll
        for (int i = 0; i < TC; i += 4) {
            if ((i & 15) == 0 && c0 + i >= npad) break;
            const float4 m4 = *reinterpret_cast<const float4*>(nm + i);
#pragma unroll
            for (int t = 0; t < NTILE; ++t)
                top = fmaxf(top, fmaxf(fmaxf(fmaf(L[t * TC + i], cscale, m4.x), fmaf(L[t * TC + i + 1], cscale, m4.y)),
                                       fmaxf(fmaf(L[t * TC + i + 2], cscale, m4.z), fmaf(L[t * TC + i + 3], cscale, m4.w))));
        }
        if (__any_sync(0xffffffffu, top > kRescaleAt)) {  // rare
#pragma unroll
            for (int qc = 0; qc < TC / 16; ++qc) {
                if (c0 + qc * 16 >= npad) break;
                float m[16];
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    m[i] = L[qc * 16 + i];
#pragma unroll
                    for (int t = 1; t < NTILE; ++t) m[i] = fmaxf(m[i], L[t * TC + qc * 16 + i]);
                }
                const float red = warp_reduce16<true>(m, lane);
                __syncwarp();
                if ((lane & 1) == 0) nm[qc * 16 + col16(lane)] = -red * cscale;
            }
            __syncwarp();
        }
    }

    // ---- exponentials (kept in registers) and their sum per query
#pragma unroll
    for (int qc = 0; qc < TC / 16; ++qc) {
        if (c0 + qc * 16 >= npad) break;
        float sum[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const float mm = nm[qc * 16 + i];
            sum[i] = 0.f;
#pragma unroll
            for (int t = 0; t < NTILE; ++t) {
                const float e = ex2_approx(fmaf(L[t * TC + qc * 16 + i], cscale, mm));
                L[t * TC + qc * 16 + i] = e;
                sum[i] += e;
            }
        }
        const float red = warp_reduce16<false>(sum, lane);
        if ((lane & 1) == 0) sm.w[kwarp][c0 + qc * 16 + col16(lane)] = red;
    }
    __syncthreads();
    before_exchange();

    // ---- one thread per query: the pairs of the CTA's warps, exchanged with the other key tiles of this (sample, head)
    cluster_wait_acquire();                   // every peer is running and has initialised its barriers
    if (tid < npad) {                         // (the other warps park at the barrier below)
        float ref[4], mx = -CUDART_INF_F, z = 0.f;
#pragma unroll
        for (int k = 0; k < 4; ++k) {         // (a warp with a key has a sum of at least one: its reference's)
            ref[k] = sm.w[k][tid] > 0.f ? -sm.m[k][tid] : -CUDART_INF_F;
            mx = fmaxf(mx, ref[k]);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (ref[k] > -CUDART_INF_F) z += sm.w[k][tid] * ex2_approx(ref[k] - mx);
        for (uint32_t r = 0; r < csize; ++r) st_async_pair(smem_u32(&sm.peer[crank][tid]), bar_x, r, make_float2(mx, z));
        const float inv_hn = 1.f / (static_cast<float>(o.n_heads) * static_cast<float>(s.n_txt));
        const bool okx = mbar_wait<true>(bar_x, 0);
        if (!okx) *reinterpret_cast<volatile int*>(o.status) = MVLA_ERR_TIMEOUT;
        mx = -CUDART_INF_F;
        for (uint32_t r = 0; r < csize; ++r) mx = fmaxf(mx, sm.peer[r][tid].x);
        z = 0.f;
        for (uint32_t r = 0; r < csize; ++r) {
            const float2 pr = sm.peer[r][tid];
            if (pr.x > -CUDART_INF_F) z += pr.y * ex2_approx(pr.x - mx);
        }
        const float iz = (tid < s.n_txt && z > 0.f && okx) ? inv_hn / z : 0.f;
#pragma unroll
        for (int k = 0; k < 4; ++k) sm.w[k][tid] = ref[k] > -CUDART_INF_F ? ex2_approx(ref[k] - mx) * iz : 0.f;
    }
    __syncthreads();

    // ---- per key: sum over queries of the normalised probabilities (this head's contribution)
    const float* const w = sm.w[kwarp] + c0;  // 0 past the text queries
    if (!o.early) pdl_wait();                 // the accumulators were read and cleared by an earlier selection
#pragma unroll
    for (int t = 0; t < NTILE; ++t) {
        if (key >= valid[t]) continue;
        if constexpr (!ALPHA) {               // (with SPLIT = 2 both halves of the queries add into the key's accumulator)
            float acc = 0.f;
#pragma unroll
            for (int i = 0; i < TC; i += 4) {
                if ((i & 15) == 0 && c0 + i >= npad) break;   // columns past the padded query count were never exponentiated
                const float4 w4 = *reinterpret_cast<const float4*>(w + i);
                acc = fmaf(L[t * TC + i], w4.x, acc);
                acc = fmaf(L[t * TC + i + 1], w4.y, acc);
                acc = fmaf(L[t * TC + i + 2], w4.z, acc);
                acc = fmaf(L[t * TC + i + 3], w4.w, acc);
            }
            atomicAdd(o.acc64 + s.vis_off + vis0[t] + key, __float2ull_rn(acc * kFixScale));
        }
        if constexpr (ALPHA) {                // the attention itself, for the per-patch indicators: this key's row of queries
            float* ap = o.alpha.ptr + static_cast<int64_t>(h) * o.alpha.stride_h + static_cast<int64_t>(s.vis_off + vis0[t] + key) * 4;
            const float hn = static_cast<float>(o.n_heads) * static_cast<float>(s.n_txt);   // the weights carry 1 / (H n_t)
#pragma unroll
            for (int i = 0; i < TC; i += 4) { // 16-byte stores: a handful of instructions
                if (c0 + i >= s.n_txt) break;
                const float4 w4 = *reinterpret_cast<const float4*>(w + i);
                *reinterpret_cast<float4*>(ap + ((c0 + i) >> 2) * o.alpha.stride_q) =
                    make_float4(L[t * TC + i] * w4.x * hn, L[t * TC + i + 1] * w4.y * hn, L[t * TC + i + 2] * w4.z * hn, L[t * TC + i + 3] * w4.w * hn);
            }
        }
    }
}

// grid = (cluster size, n_heads, samples), cluster = (cluster size, 1, 1), 128 x SPLIT threads.
// TCOL: tensor-memory columns per tile (>= padded query count); NTILE: key tiles per CTA.
// KIND: what else the kernel does.  Its code runs once per launch, from a cold instruction cache: code that a step does
// not use still costs it time (0.5 us for 1.5 KB), so the variants are compiled apart.
// SPLIT: threads per key.  1: a thread holds all the logits of its key.  2: threads t and t + 128 hold one half of the
// text queries each -- the chain through exponentials, sums and weighted sum is half as long per warp, and a scheduler
// has two warps to alternate between; both halves add into the key's accumulator.
// scores only; with the logit cache; the attention copy instead of scores; scores of a step with stable inputs, beside the kernel before
enum { kPlain = 0, kWithCache = 1, kForPatches = 2, kEarly = 3 };
template <int TCOL, int NTILE, int SPLIT, int KIND, class BD>
__global__ void __launch_bounds__(kFastThreads * SPLIT, 1)
salience_fast_kernel(const __grid_constant__ BD bd, const __grid_constant__ CUtensorMap tmap_q,
                     const __grid_constant__ CUtensorMap tmap_k, int n_heads, int kv_group, int head_dim, int esize, int npad_max,
                     unsigned long long* __restrict__ acc64,
                     int* status, const AlphaOut alpha, int32_t* __restrict__ rearm, unsigned long long* __restrict__ rearm_rec,
                     unsigned long long* __restrict__ stamps, float* __restrict__ lcache, int cache_vis, int cache_cols)
{
    constexpr bool early = KIND == kEarly;
    constexpr int CC = TCOL * NTILE;                      // tensor-memory columns of the CTA
    constexpr int TC = TCOL / SPLIT;                      // columns (text queries) of a tile that one thread holds
    constexpr int NT = kFastThreads * SPLIT;
    static_assert(TC % 16 == 0, "a thread holds whole groups of 16 queries");
    extern __shared__ uint8_t dyn_smem_raw[];
    uint8_t* dyn_smem = dyn_smem_raw + ((1024u - (smem_u32(dyn_smem_raw) & 1023u)) & 1023u);   // swizzle atoms are 1 KB
    __shared__ FastSmem sm;
    __shared__ __align__(8) uint64_t s_bar[3];
    __shared__ uint32_t s_tmem;

    const SampleDev& s = bd.at(blockIdx.z);
    const int h = blockIdx.y;
    const int tid = threadIdx.x, warp = tid >> 5;
    const int key = tid & (kFastThreads - 1);            // key of the tile(s) this thread works on
    const int kwarp = warp & 3;                           // its warp among the four that cover the 128 keys (= tensor-memory lane quarter)
    const int c0 = (tid / kFastThreads) * TC;             // first of its text queries
    // queries padded to the MMA's N granularity for THIS sample (the launch is sized for the longest text)
    const int npad = min(npad_max, (s.n_txt + 15) & ~15);
    const uint32_t crank = cluster_ctarank();
    const uint32_t csize = gridDim.x;
    const int d = head_dim;
    const int khalves = (d * esize + 127) / 128;          // 128-byte swizzle rows (64 bf16 or 128 e4m3) per key; a last partial box is zero-filled by TMA
    const int box_elems = 128 / esize;
    const float cscale = 1.4426950408889634f * rsqrtf(static_cast<float>(d));   // log2 domain
    const int tt0 = static_cast<int>(crank) * NTILE;
    uint8_t* Ks = dyn_smem;                               // [tile][khalf][128 rows x 128 B]
    uint8_t* Qs = dyn_smem + static_cast<size_t>(NTILE) * khalves * 16384;   // [khalf][npad rows x 128 B]
    const uint32_t bar_full = smem_u32(&s_bar[0]), bar_mma = smem_u32(&s_bar[1]), bar_x = smem_u32(&s_bar[2]);

    int valid[NTILE], vis0[NTILE];
    bool from_k[NTILE];                       // the tile's logits come from K (TMA + MMA); false: from the logit cache
    bool any_live = false;
    const bool caching = KIND == kWithCache && s.cache_state >= 0;
#pragma unroll
    for (int t = 0; t < NTILE; ++t) {
        const TileInfo ti = tile_info(s, tt0 + t);
        valid[t] = ti.valid;
        vis0[t] = ti.vis0;
        any_live |= ti.valid > 0;
        from_k[t] = !caching || ((s.tile_compute >> (tt0 + t)) & 1u) != 0;
    }
    // row of this thread's key in the cache: [state][head][visual index][column]
    const int64_t cache_row0 = caching ? ((static_cast<int64_t>(s.cache_state) * n_heads + h) * cache_vis) * cache_cols : 0;

    // ---- before the wait for the kernel before this one: everything that does not read its results.  In particular the
    //      cluster arrive: a release waits for all that its thread has issued, and behind the loads it took as long as
    //      they did (0.6 us behind six boxes, 1.4 us behind ten).
    const bool one = warp == 0 && elect_one();
    if (one) {
        prefetch_tensormap(&tmap_q);
        prefetch_tensormap(&tmap_k);
        mbar_init(bar_full, 1);
        mbar_init(bar_mma, 1);
        mbar_init(bar_x, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        mbar_expect_tx(bar_x, csize * static_cast<uint32_t>(npad) * 8u);     // every CTA of the cluster sends npad pairs
    }
    __syncwarp();
    cluster_arrive_release();                 // publishes this CTA's barriers; matched by the wait before the first remote store
    uint32_t tmem_cols = 32;
    while (tmem_cols < static_cast<uint32_t>(CC)) tmem_cols <<= 1;
    // Blocks until the columns are free.  Whoever holds some on this multiprocessor gives them back without waiting for
    // another CTA: this kernel before its exchange (below), the streaming kernel is never beside it, and the CTAs of the
    // generic kernel that fit beside one another never ask for more than there is (tmem_plan.h).  (Warp 3: it has no part
    // in the exchange.)
    if (warp == 3) tmem_alloc(smem_u32(&s_tmem), tmem_cols);
    // One CTA per sample re-arms the words through which the kernel after this one hands the kept list from
    // its selecting CTA to its copying CTAs (-1: not yet known).  Their last users finished long ago.
    if (rearm && blockIdx.x == 0 && blockIdx.y == 0) {
        if constexpr (KIND != kForPatches) {
            for (int i = tid; i < s.n_out; i += NT) rearm[(s.out_off + i) * kListStride] = -1;
        } else {                              // the patch-by-patch tail: its list words, and three words per patch
            for (int i = tid; i < kHandWords; i += NT) rearm[s.cap_off + i] = -1;
            for (int i = tid; i < s.n_txt + s.n_2d + s.n_3d; i += NT) rearm[s.cap_off + kHandWords + i * kListStride] = -1;
            for (int i = tid; i < 3 * s.n_2d; i += NT) rearm_rec[static_cast<int64_t>(s.vis_off / 2) * 3 + i] = ~0ull;
        }
    }
    int row0[NTILE], live = 0;                // key tiles to fetch: those that exist and do not come from the cache
#pragma unroll
    for (int t = 0; t < NTILE; ++t) {
        row0[t] = tile_info(s, tt0 + t).row0;
        live += valid[t] > 0 && from_k[t];
    }
    const int hk = h / kv_group, qrow = s.seq_off + s.off_txt, nq = npad / 16;
    const uint32_t k_smem = smem_u32(Ks), q_smem = smem_u32(Qs);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = s_tmem;

    // Logit cache: a reused tile takes the previous action step's dot products instead of K (128 bytes per key and head
    // at 32 queries: half a key row, and no MMA).  They were written two kernels ago, so they are fetched before the wait,
    // too, instead of behind the MMAs, where they are needed.
    float L[NTILE * TC];                      // L[t * TC + i]: tile t, text query c0 + i
#pragma unroll
    for (int i = 0; i < NTILE * TC; ++i) L[i] = 0.f;
    if constexpr (KIND == kWithCache) {
#pragma unroll
        for (int t = 0; t < NTILE; ++t) {
            if (!caching || from_k[t] || key >= valid[t]) continue;
            const float4* row = reinterpret_cast<const float4*>(lcache + cache_row0 + static_cast<int64_t>(vis0[t] + key) * cache_cols + c0);
#pragma unroll
            for (int i = 0; i < TC; i += 4) {
                if (c0 + i >= npad) break;
                const float4 v = __ldcg(row + i / 4);
                L[t * TC + i] = v.x; L[t * TC + i + 1] = v.y; L[t * TC + i + 2] = v.z; L[t * TC + i + 3] = v.w;
            }
        }
    }

    // Warp 0 loads and multiplies: it runs these loops as a whole warp, all values the same in every lane, and one
    // elected lane issues, so that coordinates and descriptors stay in uniform registers.  (In a single-thread branch
    // every operand is moved to a uniform register one by one: 0.1 us more for the MMAs of a tile.)
    if (warp == 0) {
        // Inputs may come from the kernel before this one (not in a step whose inputs are promised stable: `early`).
        if (!early) pdl_wait();
        // (no tile to compute: nothing is fetched, both barriers below complete at once)
        if (one) mbar_expect_tx(bar_full, live > 0 ? static_cast<uint32_t>(khalves) * (npad * 128 + live * 16384) : 0u);
#pragma unroll
        for (int t = 0; t < NTILE; ++t) {
            if (valid[t] <= 0 || !from_k[t]) continue;
            for (int kh = 0; kh < khalves; ++kh)
                if (one) tma_load_3d(k_smem + static_cast<uint32_t>(t * khalves + kh) * 16384u, &tmap_k, kh * box_elems, hk, row0[t], bar_full);
        }
        for (int kh = 0; kh < khalves && live > 0; ++kh)
            for (int c = 0; c < nq; ++c)
                if (one) tma_load_3d(q_smem + static_cast<uint32_t>(kh * npad * 128 + c * 2048), &tmap_q, kh * box_elems, h, qrow + c * 16, bar_full);
        // Whatever the kernel before this one wrote is complete: the next kernel may become resident now and may read
        // such data in its prologue.  Not with `early`: the kernel behind it (the norms, or the tail of a chained step) reads
        // promised inputs before its own wait, or nothing, and writes the norms into this step's scratch set, which the
        // step six calls back left complete: the kernel before this one could start only after that.
        pdl_trigger();
        if (stamps && one) {                  // measurement aid: when this CTA was free to start its loads
            const unsigned cta = blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z);
            if (cta < kStampSlots) stamps[2 * cta] = global_ns();
        }
    }
    // Only warp 0 polls the barriers; the other threads park at the block barrier below (a hardware
    // wait), so while a CTA waits for its predecessor, its loads or its MMAs it leaves the issue slots and
    // the shared-memory pipe of the multiprocessor to the CTAs that share it.
    bool ok = true;
    if (warp == 0) {
        bool got = mbar_wait(bar_full, 0);
        if (!got) {                           // report, then give the copies one more bounded chance to land
            *reinterpret_cast<volatile int*>(status) = MVLA_ERR_TIMEOUT;
            got = mbar_wait(bar_full, 0);
        }
        __syncwarp();
        got = __all_sync(0xffffffffu, got);
        tc_fence_after();
        if (got) {
            const uint32_t idesc = idesc_by_size(esize, npad);
            const int ksteps = (d * esize + 31) / 32;              // an instruction consumes 32 bytes of every row
            const uint64_t k_desc = smem_desc_sw128(k_smem), q_desc = smem_desc_sw128(q_smem);   // (addresses / 16 in the low bits)
#pragma unroll
            for (int t = 0; t < NTILE; ++t) {
                if (valid[t] <= 0 || !from_k[t]) continue;
                for (int kh = 0; kh < khalves; ++kh) {
                    if (one)
                        umma_box(esize, tmem_base + t * TCOL, desc_plus(k_desc, static_cast<uint32_t>(t * khalves + kh) * (16384 >> 4)),
                                 desc_plus(q_desc, static_cast<uint32_t>(kh * npad) * (128 >> 4)), idesc, min(4, ksteps - kh * 4), kh > 0);
                }
            }
        }
        if (one) umma_commit(bar_mma);        // arrives once every MMA issued above has finished
        ok = mbar_wait(bar_mma, 0);
        if (!ok) *reinterpret_cast<volatile int*>(status) = MVLA_ERR_TIMEOUT;
        __syncwarp();
    }
    ok = __syncthreads_and(ok) != 0;          // block-uniform from here on (aligned instructions follow)
    tc_fence_after();

    // ---- all logits of this thread's key(s) into registers
    if constexpr (SPLIT == 1 && KIND != kWithCache) {
        if (any_live && ok) tmem_ld_cols<CC>(tmem_base + (static_cast<uint32_t>(kwarp * 32) << 16), L);
    } else {
#pragma unroll
        for (int t = 0; t < NTILE; ++t) {
            if (!any_live || !ok || !from_k[t]) continue;                    // block-uniform
            float part_l[TC];
            tmem_ld_cols<TC>(tmem_base + static_cast<uint32_t>(t * TCOL + c0) + (static_cast<uint32_t>(kwarp * 32) << 16), part_l);
#pragma unroll
            for (int i = 0; i < TC; ++i) L[t * TC + i] = part_l[i];
        }
    }
    // Logit cache: a computed tile leaves its raw dot products for the next action step.
    if constexpr (KIND == kWithCache) {
#pragma unroll
        for (int t = 0; t < NTILE; ++t) {
            if (!caching || !ok || !from_k[t] || key >= valid[t]) continue;
            float4* row = reinterpret_cast<float4*>(lcache + cache_row0 + static_cast<int64_t>(vis0[t] + key) * cache_cols + c0);
#pragma unroll
            for (int i = 0; i < TC; i += 4) {
                if (c0 + i >= npad) break;
                row[i / 4] = make_float4(L[t * TC + i], L[t * TC + i + 1], L[t * TC + i + 2], L[t * TC + i + 3]);
            }
        }
    }
    tc_fence_before();
    softmax_scores<TCOL, NTILE, SPLIT, KIND == kForPatches>(L, s, valid, vis0, ok, npad, h, cscale, bar_x, sm,
                                       FastOut{acc64, status, n_heads, alpha, early}, [&]() {
        if (warp == 3) {
            tc_fence_after();
            tmem_dealloc(tmem_base, tmem_cols);
        }
    });
    // "This kernel is complete" implies that the one before it is, for whoever comes after: one CTA sees to that last.
    if (early && tid == 0 && blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0) pdl_wait();
    if (stamps) {
        __syncthreads();
        if (tid == 0) {
            const unsigned cta = blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z);
            if (cta < kStampSlots) stamps[2 * cta + 1] = global_ns();
        }
    }
}

// ------------------------------------------------------------------ fp32 inputs
// The same chain for fp32 q / k: plain FMAs instead of the tensor cores (their fp32 forms round the operands).  Rows
// arrive as TMA boxes of 32 floats x 128 keys (or 16 queries) with the 128-byte swizzle, in which 16-byte reads of
// neighbouring rows do not conflict; a thread computes the dot products of its key with its half of the text queries,
// the key's piece in registers against broadcasts of the queries.  Dot products are summed in element order.
// Bound by latency at the sizes this path serves (2.2 MB a step at 192 tokens, 8 heads x 64): the loads of a CTA go out at
// once, where scalar loads through registers kept a few in flight, and the step runs as chained kernels like that of the
// other types (24.6 -> 14.4 us a step at that size with a bulk copy per row, 10.3 with boxes: 144 small copies took
// their time to issue).
template <int TCOL, int NTILE, class BD>
__global__ void __launch_bounds__(kFastThreads * 2, 1)
salience_f32_kernel(const __grid_constant__ BD bd, const __grid_constant__ CUtensorMap tmap_q, const __grid_constant__ CUtensorMap tmap_k,
                    int n_heads, int kv_group, int d, int npad_max, unsigned long long* __restrict__ acc64, int* status, int32_t* __restrict__ rearm,
                    unsigned long long* __restrict__ stamps)
{
    constexpr int TC = TCOL / 2, NT = kFastThreads * 2;
    extern __shared__ uint8_t dyn_smem_raw[];
    const int boxes = d / 32;                             // head dims are multiples of 32
    // The queries come first: a thread reads a whole half of TCOL queries, rows past the padded ones (up to 2 KB past the
    // last box) included, and what it reads there must exist.
    uint8_t* Qs = dyn_smem_raw + ((1024u - (smem_u32(dyn_smem_raw) & 1023u)) & 1023u);   // [box][npad rows x 128 B]
    uint8_t* Ks = Qs + boxes * npad_max * 128;            // [tile][box][128 rows x 128 B]
    __shared__ FastSmem sm;
    __shared__ __align__(8) uint64_t s_bar[2];
    const SampleDev& s = bd.at(blockIdx.z);
    const int h = blockIdx.y, tid = threadIdx.x, warp = tid >> 5;
    const int key = tid & (kFastThreads - 1), c0 = (tid / kFastThreads) * TC;
    const int npad = min(npad_max, (s.n_txt + 15) & ~15);
    const int tt0 = static_cast<int>(cluster_ctarank()) * NTILE;
    const float cscale = 1.4426950408889634f * rsqrtf(static_cast<float>(d));   // log2 domain
    const uint32_t bar_full = smem_u32(&s_bar[0]), bar_x = smem_u32(&s_bar[1]);
    int valid[NTILE], vis0[NTILE];
    TileInfo ti[NTILE];
#pragma unroll
    for (int t = 0; t < NTILE; ++t) {
        ti[t] = tile_info(s, tt0 + t);
        valid[t] = ti[t].valid;
        vis0[t] = ti[t].vis0;
    }
    // before the wait for the kernel before this one (see salience_fast_kernel)
    const bool one = warp == 0 && elect_one();
    if (one) {
        prefetch_tensormap(&tmap_q);
        prefetch_tensormap(&tmap_k);
        mbar_init(bar_full, 1);
        mbar_init(bar_x, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        mbar_expect_tx(bar_x, gridDim.x * static_cast<uint32_t>(npad) * 8u);
    }
    __syncwarp();
    cluster_arrive_release();                 // publishes this CTA's barriers; matched by the wait before the first remote store
    if (rearm && blockIdx.x == 0 && blockIdx.y == 0)
        for (int i = tid; i < s.n_out; i += NT) rearm[(s.out_off + i) * kListStride] = -1;
    const int hk = h / kv_group, qrow = s.seq_off + s.off_txt, nq = npad / 16;
    int live = 0;
#pragma unroll
    for (int t = 0; t < NTILE; ++t) live += valid[t] > 0;
    __syncthreads();
    if (warp == 0) {
        pdl_wait();
        if (one) mbar_expect_tx(bar_full, static_cast<uint32_t>(boxes) * (npad * 128 + live * 16384));
#pragma unroll
        for (int t = 0; t < NTILE; ++t) {
            if (valid[t] <= 0) continue;
            for (int x = 0; x < boxes; ++x)
                if (one) tma_load_3d(smem_u32(Ks) + static_cast<uint32_t>(t * boxes + x) * 16384u, &tmap_k, x * 32, hk, ti[t].row0, bar_full);
        }
        for (int x = 0; x < boxes; ++x)
            for (int c = 0; c < nq; ++c)
                if (one) tma_load_3d(smem_u32(Qs) + static_cast<uint32_t>(x * npad * 128 + c * 2048), &tmap_q, x * 32, h, qrow + c * 16, bar_full);
        pdl_trigger();
        if (stamps && one) {
            const unsigned cta = blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z);
            if (cta < kStampSlots) stamps[2 * cta] = global_ns();
        }
    }
    bool ok = true;
    if (tid == 0) {
        ok = mbar_wait(bar_full, 0);
        if (!ok) {                            // report, then give the copies one more bounded chance to land
            *reinterpret_cast<volatile int*>(status) = MVLA_ERR_TIMEOUT;
            mbar_wait(bar_full, 0);
        }
    }
    ok = __syncthreads_and(ok) != 0;
    if (ok) mbar_wait(bar_full, 0);           // complete: makes the copied rows visible to every thread
    float L[NTILE * TC];
#pragma unroll
    for (int i = 0; i < NTILE * TC; ++i) L[i] = 0.f;
    if (c0 < npad) {
#pragma unroll
        for (int t = 0; t < NTILE; ++t) {
            if (valid[t] <= 0) continue;
            for (int x = 0; x < boxes; ++x) {
                const uint8_t* kr = Ks + (t * boxes + x) * 16384 + key * 128;
                const uint8_t* qr = Qs + (x * npad + c0) * 128;
#pragma unroll 2
                for (int c = 0; c < 8; ++c) {             // 16-byte piece c of row r lies at c ^ (r mod 8)
                    const float4 k4 = *reinterpret_cast<const float4*>(kr + ((c ^ (key & 7)) << 4));
#pragma unroll
                    for (int i = 0; i < TC; ++i) {        // (c0 is a multiple of 16)
                        const float4 q4 = *reinterpret_cast<const float4*>(qr + i * 128 + ((c ^ (i & 7)) << 4));
                        float& acc = L[t * TC + i];
                        acc = fmaf(k4.x, q4.x, acc);
                        acc = fmaf(k4.y, q4.y, acc);
                        acc = fmaf(k4.z, q4.z, acc);
                        acc = fmaf(k4.w, q4.w, acc);
                    }
                }
            }
        }
    }
    softmax_scores<TCOL, NTILE, 2, false>(L, s, valid, vis0, ok, npad, h, cscale, bar_x, sm,
                                   FastOut{acc64, status, n_heads, AlphaOut{nullptr, 0, 0}, false}, []() {});
    if (stamps) {
        __syncthreads();
        if (tid == 0) {
            const unsigned cta = blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z);
            if (cta < kStampSlots) stamps[2 * cta + 1] = global_ns();
        }
    }
}

// One variant of the kernel with the set-up that goes with it.
template <int TCOL, int NTILE, int SPLIT, int KIND, class BD>
struct FastVariant {
    static constexpr int kThreads = kFastThreads * SPLIT;
    static constexpr auto kern = salience_fast_kernel<TCOL, NTILE, SPLIT, KIND, BD>;
    static const void* address() { return reinterpret_cast<const void*>(kern); }
    static KernelSetup& setup()
    {
        static KernelSetup ks;
        return ks;
    }
    // dynamic shared memory of a launch, with the kernel ready for it
    static cudaError_t prepare(int head_dim, int esize, int npad, size_t* smem)
    {
        // resident CTAs x tensor-memory columns must not exceed the 512 of a multiprocessor
        const int tmem_cols = tmem_cols_for(TCOL * NTILE);
        *smem = smem_for_tmem(1024 + static_cast<size_t>((head_dim * esize + 127) / 128) * (static_cast<size_t>(NTILE) * 16384 + npad * 128), tmem_cols);
        return *smem == 0 ? cudaErrorInvalidConfiguration : setup_kernel(setup(), address(), *smem, tmem_cols);
    }
};

template <class V, class BD>
cudaError_t launch_fast_t(const BD& bd, int n_heads, int kv_group, int head_dim, int esize, const CUtensorMap* tq,
                          const CUtensorMap* tk, int cluster, int npad,
                          unsigned long long* acc64, int* status, AlphaOut alpha, int32_t* rearm, unsigned long long* rearm_rec, unsigned long long* stamps,
                          float* lcache, int cache_vis, int cache_cols, cudaStream_t stream)
{
    size_t smem = 0;
    const cudaError_t e = V::prepare(head_dim, esize, npad, &smem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(cluster, n_heads, bd.n);
    cfg.blockDim = dim3(V::kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cluster;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1] = pdl_attribute();
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, V::kern, bd, *tq, *tk, n_heads, kv_group, head_dim, esize, npad, acc64, status, alpha, rearm, rearm_rec, stamps, lcache, cache_vis, cache_cols);
}

// use(variant, descriptors) with the variant that scores a launch
template <class F>
cudaError_t with_fast_variant(const BatchDesc& bd, int npad, int tiles_per_cta, int kind, F use)
{
    const int tcol = npad <= 16 ? 16 : (npad <= 32 ? 32 : 64);
    const int split = tcol >= 32 ? 2 : 1;     // two threads per key while a thread still holds 16 queries
#define MVLA_FAST1(TC, NTL, SP, KD)                                                                             \
    if (tcol == TC && tiles_per_cta == NTL && split == SP && kind == KD)                                        \
        return with_desc(bd, [&](const auto& d) { return use(FastVariant<TC, NTL, SP, KD, std::decay_t<decltype(d)>>{}, d); });
#define MVLA_FAST(TC, NTL, SP) MVLA_FAST1(TC, NTL, SP, kPlain) MVLA_FAST1(TC, NTL, SP, kWithCache) MVLA_FAST1(TC, NTL, SP, kForPatches)
    MVLA_FAST(16, 1, 1) MVLA_FAST(16, 2, 1) MVLA_FAST(32, 1, 2) MVLA_FAST(64, 1, 2) MVLA_FAST(32, 2, 2) MVLA_FAST(64, 2, 2)
#undef MVLA_FAST1
#undef MVLA_FAST
    if (kind != kEarly || bd.n != 1 || tiles_per_cta != 1) return cudaErrorInvalidConfiguration;
    const OneDesc one = {{bd.s[0]}, 1};       // a chained step has one sample and one tile per CTA (mvla_prune_step)
    if (tcol == 16) return use(FastVariant<16, 1, 1, kEarly, OneDesc>{}, one);
    if (tcol == 32) return use(FastVariant<32, 1, 2, kEarly, OneDesc>{}, one);
    if (tcol == 64) return use(FastVariant<64, 1, 2, kEarly, OneDesc>{}, one);
    return cudaErrorInvalidConfiguration;
}

template <int TCOL, int NTILE, class BD>
cudaError_t launch_f32_t(const BD& bd, int n_heads, int kv_group, int head_dim, const CUtensorMap* tq, const CUtensorMap* tk, int cluster, int npad,
                         unsigned long long* acc64, int* status, int32_t* rearm, unsigned long long* stamps, cudaStream_t stream)
{
    const size_t smem = 1024 + static_cast<size_t>(head_dim / 32) * (NTILE * 16384 + npad * 128);
    auto kern = salience_f32_kernel<TCOL, NTILE, BD>;
    static KernelSetup ks;
    const cudaError_t e = setup_kernel(ks, reinterpret_cast<const void*>(kern), smem, 0);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(cluster, n_heads, bd.n);
    cfg.blockDim = dim3(kFastThreads * 2);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cluster;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1] = pdl_attribute();
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, kern, bd, *tq, *tk, n_heads, kv_group, head_dim, npad, acc64, status, rearm, stamps);
}

}  // namespace

// fp32: two key tiles per CTA at most, and all rows of a CTA in shared memory beside the kernel's own 7 KB.
bool f32_salience_supported(int tiles_per_cta, int npad, int head_dim)
{
    return tiles_per_cta <= 2 && 1024 + head_dim / 32 * (tiles_per_cta * 16384 + npad * 128) <= 218 * 1024;
}

cudaError_t launch_salience_f32(const BatchDesc& bd, int n_heads, int kv_group, int head_dim, const CUtensorMap* tmap_q,
                                const CUtensorMap* tmap_k, int tiles_per_cta,
                                int cluster, int npad, unsigned long long* acc64, int* status, int32_t* rearm, unsigned long long* stamps,
                                cudaStream_t stream)
{
    if (!f32_salience_supported(tiles_per_cta, npad, head_dim)) return cudaErrorInvalidConfiguration;
#define MVLA_F32(TC, NTL)                                                                                       \
    if (npad <= TC && tiles_per_cta == NTL)                                                                     \
        return with_desc(bd, [&](const auto& d) {                                                               \
            return launch_f32_t<TC, NTL>(d, n_heads, kv_group, head_dim, tmap_q, tmap_k, cluster, npad, acc64, status, rearm, stamps, stream); });
    MVLA_F32(32, 1) MVLA_F32(64, 1) MVLA_F32(32, 2) MVLA_F32(64, 2)
#undef MVLA_F32
    return cudaErrorInvalidConfiguration;
}

bool fast_salience_supported(int tiles_per_cta) { return tiles_per_cta >= 1 && tiles_per_cta <= 2; }

cudaError_t launch_salience_fast(const BatchDesc& bd, int n_heads, int kv_group, int head_dim, int esize, const CUtensorMap* tmap_q,
                                 const CUtensorMap* tmap_k, int tiles_per_cta, int cluster, int npad,
                                 unsigned long long* acc64, int* status,
                                 AlphaOut alpha, int32_t* rearm, unsigned long long* rearm_rec, unsigned long long* stamps,
                                 float* lcache, int cache_vis, int cache_cols, bool early, cudaStream_t stream)
{
    if ((acc64 == nullptr) == (alpha.ptr == nullptr)) return cudaErrorInvalidConfiguration;      // one or the other
    return with_fast_variant(bd, npad, tiles_per_cta, alpha.ptr ? kForPatches : (lcache ? kWithCache : (early ? kEarly : kPlain)), [&](auto v, const auto& d) {
        return launch_fast_t<decltype(v)>(d, n_heads, kv_group, head_dim, esize, tmap_q, tmap_k, cluster, npad, acc64, status,
                                          alpha, rearm, rearm_rec, stamps, lcache, cache_vis, cache_cols, stream);
    });
}

cudaError_t fast_salience_residency(const BatchDesc& bd, int head_dim, int esize, int tiles_per_cta, int cluster, int npad,
                                    bool for_patches, int* per_sm, int* clusters)
{
    return with_fast_variant(bd, npad, tiles_per_cta, for_patches ? kForPatches : kPlain, [&](auto v, const auto&) {
        using V = decltype(v);
        size_t smem = 0;
        const cudaError_t e = V::prepare(head_dim, esize, npad, &smem);
        if (e != cudaSuccess) return e;
        *per_sm = ctas_by_smem(smem + kFastStaticSmem);      // (registers allow two CTAs of two tiles and three of one)
        return *per_sm > 1 ? cudaSuccess : clusters_at_once(V::setup(), V::address(), V::kThreads, smem, cluster, clusters);
    });
}

}  // namespace mvla
