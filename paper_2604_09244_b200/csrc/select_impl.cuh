// Carry-over, budget split and top-k selection of ONE sample by one CTA of NT threads
// (Alg. 1 of the paper, stages 1-4; Eqs. 8, 9, 10).
//
// The work is a few KB, so the kernel is a chain of latencies; it is written around the number of dependent
// instructions on that chain (a shuffle is 24 cycles, a step of a scan 34, a shared-memory access 35, a block barrier 42, an
// IEEE division 73, an L2 hit 330) and of block-wide barriers (four on the usual path):
//   1. every thread issues ALL its global loads (scores, previous state, norms) before any dependent
//      work, then smooths the scores (Eq. 8 / Eq. 9 as  xhat = c_prev xhat + c_new x), builds
//      order-preserving 32-bit keys, kept in registers, and counts them into a histogram at once: the
//      bins are a window of eight octaves around the mean score, which is known to be 1 / n_vis, so no
//      pass over the keys has to find their range first.  One word per bin counts both modalities.  Each
//      warp leaves its partial sums in shared memory                                    [barrier A]
//   2. every warp takes the running count over its two slices of 128 bins; one warp goes on to the modality
//      sums -> the four indicators, smoothed too; dual threshold (Sec. 4.1), target-object rule
//      (Sec. 4.2), fusion (Sec. 4.4), budget split                                      [barrier B]
//   3. the number of keys in higher bins tells every thread what becomes of its keys: kept, dropped, or, in the bin where
//      the budget runs out, listed                                                      [barrier C]
//      The few listed keys are ranked by (key, lower index first) by the threads that own them.  The keys of a crowded bin
//      are counted again, over the range that they have (only then: more barriers); keys that are
//      all equal are ranked by index during the emission;
//   4. emission merged with all text positions: warp ballots rank the kept tokens, the per-warp
//      counts meet in shared memory                                                     [barrier D]
// Bound by that chain and, second, by issue slots: sixteen warps share four schedulers, so an instruction that all of them
// repeat costs four cycles.  From the wait to the list, in cycles, against a version that found the range of the keys
// first, searched the histogram with one warp per modality and ranked through shared memory: 768 tokens, host-decided
// budgets 5850 -> 3650, device-decided 7220 -> 5050; 1791 tokens 9620 -> 7300; 1280 with carried-over state 8500 -> 5530; a
// step of one frame 11.6 -> 10.7 us, eight action steps 140.8 -> 130.4.  With 256 threads 4730 instead of 3650.
#pragma once

#include "common.cuh"
#include "copy_impl.cuh"

#include <math_constants.h>

namespace mvla {

constexpr float kFixScale = 1152921504606846976.f;          // 2^60
constexpr float kFixInv = 1.f / 1152921504606846976.f;      // 2^-60, exact

// The first histogram covers [2^-6, 4) times the power of two at or below the mean score (the last bin also takes
// everything above, the first one everything below): scores that the softmax and the mean over heads and queries leave lie
// within a factor of ten below their mean but for a few strong ones above.  256 bins an octave for up to 1024 tokens, 512 for
// more, leave up to 32 keys in the bin where the budget runs out; fewer bins cost less to count up, fewer keys in one less to
// rank.  (Bins laid over the range of the keys, which needs a pass, a barrier and two reductions first, held more:
// a few strong tokens stretch the range.)
// Where the window does not fit -- scores within a percent of one another, one token with nearly all of the attention, scores that
// are not normalised -- a second histogram does.  mvla_select in us, 768 / 1791 / 3584 tokens, and in parentheses with bins laid
// over the whole range of the crowded bin instead of over its keys, in a pass that also ranked the other modality:
//   as the window expects 5.3 / 6.6 / 10.6; spread of 3e-4 6.4 / 9.6 / 13.4 (6.3 / 9.5 / 13.2);
//   one token with 99 % 6.8 / 9.6 / 14.6 (8.2 / 12.1 / 17.8); all equal 6.5 / 8.8 / 13.1 (9.0 / 15.0 / 24.1);
//   four fifths zero 6.4 / 8.6 / 12.0 (10.5 / 17.2 / 27.2).
// Keys of a warp that share a bin added up before they are counted: 0.3 to 1 us less with all keys in one bin, but 0.1 to 0.2
// more in every step.
constexpr int sel_bin_bits(int cap) { return cap <= 1024 ? 11 : 12; }
constexpr int kWindowOctaves = 8, kWindowBelow = 6;
constexpr int kSliceBins = 128;     // bins that a warp reads at once: four a lane
constexpr int kCandMax = 64;        // keys of the threshold bin ranked from a list; above that the bin is split again
// Histograms at most: every one after the second takes 11 bits off a key (32, 21, 10: then all keys of a bin are equal).
constexpr int kSelLevels = 5;

template <int NT, int EPT>
struct SelectSmem {
    static constexpr int kBits = sel_bin_bits(NT * EPT), kBins = 1 << kBits, kSlices = kBins / kSliceBins;
    static_assert(kSlices <= 32 && kSlices % (NT / 32) == 0, "");
    alignas(16) uint32_t hist[kBins];        // bin 0: largest keys; low half: keys of the 2D tokens, high half: of the 3D tokens
    alignas(16) uint32_t before[kBins];      // counts in the bins before, within the slice
    uint32_t slice[kSlices];                 // counts of every slice of the bins
    alignas(16) float red[4][NT / 32];       // per-warp partial sums: scores 2D, 3D; norms 2D, 3D
    alignas(16) uint32_t cand[2][kCandMax];          // listed keys: place in the bin, index complemented below it: larger = ranked first; unused: 0
    alignas(16) uint32_t ext[4];             // of a crowded bin: complement of its smallest key, its largest key: 2D, 3D
    int ncand[2];
    int take[2];                             // per modality: keys to take from the bin in which the budget runs out
    int wtot[NT / 32];                       // emission: kept tokens of every warp; ties by index: 2D (low half), 3D (high half)
    int budget[2];                           // kept tokens per modality
    float x[4], mhat[4];                     // the indicators, and smoothed
    int sets[3];                             // C_S1, C_S2, their fusion
};
__device__ __forceinline__ int half_of(uint32_t packed, int shift) { return static_cast<int>((packed >> shift) & 0xFFFFu); }

// fp32 -> uint32 whose unsigned order is the float order; NaN sorts below everything.
__device__ __forceinline__ uint32_t order_key(float x)
{
    if (x != x) return 0u;
    const uint32_t b = __float_as_uint(x);
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float key_to_float(uint32_t k)
{
    return __uint_as_float((k & 0x80000000u) ? (k & 0x7FFFFFFFu) : ~k);
}

__device__ __forceinline__ int warp_incl_scan(int x, int lane)
{
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int n = __shfl_up_sync(0xffffffffu, x, off);
        if (lane >= off) x += n;
    }
    return x;
}

// Sums 4 per-thread values over the 32 lanes of a warp in 6 shuffles (a butterfly that halves the number
// of values a lane carries at each of its first two stages).  On return the lanes whose bits 4..3 spell
// c hold the sum of column c.  The order of the additions is fixed.
__device__ __forceinline__ float warp_sum4(const float (&v)[4], int lane)
{
    const bool up = (lane & 16) != 0, up2 = (lane & 8) != 0;
    const float a = (up ? v[2] : v[0]) + __shfl_xor_sync(0xffffffffu, up ? v[0] : v[2], 16);
    const float b = (up ? v[3] : v[1]) + __shfl_xor_sync(0xffffffffu, up ? v[1] : v[3], 16);
    float r = (up2 ? b : a) + __shfl_xor_sync(0xffffffffu, up2 ? a : b, 8);
#pragma unroll
    for (int off = 4; off >= 1; off >>= 1) r += __shfl_xor_sync(0xffffffffu, r, off);
    return r;
}

// Exclusive block scan of one int per thread (used by the patch-by-patch emission).
template <int NT>
__device__ __forceinline__ int block_exscan(int x, int* warp_tot, int* total)
{
    constexpr int NW = NT / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int inc = warp_incl_scan(x, lane);
    __syncthreads();                                       // previous users of warp_tot are done
    if (lane == 31) warp_tot[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        const int t = lane < NW ? warp_tot[lane] : 0;
        const int winc = warp_incl_scan(t, lane);
        if (lane < NW) warp_tot[lane] = winc - t;          // exclusive prefix of the warp totals
        if (lane == 31) warp_tot[NW] = winc;               // grand total
    }
    __syncthreads();
    *total = warp_tot[NW];
    return warp_tot[warp] + inc - x;
}

// How one CTA takes part in the selection of a sample.
//   list     : optional copy of the kept list for CTAs of the same kernel, kListStride words an entry.
//   late_pdl : false: the next kernel in the stream may become resident right away and the loads of the
//              previous state and of the norms follow griddepcontrol.wait; true: the state is loaded before it
//              (the caller guarantees that it was written before this kernel could start), and the next kernel
//              is released only after the list.
//   stable   : the next kernel may become resident as soon as the kernel before this one is complete, and the previous state is
//              loaded after the wait.
//   beside   : the scoring kernel is still running; the caller has seen that this sample's scores are complete.  Norms are waited
//              for one by one, and nothing is waited for or released on behalf of the next kernel.
struct SelectRole {
    int32_t* list = nullptr;
    bool late_pdl = false;
    bool stable = false;
    bool beside = false;
    int* status = nullptr;       // beside: receives MVLA_ERR_TIMEOUT ...
    uint64_t t0 = 0;             // ... a second after this time (the CTA's start), whichever of its waits that falls in
};
struct NoHook {
    __device__ void operator()() const {}
};

// `after_list` runs as soon as the kept list is written, before the bookkeeping that nobody downstream waits for (smoothed
// state, indicators and diagnostics, optional score outputs).
// EPT: elements per thread at most.  Warp w owns the 32 ept tokens from 32 ept w on, ept = as few as cover the sample: what it
// keeps is contiguous in the output, and one number per warp says where it begins.
template <int NT, int EPT, class After = NoHook>
__device__ __forceinline__ void select_sample(const SampleDev& s, int b_local, const GateParams& gp, const SelectIO& io,
                                              SelectSmem<NT, EPT>& sm, const SelectRole role = SelectRole(), After after_list = After())
{
    constexpr int NW = NT / 32, kSelBins = SelectSmem<NT, EPT>::kBins, kSelBits = SelectSmem<NT, EPT>::kBits, kSlices = SelectSmem<NT, EPT>::kSlices;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n2 = s.n_2d, n3 = s.n_3d, nv = n2 + n3;
    const int b_glob = io.chunk_first + b_local;
    const bool carry = s.c_prev != 0.f;
    const int ept = (nv + NT - 1) / NT, j0 = warp * 32 * ept + lane;     // this thread's tokens: j0 + 32 e, as far as they are below
    const int j_end = min(nv, (warp + 1) * 32 * ept);
    // Budgets decided on the host (FIXED mode, cold start): the modality sums then only feed the smoothed state and
    // the diagnostics, and are taken after the selection, off everyone's chain.
    const bool k_fixed = s.k_2d_fixed >= 0;

    // prologue that needs nothing from the previous kernel
    if (!role.late_pdl && !role.stable) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    auto clear_hist = [&]() {
        for (int i = tid; i < kSelBins / 4; i += NT) reinterpret_cast<uint4*>(sm.hist)[i] = make_uint4(0u, 0u, 0u, 0u);
    };
    clear_hist();
    if (tid < 2 * kCandMax) (&sm.cand[0][0])[tid] = 0u;
    if (tid < 2) sm.ncand[tid] = 0;
    if (tid < 4) sm.ext[tid] = 0u;
    float a[EPT], prev[EPT], nrm[EPT];
    unsigned long long fx[EPT];
    float4 mprev = make_float4(0.f, 0.f, 0.f, 0.f);       // the smoothed indicators so far
#pragma unroll
    for (int e = 0; e < EPT; ++e) { a[e] = 0.f; prev[e] = 0.f; nrm[e] = 0.f; fx[e] = 0ull; }
    auto load_state = [&]() {
        if (!carry) return;
#pragma unroll
        for (int e = 0; e < EPT; ++e) {
            const int j = j0 + 32 * e;
            if (j < j_end) prev[e] = io.ahat_state[s.state_off + j];
        }
        if (warp == NW - 1) mprev = reinterpret_cast<const float4*>(io.mhat_state)[s.mstate_off];
    };
    if (role.late_pdl) load_state();
    // The first use of a kernel parameter is a trip to the L2 (every launch has its parameters in a place of its own); one
    // use each here, ahead of the wait, keeps those trips off the chain.
    asm volatile("" :: "l"(io.acc64), "l"(io.attn), "l"(io.part), "l"(io.l1), "l"(io.kept_idx), "l"(role.list), "r"(s.vis_off), "r"(s.out_off),
                 "r"(s.off_txt), "r"(s.off_2d), "r"(s.off_3d), "r"(s.n_txt), "r"(s.budget), "r"(s.kmin_2d), "r"(s.kmin_3d), "f"(s.c_new),
                 "r"(gp.has_l1), "f"(gp.tau_2d), "f"(gp.tau_3d), "f"(gp.eps_3d), "l"(io.z_out));
    __syncthreads();                                       // the histogram is clear
    if (!role.beside) asm volatile("griddepcontrol.wait;" ::: "memory");      // scores come from the kernel before this one
    if (role.stable) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    // norms of this thread's tokens
    auto load_norms = [&]() {
        const int* const words = reinterpret_cast<const int*>(io.l1) + s.vis_off;
        bool there = true;
#pragma unroll
        for (int e = 0; e < EPT; ++e)
            if (j0 + 32 * e < j_end) {
                nrm[e] = role.beside ? __int_as_float(ld_relaxed_gpu(words + j0 + 32 * e)) : io.l1[s.vis_off + j0 + 32 * e];
                there &= __float_as_uint(nrm[e]) != kNoNorm;
            }
        if (!role.beside || there) return;
        bool late = false;
#pragma unroll 1
        for (int j = j0; j < j_end && !late; j += 32)
            for (uint32_t it = 0; static_cast<uint32_t>(ld_relaxed_gpu(words + j)) == kNoNorm; ++it) {
                if (it >= kSpinLimit || ((it & 63u) == 63u && global_ns() - role.t0 > 1000000000ull)) {
                    *reinterpret_cast<volatile int*>(role.status) = MVLA_ERR_TIMEOUT;
                    late = true;
                    break;
                }
                __nanosleep(40);
            }
#pragma unroll
        for (int e = 0; e < EPT; ++e)
            if (j0 + 32 * e < j_end) nrm[e] = __int_as_float(ld_relaxed_gpu(words + j0 + 32 * e));
    };

    // ---- 1. all loads first
    // (Loops over a thread's tokens have no early exits: the chains of its tokens then run beside one another.)
    if (io.acc64) {
#pragma unroll
        for (int e = 0; e < EPT; ++e)
            if (j0 + 32 * e < j_end) fx[e] = __ldcg(io.acc64 + s.vis_off + j0 + 32 * e);        // written by other CTAs' atomics
    } else if (!io.part) {
#pragma unroll
        for (int e = 0; e < EPT; ++e)
            if (j0 + 32 * e < j_end) a[e] = io.attn[s.vis_off + j0 + 32 * e];
    }
    if (gp.has_l1 && !k_fixed) load_norms();
    if (!role.late_pdl) load_state();
    if (io.part && !io.acc64) {                            // per-head fp32 partials, summed in head order
#pragma unroll
        for (int e = 0; e < EPT; ++e) {
            const int j = j0 + 32 * e;
            if (j < j_end) {
                float acc = 0.f;
#pragma unroll 8
                for (int h = 0; h < io.n_heads; ++h) acc += io.part[static_cast<int64_t>(h) * io.part_stride + s.vis_off + j];
                a[e] = acc;
            }
        }
    }
    // (no array below is indexed with a run-time value: such an array would live in local memory, and every
    //  first touch of a local-memory line is a round trip to L2 on this latency chain)
    // The bins under examination, per modality: bin kSelBins - 1 - b holds the keys from lo + (b << sh) on.
    uint32_t lo2 = 0x80000000u | static_cast<uint32_t>(127 - kWindowBelow - (nv > 1 ? 32 - __clz(nv - 1) : 0)) << 23, lo3 = lo2;
    int sh2 = 23 - (kSelBits - 3), sh3 = sh2;
    static_assert(1 << 3 == kWindowOctaves, "");
    auto bin_of = [&](uint32_t k, uint32_t lo, int sh) {
        return kSelBins - 1 - static_cast<int>(k <= lo ? 0u : min((k - lo) >> sh, static_cast<uint32_t>(kSelBins - 1)));
    };
    uint32_t key[EPT];
    int bin[EPT];
    if (io.acc64) {
#pragma unroll
        for (int e = 0; e < EPT; ++e) a[e] = __ull2float_rn(fx[e]) * kFixInv;      // one rounding: the exact head sum to fp32
    }
#pragma unroll
    for (int e = 0; e < EPT; ++e) {
        const float smo = carry ? fmaf(s.c_prev, prev[e], s.c_new * a[e]) : a[e];
        key[e] = order_key(smo);
        bin[e] = bin_of(key[e], lo2, sh2);
    }
#pragma unroll
    for (int e = 0; e < EPT; ++e)
        if (j0 + 32 * e < j_end) atomicAdd(&sm.hist[bin[e]], j0 + 32 * e < n2 ? 1u : 0x10000u);
    auto partial_sums = [&](const float (&x)[EPT], const float (&norm)[EPT]) {       // of the warp, with a fixed order of additions
        float sums[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int e = 0; e < EPT; ++e) {
            if (j0 + 32 * e < n2) { sums[0] += x[e]; sums[2] += norm[e]; }
            else                  { sums[1] += x[e]; sums[3] += norm[e]; }
        }
        const float col = warp_sum4(sums, lane);
        if ((lane & 7) == 0) sm.red[lane >> 3][warp] = col;
    };
    if (!k_fixed) partial_sums(a, nrm);                        // block-uniform: the budgets need the indicators
    __syncthreads();                                                                       // ---- barrier A

    // ---- 2. indicators, gates, budget, by one warp (all lanes alike but for the sums and the divisions, which lanes share).
    //         With device-decided budgets this runs now (the threshold search needs them); with host-decided budgets at the
    //         very end.  What goes to memory is written at the end in either case.
    auto column_sum = [&]() {                                  // lanes 8 c .. 8 c + 7: column c over the warps
        float t;
        if constexpr (NW == 8) {
            t = (&sm.red[0][0])[lane];
        } else if constexpr (NW == 16) {
            const float2 v = reinterpret_cast<const float2*>(&sm.red[0][0])[lane];
            t = v.x + v.y;
        } else {
            static_assert(NW == 16 || NW == 32, "a lane holds an eighth of a column");
            const float4 v = reinterpret_cast<const float4*>(&sm.red[0][0])[lane];
            t = (v.x + v.y) + (v.z + v.w);
        }
#pragma unroll
        for (int off = 1; off <= 4; off <<= 1) t += __shfl_xor_sync(0xffffffffu, t, off);
        return t;
    };
    auto indicators = [&]() {
        const float t = column_sum();
        const float t0 = __shfl_sync(0xffffffffu, t, 0), t1 = __shfl_sync(0xffffffffu, t, 8);
        const float t2 = __shfl_sync(0xffffffffu, t, 16), t3 = __shfl_sync(0xffffffffu, t, 24);
        // Four shares by one IEEE division in four lanes, none as one minus another: the share of an only modality is exactly
        // 1, and a small one keeps its precision.  Attention (Eq. P2D / P3D): t_m / (t_2D + t_3D).  Mean feature norms
        // (Eq. 3-1): (t_m / n_m) / (t_2D / n_2D + t_3D / n_3D), all times n_2D n_3D / kMaxVis.
        const float f2 = t2 * (static_cast<float>(max(n3, 1)) / kMaxVis), f3 = t3 * (static_cast<float>(max(n2, 1)) / kMaxVis);   // (exact factors <= 1)
        const float num = lane == 0 ? f2 : (lane == 1 ? f3 : (lane == 2 ? t0 : t1));
        const float quot = num / (lane < 2 ? f2 + f3 : t0 + t1);
        const float x0 = gp.has_l1 ? __shfl_sync(0xffffffffu, quot, 0) : 0.5f, x1 = gp.has_l1 ? __shfl_sync(0xffffffffu, quot, 1) : 0.5f;
        const float x2 = __shfl_sync(0xffffffffu, quot, 2), x3 = __shfl_sync(0xffffffffu, quot, 3);
        const float mh0 = carry ? fmaf(s.c_prev, mprev.x, s.c_new * x0) : x0;
        const float mh1 = carry ? fmaf(s.c_prev, mprev.y, s.c_new * x1) : x1;
        const float mh2 = carry ? fmaf(s.c_prev, mprev.z, s.c_new * x2) : x2;
        const float mh3 = carry ? fmaf(s.c_prev, mprev.w, s.c_new * x3) : x3;
        const int c1 = mh1 < gp.tau_2d ? MVLA_SET_2D : (mh1 > gp.tau_3d ? MVLA_SET_3D : (MVLA_SET_2D | MVLA_SET_3D));
        const int c2 = mh3 < gp.eps_3d ? MVLA_SET_2D : (MVLA_SET_2D | MVLA_SET_3D);
        int cf = c2 & c1;
        if (cf == 0) cf = c2;                                     // conflict resolution (Sec. 4.4)
        int b2 = s.k_2d_fixed, b3 = s.budget - s.k_2d_fixed;
        if (!k_fixed) {
            const float w3 = cf == (MVLA_SET_2D | MVLA_SET_3D) ? mh3 : (cf == MVLA_SET_2D ? 0.f : 1.f);
            const int lo3k = max(s.kmin_3d, s.budget - n2);
            const int hi3k = min(n3, s.budget - s.kmin_2d);
            b3 = static_cast<int>(floorf(static_cast<float>(s.budget) * w3 + 0.5f));
            b3 = min(max(b3, lo3k), hi3k);
            b2 = s.budget - b3;
        }
        if (lane == 0) {
            sm.budget[0] = b2; sm.budget[1] = b3;
            sm.x[0] = x0; sm.x[1] = x1; sm.x[2] = x2; sm.x[3] = x3;
            sm.mhat[0] = mh0; sm.mhat[1] = mh1; sm.mhat[2] = mh2; sm.mhat[3] = mh3;
            sm.sets[0] = c1; sm.sets[1] = c2; sm.sets[2] = cf;
        }
    };

    // ---- 3. kept or dropped, by the number of keys in higher bins; where the budget runs out inside a bin, by rank in it
    // st[e]: 0 dropped, 1 kept, 2 undecided, 3 on the list of its bin
    int st[EPT];
#pragma unroll
    for (int e = 0; e < EPT; ++e) st[e] = j0 + 32 * e < j_end ? 2 : 0;
    int k2 = s.k_2d_fixed, k3 = s.budget - s.k_2d_fixed;
    int take2 = k2, take3 = k3;               // to be taken from the keys under examination
    bool act2 = true, act3 = true;            // the modality still has undecided keys
    bool ties = false;
    int listed2 = 0, listed3 = 0;
#pragma unroll 1
    for (int level = 0; level < kSelLevels; ++level) {
        auto count_slice = [&](int i) {                           // (both halves of a word at once: a half never exceeds kMaxVis)
            const uint4 x = reinterpret_cast<const uint4*>(sm.hist)[i * 32 + lane];
            const uint32_t b1 = x.x, b2 = b1 + x.y, b3 = b2 + x.z, mine = b3 + x.w;
            const uint32_t inc = static_cast<uint32_t>(warp_incl_scan(static_cast<int>(mine), lane)), ex = inc - mine;
            reinterpret_cast<uint4*>(sm.before)[i * 32 + lane] = make_uint4(ex, ex + b1, ex + b2, ex + b3);
            if (lane == 31) sm.slice[i] = inc;
        };
        if (level == 0 && !k_fixed && warp == NW - 1) indicators();      // its slice goes to the warp before it
        else
#pragma unroll
            for (int u = 0; u < kSlices / NW; ++u) count_slice(warp + u * NW);
        if (level == 0 && !k_fixed && warp == NW - 2)
#pragma unroll
            for (int u = 0; u < kSlices / NW; ++u) count_slice(NW - 1 + u * NW);
        __syncthreads();                                                                   // ---- barrier B
        if (level == 0 && !k_fixed) { take2 = k2 = sm.budget[0]; take3 = k3 = sm.budget[1]; }
        const int slice = lane < kSlices ? static_cast<int>(sm.slice[lane]) : 0, before_slice = warp_incl_scan(slice, lane) - slice;
        bool any_listed = false;
        int bound[EPT];                                           // keys in higher bins
#pragma unroll
        for (int e = 0; e < EPT; ++e) {
            const bool is3 = j0 + 32 * e >= n2, open = st[e] == 2 && (is3 ? act3 : act2);
            const int half = is3 ? 16 : 0, k = is3 ? take3 : take2;
            const uint32_t first = static_cast<uint32_t>(__shfl_sync(0xffffffffu, before_slice, bin[e] / kSliceBins));
            const int higher = half_of(first + sm.before[bin[e]], half), in_bin = half_of(sm.hist[bin[e]], half);
            bound[e] = higher;
            const int now = higher + in_bin <= k ? 1 : (higher >= k ? 0 : 3);
            st[e] = open ? now : st[e];
            any_listed |= open && now == 3;
        }
        if (any_listed) {                                         // (few threads)
#pragma unroll
            for (int e = 0; e < EPT; ++e) {
                const int j = j0 + 32 * e;
                const bool is3 = j >= n2;
                if (st[e] != 3 || !(is3 ? act3 : act2)) continue;
                // place in the bin and index in one word; a bin that is wider, as the open ends of the window are: as if crowded
                const bool open = (level == 0 && (bin[e] == 0 || bin[e] == kSelBins - 1)) || (is3 ? sh3 : sh2) > 20;
                const int slot = atomicAdd(&sm.ncand[is3 ? 1 : 0], open ? kCandMax + 1 : 1);
                const uint32_t place = (key[e] - (is3 ? lo3 : lo2)) & ((1u << (is3 ? sh3 : sh2)) - 1u);
                static_assert(kMaxVis == 1 << 12, "an index is 12 bits");
                if (slot < kCandMax) sm.cand[is3 ? 1 : 0][slot] = place << 12 | static_cast<uint32_t>(kMaxVis - 1 - j);
                sm.take[is3 ? 1 : 0] = (is3 ? take3 : take2) - bound[e];      // (the same from all keys of the bin)
            }
        }
        __syncthreads();                                                                   // ---- barrier C
        listed2 = act2 ? sm.ncand[0] : listed2;
        listed3 = act3 ? sm.ncand[1] : listed3;
        act2 = act2 && listed2 > kCandMax;
        act3 = act3 && listed3 > kCandMax;
        if (__builtin_expect(!act2 && !act3, 1)) break;        // block-uniform
        // The keys of a crowded bin are counted once more, over the range that they have, unless they are all equal.  (This
        // part is rare and runs from a cold instruction cache, half a microsecond for 1.5 KB: it does no more than it must.)
        if (act2) take2 = sm.take[0];
        if (act3) take3 = sm.take[1];
        uint32_t mn2 = 0u, mx2 = 0u, mn3 = 0u, mx3 = 0u;
#pragma unroll
        for (int e = 0; e < EPT; ++e) {
            const bool is3 = j0 + 32 * e >= n2;
            if (st[e] != 3 || !(is3 ? act3 : act2)) continue;
            st[e] = 2;
            if (is3) { mn3 = max(mn3, ~key[e]); mx3 = max(mx3, key[e]); }
            else     { mn2 = max(mn2, ~key[e]); mx2 = max(mx2, key[e]); }
        }
        mn2 = __reduce_max_sync(0xffffffffu, mn2); mx2 = __reduce_max_sync(0xffffffffu, mx2);
        mn3 = __reduce_max_sync(0xffffffffu, mn3); mx3 = __reduce_max_sync(0xffffffffu, mx3);
        if (lane == 0) { atomicMax(&sm.ext[0], mn2); atomicMax(&sm.ext[1], mx2); atomicMax(&sm.ext[2], mn3); atomicMax(&sm.ext[3], mx3); }
        clear_hist();
        if (tid < 2 * kCandMax && (tid < kCandMax ? act2 : act3)) (&sm.cand[0][0])[tid] = 0u;
        __syncthreads();
        const uint4 x = *reinterpret_cast<const uint4*>(sm.ext);
        if (tid < 2) sm.ncand[tid] = 0;
        auto narrow = [&](uint32_t least, uint32_t most, uint32_t& lo, int& sh) {
            lo = least;
            sh = max(0, 32 - __clz(most - least) - kSelBits);
            return most > least;
        };
        if (act2 && !narrow(~x.x, x.y, lo2, sh2)) { ties = true; act2 = false; }
        if (act3 && !narrow(~x.z, x.w, lo3, sh3)) { ties = true; act3 = false; }
        if (!act2 && !act3) break;
#pragma unroll
        for (int e = 0; e < EPT; ++e) {
            const bool is3 = j0 + 32 * e >= n2;
            if (st[e] != 2 || !(is3 ? act3 : act2)) continue;
            bin[e] = bin_of(key[e], is3 ? lo3 : lo2, is3 ? sh3 : sh2);
            atomicAdd(&sm.hist[bin[e]], is3 ? 0x10000u : 1u);
        }
        __syncthreads();
        if (tid < 4) sm.ext[tid] = 0u;
    }
    // the listed keys of a modality are ranked among themselves
#pragma unroll
    for (int e = 0; e < EPT; ++e) {
        if (st[e] != 3) continue;
        const int j = j0 + 32 * e;
        const bool is3 = j >= n2;
        const uint32_t place = (key[e] - (is3 ? lo3 : lo2)) & ((1u << (is3 ? sh3 : sh2)) - 1u);
        const uint32_t mine = place << 12 | static_cast<uint32_t>(kMaxVis - 1 - j);
        const int n = is3 ? listed3 : listed2;
        int rank = 0;
#pragma unroll 1
        for (int i = 0; i < n; i += 8) {                   // (entries past n are zero)
            const uint4 q = reinterpret_cast<const uint4*>(sm.cand[is3 ? 1 : 0])[i / 4], w = reinterpret_cast<const uint4*>(sm.cand[is3 ? 1 : 0])[i / 4 + 1];
            rank += ((q.x > mine ? 1 : 0) + (q.y > mine ? 1 : 0)) + ((q.z > mine ? 1 : 0) + (q.w > mine ? 1 : 0));
            rank += ((w.x > mine ? 1 : 0) + (w.y > mine ? 1 : 0)) + ((w.z > mine ? 1 : 0) + (w.w > mine ? 1 : 0));
        }
        st[e] = rank < sm.take[is3 ? 1 : 0] ? 1 : 0;
    }

    // ---- 4. emission.  Tokens are ranked in visual order (2D first) by warp ballots.  The three segments are contiguous,
    //         so a kept token's output row is the number of rows that the segments lying before its own contribute plus its
    //         rank inside its modality.
    const unsigned below = (1u << lane) - 1u;
    auto before_warp = [&]() {                                    // sum of the counts of the warps before this one (each warp for itself)
        return static_cast<int>(__reduce_add_sync(0xffffffffu, lane < warp ? static_cast<unsigned>(sm.wtot[lane]) : 0u));
    };
    if (ties) {                                                   // block-uniform: equal keys straddle a budget: lower index wins
        unsigned own = 0u;
#pragma unroll
        for (int e = 0; e < EPT; ++e) {
            const bool is3 = j0 + 32 * e >= n2;
            own += __popc(__ballot_sync(0xffffffffu, st[e] == 2 && !is3)) | (__popc(__ballot_sync(0xffffffffu, st[e] == 2 && is3)) << 16);
        }
        if (lane == 0) sm.wtot[warp] = static_cast<int>(own);
        __syncthreads();
        int r2 = before_warp(), r3 = static_cast<int>(static_cast<unsigned>(r2) >> 16);
        r2 &= 0xFFFF;
#pragma unroll
        for (int e = 0; e < EPT; ++e) {
            const bool is3 = j0 + 32 * e >= n2;
            const unsigned b2 = __ballot_sync(0xffffffffu, st[e] == 2 && !is3), b3 = __ballot_sync(0xffffffffu, st[e] == 2 && is3);
            if (st[e] == 2) st[e] = is3 ? (r3 + __popc(b3 & below) < take3 ? 1 : 0) : (r2 + __popc(b2 & below) < take2 ? 1 : 0);
            r2 += __popc(b2);
            r3 += __popc(b3);
        }
        __syncthreads();                                          // sm.wtot is reused below
    }
    unsigned kept[EPT];
    int own = 0;
#pragma unroll
    for (int e = 0; e < EPT; ++e) {
        kept[e] = __ballot_sync(0xffffffffu, st[e] == 1);
        own += __popc(kept[e]);
    }
    if (lane == 0) sm.wtot[warp] = own;
    // row of the sample's output = rank among its kept tokens + what lies before, index inside the sample = j + a constant
    const int row2 = (s.off_txt < s.off_2d ? s.n_txt : 0) + (s.off_3d < s.off_2d ? k3 : 0);
    const int row3 = (s.off_txt < s.off_3d ? s.n_txt : 0) + (s.off_2d < s.off_3d ? k2 : 0) - k2;
    int32_t* const list = role.list;
    int32_t* const kept_idx = io.kept_idx + s.out_off;
    __syncthreads();                                                                       // ---- barrier D
    int r = before_warp();
#pragma unroll
    for (int e = 0; e < EPT; ++e) {
        const int j = j0 + 32 * e;
        const bool is3 = j >= n2;
        const int pos = r + __popc(kept[e] & below) + (is3 ? row3 : row2), val = j + (is3 ? s.off_3d - n2 : s.off_2d);
        if (list && st[e] == 1) list[pos * kListStride] = val;
        if (st[e] == 1) kept_idx[pos] = val;
        r += __popc(kept[e]);
    }
    const int baset = (s.off_2d < s.off_txt ? k2 : 0) + (s.off_3d < s.off_txt ? k3 : 0);
    for (int i = tid; i < s.n_txt; i += NT) {
        if (list) list[(baset + i) * kListStride] = s.off_txt + i;
        kept_idx[baset + i] = s.off_txt + i;
    }
    after_list();
    if (role.late_pdl && !role.beside) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    // ---- 5. what nobody downstream waits for
#pragma unroll
    for (int e = 0; e < EPT; ++e) {
        const int j = j0 + 32 * e;
        if (j < j_end) {
            if (io.acc64) io.acc64[s.vis_off + j] = 0ull;         // ready for the next call
            if (io.attn_out) io.attn_out[s.vis_off + j] = a[e];
            if (s.update_state) io.ahat_state[s.state_off_w + j] = key_to_float(key[e]);
            if (io.ahat_out) io.ahat_out[s.vis_off + j] = key_to_float(key[e]);
        }
    }
    if (k_fixed) {                                            // host-decided budgets: the indicators come now
        if (gp.has_l1) load_norms();
        partial_sums(a, nrm);
        __syncthreads();
        if (warp == NW - 1) indicators();
    }
    __syncwarp();
    if (tid == NT - 32) {                                     // the lane of the indicators' warp that left them in shared memory
        if (s.update_state) reinterpret_cast<float4*>(io.mhat_state)[s.mstate_off_w] = make_float4(sm.mhat[0], sm.mhat[1], sm.mhat[2], sm.mhat[3]);
        if (io.budgets) {
            io.budgets[b_glob * 2 + 0] = k2;
            io.budgets[b_glob * 2 + 1] = k3;
        }
        if (io.diag) {
            mvla_diag dg;
            dg.t = s.t; dg.c_s1 = sm.sets[0]; dg.c_s2 = sm.sets[1]; dg.c_final = sm.sets[2];
            dg.budget = s.budget; dg.k_2d = k2; dg.k_3d = k3; dg.reserved = 0;
#pragma unroll
            for (int c = 0; c < 4; ++c) { dg.x[c] = sm.x[c]; dg.mhat[c] = sm.mhat[c]; }
            io.diag[b_glob] = dg;
        }
        io.out_offsets[b_glob] = s.out_off;
        if (io.write_total && b_local == io.n_in_launch - 1) io.out_offsets[b_glob + 1] = io.total_out;
    }
    // optional: the smoothed scores normalised to mean one inside each modality.  The ranking above
    // uses the smoothed scores themselves; a positive per-modality factor cannot change it.
    if (io.z_out) {
        float smo[EPT];
#pragma unroll
        for (int e = 0; e < EPT; ++e) smo[e] = j0 + 32 * e < j_end ? key_to_float(key[e]) : 0.f;
        __syncthreads();                                          // the indicators' warp is done with the sums
        partial_sums(smo, nrm);
        __syncthreads();
        const float t = column_sum();
        const float f2 = static_cast<float>(n2) / __shfl_sync(0xffffffffu, t, 0), f3 = static_cast<float>(n3) / __shfl_sync(0xffffffffu, t, 8);
#pragma unroll
        for (int e = 0; e < EPT; ++e) {
            const int j = j0 + 32 * e;
            if (j < j_end) io.z_out[s.vis_off + j] = smo[e] * (j < n2 ? f2 : f3);
        }
    }
}

}  // namespace mvla
