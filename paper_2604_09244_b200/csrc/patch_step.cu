// Tail of the patch-by-patch step (Alg. 1 taken literally) as ONE kernel after the scoring kernel:
//   * CTAs [0, n_ind): indicators of a block of patches each (Eq. 3-1, Eq. 3-4, Eq. P2D, Eq. P3D) from the
//     attention copy that the scoring kernel left in L2; each patch's result also goes, as three 8-byte
//     words, to the CTA that runs the stages after it;
//   * one CTA per sample: temporal predictor, dual threshold, K-Means, semantic rules, fusion, masks
//     (stages 1-4), reading each patch's words as they appear; it writes the kept list as 4-byte words;
//   * the remaining CTAs copy the surviving rows, each warp polling the word of the row it is to move.  Output rows are
//     dealt out over all of them, whatever sample they belong to: which samples keep many rows shows only here, and with CTAs of
//     its own per sample the one with the most rows was copied 17 us longer than the median one (16 samples of 512 tokens).
// No kernel boundary, fence or flag lies between the three roles: every word is its own signal, re-armed
// (all ones) by the scoring kernel of the same step.  The roles go by ticket (cta_ticket: the order in which the
// CTAs started), so a consumer only ever waits for CTAs that are already running; every wait is bounded all the same.
#include "copy_impl.cuh"
#include "patch_impl.cuh"

#include <algorithm>

namespace mvla {
namespace {

constexpr int kTailThreads = kIndThreads;

struct PatchTailPlan {
    int16_t ind0[kMaxChunk + 1];      // first indicator CTA of every sample; ind0[n] = their number
    int16_t lag;                      // see the kernel
    int16_t copiers;                  // copying CTAs
    int32_t rows;                     // rows that the samples may keep
};

template <typename T, int PP, bool NORMS, class BD>
__global__ void __launch_bounds__(kTailThreads, 1)
patch_tail_kernel(const __grid_constant__ BD bd, const __grid_constant__ PatchTailPlan tp, int n_heads,
                  const AlphaOut alpha, const T* __restrict__ hidden, const float* __restrict__ l1, int d_model, float* __restrict__ x_out,
                  float* __restrict__ attn_out, unsigned long long* rec, const PatchParams pp, const PatchIO io,
                  const __grid_constant__ CompactArgs ca, int32_t* list, unsigned int* ticket_counter)
{
    // Roles by ticket: the indicator CTAs of sample after sample, behind those of sample b the selecting CTA of sample b - lag
    // (whose indicators are then about done: a selecting CTA that waits keeps a multiprocessor from the others), the selecting CTAs of
    // the last samples, the copying CTAs.  With all selecting CTAs behind all indicator CTAs the first list of 16 samples of 512
    // tokens came when the last indicators were done: 78.7 -> 74.2 us (74.0 with a lag of 3 samples instead of 6, 76.4 with 9).
    const int n = bd.count(), n_ind = tp.ind0[n];
    int c = cta_ticket(ticket_counter);
    int sel = -1;
    if (c < n_ind + max(0, n - tp.lag)) {
        int b = 0;
        while (b + 1 < n && c >= tp.ind0[b + 1] + max(0, b + 1 - tp.lag)) ++b;
        const int at = c - tp.ind0[b] - max(0, b - tp.lag);
        if (at < tp.ind0[b + 1] - tp.ind0[b]) {
            patch_indicators_block<T, PP, NORMS>(bd.at(b), at, n_heads, alpha, hidden, l1, d_model, x_out, attn_out, rec, true);
            return;
        }
        sel = b - tp.lag;
    } else if (c < n_ind + n) {
        sel = c - n_ind;
    }
    if (sel >= 0) {
        __shared__ PatchSmemT<kTailThreads> sm;
        patch_select_block<kTailThreads>(bd.at(sel), sel, n, pp, io, sm, rec, tp.copiers > 0 ? list + bd.at(0).cap_off : nullptr);
        return;
    }
    c -= n_ind + n;
    // ---- row copy
    const int tid = threadIdx.x, lane = tid & 31;
    const int w = c * (kTailThreads / 32) + (tid >> 5), nw = tp.copiers * (kTailThreads / 32);
    asm volatile("griddepcontrol.wait;" ::: "memory");      // the words were re-armed by the kernel before this one
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    // One warp of the CTA waits, at a low rate, for the hint that a list is about to be written (its own copy of it); only
    // then do all warps poll the words of their rows.  Thousands of warps polling while the selecting CTAs work would slow
    // those CTAs' own memory traffic.
    const int32_t* words = list + bd.at(0).cap_off;
    const int32_t* mine = words + 32 * (c % kHandLines);
    const uint64_t t0 = global_ns();
    constexpr uint64_t kLimitNs = 1000000000ull;
    __shared__ int s_hint, s_rows;
    if (tid < 32) {
        int hint = -1, rows = -1;
        for (uint32_t it = 0; it < kSpinLimit; ++it) {
            if (hint < 0) hint = ld_relaxed_gpu(mine);
            if (hint >= 0) rows = ld_relaxed_gpu(mine + 1);
            if (rows >= 0 || (hint >= 0 && bd.count() > 1)) break;      // (a sample alone: its count comes with the hint)
            if ((it & 63u) == 63u && global_ns() - t0 > kLimitNs) break;
            __nanosleep(hint < 0 ? 200 : 40);
        }
        if (lane == 0) { s_hint = hint; s_rows = rows; }
    }
    __syncthreads();
    int n_rows = s_rows;                                    // rows that the batch keeps, once this warp knows
    if (s_hint < 0 || (n_rows < 0 && bd.count() == 1)) {
        if (tid == 0) *reinterpret_cast<volatile int*>(io.status) = MVLA_ERR_TIMEOUT;
        return;
    }
    words += kHandWords;
    if (bd.count() == 1) {                                  // (known when the kernel is compiled)
        copy_rows(ca, n_rows, w, nw, lane, [&](int i, int64_t& srow, int64_t& drow) {
            const int v = poll_word(words + i * kListStride, t0, kLimitNs);     // the whole warp reads one word: one request
            if (v < 0) {                                                   // gave up: report, leave the row alone
                *reinterpret_cast<volatile int*>(io.status) = MVLA_ERR_TIMEOUT;
                return false;
            }
            srow = v;
            drow = i;
            return true;
        });
        return;
    }
    bool ended = false;
    copy_rows(ca, n_rows >= 0 ? n_rows : tp.rows, w, nw, lane, [&](int i, int64_t& srow, int64_t& drow) {
        int v = ended ? -1 : ld_relaxed_gpu(words + i * kListStride);
        for (uint32_t it = 0; v < 0 && !ended; ++it) {
            if (n_rows < 0) n_rows = ld_relaxed_gpu(mine + 1);
            if (n_rows >= 0 && i >= n_rows) {               // no such row, nor any after it
                ended = true;
                break;
            }
            if (it >= kSpinLimit || ((it & 63u) == 63u && global_ns() - t0 > kLimitNs)) {
                *reinterpret_cast<volatile int*>(io.status) = MVLA_ERR_TIMEOUT;       // gave up: report, leave the rows alone
                ended = true;
                break;
            }
            __nanosleep(20);
            v = ld_relaxed_gpu(words + i * kListStride);
        }
        if (v < 0) return false;
        srow = v;
        drow = i;
        return true;
    }, [&]() { return ended; });
}

}  // namespace

bool patch_tail_supported(const BatchDesc& bd)
{
    int blocks = 0;
    for (int b = 0; b < bd.n; ++b) blocks += (bd.s[b].n_2d + 1) / 2;
    return bd.n >= 1 && blocks + bd.n < 30000;
}

cudaError_t launch_patch_tail(const BatchDesc& bd, int n_heads, AlphaOut alpha, int dtype, int d_model, const void* hidden, const float* l1,
                              float* x_out, float* attn_out, unsigned long long* rec, const PatchParams& pp, const PatchIO& io,
                              const CompactJob& job, int32_t* list, int sm_count, unsigned int* ticket_counter, cudaStream_t stream)
{
    if (!patch_tail_supported(bd)) return cudaErrorInvalidConfiguration;
    // as many patches per CTA as still give every multiprocessor a CTA
    int per = 8;
    auto blocks_at = [&](int p) {
        int n = 0;
        for (int b = 0; b < bd.n; ++b) n += (bd.s[b].n_2d + p - 1) / p;
        return n;
    };
    while (per > 2 && blocks_at(per) < sm_count) per >>= 1;
    PatchTailPlan tp;
    int next = 0;
    for (int b = 0; b < bd.n; ++b) {
        tp.ind0[b] = static_cast<int16_t>(next);
        next += (bd.s[b].n_2d + per - 1) / per;
    }
    for (int b = bd.n; b <= kMaxChunk; ++b) tp.ind0[b] = static_cast<int16_t>(next);
    // samples whose indicators fill the multiprocessors, and one more
    tp.lag = static_cast<int16_t>(1 + (sm_count * bd.n + next - 1) / std::max(next, 1));
    const CompactArgs ca = compact_args(job);
    // together with the selecting CTAs they fill the multiprocessors once the indicator CTAs have retired
    const int copiers = ca.seg_begin[3] > 0 ? std::max(sm_count - bd.n, 1) : 0;
    tp.copiers = static_cast<int16_t>(copiers);
    tp.rows = 0;
    for (int b = 0; b < bd.n; ++b) tp.rows += bd.s[b].n_txt + bd.s[b].n_2d + bd.s[b].n_3d;

    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(next + bd.n + copiers));
    cfg.blockDim = dim3(kTailThreads);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1] = {pdl_attribute()};
    cfg.attrs = attr;
    cfg.numAttrs = 1;
#define MVLA_TAIL1(T, PPV, NORMS)                                                                             \
    if (per == PPV && (l1 == nullptr) == NORMS)                                                               \
        return with_desc(bd, [&](const auto& d) {                                                             \
            return cudaLaunchKernelEx(&cfg, patch_tail_kernel<T, PPV, NORMS, std::decay_t<decltype(d)>>, d, tp, n_heads, alpha, \
                                      static_cast<const T*>(hidden), l1, d_model, x_out, attn_out, rec, pp, io, ca, list, ticket_counter); });
#define MVLA_TAIL(T, PPV) MVLA_TAIL1(T, PPV, true)
    if (dtype == MVLA_DTYPE_BF16) {
        MVLA_TAIL(__nv_bfloat16, 8) MVLA_TAIL(__nv_bfloat16, 4) MVLA_TAIL(__nv_bfloat16, 2)
        MVLA_TAIL1(__nv_bfloat16, 8, false) MVLA_TAIL1(__nv_bfloat16, 4, false) MVLA_TAIL1(__nv_bfloat16, 2, false)
    } else { MVLA_TAIL(float, 8) MVLA_TAIL(float, 4) MVLA_TAIL(float, 2) }
#undef MVLA_TAIL1
#undef MVLA_TAIL
    return cudaErrorInvalidConfiguration;
}

}  // namespace mvla
