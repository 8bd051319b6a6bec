// Tail of the fused prune step: carry-over, gates, budget split, top-k selection (Alg. 1 stages 1-4,
// Eqs. 8-10) AND the compaction of the surviving rows (Sec. 4.4) in one kernel.
//
// A step on one sample is a chain of latencies, not a bandwidth problem: a kernel boundary costs a
// microsecond or two, a device-wide fence about one.  Here one CTA per sample runs the selection and the
// other CTAs of the grid copy rows:
//   * while the scores are still being computed the copying CTAs move the text rows, whose output
//     positions the host knows;
//   * the selecting CTA writes every entry of the kept list as one 4-byte word into library scratch; a
//     copying warp polls the word of the row it is to move (-1: not yet known) and starts the moment the
//     word is there.  No fence, flag or barrier lies between the two roles: each word is its own signal;
//   * what nobody waits for (smoothed state, indicators and diagnostics when the budgets came from the
//     host, optional score outputs) is written after the list.
// The scoring kernel that runs before this one re-arms the words, so nothing is left to do at the end.
// A word is polled by the dozen warps that move its row's segments, and polls of one line of the L2 are served one
// after another: neighbouring rows' words lie kListStride words apart (8 words a line instead of 32: eight action steps
// 143.5 -> 141.2 us, three views 20.8 -> 20.4; 4 words a line were no better).
#include "common.cuh"
#include "device_utils.cuh"
#include "copy_impl.cuh"
#include "lots.h"
#include "select_impl.cuh"

#include <algorithm>

namespace mvla {
namespace {

struct TailPlan {
    int16_t cta0[kMaxChunk + 1];      // first CTA of every sample; cta0[n] = grid size
};

// The same wait on a word that nothing ever sets, with a short limit: lets a test (or a health check) see
// the whole failure path -- the wait gives up, the kernel returns, the status word holds the error --
// without any kernel being made to hang.
__global__ void wait_probe_kernel(const int* never_set, uint64_t limit_ns, int* status)
{
    if (poll_word(never_set, global_ns(), limit_ns) < 0) *reinterpret_cast<volatile int*>(status) = MVLA_ERR_TIMEOUT;
}

// grid: CTAs 0 .. n-1 select (CTA b for sample b of the launch), the CTAs after them copy; tp.cta0[b] is the
// first copying CTA of sample b.  `list`: the kept list in library scratch (one word per output row of the
// launch's samples, -1 = not yet known; the scoring kernel before this one has set them all to -1).
// The roles go by block index.  The launcher never asks for more CTAs than fit on the device together
// (`ctas` = multiprocessors x CTAs per multiprocessor), and the kernel after this one cannot start before
// every CTA of this one has started, so all CTAs of the grid become resident whatever order they are
// dispatched in: a copying CTA never keeps its selecting CTA from running.  (Taking the roles in the order
// in which the CTAs start, by a ticket from an atomic counter as the patch-by-patch tail does, cost 0.4 us per
// step here: 296 atomics on one word.)  All waits are bounded all the same.
template <int NT, int CAP, bool STABLE, class BD>
__global__ void __launch_bounds__(NT, 1024 / NT)      // as many CTAs to a multiprocessor as the launcher counts on
select_copy_kernel(const __grid_constant__ BD bd, const __grid_constant__ TailPlan tp, const GateParams gp,
                   const SelectIO io, const __grid_constant__ CompactArgs ca, int32_t* __restrict__ list, int* status,
                   unsigned long long* __restrict__ stamps)
{
    const int tid = threadIdx.x, lane = tid & 31;
    const int cta = blockIdx.x;
    if (cta < bd.count()) {
        // ---- selection of one sample, by one CTA
        __shared__ SelectSmem<NT, CAP / NT> sm;
        const int b = cta;
        SelectRole role;
        role.late_pdl = !STABLE;
        role.stable = STABLE;
        if (tp.cta0[bd.count()] > 0) role.list = list + bd.at(b).out_off * kListStride;   // every word is its own "ready" signal
        select_sample<NT, CAP / NT>(bd.at(b), b, gp, io, sm, role, [&]() {
            if (stamps && tid == 0 && cta < kStampSlots) stamps[2 * cta + 1] = global_ns();
        });
        if (stamps && tid == 0 && cta < kStampSlots) stamps[2 * cta] = stamps[2 * cta + 1];   // placeholder start, see the copiers
        return;
    }
    // ---- row copy
    const int c = cta - bd.count();
    int b = 0;
    while (b + 1 < bd.count() && c >= tp.cta0[b + 1]) ++b;
    const int part = c - tp.cta0[b], nparts = tp.cta0[b + 1] - tp.cta0[b];
    const SampleDev& s = bd.at(b);
    const int w = part * (NT / 32) + (tid >> 5), nw = nparts * (NT / 32);

    // Output position of the text rows: known on the host when the split is (FIXED budgets, cold start),
    // or when the text segment lies before or behind both visual segments (then only the total counts).
    const bool b2 = s.n_2d > 0 && s.off_2d < s.off_txt, b3 = s.n_3d > 0 && s.off_3d < s.off_txt;
    int baset = -1;
    if (s.k_2d_fixed >= 0) baset = (b2 ? s.k_2d_fixed : 0) + (b3 ? s.budget - s.k_2d_fixed : 0);
    else if (b2 == b3) baset = b2 ? s.budget : 0;
    const bool text_early = baset >= 0;
    auto copy_text = [&]() {
        copy_rows(ca, s.n_txt, w, nw, lane, [&](int i, int64_t& srow, int64_t& drow) {
            srow = static_cast<int64_t>(s.seq_off) + s.off_txt + i;
            drow = static_cast<int64_t>(s.out_off) + baset + i;
            return true;
        });
    };
    if (!STABLE && text_early) copy_text();                 // while the scores are still being computed
    asm volatile("griddepcontrol.wait;" ::: "memory");      // keeps the chain of dependencies whole: the kernel after
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");   // this one may rely on the one before it being complete
    if (stamps && tid == 0 && cta < kStampSlots) stamps[2 * cta] = global_ns();
    if (STABLE && text_early) copy_text();

    {
        const int n_rows = s.n_out - (text_early ? s.n_txt : 0);
        const int32_t* kept = list + s.out_off * kListStride;
        const uint64_t t0 = global_ns();
        copy_rows(ca, n_rows, w, nw, lane, [&](int i, int64_t& srow, int64_t& drow) {
            const int r = (text_early && i >= baset) ? i + s.n_txt : i;       // skip the text rows copied before
            const int v = poll_word(kept + r * kListStride, t0, 1000000000ull);   // the whole warp reads one word: one request
            if (v < 0) {                                    // gave up: report, leave the row alone
                *reinterpret_cast<volatile int*>(status) = MVLA_ERR_TIMEOUT;
                return false;
            }
            srow = static_cast<int64_t>(s.seq_off) + v;
            drow = static_cast<int64_t>(s.out_off) + r;
            return true;
        });
    }
    if (stamps && cta < kStampSlots) {
        __syncthreads();
        if (tid == 0) stamps[2 * cta + 1] = global_ns();
    }
}

template <int NT, int CAP, bool STABLE, class BD>
cudaError_t launch_t(const BD& bd, const TailPlan& tp, const GateParams& gp, const SelectIO& io, const CompactArgs& ca,
                     int32_t* list, int* status, unsigned long long* stamps, cudaStream_t stream)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(bd.n + tp.cta0[bd.n]));
    cfg.blockDim = dim3(NT);
    cfg.stream = stream;
    // With its own small need a multiprocessor is left with little shared memory while this kernel runs, and only one scoring CTA
    // of the next step fits beside it: the others come when it is done.  All of it as shared memory, eight requests in a row, per request: 768
    // tokens, 32 heads of 128, fixed, 10.9 -> 10.0 us, 500 of 128 10.1 -> 8.6, 630 of 64 9.1 -> 7.6; up to 148 scoring CTAs as before.
    cudaLaunchAttribute attr[2] = {pdl_attribute()};
    attr[1].id = cudaLaunchAttributePreferredSharedMemoryCarveout;
    attr[1].val.sharedMemCarveout = cudaSharedmemCarveoutMaxShared;
    cfg.attrs = attr;
    cfg.numAttrs = STABLE ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, select_copy_kernel<NT, CAP, STABLE, BD>, bd, tp, gp, io, ca, list, status, stamps);
}

// ------------------------------------------------------------------ beside the scoring kernel
constexpr int kPieceSegs = 2;         // segments of rows that a warp takes at a time
// Pieces that a CTA takes at a time.  Smaller lots end together: with 16 pieces of four segments the rows of a dozen samples were 333 lots for 288
// CTAs, and some copied
// two where most had one.  Whole steps in us, behind the scoring kernel / 16 of 4 / 8 of 4 / 16 of 2 / 8 of 2 / 4 of 2: fixed budgets, 768 tokens, 8
// key heads, 10 samples 39.0 / 45.5 / 41.9 /
// 38.7 / 37.3 / 36.0, 16 53.1 / 54.9 / 51.3 / 49.6 / 48.9 / 48.6; 32 key heads, 16 72.1 / 68.7 / 66.7 / 68.5 / 67.1 / 67.0; adaptive, 16 93.7 / 88.4
// / 88.5 / 89.5 / 88.4 / 88.3, 5 of 228
// and one of 3584 tokens 55.4 / 59.2 / 57.3 / 56.2 / 55.1 / 55.2; 8 of 3584 (CTAs of 32 warps) 163.6 / 157.0 / 156.1 / 156.8 / 156.0 / 158.8.
constexpr int kLotPieces = 8;

// Work of the row copy, in segments (kSegBytes): the text rows of every sample whose place the host knows, then every sample's other rows.
struct BesidePlan {
    int32_t begin[2 * kMaxChunk + 1];
    int32_t baset[kMaxChunk];         // first output row of a sample's text rows inside the sample; -1: not known yet
    int32_t n, selectors, parts;
    int32_t lots;
};

// The tail of a batch scored by the streaming kernel, beside that kernel: it lives on the multiprocessors that the scoring kernel leaves free
// and, as that kernel's CTAs end, on all of them.  CTAs take their roles by ticket: the first ones select, sample after sample, as the
// samples' counters say that their scores are complete; all others copy rows, whose words the selecting CTAs write (select_copy_kernel).
// Scoring is then bound by the memory for all of its time and the row copy for its own, where in turn a batch left the memory
// idle from the drain of the one to the first list of the other.  Rows are given out in lots from one counter, samples in
// order, because CTAs join while it runs.  A CTA waits only for the scoring kernel, all of whose CTAs run when this one starts, and for the selecting
// CTAs, which have the lower tickets.
template <int NT, int CAP>
__global__ void __launch_bounds__(NT, 1024 / NT)
select_copy_beside_kernel(const __grid_constant__ BatchDesc bd, const __grid_constant__ BesidePlan bp, const GateParams gp, const SelectIO io,
                          const __grid_constant__ CompactArgs ca, int32_t* __restrict__ list, int32_t* hand, int* status,
                          unsigned long long* __restrict__ stamps)
{
    const int tid = threadIdx.x, lane = tid & 31;
    const int cta = cta_ticket(reinterpret_cast<unsigned int*>(hand + kHandTicket));
    const uint64_t t0 = global_ns();
    if (cta < bp.selectors) {
        __shared__ SelectSmem<NT, CAP / NT> sm;
        for (int b = cta; b < bp.n; b += bp.selectors) {
            if (tid == 0) {
                int done = 0;
                for (uint32_t it = 0; it < kSpinLimit; ++it) {
                    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(done) : "l"(hand + b) : "memory");
                    if (done == bp.parts || ((it & 63u) == 63u && global_ns() - t0 > 1000000000ull)) break;
                    __nanosleep(100);
                }
                if (done != bp.parts) *reinterpret_cast<volatile int*>(status) = MVLA_ERR_TIMEOUT;
                hand[b] = 0;                                // for the next launch
            }
            __syncthreads();                                // (and the sample before is done with the shared memory)
            SelectRole role;
            role.late_pdl = true;
            role.beside = true;
            role.status = status;
            role.t0 = t0;
            if (bp.lots > 0) role.list = list + bd.s[b].out_off * kListStride;
            select_sample<NT, CAP / NT>(bd.s[b], b, gp, io, sm, role, [&]() {
                if (stamps && tid == 0 && cta < kStampSlots) stamps[2 * cta + 1] = global_ns();
            });
            __syncthreads();
        }
        if (stamps && tid == 0 && cta < kStampSlots) stamps[2 * cta] = stamps[2 * cta + 1];   // of its last list, as in select_copy_kernel
        // "This kernel is complete" implies that the scoring kernel is.
        asm volatile("griddepcontrol.wait;" ::: "memory");
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
        return;
    }
    if (stamps && tid == 0 && cta < kStampSlots) stamps[2 * cta] = t0;
    // ---- row copy.  What a warp knows of the span of segments it is in stays in registers (an index into the parameters costs some hundred cycles).
    const int per_row = ca.seg_begin[3], n = bp.n;
    unsigned int* const counter = reinterpret_cast<unsigned int*>(hand + kHandLots);
    // Pieces come in lots (lots.h): 11000 pieces of six segments straight from one counter, by 4700 warps, made that counter the limit (the rows of
    // 16 requests moved
    // at 4.8 instead of 6.8 TB/s).
    __shared__ unsigned int s_lot;
    __shared__ volatile int s_next;
    if (tid == 0) {
        s_lot = atomicAdd(counter, 1u) << 12;
        s_next = static_cast<int>(atomicAdd(counter, 1u));
    }
    __syncthreads();
    struct Cell {
        unsigned int *word, *counter;
        volatile int* ahead;
        __device__ __forceinline__ uint32_t add() { return atomicAdd(word, 1u); }
        __device__ __forceinline__ void swap(uint32_t x) { __threadfence_block(); atomicExch(word, x); }
        __device__ __forceinline__ uint32_t peek() { return *reinterpret_cast<volatile unsigned int*>(word); }
        __device__ __forceinline__ int32_t next() { return *ahead; }
        __device__ __forceinline__ void put(int32_t x) { *ahead = x; }
        __device__ __forceinline__ int32_t ask() { return static_cast<int32_t>(atomicAdd(counter, 1u)); }
    } cell = {&s_lot, counter, &s_next};
    auto take = [&]() {
        uint32_t piece = 0;
        if (lane == 0) {
            bool gave_up = false;
            piece = take_piece(cell, kLotPieces, static_cast<uint32_t>(bp.lots), kSpinLimit, &gave_up);
            if (gave_up) *reinterpret_cast<volatile int*>(status) = MVLA_ERR_TIMEOUT;
        }
        return static_cast<int>(__shfl_sync(0xffffffffu, piece, 0));
    };
    int span = -1, begin = 0, end = 0, src0 = 0, dst0 = 0, skip_at = 0, skip = 0, row = -1, from = 0;
    bool polled = false, released = false;
    const int32_t* words = nullptr;
    const int all = bp.begin[2 * n];
    for (;;) {
        const int first = take() * kPieceSegs;
        if (first >= all) break;
        const int u1 = min(first + kPieceSegs, all);
        for (int u0 = first; u0 < u1; u0 += 2) {
            uint4 v[2][4];
            const uint4* sp[2];
            uint4* dp[2];
            int nvec[2];
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const int u = u0 + k;
                nvec[k] = 0;
                sp[k] = nullptr;
                dp[k] = nullptr;
                if (u >= u1) continue;
                if (u >= end) {                             // the span that holds the segment (spans may be empty)
                    do ++span; while (u >= bp.begin[span + 1]);
                    begin = bp.begin[span];
                    end = bp.begin[span + 1];
                    row = -1;
                    polled = span >= n;
                    const int b = polled ? span - n : span, baset = bp.baset[b];
                    const SampleDev& s = bd.s[b];
                    dst0 = s.out_off + (polled ? 0 : baset);
                    src0 = s.seq_off + (polled ? 0 : s.off_txt);
                    skip_at = baset >= 0 ? baset : s.n_out;
                    skip = baset >= 0 ? s.n_txt : 0;
                    words = list + s.out_off * kListStride;
                }
                const int r = (u - begin) / per_row, g = u - begin - r * per_row;
                int drow = r;
                if (polled) {
                    drow = r >= skip_at ? r + skip : r;     // the text rows have a span of their own
                    if (r != row) {
                        row = r;
                        from = poll_word(words + drow * kListStride, t0, 1000000000ull);
                        if (from < 0) *reinterpret_cast<volatile int*>(status) = MVLA_ERR_TIMEOUT;
                    }
                    if (from < 0) continue;                 // gave up: leave the row alone
                } else {
                    from = r;
                }
                const int tsel = g >= ca.seg_begin[2] ? 2 : (g >= ca.seg_begin[1] ? 1 : 0);
                const int seg = g - ca.seg_begin[tsel], rb = ca.row_bytes[tsel];
                sp[k] = reinterpret_cast<const uint4*>(ca.src[tsel] + static_cast<int64_t>(src0 + from) * rb + static_cast<int64_t>(seg) * kSegBytes);
                dp[k] = reinterpret_cast<uint4*>(ca.dst[tsel] + static_cast<int64_t>(dst0 + drow) * rb + static_cast<int64_t>(seg) * kSegBytes);
                nvec[k] = min(kSegBytes, rb - seg * kSegBytes) >> 4;
            }
#pragma unroll
            for (int k = 0; k < 2; ++k)
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (lane + i * 32 < nvec[k]) v[k][i] = ld_row(sp[k] + lane + i * 32);
#pragma unroll
            for (int k = 0; k < 2; ++k)
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (lane + i * 32 < nvec[k]) st_row(dp[k] + lane + i * 32, v[k][i]);
        }
        if (!released && span == 2 * n - 1) {               // the last sample's list is there: the scoring kernel is about done
            released = true;
            asm volatile("griddepcontrol.wait;" ::: "memory");
            asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
        }
    }
    __syncthreads();                                        // no warp of this CTA asks for a lot any more
    if (tid == 0) {
        if (atomicInc(reinterpret_cast<unsigned int*>(hand + kHandLeft), gridDim.x - bp.selectors - 1) == gridDim.x - bp.selectors - 1) *counter = 0u;
        if (stamps && cta < kStampSlots) stamps[2 * cta + 1] = global_ns();
    }
}

int max_vis_of(const BatchDesc& bd)
{
    int m = 0;
    for (int b = 0; b < bd.n; ++b) m = std::max(m, bd.s[b].n_2d + bd.s[b].n_3d);
    return m;
}

template <int NT, int CAP>
cudaError_t launch_beside_t(const BatchDesc& bd, const BesidePlan& bp, const GateParams& gp, const SelectIO& io, const CompactArgs& ca, int32_t* list,
                            int32_t* hand, int ctas, int* status, unsigned long long* stamps, cudaStream_t stream)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(ctas));
    cfg.blockDim = dim3(NT);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1] = {pdl_attribute()};
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, select_copy_beside_kernel<NT, CAP>, bd, bp, gp, io, ca, list, hand, status, stamps);
}

// First output row of a sample's text rows inside the sample, where the host knows it (see select_copy_kernel); else -1.
int text_base(const SampleDev& s)
{
    const bool b2 = s.n_2d > 0 && s.off_2d < s.off_txt, b3 = s.n_3d > 0 && s.off_3d < s.off_txt;
    if (s.k_2d_fixed >= 0) return (b2 ? s.k_2d_fixed : 0) + (b3 ? s.budget - s.k_2d_fixed : 0);
    return b2 == b3 ? (b2 ? s.budget : 0) : -1;
}

}  // namespace

cudaError_t launch_select_copy_beside(const BatchDesc& bd, const GateParams& gp, const SelectIO& io, const CompactJob& job, int32_t* list,
                                      int32_t* hand, int parts, int free_sms, int* status, unsigned long long* stamps, cudaStream_t stream)
{
    const CompactArgs ca = compact_args(job);
    const int nv = max_vis_of(bd), per_sm = nv > 2048 ? 1 : 2, per_row = ca.seg_begin[3];
    BesidePlan bp;
    bp.n = bd.n;
    bp.parts = parts;
    int at = 0;
    for (int b = 0; b < bd.n; ++b) {
        bp.baset[b] = text_base(bd.s[b]);
        bp.begin[b] = at;
        if (bp.baset[b] >= 0) at += bd.s[b].n_txt * per_row;
    }
    for (int b = 0; b < bd.n; ++b) {
        bp.begin[bd.n + b] = at;
        at += (bd.s[b].n_out - (bp.baset[b] >= 0 ? bd.s[b].n_txt : 0)) * per_row;
    }
    bp.begin[2 * bd.n] = at;
    bp.lots = (at + kPieceSegs * kLotPieces - 1) / (kPieceSegs * kLotPieces);
    bp.selectors = std::min(bd.n, std::max(1, std::min(8, free_sms * per_sm / 4)));
    const int ctas = at > 0 ? std::max(sm_count_of_current_device() * per_sm, bp.selectors + 1) : bp.selectors;
    if (nv <= 1024) return launch_beside_t<512, 1024>(bd, bp, gp, io, ca, list, hand, ctas, status, stamps, stream);
    if (nv <= 2048) return launch_beside_t<512, 2048>(bd, bp, gp, io, ca, list, hand, ctas, status, stamps, stream);
    return launch_beside_t<1024, kMaxVis>(bd, bp, gp, io, ca, list, hand, ctas, status, stamps, stream);
}

cudaError_t launch_wait_probe(const int32_t* never_set, uint64_t limit_ns, int* status, cudaStream_t stream)
{
    wait_probe_kernel<<<1, 32, 0, stream>>>(never_set, limit_ns, status);
    return cudaGetLastError();
}

cudaError_t launch_select_copy(const BatchDesc& bd, const GateParams& gp, const SelectIO& io, const CompactJob& job,
                               int32_t* list, int* status, bool stable, unsigned long long* stamps, cudaStream_t stream)
{
    if (bd.n < 1) return cudaErrorInvalidConfiguration;
    const CompactArgs ca = compact_args(job);
    // CTAs on the device at once: two of 512 threads to a multiprocessor, or one of 1024 (more than 2048 visual tokens); one of
    // 512 where the scoring CTAs of the next step are to run beside them (two: eight requests of 671 tokens 73 -> 79 us)
    int ctas = sm_count_of_current_device() * (max_vis_of(bd) > 2048 || stable ? 1 : 2) - bd.n;
    TailPlan tp;
    int next = 0;
    if (ca.seg_begin[3] > 0) {
        // copying CTAs per sample in proportion to its kept rows (rounded down), at least one each, and never more
        // than `ctas` in all -- the grid must fit on the device at once, see the kernel -- unless there are more
        // samples than that
        ctas = std::min(std::max(ctas, bd.n), 30000);
        int64_t rows = 0;
        for (int b = 0; b < bd.n; ++b) rows += bd.s[b].n_out;
        int share[kMaxChunk];
        int total = 0;
        for (int b = 0; b < bd.n; ++b) {
            share[b] = static_cast<int>(std::max<int64_t>(1, rows > 0 ? static_cast<int64_t>(ctas) * bd.s[b].n_out / rows : 1));
            total += share[b];
        }
        while (total > ctas) {                               // the minimum of one pushed it over: take from the largest
            int big = 0;
            for (int b = 1; b < bd.n; ++b) big = share[b] > share[big] ? b : big;
            if (share[big] <= 1) break;
            --share[big];
            --total;
        }
        for (int b = 0; b < bd.n; ++b) {
            tp.cta0[b] = static_cast<int16_t>(next);
            next += share[b];
        }
    } else {
        for (int b = 0; b < bd.n; ++b) tp.cta0[b] = 0;       // nothing to copy: selection only
    }
    for (int b = bd.n; b <= kMaxChunk; ++b) tp.cta0[b] = static_cast<int16_t>(next);
    const int nv = max_vis_of(bd);
    return with_desc(bd, [&](const auto& d) {
        if constexpr (std::is_same_v<std::decay_t<decltype(d)>, OneDesc>) {
            if (stable && nv <= 1024) return launch_t<512, 1024, true>(d, tp, gp, io, ca, list, status, stamps, stream);
        }
        if (stable) return cudaErrorInvalidConfiguration;
        if (nv <= 1024) return launch_t<512, 1024, false>(d, tp, gp, io, ca, list, status, stamps, stream);
        if (nv <= 2048) return launch_t<512, 2048, false>(d, tp, gp, io, ca, list, status, stamps, stream);
        return launch_t<1024, kMaxVis, false>(d, tp, gp, io, ca, list, status, stamps, stream);
    });
}

}  // namespace mvla
