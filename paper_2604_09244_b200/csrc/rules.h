// Rules of the host that choose between two ways of doing the same work, by sizes alone, and what they were measured with.
#pragma once

#include <stddef.h>
#include <stdint.h>

namespace mvla {

// Whether the streaming scoring kernel takes the feature norms of an adaptive batch itself, by two more warps, or a kernel
// beside it does.  A piece of a row (kNormPiece) takes a norm warp the same time whatever its bytes: it waits for the piece, and three
// are in flight.  The scores hide that as far as they go, one unit per (head, text query); the kernel beside them costs bandwidth, by the bytes of a
// row; and inside saves its launch and boundary, a fixed gain.  In units: 2048 a piece, 15 / 64 a byte, 300 000 for the launch; these put
// the line where 800 pairs of measurements have it with the fewest calls on the wrong side.  Whole steps in us, beside / inside, 768 tokens a
// sample unless said otherwise, texts of up to 64 | of up to 14 (16 queries):
//   rows of 2 KB, 8 heads of 128: 6 samples 15.9 / 15.7, 10 22.9 / 26.5, 15 25.3 / 35.3 | 10 18.9 / 26.3
//   rows of 4 KB, 16 heads of 128: 16 of 228 tokens 21.5 / 20.8, 16 46.6 / 50.5, with 4 key heads 32.3 / 38.6 | 26 of 228 22.6 / 27.9, 15 40.8 / 46.0
//                 32 heads of 64: 12 39.8 / 39.6, 16 with 8 key heads 43.5 / 42.8 | 15 42.0 / 46.1, with 8 key heads 29.6 / 37.0
//   rows of 6 KB, 32 heads of 96: | 15 59.6 / 62.2, with 8 key heads, 10 29.8 / 32.8
//   rows of 8 KB, 32 heads of 128: 4 24.0 / 23.1, 16 83.0 / 81.5, e4m3 67.3 / 62.4 | 10 48.5 / 42.4
//                 16 heads of 256: 16 81.3 / 80.3, 16 of 228 33.8 / 27.6, e4m3 with 8 key heads 54.2 / 52.4 | e4m3, 26 of 228 33.3 / 31.9
//   rows of 10 KB, 40 heads of 128: 6 49.1 / 43.7 | 15 88.0 / 99.2; 20 heads: 6 28.0 / 33.5
//   rows of 16 KB, 16 heads of 128: 6 45.6 / 38.4, 10 66.8 / 61.2 | 6 45.8 / 37.6
// Above 88 tokens a multiprocessor inside loses whatever the texts (32 heads of 128: 18 samples 90.4 / 92.6, 32 153 / 163), and samples of more
// than 16 key tiles go either way (2 x 3426 77.4 / 73.3, 7 x 2584 115.4 / 119); with the tail behind the kernel, that is: where it runs beside (tail_beside_pays, as
// for most of these now) the norms are inside whatever this rule says.  Rows of eight times the keys' bytes, where the
// scores of few jobs end early: e4m3, 16 heads of 256, 4 key heads, 12 x 435 (192 jobs) 26.5 / 27.3, 20 x 350 (320 jobs) 37.8 / 34.8.
constexpr uint32_t kNormPiece = 8192;        // bytes of a row that a norm warp fetches at once
struct NormsInsideSizes {
    int64_t rows;               // visual tokens of the launch
    int padded_text, max_tiles; // longest text rounded up to 16, key tiles of the largest sample
    int jobs;                   // samples x heads
    int n_heads;
    int64_t row_bytes, key_bytes;   // of a token: its hidden row, its keys
    int sm_count;
};
inline bool norms_inside_pays(const NormsInsideSizes& c)
{
    if (c.max_tiles > 16 || c.rows > 88 * c.sm_count) return false;
    if (c.row_bytes >= 8 * c.key_bytes && c.jobs < 2 * c.sm_count) return false;
    const int64_t pieces = (c.row_bytes + kNormPiece - 1) / kNormPiece;
    return c.rows * (2048 * pieces - 15 * c.row_bytes / 64 - static_cast<int64_t>(c.n_heads) * c.padded_text) < 300000;
}

// The same of patch-by-patch batches, whose norms otherwise come from the indicators.  The scoring kernel writes the attention copy there, which
// takes as long as (heads x text) does, whatever the heads' size.  Indicators / inside, samples of 256 patches unless said otherwise:
//   640 and more: 32 heads x 32 queries, heads of 64, 8 samples 35.2 / 33.2, 16 64.0 / 57.4; of 128, 8 39.8 / 36.4, 16 68.4 / 67.9; 16 x 48, 12 of
//     600 patches 97.4 / 84.9 (rows of 4 KB 87.9 / 80.7);
//   512: 32 x 16, 16 of 500 patches 93.5 / 94.8; 16 x 32, 16 52.0 / 49.6, 8 41.2 / 43.0, rows of 4 KB 43.2 / 45.2; 16 of 100 27.2 / 29.1;
//   256: 8 x 32, 16 42.7 / 45.0, rows of 4 KB 35.2 / 44.4; 16 x 16, 16 of 500 patches, rows of 4 KB 70.6 / 78.8.
inline bool patch_norms_inside_pays(int n_heads, int padded_text) { return n_heads * padded_text >= 640; }

// Whether a step of one sample with stable inputs and one key tile per scoring CTA is chained on the caller's stream, with its
// scores taken beside the selection and row copy of the step before, or forked to a side stream: two or three launches against three or four
// and four event calls (10 to 14 us of host time).  `moved`: bytes of keys, feature rows, text queries and surviving rows in and out.
// Per request of eight in a row, fork / chain in us, on a fast host (fork at the host's 9.6 to 10 us with fixed budgets, 11.5 to
// 12 adaptive, at any size):
//   fixed, up to 1.5 scoring CTAs a multiprocessor: 160 tokens 9.8 / 6.5, 32 heads of 64, 768 tokens 9.7 / 7.9; of 96 (15 MB) 9.7 / 9.4; of 128, 640
//     (17 MB) 9.7 / 9.9, 768 (20 MB) 9.6 / 9.9; 16 heads of 256, 768 (20 MB) 9.9 / 9.3, 850 (22 MB) 10.0 / 9.9, 950 (24 MB) 10.0 / 10.3;
//   fixed, more CTAs: 32 heads of 64, 950 tokens (12 MB) 9.8 / 9.1; of 96, 800 (15.4 MB) 9.9 / 10.3, 900 (17.1 MB) 10.0 / 10.5,
//     950 (18 MB) 9.7 / 11.0; of 128, 850 (22 MB) 9.8 / 11.1, 1010 (27 MB) 11.3 / 15.1;
//   adaptive: 32 heads of 64, 950 (15 MB) 11.8 / 9.8; of 96, 800 (19 MB) 11.7 / 12.0; of 128, 600 (20 MB) 11.9 / 10.6, 700 (22.5 MB) 12.0 / 12.3, 768
//     (24.5 MB) 11.8 / 12.7, 850 (27 MB) 12.0 / 13.4;
// on a slow host 768 of 128 fixed 13.4 / 9.8, 1010 of 96 adaptive 14.0 / 11.8.  The first pass of a new context gains more, eight requests of 768
// tokens 167 / 106 us, of 800 tokens and heads of 96 165 / 106: a step that loses 3 % later is left chained.  Two tiles per CTA:
// 1280 tokens of 64 (17 MB) 11.3 / 12.1, of 96 11.4 / 14.3, adaptive 14.0 / 18.5.  (In a CUDA graph launches cost nothing: always the fork.)
inline bool chain_pays(int64_t moved, int ctas, bool adaptive, int sm_count)
{
    const bool all_at_once = 2 * ctas <= 3 * sm_count;      // scoring CTAs that run beside the tail before it
    return moved <= (all_at_once || adaptive ? 20 : 17) * (int64_t(1) << 20);
}

// Jobs of the streaming scoring kernel go round the clusters in order, sample after sample.  The fullest cluster's costs in all, where `cost[b]` is that of a job of
// sample b: what the samples' order can make larger than it has to be, when clusters with a job more than others get one of the long ones last.
// The samples whose jobs take longest come first where that makes it smaller.  Elsewhere the order given stays: a long job
// behind short ones has its keys loaded while those are worked on.  Whole steps in us, order given / longest first, batches of 32 heads:
//   smaller: 16 of 228 tokens, texts of 16 to 64, 38.8 / 37.3, of 128 to 768 59.4 / 57.8, e4m3 45.6 / 44.4; five of 228 and one of 1500, twice, 64.6
//   / 60.6; patch by patch
//     16 of 512 77.6 / 74.6, 10 of 600 65.8 / 62.1, 16 of 128 to 800 74.4 / 70.4;
//   the same: eleven of 300 and one of 4048 87.5 / 90.8, fixed budgets 78.5 / 81.3; patch by patch seven of 128 and one of 1200 39.9 / 41.4, 8 of 1000 71.3 / 71.5.
// The cost is that of the softmax, by tiles and padded text queries, and of the keys, by tiles (with 0, 16, 32 or 64 queries' worth the choice is
// the same at all of these).
inline int job_cost(int tiles, int padded_text) { return tiles * (padded_text + 32); }
constexpr int kMostClusters = 256;
inline int64_t fullest_cluster(const int* cost, int samples, int heads, int clusters)
{
    if (clusters < 1 || clusters > kMostClusters) return 0;
    int64_t step[kMostClusters + 1] = {}, all = 0, load = 0, most = 0;
    int at = 0;                          // cluster of the sample's first job
    for (int b = 0; b < samples; ++b) {
        all += static_cast<int64_t>(heads / clusters) * cost[b];
        const int end = at + heads % clusters;
        step[at] += cost[b];
        step[end < clusters ? end : clusters] -= cost[b];
        if (end > clusters) { step[0] += cost[b]; step[end - clusters] -= cost[b]; }
        at = end % clusters;
    }
    for (int c = 0; c < clusters; ++c) {
        load += step[c];
        most = load > most ? load : most;
    }
    return all + most;
}
// `order`: the samples by falling cost, those of one cost as they were; whether that order is to be taken.
inline bool longest_first_pays(const int* cost, int samples, int heads, int clusters, uint8_t* order)
{
    int sorted[256];
    if (samples > 256) return false;
    bool same = true;
    for (int b = 0; b < samples; ++b) {
        int i = b;
        for (; i > 0 && sorted[i - 1] < cost[b]; --i) { sorted[i] = sorted[i - 1]; order[i] = order[i - 1]; }
        same &= i == b;
        sorted[i] = cost[b];
        order[i] = static_cast<uint8_t>(b);
    }
    return !same && fullest_cluster(sorted, samples, heads, clusters) < fullest_cluster(cost, samples, heads, clusters);
}

// Whether the tail of a batch runs beside the streaming kernel that scores it (launch_select_copy_beside): where the jobs fill more than two rounds, so that
// some samples are scored well before the others; where a job is long enough that the multiprocessors given to the tail and the words that pass between
// the kernels cost less than the idle memory between them; and where the scoring kernel's two norm warps, which take the feature norms then,
// keep up with its scores.  Whole steps in us, behind / beside, 32 heads of 128, texts of 16 to 64, unless said otherwise:
//   768 tokens (196 KB of keys a job): 10 samples 62.4 / 56.6, 16 93.7 / 88.4, 24 139.8 / 133.2; fixed budgets 12 56.0 / 51.9, 16 72.1 / 67.1; with 8
//   key heads, fixed, 10
//     39.0 / 37.3, 16 53.1 / 48.9, 32 90.6 / 86.1, short texts 42.0 / 41.4; 16 heads, fixed, short texts, 24 50.4 / 49.1; 640 tokens (160 KB), few
//     kept, 16 55.0 / 54.5;
//   3000 tokens: 5 samples 105.0 / 99.0; 3584: 8 163.6 / 156.0; e4m3, fixed, short texts, 12 of 1300 57.7 / 54.5, with 8 key heads 44.7 / 43.8; 32
//   heads of 64, fixed, short texts, 12 of 1500
//     55.6 / 52.2, with 8 key heads 40.3 / 39.6;
//   long and short samples: 5 of 228 and one of 3584 55.4 / 55.1, the long one first 61.1 / 55.4, 5 of 768 and one of 3584 67.5 / 65.5, 10 of 500 and
//   two of 1800 82.8 / 76.2.
// Of the other side of the lines, with rows copied in larger lots than now (kLotPieces in step.cu; between 98 and 160 KB nothing has been timed):
//   98 KB: e4m3 with 8 key heads 53.7 / 54.9, 32 heads of 64 56.9 / 57.8; 58 KB (228 tokens): 11 samples 31.1 / 38.4, 32 68.0 / 75.9;
//   16 heads of 128 (4 KB of keys a token), 24 samples 74.0 / 78.3: the norms take longer than the scores; two rounds and a bit of clusters of two, 6
//   of 1700 tokens with short
//   texts 68.5 / 68.5.
struct TailBesideSizes {
    int64_t tokens;             // visual tokens of the launch
    int samples, jobs;          // jobs: samples x heads
    int at_once;                // clusters that run at once
    int64_t head_bytes, key_bytes, row_bytes;   // of a token: its keys of one head, of all, its hidden row (0: no norms)
};
inline bool tail_beside_pays(const TailBesideSizes& c)
{
    if (c.samples < 2 || c.jobs <= 2 * c.at_once || c.tokens * c.head_bytes < (int64_t(160) << 10) * c.samples) return false;
    return c.key_bytes >= 6144 * ((c.row_bytes + kNormPiece - 1) / kNormPiece);
}

// Clusters of the streaming scoring kernel when the tail of the step runs beside it: at least kTailSms multiprocessors are the tail's, and of the others no
// more are taken than the rounds of jobs on them need (what a last round leaves idle is the tail's, too).  Counting the rounds on all multiprocessors and
// leaving kTailSms out afterwards, 32 heads, fixed budgets, us a step: 18 samples (576 jobs: five rounds on 136) 77.9, five rounds on 116 75.2, four on 144 with
// four left for the tail 80.3 (behind the scoring kernel 77.2); 27 samples 112.6 / 109.8 / 114.2; adaptive, 13 samples 74.1 / 72.5 / 74.5, 22 124.1 / 120.2 / 125.0,
// 32 174.1 / 172.7; 13 of 1280 tokens (clusters of two) 127.7 / 125.1 / 128.2.
constexpr int kTailSms = 12;
inline int clusters_beside_tail(int jobs, int at_once, int cluster, int sm_count)
{
    const int left = (sm_count - kTailSms) / cluster, most = left < 1 ? 1 : (left < at_once ? left : at_once);
    const int rounds = (jobs + most - 1) / most;
    return (jobs + rounds - 1) / rounds;
}

}  // namespace mvla
