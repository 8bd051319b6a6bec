"""The rules by which the host chooses between two ways of the same work (csrc/rules.h), at sizes on both sides of their lines
where both ways were timed.  Checked by a small C++ program built from the header itself (no GPU needed)."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def run_program(tmp_path, text):
    src, exe = tmp_path / "rules.cpp", tmp_path / "rules"
    src.write_text(text)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_2604_09244_b200", "csrc"),
                    "-o", str(exe), str(src)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout


NORMS = r"""
#include <cstdio>
#include "rules.h"
using namespace mvla;
// (bytes of an element of k, heads, head dim, key heads, bytes of a hidden row, padded text, samples, tokens and key tiles of a sample)
struct Point { int esize, heads, dim, kv, row, text, batch, tokens, tiles; bool inside; };
static const Point points[] = {
    {2, 8, 128, 8, 2048, 64, 10, 768, 6, false}, {2, 8, 128, 8, 2048, 16, 10, 768, 6, false},
    {2, 16, 128, 16, 4096, 64, 16, 228, 3, true}, {2, 16, 128, 16, 4096, 64, 16, 768, 6, false}, {2, 16, 128, 4, 4096, 64, 16, 768, 6, false},
    {1, 16, 128, 16, 4096, 64, 8, 768, 6, false}, {2, 16, 128, 16, 4096, 16, 26, 228, 3, false},
    {2, 32, 64, 8, 4096, 64, 16, 768, 6, true}, {2, 32, 64, 8, 4096, 16, 15, 768, 6, false}, {1, 32, 64, 8, 4096, 32, 15, 768, 6, false},
    {2, 32, 96, 32, 6144, 16, 15, 768, 6, false}, {2, 32, 96, 8, 6144, 16, 10, 768, 6, false}, {2, 32, 96, 32, 6144, 64, 15, 768, 6, true},
    {2, 32, 128, 32, 8192, 64, 16, 768, 6, true}, {2, 32, 128, 32, 8192, 64, 18, 768, 6, false}, {2, 32, 128, 8, 8192, 64, 16, 768, 6, true},
    {1, 32, 128, 32, 8192, 64, 16, 768, 6, true}, {2, 32, 128, 32, 8192, 16, 10, 768, 6, true}, {2, 16, 256, 16, 8192, 64, 16, 768, 6, true},
    {1, 16, 256, 8, 8192, 64, 16, 768, 6, true}, {1, 16, 256, 16, 8192, 16, 26, 228, 3, true}, {1, 16, 256, 4, 8192, 64, 12, 435, 5, false},
    {2, 40, 128, 40, 10240, 64, 6, 768, 6, true}, {2, 40, 128, 40, 10240, 16, 15, 768, 6, false}, {2, 20, 128, 20, 10240, 64, 6, 768, 6, false},
    {2, 16, 128, 16, 16384, 64, 10, 768, 6, true}, {2, 16, 128, 16, 16384, 16, 6, 768, 6, true}, {2, 32, 128, 32, 8192, 64, 5, 2224, 18, false},
};
int main()
{
    for (const Point& p : points) {
        const NormsInsideSizes c = {static_cast<int64_t>(p.batch) * p.tokens, p.text, p.tiles, p.batch * p.heads, p.heads, p.row,
                                   static_cast<int64_t>(p.kv) * p.dim * p.esize, 148};
        if (norms_inside_pays(c) != p.inside) { std::printf("%d heads of %d, %d x %d, text %d\n", p.heads, p.dim, p.batch, p.tokens, p.text); return 1; }
    }
    if (!patch_norms_inside_pays(32, 32) || !patch_norms_inside_pays(16, 48) || patch_norms_inside_pays(32, 16) || patch_norms_inside_pays(16, 32) ||
        patch_norms_inside_pays(8, 32)) { std::printf("patch by patch\n"); return 1; }
    std::printf("ok\n");
    return 0;
}
"""


def test_norms_are_taken_by_the_scoring_kernel_only_where_the_scores_hide_them(tmp_path):
    run_program(tmp_path, NORMS)


CHAIN = r"""
#include <cstdio>
#include "rules.h"
using namespace mvla;
struct Point { double mb; int ctas; bool adaptive, chained; };
static const Point points[] = {
    {5.5, 64, false, true}, {14.8, 192, false, true}, {19.8, 192, false, true}, {24.0, 128, false, false},
    {12.0, 256, false, true}, {15.4, 256, false, true}, {17.1, 256, false, false}, {18.0, 256, false, false}, {21.7, 256, false, false},
    {15.0, 256, true, true}, {19.1, 256, true, true}, {19.6, 192, true, true}, {22.5, 192, true, false}, {27.0, 256, true, false},
};
int main()
{
    for (const Point& p : points)
        if (chain_pays(static_cast<int64_t>(p.mb * (1 << 20)), p.ctas, p.adaptive, 148) != p.chained) {
            std::printf("%.1f MB, %d CTAs, adaptive %d\n", p.mb, p.ctas, p.adaptive);
            return 1;
        }
    std::printf("ok\n");
    return 0;
}
"""


def test_small_stable_steps_are_chained_only_where_the_gpu_keeps_up(tmp_path):
    run_program(tmp_path, CHAIN)


CLUSTERS = r"""
#include <cstdio>
#include "rules.h"
using namespace mvla;
int main()
{
    const int sizes[] = {1, 2, 4, 8}, at_once[] = {148, 74, 35, 16}, left[] = {136, 68, 34, 17};
    for (int s = 0; s < 4; ++s)
        for (int jobs = 1; jobs <= 2048; ++jobs) {
            const int most = at_once[s] < left[s] ? at_once[s] : left[s], n = clusters_beside_tail(jobs, at_once[s], sizes[s], 148);
            // no more than run at once beside the tail, as many rounds as on all of those, and no fewer clusters do
            const int rounds = (jobs + most - 1) / most;
            if (n < 1 || n > most || (jobs + n - 1) / n != rounds || (n > 1 && (jobs + n - 2) / (n - 1) == rounds)) {
                std::printf("%d jobs, clusters of %d: %d\n", jobs, sizes[s], n);
                return 1;
            }
        }
    if (clusters_beside_tail(512, 148, 1, 148) != 128 || clusters_beside_tail(576, 148, 1, 148) != 116 || clusters_beside_tail(256, 35, 4, 148) != 32 ||
        clusters_beside_tail(64, 4, 4, 16) != 1) { std::printf("points\n"); return 1; }
    std::printf("ok\n");
    return 0;
}
"""


def test_clusters_beside_a_tail_are_those_that_their_rounds_need(tmp_path):
    run_program(tmp_path, CLUSTERS)


ORDER = r"""
#include <cstdio>
#include <algorithm>
#include <random>
#include <vector>
#include "rules.h"
using namespace mvla;
struct Point { int clusters; bool first; std::vector<int> cost; };      // 32 heads; costs of a sample's jobs (tiles x (padded text + 32))
static const Point points[] = {
    {148, true, {160, 160, 160, 160, 160, 128, 160, 128, 128, 192, 192, 160, 128, 192, 192, 160}},
    {148, true, {160, 400, 160, 560, 160, 320, 160, 448, 128, 480, 192, 560, 128, 480, 192, 560}},
    {74, true, {192, 192, 192, 192, 192, 1248, 192, 192, 192, 192, 192, 1248}},
    {148, true, {480, 480, 480, 480, 480, 384, 480, 384, 384, 576}},
    {148, true, {320, 160, 640, 160, 320, 128, 640, 128, 256, 192, 768, 160, 256, 192, 768, 160}},
    {33, false, {288, 288, 288, 288, 288, 288, 288, 288, 288, 288, 288, 3072}},
    {33, false, {192, 192, 192, 192, 192, 2688}},
    {148, false, {160, 160, 160, 160, 160, 128, 160, 640}},
    {148, false, {640, 640, 640, 640, 640, 512, 640, 512}}, {148, false, {480, 480, 480}},
};
int main()
{
    uint8_t order[32];
    for (const Point& p : points)
        if (longest_first_pays(p.cost.data(), static_cast<int>(p.cost.size()), 32, p.clusters, order) != p.first) {
            std::printf("%d samples on %d clusters\n", static_cast<int>(p.cost.size()), p.clusters);
            return 1;
        }
    std::mt19937 rng(5);
    for (int k = 0; k < 4000; ++k) {                     // the sum against jobs dealt out one by one; the order a falling one, and stable
        const int n = 1 + rng() % 32, heads = 1 + rng() % 64, clusters = 1 + rng() % 160;
        std::vector<int> cost(n);
        std::vector<int64_t> load(clusters, 0);
        for (int& c : cost) c = 1 + rng() % 5 * 100;
        for (int j = 0; j < n * heads; ++j) load[j % clusters] += cost[j / heads];
        const int64_t most = *std::max_element(load.begin(), load.end());
        if (fullest_cluster(cost.data(), n, heads, clusters) != most) { std::printf("%d x %d jobs on %d clusters\n", n, heads, clusters); return 1; }
        longest_first_pays(cost.data(), n, heads, clusters, order);
        std::vector<int> by(n);
        for (int b = 0; b < n; ++b) by[b] = b;
        std::stable_sort(by.begin(), by.end(), [&](int x, int y) { return cost[x] > cost[y]; });
        if (!std::equal(by.begin(), by.end(), order)) { std::printf("order\n"); return 1; }
    }
    std::printf("ok\n");
    return 0;
}
"""


def test_samples_with_long_jobs_come_first_only_where_the_fullest_cluster_gets_less(tmp_path):
    run_program(tmp_path, ORDER)


BESIDE = r"""
#include <cstdio>
#include "rules.h"
using namespace mvla;
// (bytes of an element of k, heads, head dim, key heads, bytes of a hidden row, samples, tokens of a sample, clusters at once; norms: adaptive budgets)
struct Point { int esize, heads, dim, kv, row, batch, tokens, at_once; bool norms, beside; };
static const Point points[] = {
    {2, 32, 128, 32, 8192, 10, 768, 148, true, true}, {2, 32, 128, 32, 8192, 16, 768, 148, true, true}, {2, 32, 128, 32, 8192, 32, 768, 148, true, true},
    {2, 32, 128, 32, 8192, 9, 768, 148, true, false},          // 288 jobs: two rounds
    {2, 32, 128, 32, 8192, 16, 640, 148, true, true}, {2, 32, 128, 32, 8192, 16, 639, 148, true, false},       // keys of a job on both sides of 160 KB
    {2, 32, 128, 32, 8192, 16, 228, 148, true, false}, {2, 32, 128, 32, 8192, 32, 228, 148, false, false},
    {2, 32, 128, 32, 8192, 5, 1280, 74, true, true}, {2, 32, 128, 32, 8192, 4, 1280, 74, true, false}, {2, 32, 128, 32, 8192, 3, 3000, 33, true, true},
    {2, 32, 128, 32, 8192, 2, 3000, 33, true, false}, {2, 32, 128, 32, 8192, 1, 4096, 8, true, false},
    {2, 16, 256, 16, 8192, 24, 768, 148, true, true}, {2, 32, 96, 32, 6144, 12, 900, 148, true, true},
    {1, 32, 128, 32, 8192, 12, 1300, 148, false, true}, {1, 32, 128, 32, 8192, 12, 1300, 148, true, false}, {1, 32, 128, 8, 8192, 16, 768, 148, false, false},
    {2, 32, 64, 32, 4096, 16, 768, 148, true, false}, {2, 32, 64, 32, 4096, 12, 1500, 148, false, true},
    {2, 16, 128, 16, 4096, 24, 768, 148, true, false}, {2, 16, 128, 16, 4096, 24, 768, 148, false, true},      // the norms would take longer than the scores
    {2, 32, 128, 8, 8192, 10, 768, 148, false, true}, {2, 32, 128, 8, 8192, 16, 768, 148, true, false},
    {2, 48, 128, 48, 8208, 7, 700, 148, true, true}, {2, 40, 128, 40, 10240, 8, 768, 148, true, false},        // rows of two pieces
};
int main()
{
    for (const Point& p : points) {
        const TailBesideSizes c = {static_cast<int64_t>(p.batch) * p.tokens, p.batch, p.batch * p.heads, p.at_once, p.dim * p.esize,
                                   static_cast<int64_t>(p.kv) * p.dim * p.esize, p.norms ? p.row : 0};
        if (tail_beside_pays(c) != p.beside) { std::printf("%d heads of %d, %d x %d, norms %d\n", p.heads, p.dim, p.batch, p.tokens, p.norms); return 1; }
    }
    std::printf("ok\n");
    return 0;
}
"""


def test_the_tail_runs_beside_the_scoring_kernel_only_where_jobs_are_long_and_many(tmp_path):
    run_program(tmp_path, BESIDE)
