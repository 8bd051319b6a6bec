"""Pieces of work handed to the warps of CTAs that join while it runs (csrc/lots.h): every piece goes to one caller, and every
caller gets away, whatever the order in which the callers' steps come.  Checked by a small C++ program built from the header
itself, whose callers are coroutines that change places at every access to a shared word (no GPU needed)."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <random>
#include <vector>
#include <ucontext.h>
#include "lots.h"
static ucontext_t home;
struct Fiber { ucontext_t at; std::vector<char> stack; bool over; };
static std::vector<Fiber> fibers;
static int now;
static void turn() { swapcontext(&fibers[now].at, &home); }
static int32_t counter;
struct Cta { uint32_t word; int32_t ahead; };
struct Cell {
    Cta* c;
    uint32_t add() { turn(); return c->word++; }
    void swap(uint32_t x) { turn(); c->word = x; }
    uint32_t peek() { turn(); return c->word; }
    int32_t next() { turn(); return c->ahead; }
    void put(int32_t x) { turn(); c->ahead = x; }
    int32_t ask() { turn(); return counter++; }
};
static std::vector<Cta> ctas;
static std::vector<int> given;
static int warps, pieces, lots, stuck;
static void body(int f)
{
    Cell cell = {&ctas[f / warps]};
    for (;;) {
        bool gave_up = false;
        const uint32_t p = mvla::take_piece(cell, pieces, lots, 3000, &gave_up);
        stuck += gave_up;
        if (p >= given.size()) break;
        ++given[p];
        for (int k = 0; k < 4; ++k) turn();          // the piece's work
    }
    fibers[f].over = true;
}
int main(int argc, char** argv)
{
    const int n_ctas = std::atoi(argv[1]), seeds = std::atoi(argv[5]);
    warps = std::atoi(argv[2]); pieces = std::atoi(argv[3]); lots = std::atoi(argv[4]);
    for (int seed = 0; seed < seeds; ++seed) {
        std::mt19937 rng(seed);
        counter = 0;
        stuck = 0;
        given.assign(lots * pieces, 0);
        ctas.assign(n_ctas, Cta{0, 0});
        for (Cta& c : ctas) { c.word = static_cast<uint32_t>(counter++) << 12; c.ahead = counter++; }
        fibers.assign(n_ctas * warps, Fiber());
        for (int f = 0; f < n_ctas * warps; ++f) {
            Fiber& b = fibers[f];
            b.stack.resize(32768);
            b.over = false;
            getcontext(&b.at);
            b.at.uc_stack.ss_sp = b.stack.data();
            b.at.uc_stack.ss_size = b.stack.size();
            b.at.uc_link = &home;
            makecontext(&b.at, reinterpret_cast<void (*)()>(body), 1, f);
        }
        for (int left = n_ctas * warps; left > 0;) {
            do now = rng() % fibers.size(); while (fibers[now].over);
            // some callers get many turns in a row, others wait for theirs
            for (int k = 1 << rng() % 6; k > 0 && !fibers[now].over; --k) swapcontext(&home, &fibers[now].at);
            left -= fibers[now].over;
        }
        int wrong = 0;
        for (int g : given) wrong += g != 1;
        if (stuck || wrong) { std::printf("order %d: %d callers gave up, %d pieces not given once\n", seed, stuck, wrong); return 1; }
    }
    std::printf("ok\n");
    return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("lots")
    (d / "lots.cpp").write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_2604_09244_b200", "csrc"), "-o", str(d / "lots"), str(d / "lots.cpp")],
                   check=True)
    return str(d / "lots")


@pytest.mark.parametrize("ctas,warps,pieces,lots", [
    (1, 3, 1, 2), (1, 4, 2, 1), (1, 5, 2, 3), (2, 4, 2, 5),       # more callers than pieces in a lot
    (1, 32, 16, 3), (2, 16, 8, 7),                                 # ... by half, as CTAs of 32 warps have
    (3, 16, 16, 8), (2, 3, 8, 4),                                  # as many, and fewer
    (4, 2, 2, 1), (3, 4, 4, 0)])                                   # fewer lots than CTAs, and none
def test_every_piece_is_given_once_and_every_caller_gets_away(program, ctas, warps, pieces, lots):
    r = subprocess.run([program, str(ctas), str(warps), str(pieces), str(lots), "600" if ctas * warps <= 8 else "300"], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout
