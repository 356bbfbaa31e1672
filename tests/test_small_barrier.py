"""The grid barrier of the one-launch path, stepped through in every order on the CPU.

A program built from csrc/small_barrier.h lets four CTAs (one of which clears the slots) take their steps - clear, arrive,
read the word - in every possible order over several rounds, and checks that every CTA leaves a round only when all have
arrived and with exactly that round's number of active vertices.  A word that all rounds share, which counts on, fails
the same check: a CTA may read it after a faster one has arrived at the next round."""
import os
import shutil
import subprocess

import numpy as np
import pytest

import graphgen as gg
import oracle as O

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1806_08092_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cstring>
#include <set>
#include <vector>
#include "small_barrier.h"
using namespace gpop;
constexpr uint32_t N = 4, ROUNDS = 7;
// vertices a CTA leaves active for a round: frontiers of one vertex, of one CTA, of all
uint32_t active(uint32_t cta, uint32_t round) {
    static const uint32_t a[ROUNDS][N] = {{1, 0, 0, 0}, {0, 5, 0, 0}, {0, 0, 1, 0}, {1u << 18, 2, 0, 7}, {0, 0, 0, 1},
                                          {1, 0, 0, 0}, {0, 0, 0, 0}};
    return a[round][cta];
}
uint32_t frontier(uint32_t round) { uint32_t s = 0; for (uint32_t c = 0; c < N; ++c) s += active(c, round); return s; }
struct State {
    unsigned long long word[kSmallSlots];
    uint32_t round[N], phase[N], seen[N];  // phase 0: arrives next (CTA 0: clears first), 1: arrives, 2: reads the word
};
bool less_(const State &a, const State &b) { return std::memcmp(&a, &b, sizeof a) < 0; }
struct Slots {  // the header's protocol
    static constexpr bool clears = true;
    static uint32_t slot(uint32_t r) { return small_slot_of(r); }
    static bool all(unsigned long long w, uint32_t) { return small_all_arrived(w, N); }
    static uint32_t got(unsigned long long w, uint32_t) { return small_active(w); }
};
struct OneWord {  // one running word for all rounds
    static constexpr bool clears = false;
    static uint32_t slot(uint32_t) { return 0; }
    static bool all(unsigned long long w, uint32_t r) { return (uint32_t)w >= (r + 1) * N; }
    static uint32_t got(unsigned long long w, uint32_t seen) { return small_active(w) - seen; }
};
template <class P> int check(size_t &states) {
    auto cmp = [](const State &a, const State &b) { return less_(a, b); };
    std::set<State, decltype(cmp)> done(cmp);
    std::vector<State> todo(1);
    std::memset(&todo[0], 0, sizeof(State));
    done.insert(todo[0]);
    bool ends = false;
    while (!todo.empty()) {
        const State s = todo.back();
        todo.pop_back();
        uint32_t stuck = 0, finished = 0;
        for (uint32_t c = 0; c < N; ++c) {
            State t = s;
            const uint32_t r = s.round[c];
            if (r == ROUNDS) { ++finished; continue; }
            if (s.phase[c] == 0) {
                if (P::clears && c == 0 && r > 0) t.word[small_slot_to_clear(r)] = 0;
                t.phase[c] = 1;
            } else {
                if (s.phase[c] == 1) t.word[P::slot(r)] += small_arrival(active(c, r));
                const unsigned long long w = t.word[P::slot(r)];
                if (P::all(w, r)) {
                    for (uint32_t o = 0; o < N; ++o)  // nobody is still before this round's arrival
                        if (o != c && (s.round[o] < r || (s.round[o] == r && s.phase[o] < 2))) return 1;
                    if (P::got(w, s.seen[c]) != frontier(r)) return 2;
                    t.seen[c] = small_active(w);
                    t.round[c] = r + 1;
                    t.phase[c] = 0;
                } else {
                    t.phase[c] = 2;
                    if (s.phase[c] == 2) { ++stuck; continue; }
                }
            }
            if (done.insert(t).second) todo.push_back(t);
        }
        if (finished == N) ends = true;
        else if (stuck + finished == N) return 3;  // all wait for ever
    }
    states = done.size();
    return ends ? 0 : 4;
}
int main() {
    size_t n = 0, m = 0;
    const int a = check<Slots>(n), b = check<OneWord>(m);
    std::printf("%d %zu %d\n", a, n, b);
    return 0;
}
"""


def test_every_order_of_steps(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    src = tmp_path / "barrier.cpp"
    src.write_text(PROGRAM)
    exe = tmp_path / "barrier"
    subprocess.run([cxx, "-std=c++17", "-O1", "-Wall", "-Werror", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    result, states, one_word = map(int, subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split())
    assert result == 0 and states > 500  # 1: left too early, 2: another frontier, 3: all wait, 4: never ends
    assert one_word == 2


@pytest.mark.gpu
@pytest.mark.parametrize("n", [2, 300, 20001])
def test_rounds_of_one_vertex(n):
    # a path: every round's frontier is one vertex, the last one's is empty
    torch = pytest.importorskip("torch")
    import paper_1806_08092_gb300 as gp
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    gp.build()
    g = gg.path(n)
    G = gp.Graph.from_csr(g.row_ptr, g.col, partition_size=32)
    level, parent = O.bfs(g, 0)
    for _ in range(20 if n <= 300 else 2):
        r = G.run("bfs", source=0, max_iters=2 * n)
        assert r.stats["iterations"] == n and r.stats["converged"] == 1 and r.stats["vertices_scattered"] == n
        assert np.array_equal(r.values.cpu().numpy(), level) and np.array_equal(r.parent.cpu().numpy(), parent)
    G.close()
