"""The ends of the tensor-core products on the CPU (csrc/gemm_ring.h): a model of the CTA pair's and the
single CTA's barriers - copies and commits that land later in any order, agents scheduled at random,
waits that give up at random - shows that after the final waits nothing can land in a CTA that has left,
that each of those waits ends, and that without them something is left over."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1911_10274_gb300", "csrc")

MODEL = r"""
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <functional>
#include <random>
#include <vector>
#include "gemm_ring.h"
using namespace titan;

struct Bar {                                  // an mbarrier
    int init = 1, pending = 1;
    long tx = 0;
    unsigned phase = 0;
    void set(int c) { init = pending = c; tx = 0; phase = 0; }
    void settle() { if (!pending && !tx) { ++phase; pending = init; } }
    void arrive() { --pending; settle(); }
    void expect(long b) { tx += b; --pending; settle(); }
    void complete(long b) { tx -= b; settle(); }
    bool done(unsigned parity) const { return (phase & 1) != parity; }
};

constexpr int S = 6, EACH = 4;                // ring stages, bytes of a CTA's copies

struct Event { int cta; std::function<void()> land; };   // under way, lands in shared memory of CTA `cta`

// One pair (ctas = 2) or one CTA; `tiles` of `num_kb` k-blocks, accumulators in a ring of two; `give_up`: chance
// that a wait that is not over expires.  Returns what is still under way when the CTAs leave, or -1: a final
// wait could not end.
int run(int ctas, int tiles, int num_kb, double give_up, bool drain, unsigned seed) {
    std::mt19937 rng(seed);
    auto chance = [&](double p) { return std::uniform_real_distribution<>(0, 1)(rng) < p; };
    Bar full[S], empty[2][S], acc_full[2][2], acc_empty[2], over[2];
    for (auto &b : full) b.set(1);
    for (auto &c : empty) for (auto &b : c) b.set(1);
    for (auto &c : acc_full) for (auto &b : c) b.set(1);
    for (auto &b : acc_empty) b.set(ctas);    // one epilogue warp a CTA stands for its four
    for (auto &b : over) b.set(1);
    std::vector<Event> copies, commits;       // commits land in any order once their products are done
    auto commit = [&](std::function<void(int)> on) {
        for (int c = 0; c < ctas; ++c) commits.push_back({c, [=] { on(c); }});
    };
    const int total = tiles * num_kb;
    int issued[2] = {0, 0}, mma = 0, acc = 0, epi[2] = {0, 0};
    bool failed[2] = {false, false}, prod_end[2] = {false, ctas == 1}, issuer_end = false, epi_end[2] = {false, ctas == 1};
    bool in_tile = false;
    auto land = [&](std::vector<Event> &q) {
        const size_t k = rng() % q.size();
        Event e = q[k];
        q.erase(q.begin() + k);
        e.land();
    };
    for (long guard = 0; guard < 4000000; ++guard) {
        if (prod_end[0] && prod_end[1] && issuer_end && epi_end[0] && epi_end[1]) break;
        const int who = rng() % 7;
        if (who < 2 && !prod_end[who]) {      // TMA producer
            const int j = issued[who];
            if (j == total) { prod_end[who] = true; continue; }
            if (j >= S && !empty[who][ring_slot(j, S)].done(ring_parity(j - S, S))) {
                if (chance(give_up)) { failed[who] = true; prod_end[who] = true; }
                continue;
            }
            Bar *b = &full[ring_slot(j, S)];
            if (who == 0) b->expect(ctas * EACH);
            copies.push_back({who, [b] { b->complete(EACH); }});
            ++issued[who];
        } else if (who == 2 && !issuer_end) { // MMA issuer
            auto end = [&](bool ok) {
                commit([&](int c) { over[c].arrive(); });
                issuer_end = true;
                if (!ok) failed[0] = true;
            };
            if (!in_tile) {
                if (acc == tiles) { end(true); continue; }
                if (acc >= 2 && !acc_empty[acc & 1].done(((acc >> 1) & 1) ^ 1)) {
                    if (chance(give_up)) end(false);
                    continue;
                }
                in_tile = true;
            }
            if (!full[ring_slot(mma, S)].done(ring_parity(mma, S))) {
                if (chance(give_up)) {
                    const int b = acc & 1;
                    commit([&, b](int c) { acc_full[c][b].arrive(); });
                    ++acc;
                    end(false);
                }
                continue;
            }
            const int s = ring_slot(mma, S), b = acc & 1;
            commit([&, s](int c) { empty[c][s].arrive(); });
            if (++mma % num_kb == 0) {
                commit([&, b](int c) { acc_full[c][b].arrive(); });
                ++acc;
                in_tile = false;
            }
        } else if (who >= 3 && who < 5 && !epi_end[who - 3]) {
            const int c = who - 3, i = epi[c];
            if (i == tiles) { epi_end[c] = true; continue; }
            if (!acc_full[c][i & 1].done((i >> 1) & 1)) {
                if (chance(give_up)) { failed[c] = true; epi_end[c] = true; }
                continue;
            }
            acc_empty[i & 1].arrive();
            ++epi[c];
        } else if (who == 5 && !copies.empty()) {
            land(copies);
        } else if (who == 6 && !commits.empty()) {
            land(commits);
        }
    }
    if (!issuer_end) return -2;
    const bool bad = failed[0] || failed[1];
    // a final wait: what is under way lands until it is over
    auto wait = [&](const Bar &b, unsigned parity) {
        while (!b.done(parity)) {
            if (copies.empty() && commits.empty()) return false;
            if (!commits.empty() && (copies.empty() || chance(0.5))) land(commits);
            else land(copies);
        }
        return true;
    };
    if (drain) {
        for (int c = 0; c < ctas; ++c) {
            if (!wait(over[c], 0)) return -1;
            for (int j = ring_tail(mma, S); j < mma; ++j)
                if (!wait(empty[c][ring_slot(j, S)], ring_parity(j, S))) return -1;
            if (bad)
                for (int j = ring_tail(acc, 2); j < acc; ++j)
                    if (!wait(acc_full[c][ring_slot(j, 2)], ring_parity(j, 2))) return -1;
        }
        if (bad)
            for (int j = mma; j < std::max(issued[0], issued[1]); ++j) {
                Bar &b = full[ring_slot(j, S)];
                if (ctas == 2) {
                    const PairSettle f = pair_settle(j, issued[0], issued[1], EACH);
                    if (f.expect) b.expect(f.expect);
                    if (f.cancel) b.complete(f.cancel);
                }
                if (!wait(b, ring_parity(j, S))) return -1;
            }
    }
    return (int)(copies.size() + commits.size());
}

int main() {
    int left_without = 0, failures = 0;
    for (unsigned seed = 0; seed < 4000; ++seed) {
        const int ctas = 1 + seed % 2, tiles = 1 + seed / 2 % 5, num_kb = 1 + seed / 7 % 17;
        const double give_up = seed % 3 ? 0.02 * (seed % 5) : 0.0;
        const int r = run(ctas, tiles, num_kb, give_up, true, seed);
        if (r) {
            printf("ctas %d tiles %d k-blocks %d give_up %g seed %u: %d\n", ctas, tiles, num_kb, give_up, seed, r);
            ++failures;
        }
        left_without += run(ctas, tiles, num_kb, 0.0, false, seed) > 0;
    }
    printf("left over without the final waits: %d\n", left_without);
    return failures || !left_without;
}
"""


def test_nothing_lands_after_a_cta_has_left(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("no host C++ compiler")
    (tmp_path / "model.cpp").write_text(MODEL)
    exe = str(tmp_path / "model")
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", CSRC, str(tmp_path / "model.cpp"), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout
