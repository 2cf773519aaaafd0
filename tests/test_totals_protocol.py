"""The counted totals of the persistent solver (csrc/sk_totals.h), stepped on the host.

A model of a group of CTAs takes one addition or one read of a word at a time, in orders that no
GPU run can be made to take: a CTA that moves only when all others are stuck, the CTAs without
a partition last, random ones.  Every CTA has to get the exact totals of every sweep, and none may
be left waiting.  The counting rules are the header's, which the kernel uses.
"""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1805_01559_gb300", "csrc")

MODEL = r"""
#include <cstdio>
#include <cstdlib>
#include <random>
#include <vector>
#include "sk_totals.h"
using namespace ota;
static const int W = 3, SWEEPS = 6;  // column words of a row, sweeps of a solve
static int V, nb;
static uint64_t row[2][W + 1];
static uint64_t value(int s, int v, int w) {  // of partition v in sweep s: up to the largest a word takes
    uint64_t h = (uint64_t)(s * 1000003 + v * 7919 + w * 104729 + 1) * 0x9e3779b97f4a7c15ull;
    return h % ((1ull << FX_TOP) + 1);
}
static uint64_t total(int s, int w) {
    uint64_t t = 0;
    for (int v = 0; v < V; ++v) t += value(s, v, w);
    return t;
}
#ifdef NO_BARE_COUNT
static const bool bare = false;
static int due_err() { return V; }
#else
static const bool bare = true;
static int due_err() { return fx_due_err(V, nb); }
#endif
struct Cta {
    int v0, v1, s = 0, add = 0, wait = 0;
    uint64_t was[2][W + 1] = {};
    std::vector<int> order;  // in which it reads the words of a row
    bool done() const { return s == SWEEPS; }
    bool owns() const { return v0 < v1; }
    // one addition or one complete read; false when it has to wait
    bool step() {
        uint64_t* r = row[s & 1];
        const int adds = owns() ? (v1 - v0) * (W + 1) : (bare ? 1 : 0);
        if (add < adds) {
            if (owns()) r[add % (W + 1)] += FX_ONE + value(s, v0 + add / (W + 1), add % (W + 1));
            else r[W] += FX_ONE;
            ++add;
            return true;
        }
        const int w = order[wait];
        uint64_t& b = was[s & 1][w];
        if (!fx_complete(r[w], b, w < W ? fx_due_col(V) : due_err())) return false;
        if (fx_value(r[w], b) != total(s, w)) {
            printf("wrong\n");
            exit(0);
        }
        b = r[w];
        if (++wait == W + 1) {
            ++s;
            add = wait = 0;
        }
        return true;
    }
};
int main(int argc, char** argv) {
    V = atoi(argv[1]);
    nb = atoi(argv[2]);
    const int mode = atoi(argv[3]), seed = atoi(argv[4]);  // 0: CTAs without a partition last, 1: CTA `seed` last, 2: random
    std::mt19937 rng(seed);
    std::vector<Cta> c(nb);
    for (int b = 0; b < nb; ++b) {
        cta_parts(V, b, nb, &c[b].v0, &c[b].v1);
        for (int w = 0; w <= W; ++w) c[b].order.push_back(w);
        for (int w = W; w > 0; --w) std::swap(c[b].order[w], c[b].order[rng() % (w + 1)]);
    }
    for (;;) {
        bool moved = false, all = true;
        auto run = [&](Cta& x) {
            if (x.done()) return;
            all = false;
            if (x.step()) moved = true;
        };
        if (mode == 2) {
            for (int k = 0; k < 4 * nb; ++k) run(c[rng() % nb]);
            for (auto& x : c) run(x);
        } else {
            for (int b = 0; b < nb; ++b)
                if (mode == 0 ? c[b].owns() : b != seed % nb) run(c[b]);
            if (!moved)
                for (int b = 0; b < nb; ++b)
                    if (mode == 0 ? !c[b].owns() : b == seed % nb) run(c[b]);
            if (!moved) {
                all = true;
                for (auto& x : c) all = all && x.done();
            }
        }
        if (all) {
            printf("ok\n");
            return 0;
        }
        if (!moved) {
            printf("stuck\n");
            return 0;
        }
    }
}
"""


@pytest.fixture(scope="module")
def model(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("totals")
    src = d / "model.cpp"
    src.write_text(MODEL)

    def compiled(name, *flags):
        exe = d / name
        subprocess.run([cxx, "-O1", "-std=c++17", "-I", CSRC, *flags, str(src), "-o", str(exe)], check=True)
        return lambda *a: subprocess.run([str(exe), *map(str, a)], check=True, capture_output=True, text=True,
                                         timeout=120).stdout.strip()
    return compiled("model"), compiled("without", "-DNO_BARE_COUNT")


# fewer partitions than CTAs, as many, more; 128 partitions, at which the 8-bit count of three
# sweeps equals that of one; the largest group with one partition and with one short of it
GROUPS = [(1, 1), (1, 2), (3, 8), (3, 152), (8, 8), (20, 8), (128, 152), (151, 152), (1, 152), (152, 38), (152, 152)]


@pytest.mark.parametrize("V,nb", GROUPS)
def test_every_cta_gets_every_total(model, V, nb):
    run, _ = model
    for mode, seeds in ((0, range(2)), (1, (0, nb // 2, nb - 1)), (2, range(6))):
        for seed in seeds:
            assert run(V, nb, mode, seed) == "ok", (mode, seed)


@pytest.mark.parametrize("V,nb,fails", [(3, 8, "stuck"), (3, 152, "stuck"), (128, 152, "wrong")])
def test_model_sees_a_missing_count(model, V, nb, fails):
    """Without the bare count of CTAs that own no partition the same orders break the protocol."""
    _, run = model
    assert run(V, nb, 0, 0) == fails
