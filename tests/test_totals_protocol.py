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
static const int NC = 3, W = NC + 2, SWEEPS = 6;  // columns, words of a row (two of the residual), sweeps
static int V, nb;
static uint64_t row[2][W];
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
    uint64_t was[2][W] = {};
    std::vector<int> order;  // in which it reads the words of a row
    bool done() const { return s == SWEEPS; }
    bool owns() const { return v0 < v1; }
    // one addition or one complete read; false when it has to wait
    bool step() {
        uint64_t* r = row[s & 1];
        const int adds = owns() ? (v1 - v0) * W : (bare ? W - NC : 0);
        if (add < adds) {
            if (owns()) r[add % W] += FX_ONE + value(s, v0 + add / W, add % W);
            else r[NC + add] += FX_ONE;
            ++add;
            return true;
        }
        const int w = order[wait];
        uint64_t& b = was[s & 1][w];
        if (!fx_complete(r[w], b, w < NC ? fx_due_col(V) : due_err())) return false;
        if (fx_value(r[w], b) != total(s, w)) {
            printf("wrong\n");
            exit(0);
        }
        b = r[w];
        if (++wait == W) {
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
        for (int w = 0; w < W; ++w) c[b].order.push_back(w);
        for (int w = W - 1; w > 0; --w) std::swap(c[b].order[w], c[b].order[rng() % (w + 1)]);
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


def _compiled(folder, name, code, *flags):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src, exe = folder / (name + ".cpp"), folder / name
    src.write_text(code)
    subprocess.run([cxx, "-O1", "-std=c++17", "-I", CSRC, *flags, str(src), "-o", str(exe)], check=True)
    return lambda *a: subprocess.run([str(exe), *map(str, a)], check=True, capture_output=True, text=True,
                                     timeout=120).stdout.strip()


@pytest.fixture(scope="module")
def model(tmp_path_factory):
    d = tmp_path_factory.mktemp("totals")
    return _compiled(d, "model", MODEL), _compiled(d, "without", MODEL, "-DNO_BARE_COUNT")


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


RESIDUAL = r"""
#include <cstdio>
#include <cstdlib>
#include "sk_totals.h"
using namespace ota;
// residual V nb e tol: V partitions of residual e (units) each; prints whether the words are
// complete before and after the last addition, the total, and whether the loop test passes
int main(int, char** argv) {
    const int V = atoi(argv[1]), nb = atoi(argv[2]);
    const uint64_t e = strtoull(argv[3], nullptr, 10), was = 0xfedcba9876543210ull;
    uint64_t lo = was, hi = was;
    int early = 0;
    const int n = fx_due_err(V, nb);
    for (int k = 0; k < n; ++k) {
        early |= fx_complete(lo, was, n) || fx_complete(hi, was, n);
        lo += FX_ONE + (k < V ? fx_err_low(e) : 0);
        hi += FX_ONE + (k < V ? fx_err_high(e) : 0);
    }
    const bool full = fx_complete(lo, was, n) && fx_complete(hi, was, n);
    const uint64_t t = fx_err(fx_value(lo, was), fx_value(hi, was));
    printf("%d %d %llu %d", early, (int)full, (unsigned long long)t, (int)(t <= fx_stop_units(atof(argv[4]) * 0x1p50)));
}
"""

UNIT = 1 << 50   # residual 1
BROKEN = 1 << 52  # what a row that is not a number, infinite or 4 or more counts as


@pytest.mark.parametrize("V,nb,e,tol,passes", [
    (152, 152, 0, 0.0, True), (1, 1, 1, 0.0, False), (152, 152, 7, 1e-6, True), (152, 38, UNIT // 4, 0.3, False),
    (1, 152, 2 * UNIT, 2.5, True), (1, 152, 2 * UNIT, 1.9, False), (1, 1, 2 * UNIT, float("inf"), True),
    (1, 1, BROKEN, 0.3, False), (1, 1, BROKEN, 1e30, False), (152, 152, BROKEN, float("inf"), False),
    (16, 16, BROKEN - 1, 10.0, False), (152, 152, BROKEN - 1, float("inf"), False), (152, 152, 16 * BROKEN, 100.0, False)])
def test_residual_words(tmp_path, V, nb, e, tol, passes):
    """The residual words hold any residuals exactly and never count an addition too many, and a
    total that no plan of unit mass can have does not pass the loop test, whatever the tolerance."""
    early, full, total, stop = map(int, _compiled(tmp_path, "residual", RESIDUAL)(V, nb, e, tol).split())
    assert not early and full and total == V * e
    assert bool(stop) == passes
