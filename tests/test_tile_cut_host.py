"""Cutting a gate list into groups that share a tile (host C++, compiled here by itself): the order of gates that share a
qubit is kept, a group's targets fit the tile, and the time is linear in the number of gates."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

DRIVER = r"""
#include <chrono>
#include <cstdio>
#include <cstdlib>
#include <random>
#include "tile_cut.h"
using namespace qsim;
// n, tile bits, low bits, gates, per mille of diagonal / controlled / not ok gates, number of qubits in use
int main(int, char** v) {
    const int n = atoi(v[1]), bits = atoi(v[2]), low = atoi(v[3]), G = atoi(v[4]), pd = atoi(v[5]), pc = atoi(v[6]), px = atoi(v[7]);
    const int used = atoi(v[8]);
    std::mt19937 r(7);
    std::vector<TileGate> g(G);
    for (TileGate& c : g) {
        int q[4];
        for (int j = 0; j < 4; ++j) {
            bool again = true;
            while (again) {
                q[j] = (int)(r() % used);
                again = false;
                for (int i = 0; i < j; ++i) again = again || q[i] == q[j];
            }
        }
        c.ok = (int)(r() % 1000) >= px;
        c.diag = (int)(r() % 1000) < pd;
        c.k = 1 + (int)(r() & 1);
        c.nc = !c.diag && (int)(r() % 1000) < pc ? 2 : 0;
        for (int j = 0; j < c.k; ++j) { c.q[j] = q[j]; c.tmask |= 1ull << q[j]; }
        c.all = c.tmask;
        for (int j = 0; j < c.nc; ++j) { c.ctl[j] = q[2 + j]; c.all |= 1ull << q[2 + j]; }
    }
    const auto t0 = std::chrono::steady_clock::now();
    const auto cuts = tile_cut(g, bits, (1ull << low) - 1, [](const TileGate& c) { return c.k == 2 ? 26 : 14; }, 1535, 256);
    const double s = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
    // per qubit: the last dense gate placed, and the last gate of either kind
    std::vector<int> seen(G, 0), dense(64, -1), any(64, -1);
    for (const TileCut& c : cuts) {
        if (c.members.empty() || __builtin_popcountll(c.set) > bits) return 1;
        for (int i : c.members) {
            if (seen[i]++) return 2;
            if (!g[i].ok && c.members.size() != 1) return 3;
            if (g[i].ok && !g[i].diag && (g[i].tmask & ~c.set)) return 4;
            for (int q = 0; q < n; ++q) {
                if (!((g[i].all >> q) & 1)) continue;
                if (i < dense[q] || (!g[i].diag && i < any[q])) return 5;
                if (!g[i].diag && i > dense[q]) dense[q] = i;
                if (i > any[q]) any[q] = i;
            }
        }
    }
    for (int x : seen) if (x != 1) return 6;
    printf("%zu %.6f\n", cuts.size(), s);
    return 0;
}
"""


@pytest.fixture(scope="module")
def cut(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("tile_cut")
    (d / "driver.cpp").write_text(DRIVER)
    exe = str(d / "driver")
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", os.path.join(ROOT, "paper_2511_14664_gb300", "csrc"), str(d / "driver.cpp"),
                    "-o", exe], check=True)

    def run(*args):
        out = subprocess.run([exe, *map(str, args)], capture_output=True, text=True)
        assert out.returncode == 0, out.returncode
        groups, seconds = out.stdout.split()
        return int(groups), float(seconds)
    return run


@pytest.mark.parametrize("diag", [0, 300, 1000])
@pytest.mark.parametrize("ctl,wide", [(0, 0), (300, 0), (200, 50), (0, 1000)])
@pytest.mark.parametrize("n,bits,low,used", [(14, 9, 0, 14), (17, 11, 2, 17), (25, 12, 3, 25), (20, 12, 3, 6)])
def test_order_and_targets(cut, n, bits, low, used, diag, ctl, wide):
    for gates in (1, 5, 300, 5000):
        cut(n, bits, low, gates, diag, ctl, wide, used)


@pytest.mark.parametrize("n,bits,low,used", [(14, 9, 0, 14), (20, 12, 3, 20), (33, 12, 3, 33), (25, 12, 3, 8)])
@pytest.mark.parametrize("diag,wide", [(0, 0), (500, 0), (0, 900)])
def test_time_is_linear(cut, n, bits, low, used, diag, wide):
    """200 000 gates take at most 2 s (17 to 32 s when every group looked at all of the rest), and about ten times as
    long as 20 000."""
    _, t1 = cut(n, bits, low, 20000, diag, 0, wide, used)
    _, t2 = cut(n, bits, low, 200000, diag, 0, wide, used)
    assert t2 < 2.0
    assert t2 < 30 * t1 + 0.1
