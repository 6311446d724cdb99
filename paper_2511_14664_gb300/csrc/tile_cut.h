// tile_cut.h -- which gates of a list share a tile of the state (host only; k_tilegates.cu and k_small_tiles.cu run them).
#pragma once
#include <stdint.h>

#include <algorithm>
#include <functional>
#include <vector>

#include "../../include/qsim.h"

namespace qsim {

struct TileGate {
    bool ok = false;             // tile_gate_ok: may join a group
    bool diag = false;
    int k = 0, nc = 0;
    int q[2] = {0, 0};           // targets; for a diagonal (k = 1 or 2, nc = 0) all its qubits
    int ctl[QSIM_MAX_CONTROLS] = {0};
    uint64_t tmask = 0, all = 0; // targets; targets and controls
    std::vector<double> mat;     // 2^k x 2^k, or the diagonal's 2^k entries (interleaved)
};

// Gates of `und` ready in order: each takes its place unless one left behind shares a qubit (diagonals pass diagonals),
// and its targets, all in `within`, grow `set` up to `limit` bits (diagonals have no targets here: they go anywhere). `every`:
// the qubits of all gates; once dense gates left behind block them all, none of the rest can join.
inline std::vector<int> tile_collect(const std::vector<TileGate>& g, const std::vector<int>& und, int seed, uint64_t& set, int limit,
                                     uint64_t within, uint64_t every) {
    std::vector<int> out;
    uint64_t bany = 0, bdiag = 0;
    if (seed >= 0) set |= g[seed].tmask;
    for (int i : und) {
        const bool blocked = g[i].diag ? (g[i].all & bany) != 0 : (g[i].all & (bany | bdiag)) != 0;
        const uint64_t want = g[i].diag ? 0 : g[i].tmask;
        if (g[i].ok && !blocked && (want & ~within) == 0 && __builtin_popcountll(set | want) <= limit) {
            set |= want;
            out.push_back(i);
        } else {
            (g[i].diag ? bdiag : bany) |= g[i].all;
            if (bany == every) break;
        }
    }
    return out;
}

// Gates cut into groups of which each acts on `bits` qubits at most (diagonals and controls on any), in an order that keeps
// that of gates that share a qubit (diagonals among themselves excepted). The qubits in lowset count in every group;
// `size` adds up to max_size at most, gates to max_ops. A gate that is not ok is a group of its own. A group is looked for
// among the first kTileAhead gates that have no place yet, so that the time is linear in the number of gates (50 000 random
// ones: 0.01 s at 14 and at 20 qubits; over all of the rest 1.0 and 1.25 s).
constexpr int kTileAhead = 1024;
struct TileCut { std::vector<int> members; uint64_t set = 0; };
inline std::vector<TileCut> tile_cut(const std::vector<TileGate>& g, int bits, uint64_t lowset,
                                     const std::function<int(const TileGate&)>& size, int max_size, int max_ops) {
    std::vector<TileCut> out;
    uint64_t every = 0;
    for (const TileGate& c : g) every |= c.all;
    std::vector<int> und, rest;  // the window: gates without a place, in order
    size_t next = 0;             // the first gate behind it
    for (;;) {
        while (next < g.size() && und.size() < (size_t)kTileAhead) und.push_back((int)next++);
        if (und.empty()) break;
        TileCut cut;
        if (!g[und[0]].ok) {  // no group takes it: alone
            cut.members = {und[0]};
        } else {
            uint64_t seen = 0;
            int tried = 0;
            for (size_t u = 0; u < und.size() && tried < 12 && seen != every; ++u) {
                const TileGate& c = g[und[u]];
                const bool free_ = (c.all & seen) == 0;
                seen |= c.all;
                if (!c.ok || !free_ || (u > 0 && c.diag)) continue;
                ++tried;
                uint64_t set = lowset;
                std::vector<int> got = tile_collect(g, und, c.diag ? -1 : und[u], set, bits, ~0ull, every);
                if (got.size() > cut.members.size()) { cut.members.swap(got); cut.set = set; }
            }
            // a program larger than the room set aside for it is cut short
            int used = 0;
            for (size_t m = 0; m < cut.members.size(); ++m) {
                used += size(g[cut.members[m]]);
                if ((used > max_size || m >= (size_t)max_ops) && m > 0) { cut.members.resize(m); break; }
            }
        }
        rest.clear();
        size_t m = 0;
        for (int i : und) {
            if (m < cut.members.size() && cut.members[m] == i) ++m;
            else rest.push_back(i);
        }
        und.swap(rest);
        out.push_back(std::move(cut));
    }
    return out;
}

}  // namespace qsim
