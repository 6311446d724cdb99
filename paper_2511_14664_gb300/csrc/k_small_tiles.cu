// k_small_tiles.cu -- a whole plan of a small state in one launch, many gates between two grid barriers (paper Sec. 2.1
// "State-Vector Simulation").
//
// k_small.cu runs such a plan one pass at a time with a grid barrier after each: about 2.5 us of barrier and L2 round
// trips a pass (22 passes for the 14-qubit brickwork of 410 gates fused at 5 qubits, 410 passes gate by gate), and its
// 5-qubit blocks are 128 FMAs an amplitude, which FP64 (1.67 FMAs a cycle and SM) makes 5 us. Here a CTA owns a tile of
// 2^T amplitudes (T = 7 for 14 complex128 qubits: 128 tiles) and applies every gate of a group whose targets lie in the
// tile's T bits; controls and diagonals may lie anywhere. The state goes through L2 once a group (10 groups for that
// brickwork). Each thread keeps its amplitudes in registers; a gate publishes them in shared memory, waits once, and
// computes its rows from its partners' amplitudes (two buffers in turn, so one CTA barrier a gate); diagonals touch no
// shared memory.
//
// Fused plans combine gates into products on at most two qubits first, where that is less arithmetic: 16 FMAs an
// amplitude for a product of four Haar gates and a CZ. (Wider products cost more: 32 FMAs at 3 qubits for about 7 gates,
// 128 at 5 for 19.) Per-gate plans apply the gates as they are.
// A complex64 state may be computed in FP64 between the grid barriers (its amplitudes are rounded once a group then);
// plan.cu has the rule.
// Bound: FP64 in complex128, the CTA barrier of each gate in complex64.
// Measured, against k_small.cu (us): complex128 14-qubit brickwork of 410 gates
// 97 against 163 fused and 174 against 1052 gate by gate; complex64 10 to 16 qubits 37..64 against 50..117 and 68..113
// against 642..1233; 12-qubit TFIM gate by gate 35 against 354; the 14-qubit QFT gate by gate 31 against 256. One-shot
// runs, 6 to 16 qubits, 1.3 to 4 times as fast (they compose no blocks).
// The grid barrier is bounded (2 s); on expiry the kernel records DEVERR_TIMEOUT and returns.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "common.cuh"
#include "internal.h"

namespace qsim {
namespace stile {

// complex128: a warp for each of the SM's four FP64 units, 1 to 4 amplitudes a thread; complex64: one amplitude a thread
// (with four, a gate took 0.4 us at 14 qubits, twice as long)
template <typename R> constexpr int kThrBits = sizeof(R) == 4 ? 9 : 7;
template <typename R> constexpr int kThreads = 1 << kThrBits<R>;
constexpr int kMaxBits = 9;
constexpr int kMaxProg = 40960;              // bytes of a group's program (two buffers in shared memory)
constexpr size_t kHeader = 256;              // the barrier word, padded

enum Code { kDense1 = 0, kReal1, kRx1, kDense2, kSwap2, kDiag };

struct Op {
    uint32_t code, coef;      // coefficients start at this complex value of the group's
    uint32_t t0, t1;          // tile bits of the targets (masks)
    uint32_t tctl, gctl;      // tile bits and index bits outside the tile that must be set
    uint32_t am, bm, ag, bg;  // diagonal: the qubits a and b of the table's index, as tile bits or index bits outside
    uint32_t flags;           // diagonal: bits 0..3 entry m differs from 1, bit 4 those are all -1
    uint32_t pad;
};
struct alignas(16) Group {
    int32_t ops, chunks, next_chunks, bits;  // 16-byte chunks of this group and of the next
    int32_t pos[12];                         // index bits of the tile, ascending
};
static_assert(sizeof(Op) == 48 && sizeof(Group) == 64, "");

__device__ __forceinline__ float fmar(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fmar(double a, double b, double c) { return __fma_rn(a, b, c); }

__device__ __forceinline__ uint64_t gtimer() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// The grid barrier of k_small.cu: the word counts arrivals, epoch by epoch.
__device__ __forceinline__ bool grid_sync(unsigned* bar, unsigned target, unsigned* err, int* s_stop) {
    __syncthreads();
    if (threadIdx.x == 0) {
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" :: "l"(bar) : "memory");
        const uint64_t t0 = gtimer();
        int stop = 0;
        for (;;) {
            unsigned v;
            asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
            if ((int)(v - target) >= 0) break;
            if (gtimer() - t0 > 2000000000ull) {
                atomicOr(err, DEVERR_TIMEOUT);
                stop = 1;
                break;
            }
        }
        asm volatile("fence.acq_rel.gpu;" ::: "memory");  // acquire: the other CTAs' writes before our reads
        *s_stop = stop;
    }
    __syncthreads();
    return *s_stop == 0;
}

__device__ __forceinline__ void copy_async(unsigned char* dst, const unsigned char* src, int chunks) {
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    for (int i = threadIdx.x; i < chunks; i += blockDim.x)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" :: "r"(d + 16 * i), "l"(src + 16 * i) : "memory");
}

// Row `row` of a 2 x 2 or 4 x 4 matrix against amplitudes x: the FMA chain of the other per-gate kernels.
template <typename R, int D>
__device__ __forceinline__ typename Amp<R>::T row_product(const typename Amp<R>::T* u, const typename Amp<R>::T (&x)[D]) {
    R re = 0, im = 0;
#pragma unroll
    for (int c = 0; c < D; ++c) {
        const typename Amp<R>::T w = u[c];
        re = fmar(w.x, x[c].x, re);
        re = fmar(-w.y, x[c].y, re);
        im = fmar(w.x, x[c].y, im);
        im = fmar(w.y, x[c].x, im);
    }
    return make_amp<R>(re, im);
}

// R: arithmetic, S: the state's type.
template <typename R, typename S, int NA>
__global__ void __launch_bounds__(kThreads<R>) k_small_tiles(typename Amp<S>::T* __restrict__ psi, uint32_t ntiles,
                                                          const unsigned char* __restrict__ prog, int groups, int prog_bytes,
                                                          unsigned* bar, unsigned* err, int from_basis, uint32_t basis) {
    using T = typename Amp<R>::T;
    constexpr int THR = kThreads<R>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* const buf = reinterpret_cast<T*>(smem_raw);                       // [2][NA * THR]
    unsigned char* const sp = smem_raw + 2 * NA * THR * sizeof(T);  // [2][prog_bytes]
    __shared__ int s_stop;
    const unsigned tid = threadIdx.x, G = gridDim.x;
    const unsigned char* src = prog;
    copy_async(sp, src, (int)(sizeof(Group) / 16));
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    copy_async(sp, src, reinterpret_cast<const Group*>(sp)->chunks);
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    int cur = 0;
    for (int g = 0; g < groups; ++g) {
        const Group& gr = *reinterpret_cast<const Group*>(sp + (g & 1) * prog_bytes);
        const Op* const ops = reinterpret_cast<const Op*>(&gr + 1);
        const T* const coefs = reinterpret_cast<const T*>(ops + gr.ops);
        src += 16 * gr.chunks;
        if (g + 1 < groups) copy_async(sp + ((g + 1) & 1) * prog_bytes, src, gr.next_chunks);  // waited for below
        const bool act = tid < (1u << gr.bits);  // states narrower than the threads
        for (uint32_t t = blockIdx.x; t < ntiles; t += G) {
            const uint32_t base = (uint32_t)insert_zeros(t, gr.pos, gr.bits);
            uint32_t at[NA];
            T v[NA];
#pragma unroll
            for (int j = 0; j < NA; ++j) {
                at[j] = base | (uint32_t)deposit(tid + THR * j, gr.pos, gr.bits);
                v[j] = make_amp<R>(0, 0);
                if (act) {
                    if (g == 0 && from_basis) v[j].x = at[j] == basis ? (R)1 : (R)0;
                    else {
                        const typename Amp<S>::T w = __ldcg(psi + at[j]);
                        v[j] = make_amp<R>((R)w.x, (R)w.y);
                    }
                }
            }
            for (int o = 0; o < gr.ops; ++o) {
                const Op op = ops[o];
                if ((base & op.gctl) != op.gctl) continue;
                const T* const u = coefs + op.coef;
                if (op.code == kDiag) {
                    const uint32_t pa = base & op.ag ? 1 : 0, pb = base & op.bg ? 2 : 0;
#pragma unroll
                    for (int j = 0; j < NA; ++j) {
                        const uint32_t i = tid + THR * j;
                        const uint32_t m = (i & op.am ? 1u : pa) | (i & op.bm ? 2u : pb);
                        if (!((op.flags >> m) & 1)) continue;
                        if (op.flags & 16) {
                            v[j] = make_amp<R>(-v[j].x, -v[j].y);
                        } else {
                            const T d = u[m];
                            v[j] = make_amp<R>(fmar(d.x, v[j].x, -d.y * v[j].y), fmar(d.x, v[j].y, d.y * v[j].x));
                        }
                    }
                    continue;
                }
                T* const b = buf + cur * (NA * THR);
                cur ^= 1;  // the buffer before last is free: every thread has passed the barrier after reading it
#pragma unroll
                for (int j = 0; j < NA; ++j) b[tid + THR * j] = v[j];
                __syncthreads();
#pragma unroll
                for (int j = 0; j < NA; ++j) {
                    const uint32_t i = tid + THR * j;
                    if ((i & op.tctl) != op.tctl) continue;
                    if (op.code <= kRx1) {
                        const bool hi = i & op.t0;
                        const T y = b[i ^ op.t0];
                        if (op.code == kDense1) {
                            const T x[2] = {hi ? y : v[j], hi ? v[j] : y};
                            v[j] = row_product<R, 2>(u + (hi ? 2 : 0), x);
                        } else if (op.code == kReal1) {
                            const R c0 = hi ? u[2].x : u[0].x, c1 = hi ? u[3].x : u[1].x;
                            const T x = hi ? y : v[j], z = hi ? v[j] : y;
                            v[j] = make_amp<R>(fmar(c1, z.x, c0 * x.x), fmar(c1, z.y, c0 * x.y));
                        } else {
                            // real diagonal, imaginary off-diagonal: both rows by selection (a branch would take a warp
                            // through both), the first column's product first
                            const R c0 = hi ? u[2].y : u[0].x, c1 = hi ? u[3].x : u[1].y;
                            const T x = hi ? y : v[j], z = hi ? v[j] : y;
                            const R xr = hi ? -x.y : x.x, xi = hi ? x.x : x.y, zr = hi ? z.x : -z.y, zi = hi ? z.y : z.x;
                            v[j] = make_amp<R>(fmar(c1, zr, c0 * xr), fmar(c1, zi, c0 * xi));
                        }
                    } else {
                        const uint32_t z = i & ~(op.t0 | op.t1);
                        const int row = (i & op.t0 ? 1 : 0) | (i & op.t1 ? 2 : 0);
                        if (op.code == kSwap2) {
                            v[j] = b[z | (row & 1 ? op.t1 : 0u) | (row & 2 ? op.t0 : 0u)];
                        } else {
                            const T x[4] = {b[z], b[z | op.t0], b[z | op.t1], b[z | op.t0 | op.t1]};
                            v[j] = row_product<R, 4>(u + 4 * row, x);
                        }
                    }
                }
            }
            if (act) {
#pragma unroll
                for (int j = 0; j < NA; ++j) psi[at[j]] = make_amp<S>((S)v[j].x, (S)v[j].y);
            }
        }
        if (g + 1 < groups) {
            asm volatile("cp.async.wait_all;" ::: "memory");  // the barrier below orders the copies for all threads
            if (G > 1) {
                if (!grid_sync(bar, (unsigned)(g + 1) * G, err, &s_stop)) return;
            } else {
                __threadfence();
                __syncthreads();
            }
        }
    }
}

static int tile_bits(int arith, int n) {
    // complex128: as many tiles as SMs, and all four FP64 units of an SM busy (128 amplitudes or more); complex64, which
    // the barriers bound: 512 amplitudes, so that a group holds more gates
    const int want = arith == QSIM_C64 ? kMaxBits : std::max(kThrBits<double>, n - 7);
    return std::min(n, std::min(want, kMaxBits));
}

}  // namespace stile

// ---- products on at most two qubits -------------------------------------------------------------------------------
namespace {

using Mat4 = double[32];  // 4 x 4, interleaved

bool exact_one(double re, double im) { return re == 1.0 && im == 0.0; }

// The gate (at most two qubits in all, diagonals as tables) as a 4 x 4 matrix on (a, b); b = -1: on (a, an idle qubit).
void embed(const TileGate& g, int a, int b, Mat4& m) {
    std::memset(m, 0, sizeof(Mat4));
    auto bit = [&](int idx, int q) { return q == a ? idx & 1 : (q == b ? idx >> 1 : 0); };
    for (int r = 0; r < 4; ++r)
        for (int c = 0; c < 4; ++c) {
            bool same = true, ctl = true;  // the bits the gate does not act on agree; its controls are set
            int gr = 0, gc = 0, mine = 0;
            for (int j = 0; j < g.k; ++j) {
                gr |= bit(r, g.q[j]) << j;
                gc |= bit(c, g.q[j]) << j;
                mine |= g.q[j] == a ? 1 : 2;
            }
            same = ((r ^ c) & ~mine) == 0;
            for (int j = 0; j < g.nc; ++j) ctl = ctl && bit(r, g.ctl[j]) && bit(c, g.ctl[j]);
            double re = 0, im = 0;
            if (same && g.nc > 0 && !ctl) {
                re = r == c ? 1.0 : 0.0;
            } else if (same) {
                if (g.diag) {
                    if (gr == gc) { re = g.mat[2 * gr]; im = g.mat[2 * gr + 1]; }
                } else {
                    re = g.mat[2 * ((gr << g.k) + gc)];
                    im = g.mat[2 * ((gr << g.k) + gc) + 1];
                }
            }
            m[2 * (4 * r + c)] = re;
            m[2 * (4 * r + c) + 1] = im;
        }
}

struct Kind1 { bool real, rx; };  // a 2 x 2 matrix: real; real diagonal with imaginary off-diagonal
Kind1 kind1(const double* m) {
    return {m[1] == 0 && m[3] == 0 && m[5] == 0 && m[7] == 0,
            m[1] == 0 && m[7] == 0 && m[2] == 0 && m[4] == 0};
}

// FMAs an amplitude (diagonals: a complex factor, free when it is a sign).
int fmas(const TileGate& g) {
    if (g.diag) {
        for (size_t m = 0; m < g.mat.size() / 2; ++m)
            if (!exact_one(g.mat[2 * m], g.mat[2 * m + 1]) && !(g.mat[2 * m] == -1.0 && g.mat[2 * m + 1] == 0.0)) return 4;
        return 0;
    }
    if (g.k == 2) return 16;
    const Kind1 k = kind1(g.mat.data());
    return k.real || k.rx ? 4 : 8;
}

}  // namespace

std::vector<TileGate> fuse_pairs(int arith, const std::vector<TileGate>& gates) {
    struct Item {
        int a = -1, b = -1;
        std::vector<int> members;  // empty: merged into a later item
    };
    // what an operation costs besides its FMAs, in FMAs an amplitude: a CTA barrier and its latency
    const int per_op = arith == QSIM_C64 ? 40 : 2;
    std::vector<Item> items;
    int open[64];
    std::fill(open, open + 64, -1);  // the last item on a qubit, while gates on that qubit may still join it
    for (int i = 0; i < (int)gates.size(); ++i) {
        const TileGate& g = gates[i];
        int q[2] = {g.q[0], g.k > 1 ? g.q[1] : (g.nc > 0 ? g.ctl[0] : -1)};
        const int nq = g.k + g.nc;
        if (nq > 2) {  // wider: alone
            items.push_back({});
            items.back().members = {i};
            for (int b = 0; b < 64; ++b)
                if ((g.all >> b) & 1) open[b] = -1;
            continue;
        }
        if (nq == 1) {
            if (open[q[0]] < 0) {
                items.push_back({});
                items.back().a = q[0];
                open[q[0]] = (int)items.size() - 1;
            }
            items[open[q[0]]].members.push_back(i);
            continue;
        }
        const int oa = open[q[0]], ob = open[q[1]];
        if (oa >= 0 && oa == ob) {
            items[oa].members.push_back(i);
            continue;
        }
        const bool sa = oa >= 0 && items[oa].b < 0, sb = ob >= 0 && items[ob].b < 0;  // open items on one qubit
        Item it;
        it.a = q[0];
        it.b = q[1];
        if (g.diag && !(sa && sb)) {  // between products: a diagonal of its own, which ends both
            it.members = {i};
            items.push_back(std::move(it));
            open[q[0]] = open[q[1]] = -1;
            continue;
        }
        for (int o : {sa ? oa : -1, sb ? ob : -1}) {
            if (o < 0) continue;
            it.members.insert(it.members.end(), items[o].members.begin(), items[o].members.end());
            items[o].members.clear();
        }
        it.members.push_back(i);
        items.push_back(std::move(it));
        open[q[0]] = open[q[1]] = (int)items.size() - 1;
    }
    std::vector<TileGate> out;
    for (const Item& it : items) {
        if (it.members.size() < 2 || it.a < 0) {
            for (int i : it.members) out.push_back(gates[i]);
            continue;
        }
        Mat4 m, e, t;
        embed(gates[it.members[0]], it.a, it.b, m);
        int apart = 0;
        for (size_t x = 0; x < it.members.size(); ++x) {
            apart += fmas(gates[it.members[x]]) + (gates[it.members[x]].diag ? 0 : per_op);
            if (x == 0) continue;
            embed(gates[it.members[x]], it.a, it.b, e);
            for (int r = 0; r < 4; ++r)
                for (int c = 0; c < 4; ++c) {
                    double re = 0, im = 0;
                    for (int k = 0; k < 4; ++k) {
                        const double ar = e[2 * (4 * r + k)], ai = e[2 * (4 * r + k) + 1];
                        const double br = m[2 * (4 * k + c)], bi = m[2 * (4 * k + c) + 1];
                        re = std::fma(ar, br, std::fma(-ai, bi, re));
                        im = std::fma(ar, bi, std::fma(ai, br, im));
                    }
                    t[2 * (4 * r + c)] = re;
                    t[2 * (4 * r + c) + 1] = im;
                }
            std::memcpy(m, t, sizeof(Mat4));
        }
        TileGate p;
        p.ok = true;
        p.k = it.b >= 0 ? 2 : 1;
        p.q[0] = it.a;
        p.q[1] = it.b >= 0 ? it.b : 0;
        p.tmask = p.all = (1ull << it.a) | (it.b >= 0 ? 1ull << it.b : 0);
        const int D = 1 << p.k;
        p.diag = true;
        for (int r = 0; r < D; ++r)
            for (int c = 0; c < D; ++c) {
                p.mat.push_back(m[2 * (4 * r + c)]);
                p.mat.push_back(m[2 * (4 * r + c) + 1]);
                p.diag = p.diag && (r == c || (m[2 * (4 * r + c)] == 0 && m[2 * (4 * r + c) + 1] == 0));
            }
        if (p.diag) {
            std::vector<double> d;
            for (int r = 0; r < D; ++r) {
                d.push_back(p.mat[2 * (r * D + r)]);
                d.push_back(p.mat[2 * (r * D + r) + 1]);
            }
            p.mat.swap(d);
        }
        if (fmas(p) + (p.diag ? 0 : per_op) <= apart) out.push_back(std::move(p));
        else
            for (int i : it.members) out.push_back(gates[i]);
    }
    return out;
}

namespace stile {

template <typename R>
static bool build_t(int arith, int n, const std::vector<TileGate>& g, std::vector<unsigned char>& prog, int* groups) {
    using T = typename Amp<R>::T;
    const int B = tile_bits(arith, n);
    auto size = [](const TileGate& c) { return (int)(sizeof(Op) + sizeof(T) * (!c.diag && c.k == 2 ? 16 : 4)); };
    const auto cuts = tile_cut(g, B, 0, size, kMaxProg - (int)sizeof(Group) - 16, 1 << 20);
    prog.assign(kHeader, 0);
    std::vector<size_t> starts;
    for (const TileCut& cut : cuts) {
        uint64_t set = cut.set;
        for (int q = 0; q < n && __builtin_popcountll(set) < B; ++q) set |= 1ull << q;
        Group gr;
        std::memset(&gr, 0, sizeof(gr));
        gr.bits = B;
        int tb[64], nb = 0;
        for (int q = 0; q < n; ++q)
            if ((set >> q) & 1) { tb[q] = nb; gr.pos[nb++] = q; }
        std::vector<Op> ops;
        std::vector<T> coefs;
        for (int i : cut.members) {
            const TileGate& c = g[i];
            if (!c.ok) return false;
            Op op;
            std::memset(&op, 0, sizeof(op));
            op.coef = (uint32_t)coefs.size();
            auto place = [&](int q, uint32_t& tm, uint32_t& gm) {
                if ((set >> q) & 1) tm |= 1u << tb[q];
                else gm |= 1u << q;
            };
            auto put = [&](double re, double im) {
                T v;
                v.x = (R)re;
                v.y = (R)im;
                coefs.push_back(v);
            };
            const double* m = c.mat.data();
            if (c.diag) {
                op.code = kDiag;
                place(c.q[0], op.am, op.ag);
                if (c.k > 1) place(c.q[1], op.bm, op.bg);
                bool neg = true;
                for (int x = 0; x < 4; ++x) {
                    const int o = c.k > 1 ? x : x & 1;
                    put(m[2 * o], m[2 * o + 1]);
                    if (!exact_one(m[2 * o], m[2 * o + 1])) {
                        op.flags |= 1u << x;
                        neg = neg && m[2 * o] == -1.0 && m[2 * o + 1] == 0.0;
                    }
                }
                if (neg) op.flags |= 16;
            } else {
                for (int j = 0; j < c.nc; ++j) place(c.ctl[j], op.tctl, op.gctl);
                op.t0 = 1u << tb[c.q[0]];
                if (c.k == 1) {
                    const Kind1 kd = kind1(m);
                    op.code = kd.real ? kReal1 : (kd.rx ? kRx1 : kDense1);
                    for (int x = 0; x < 4; ++x) put(m[2 * x], m[2 * x + 1]);
                } else {
                    op.t1 = 1u << tb[c.q[1]];
                    bool swap = true;
                    for (int r = 0; r < 4; ++r)
                        for (int k = 0; k < 4; ++k) {
                            put(m[2 * (4 * r + k)], m[2 * (4 * r + k) + 1]);
                            const double want = (r == 0 || r == 3 ? r : 3 - r) == k ? 1.0 : 0.0;
                            swap = swap && m[2 * (4 * r + k)] == want && m[2 * (4 * r + k) + 1] == 0.0;
                        }
                    op.code = swap ? kSwap2 : kDense2;
                }
            }
            ops.push_back(op);
        }
        gr.ops = (int)ops.size();
        const size_t bytes = sizeof(Group) + sizeof(Op) * ops.size() + sizeof(T) * coefs.size();
        gr.chunks = (int)((bytes + 15) / 16);
        if (16 * gr.chunks > kMaxProg) return false;
        const size_t at = prog.size();
        prog.resize(at + 16 * (size_t)gr.chunks, 0);
        std::memcpy(prog.data() + at, &gr, sizeof(gr));
        std::memcpy(prog.data() + at + sizeof(gr), ops.data(), sizeof(Op) * ops.size());
        std::memcpy(prog.data() + at + sizeof(gr) + sizeof(Op) * ops.size(), coefs.data(), sizeof(T) * coefs.size());
        starts.push_back(at);
    }
    for (size_t i = 0; i + 1 < starts.size(); ++i)
        reinterpret_cast<Group*>(prog.data() + starts[i])->next_chunks = reinterpret_cast<Group*>(prog.data() + starts[i + 1])->chunks;
    *groups = (int)starts.size();
    return *groups > 0;
}

template <typename R, typename S, int NA>
static cudaError_t run_t(void* psi, int n, int bits, unsigned char* dprog, int groups, unsigned* dev_err, cudaStream_t s,
                         const DevInfo& d, const uint64_t* from_basis) {
    using T = typename Amp<R>::T;
    auto kern = k_small_tiles<R, S, NA>;
    const size_t smem = 2 * NA * kThreads<R> * sizeof(T) + 2 * (size_t)kMaxProg;
    cudaError_t e = smem_optin(reinterpret_cast<const void*>(kern), (int)smem);
    if (e != cudaSuccess) return e;
    const uint32_t ntiles = 1u << (n - bits);
    const unsigned grid = std::min<unsigned>(ntiles, (unsigned)std::max(1, d.num_sms));
    if ((uint64_t)groups * grid >= (1ull << 31)) return cudaErrorInvalidValue;
    unsigned* bar = reinterpret_cast<unsigned*>(dprog);
    const bool coop = grid > 1 && groups > 1;  // only then do CTAs wait for one another
    if (coop && (e = cudaMemsetAsync(bar, 0, sizeof(unsigned), s)) != cudaSuccess) return e;
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.gridDim = dim3(grid, 1, 1);
    cfg.blockDim = dim3(kThreads<R>, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = coop ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<typename Amp<S>::T*>(psi), ntiles, (const unsigned char*)(dprog + kHeader), groups, kMaxProg,
                              bar, dev_err, from_basis ? 1 : 0, from_basis ? (uint32_t)*from_basis : 0u);
}

template <typename R, typename S>
static cudaError_t run_n(int arith, void* psi, int n, unsigned char* dprog, int groups, unsigned* dev_err, cudaStream_t s,
                         const DevInfo& d, const uint64_t* from_basis) {
    const int bits = tile_bits(arith, n);
    if constexpr (sizeof(R) == 8) {
        if (bits == kThrBits<R> + 1) return run_t<R, S, 2>(psi, n, bits, dprog, groups, dev_err, s, d, from_basis);
        if (bits == kThrBits<R> + 2) return run_t<R, S, 4>(psi, n, bits, dprog, groups, dev_err, s, d, from_basis);
    }
    return run_t<R, S, 1>(psi, n, bits, dprog, groups, dev_err, s, d, from_basis);
}

}  // namespace stile

bool small_tiles_build(int arith, int n, const std::vector<TileGate>& gates, std::vector<unsigned char>& prog,
                       SmallTiles* out) {
    if (n < 1 || n > kSmallMaxQubits || gates.empty()) return false;
    out->arith = arith;
    if (!(arith == QSIM_C64 ? stile::build_t<float>(arith, n, gates, prog, &out->groups)
                            : stile::build_t<double>(arith, n, gates, prog, &out->groups)))
        return false;
    // measured over brickwork, random, U(4), TFIM and QFT circuits of 6 to 16 qubits: within 30 % of the times
    out->us = 2.7 * out->groups;
    out->roundings = 0.0;
    const double fp64 = std::ldexp(1.0, std::max(7, stile::tile_bits(arith, n))) / 3170.0;  // us per FMA an amplitude, one SM
    for (const TileGate& g : gates) {
        const int f = fmas(g);
        if (arith == QSIM_C64) out->us += g.diag ? (f ? 0.15 : 0.12) : (g.k == 2 ? 0.37 : 0.25);
        else out->us += 0.15 + 1.2 * fp64 * f;
        out->roundings += f ? 1.0 + f / 4.0 : 0.0;
    }
    return true;
}

cudaError_t launch_small_tiles(int dtype, const SmallTiles& t, void* psi, int n, void* dprog, unsigned* dev_err,
                               cudaStream_t s, const DevInfo& d, const uint64_t* from_basis) {
    if (n < 1 || n > kSmallMaxQubits || t.groups < 1 || !dev_err || (reinterpret_cast<uintptr_t>(dprog) & 15) != 0)
        return cudaErrorInvalidValue;
    unsigned char* p = static_cast<unsigned char*>(dprog);
    if (dtype == QSIM_C128) return stile::run_n<double, double>(t.arith, psi, n, p, t.groups, dev_err, s, d, from_basis);
    return t.arith == QSIM_C64 ? stile::run_n<float, float>(t.arith, psi, n, p, t.groups, dev_err, s, d, from_basis)
                               : stile::run_n<double, float>(t.arith, psi, n, p, t.groups, dev_err, s, d, from_basis);
}

}  // namespace qsim
