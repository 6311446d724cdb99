// k_tilegates.cu -- many gates of a per-gate plan in one pass over the state (paper Sec. 2.1 "State-Vector
// Simulation": the gates applied one after another to the state vector).
//
// A gate by itself is one read and one write of the state for 8 FMAs an amplitude or fewer, so a per-gate plan is
// bound by memory: 750 gates on 25 qubits took 53.2 ms, 79 us a pass. Gates that act on a common small set of
// qubits need not go through memory one by one: a tile of 2^12 complex64 (2^11 complex128) amplitudes, all
// combinations of 12 (11) index bits, is closed under every gate whose targets lie among those bits. Controls and
// diagonal gates put no condition on the tile: a control or a diagonal qubit outside it has one value in the whole
// tile. One pass loads each tile into shared memory, applies a group of gates in circuit order (gates on other
// qubits may move past one another), and writes it back; each gate still does its own arithmetic in the state's
// precision (the FMA chains of k_dense_small and k_diag, terms with a zero coefficient left out).
//
// Inside a tile the group is cut into steps of up to 4 register bits: a thread holds the 16 amplitudes that differ
// in those bits and applies every gate of the step in registers, so that a gate costs its FMAs and not a trip
// through shared memory. The amplitude index is XOR-swizzled (one 4-bit vector per tile bit, all different; 3-bit
// for complex128), and a step's lanes take tile bits whose vectors are independent, so every access is free of
// bank conflicts whatever the register bits. Steps and gates are a small program that travels as a kernel
// parameter.
//
// The lowest bits of the index (3 in complex64, 2 in complex128) always belong to the tile: 64-byte runs.
// Bound: instruction issue in complex64 (24 qubits, 720 random-circuit gates: 2.9 ms; per gate and thread 64 FMAs or
// fewer and about 45 other instructions), FP64 in complex128. Measured and left: every thread decoding the program
// from shared memory (4.1 ms, against 3.1 at the time) or from the parameter (3.9 ms).
#include <algorithm>
#include <cstring>

#include "common.cuh"
#include "internal.h"

namespace qsim {
namespace tile {

constexpr int kReg = 4, NV = 1 << kReg;   // register bits, amplitudes per thread
template <typename R> constexpr int kThrBits = sizeof(R) == 4 ? 8 : 7;
template <typename R> constexpr int kThreads = 1 << kThrBits<R>;
template <typename R> constexpr int kBits = kReg + kThrBits<R>;   // tile bits
template <typename R> constexpr int kLow = sizeof(R) == 4 ? 3 : 2;  // always in the tile
constexpr int kMaxBits = 12;
constexpr int kMaxProg = 1536;      // 64-bit words of a group's program

constexpr int kMaxOps = 256;        // and its operations

// What an operation does, and on which register bits: one number, so that the threads take one branch to its code.
enum Code { kDense1 = 0, kReal1 = 4, kRx1 = 8, kCtl1 = 12 /* any gate with a control among the tile's bits */,
            kDense2 = 16, kSwap2 = 22, kDiag2 = 28, kDiag1 = 34, kDiag0 = 38, kSkip = 39 };
// register-bit pairs in order: 01 02 03 12 13 23
__host__ __device__ constexpr int pair_index(int r0, int r1) { return r0 == 0 ? r1 - 1 : r0 + r1; }

// The program travels as a kernel parameter and is copied to shared memory once per CTA: steps, operations,
// coefficients. A step is 64 bytes: the byte offset in the tile that each thread bit and each register bit adds (by
// XOR: the index is swizzled), its first operation and the one after its last.
struct Step { uint32_t pv[8], pr[4], first, end, pad[2]; };
constexpr int kStepWords = sizeof(Step) / 8;
// Words of an operation: code | rctl << 8 (register bits that must be set: controls) | diagonal flags << 16 (bits 0..3:
// entry m differs from 1; bit 4: those are all -1) | first coefficient << 32; thread bits that must be set | thread bits
// of the diagonal's qubits a << 8 and b << 16 that are not register bits; index bits outside the tile that must be
// set; a and b among those.
constexpr int kOpWords = 5;

// An operation as a tile's threads use it, decoded once per tile (by one thread each) from the bits outside the tile:
// decoding by every thread was a third of all instructions. x: code | rctl << 8 | flags << 16 | a << 24 | b << 25 (the
// values outside the tile); y: the thread bits of the program's second word; z: first coefficient.
struct Rec { uint32_t x, y, z, w; };

struct Args {
    int pos[kMaxBits];   // index bits of the tile, ascending
    uint64_t ntiles;
    int steps, ops;
    int words;           // of the program
    uint64_t prog[kMaxProg];
};

__device__ __forceinline__ float fmar(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fmar(double a, double b, double c) { return __fma_rn(a, b, c); }

template <typename T> __device__ __forceinline__ T cscale(T d, T v) {
    T o;
    o.x = fmar(d.x, v.x, -d.y * v.y);
    o.y = fmar(d.x, v.y, d.y * v.x);
    return o;
}

// A single-qubit gate on register bit RB; KIND 0 any, 1 real, 2 real diagonal with imaginary off-diagonal.
template <typename R, int RB, int KIND, bool CTL>
__device__ __forceinline__ void apply1(typename Amp<R>::T (&v)[NV], const typename Amp<R>::T* c, int rctl) {
    using T = typename Amp<R>::T;
    R a0, a1, b0, b1, c0, c1, d0, d1;
    if constexpr (sizeof(R) == 4) {
        const float4 ab = reinterpret_cast<const float4*>(c)[0], cd = reinterpret_cast<const float4*>(c)[1];
        a0 = ab.x; a1 = ab.y; b0 = ab.z; b1 = ab.w; c0 = cd.x; c1 = cd.y; d0 = cd.z; d1 = cd.w;
    } else {
        const T u0 = c[0], u1 = c[1], u2 = c[2], u3 = c[3];
        a0 = u0.x; a1 = u0.y; b0 = u1.x; b1 = u1.y; c0 = u2.x; c1 = u2.y; d0 = u3.x; d1 = u3.y;
    }
#pragma unroll
    for (int p = 0; p < NV / 2; ++p) {
        const int i = ((p >> RB) << (RB + 1)) | (p & ((1 << RB) - 1)), j = i | (1 << RB);
        if (CTL && (i & rctl) != rctl) continue;
        const T x = v[i], y = v[j];
        if constexpr (KIND == 1) {
            v[i].x = fmar(b0, y.x, a0 * x.x);
            v[i].y = fmar(b0, y.y, a0 * x.y);
            v[j].x = fmar(d0, y.x, c0 * x.x);
            v[j].y = fmar(d0, y.y, c0 * x.y);
        } else if constexpr (KIND == 2) {
            v[i].x = fmar(-b1, y.y, a0 * x.x);
            v[i].y = fmar(b1, y.x, a0 * x.y);
            v[j].x = fmar(d0, y.x, -c1 * x.y);
            v[j].y = fmar(d0, y.y, c1 * x.x);
        } else {
            v[i].x = fmar(-b1, y.y, fmar(b0, y.x, fmar(-a1, x.y, a0 * x.x)));
            v[i].y = fmar(b1, y.x, fmar(b0, y.y, fmar(a1, x.x, a0 * x.y)));
            v[j].x = fmar(-d1, y.y, fmar(d0, y.x, fmar(-c1, x.y, c0 * x.x)));
            v[j].y = fmar(d1, y.x, fmar(d0, y.y, fmar(c1, x.x, c0 * x.y)));
        }
    }
}
// A two-qubit gate on register bits R0 < R1 (matrix bit 0 <-> R0); SWAP exchanges them. Without controls complex64 takes
// two groups of four at a time and reads the matrix two columns at a time: 16 shared-memory loads for 256 FMAs instead
// of 64 (24 qubits, 96 U(4) gates: 1.75 -> 1.60 ms; 25 qubits, 750 random-circuit gates, where a one-qubit matrix is two
// loads instead of four: 6.31 -> 5.88 ms).
template <typename R, int R0, int R1, bool SWAP>
__device__ __forceinline__ void apply2(typename Amp<R>::T (&v)[NV], const typename Amp<R>::T* c, int rctl) {
    using T = typename Amp<R>::T;
    if constexpr (!SWAP && sizeof(R) == 4) {
        if (rctl == 0) {
#pragma unroll
            for (int h = 0; h < NV / 8; ++h) {
                int at[2][4];
                T x[2][4];
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int g = 2 * h + e;
                    int i = ((g >> R0) << (R0 + 1)) | (g & ((1 << R0) - 1));
                    i = ((i >> R1) << (R1 + 1)) | (i & ((1 << R1) - 1));
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        at[e][r] = i | ((r & 1) << R0) | ((r >> 1) << R1);
                        x[e][r] = v[at[e][r]];
                    }
                }
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    R re[2] = {0, 0}, im[2] = {0, 0};
#pragma unroll
                    for (int k = 0; k < 4; k += 2) {
                        const float4 u = *reinterpret_cast<const float4*>(c + 4 * r + k);
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            re[e] = fmar(u.x, x[e][k].x, re[e]);
                            re[e] = fmar(-u.y, x[e][k].y, re[e]);
                            im[e] = fmar(u.x, x[e][k].y, im[e]);
                            im[e] = fmar(u.y, x[e][k].x, im[e]);
                            re[e] = fmar(u.z, x[e][k + 1].x, re[e]);
                            re[e] = fmar(-u.w, x[e][k + 1].y, re[e]);
                            im[e] = fmar(u.z, x[e][k + 1].y, im[e]);
                            im[e] = fmar(u.w, x[e][k + 1].x, im[e]);
                        }
                    }
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        v[at[e][r]].x = re[e];
                        v[at[e][r]].y = im[e];
                    }
                }
            }
            return;
        }
    }
#pragma unroll
    for (int g = 0; g < NV / 4; ++g) {
        int i = ((g >> R0) << (R0 + 1)) | (g & ((1 << R0) - 1));
        i = ((i >> R1) << (R1 + 1)) | (i & ((1 << R1) - 1));
        if ((i & rctl) != rctl) continue;
        if constexpr (SWAP) {
            const T t = v[i | (1 << R0)];
            v[i | (1 << R0)] = v[i | (1 << R1)];
            v[i | (1 << R1)] = t;
        } else {
            const T x[4] = {v[i], v[i | (1 << R0)], v[i | (1 << R1)], v[i | (1 << R0) | (1 << R1)]};
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                R re = 0, im = 0;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const T u = c[4 * r + k];
                    const R ur = u.x, ui = u.y;
                    re = fmar(ur, x[k].x, re);
                    re = fmar(-ui, x[k].y, re);
                    im = fmar(ur, x[k].y, im);
                    im = fmar(ui, x[k].x, im);
                }
                T o;
                o.x = re;
                o.y = im;
                v[i | ((r & 1) << R0) | ((r >> 1) << R1)] = o;
            }
        }
    }
}
// A diagonal whose table index has bit 0 <-> register bit M0 (or, M0 < 0, the value pa) and bit 1 <-> M1 (or pb).
// pa and pb differ from thread to thread, so their entries are selected, not branched on.
template <typename R, int M0, int M1>
__device__ __forceinline__ void diagonal(typename Amp<R>::T (&v)[NV], const typename Amp<R>::T* c, uint32_t flags, int pa, int pb) {
    using T = typename Amp<R>::T;
    constexpr int C0 = M0 >= 0 ? 2 : 1, C1 = M1 >= 0 ? 2 : 1;
    constexpr int mask = (M0 >= 0 ? 1 << (M0 & 3) : 0) | (M1 >= 0 ? 1 << (M1 & 3) : 0);
    const bool neg = (flags >> 4) & 1;
#pragma unroll
    for (int x1 = 0; x1 < C1; ++x1)
#pragma unroll
        for (int x0 = 0; x0 < C0; ++x0) {
            // the entries any thread may want here: skipped when all are 1
            const uint32_t any = (M0 >= 0 ? 1u << x0 : 3u) << (M1 >= 0 ? 2 * x1 : 0);
            if (!(flags & (M1 >= 0 ? any : any | any << 2))) continue;
            const int m = (M0 >= 0 ? x0 : pa) | ((M1 >= 0 ? x1 : pb) << 1);
            const int w = (M0 >= 0 && x0 ? 1 << (M0 & 3) : 0) | (M1 >= 0 && x1 ? 1 << (M1 & 3) : 0);
            if (neg) {
                const R sg = (flags >> m) & 1 ? (R)-1 : (R)1;
#pragma unroll
                for (int j = 0; j < NV; ++j)
                    if ((j & mask) == w) { v[j].x *= sg; v[j].y *= sg; }
            } else {
                const T d = c[m];
#pragma unroll
                for (int j = 0; j < NV; ++j)
                    if ((j & mask) == w) v[j] = cscale(d, v[j]);
            }
        }
}

template <typename R>
__global__ void __launch_bounds__(kThreads<R>, sizeof(R) == 4 ? 3 : 4)
k_tile_gates(typename Amp<R>::T* __restrict__ psi, const __grid_constant__ Args a) {
    using T = typename Amp<R>::T;
    constexpr int THR = kThreads<R>, TB = kThrBits<R>, B = kBits<R>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* sT = reinterpret_cast<T*>(smem_raw);
    Rec* recs = reinterpret_cast<Rec*>(sT + (1 << B));
    uint64_t* prog = reinterpret_cast<uint64_t*>(recs + a.ops);
    const Step* const steps = reinterpret_cast<const Step*>(prog);
    const uint64_t* const opw = prog + kStepWords * a.steps;
    const T* const coefs = reinterpret_cast<const T*>(opw + kOpWords * a.ops + ((kOpWords * a.ops) & 1));
    __shared__ uint64_t joff[NV];   // index offset of tile bits TB.. = j
    const int tid = threadIdx.x;
    for (int i = tid; i < a.words; i += THR) prog[i] = a.prog[i];
    if (tid < NV) joff[tid] = deposit((uint64_t)tid, a.pos + TB, kReg);
    const uint64_t toff = deposit((uint64_t)tid, a.pos, TB);
    // swizzle of the linear index j * THR + tid: low bits XOR-ed with one vector per set bit (see tile_vec)
    constexpr uint64_t kVec = sizeof(R) == 4 ? 0xCBA97653ull : 0x34217653ull;  // vectors of bits LB.., 4 bits each
    constexpr int LB = sizeof(R) == 4 ? 4 : 3;
    auto swz = [&](uint32_t i) {
        uint32_t x = i;
#pragma unroll
        for (int b = LB; b < B; ++b) x ^= ((i >> b) & 1) ? (uint32_t)((kVec >> (4 * (b - LB))) & 15) : 0u;
        return x;
    };
    const uint32_t ts = swz((uint32_t)tid);
    __syncthreads();
    for (uint64_t t = blockIdx.x; t < a.ntiles; t += gridDim.x) {
        const uint64_t base = insert_zeros(t, a.pos, B);
        T* const p = psi + base + toff;
#pragma unroll
        for (int j = 0; j < NV; ++j)
            asm volatile("cp.async.ca.shared.global [%0], [%1], %2;"
                         :: "r"((uint32_t)__cvta_generic_to_shared(sT + (ts ^ swz((uint32_t)(j * THR))))), "l"(p + joff[j]),
                            "n"((int)sizeof(T)) : "memory");
        for (int o = tid; o < a.ops; o += THR) {
            const uint64_t* q = opw + kOpWords * o;
            const uint64_t h = q[0];
            const uint32_t x = (uint32_t)h | (base & q[3] ? 1u << 24 : 0u) | (base & q[4] ? 1u << 25 : 0u);
            recs[o] = {(base & q[2]) != q[2] ? (uint32_t)kSkip : x, (uint32_t)q[1], (uint32_t)(h >> 32), 0u};
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
        for (int s = 0; s < a.steps; ++s) {
            const Step& st = steps[s];
            uint32_t pt = 0;
#pragma unroll
            for (int i = 0; i < TB; ++i) pt ^= ((tid >> i) & 1) ? st.pv[i] : 0u;
            const uint32_t q[kReg] = {st.pr[0], st.pr[1], st.pr[2], st.pr[3]};
            auto slot = [&](int j) {
                uint32_t x = pt;
#pragma unroll
                for (int i = 0; i < kReg; ++i)
                    if ((j >> i) & 1) x ^= q[i];
                return reinterpret_cast<T*>(smem_raw + x);
            };
            T v[NV];
#pragma unroll
            for (int j = 0; j < NV; ++j) v[j] = *slot(j);
            const int end = (int)st.end;
            for (int o = (int)st.first; o < end; ++o) {
                const Rec rec = recs[o];
                const T* const c = coefs + rec.z;
                // what only some operations need
                auto rctl = [&] { return (int)((rec.x >> 8) & 0xFF); };
                auto flags = [&] { return (rec.x >> 16) & 0x1F; };
                auto on = [&] { return (tid & rec.y & 0xFF) == (rec.y & 0xFF); };
                auto pa = [&] { return (((tid << 8) & rec.y & 0xFF00u) | (rec.x & (1u << 24))) ? 1 : 0; };
                auto pb = [&] { return (((tid << 16) & rec.y & 0xFF0000u) | (rec.x & (1u << 25))) ? 1 : 0; };
                switch (rec.x & 0xFF) {
                    case kDense1: apply1<R, 0, 0, false>(v, c, 0); break;
                    case kDense1 + 1: apply1<R, 1, 0, false>(v, c, 0); break;
                    case kDense1 + 2: apply1<R, 2, 0, false>(v, c, 0); break;
                    case kDense1 + 3: apply1<R, 3, 0, false>(v, c, 0); break;
                    case kReal1: apply1<R, 0, 1, false>(v, c, 0); break;
                    case kReal1 + 1: apply1<R, 1, 1, false>(v, c, 0); break;
                    case kReal1 + 2: apply1<R, 2, 1, false>(v, c, 0); break;
                    case kReal1 + 3: apply1<R, 3, 1, false>(v, c, 0); break;
                    case kRx1: apply1<R, 0, 2, false>(v, c, 0); break;
                    case kRx1 + 1: apply1<R, 1, 2, false>(v, c, 0); break;
                    case kRx1 + 2: apply1<R, 2, 2, false>(v, c, 0); break;
                    case kRx1 + 3: apply1<R, 3, 2, false>(v, c, 0); break;
                    case kCtl1: if (on()) apply1<R, 0, 0, true>(v, c, rctl()); break;
                    case kCtl1 + 1: if (on()) apply1<R, 1, 0, true>(v, c, rctl()); break;
                    case kCtl1 + 2: if (on()) apply1<R, 2, 0, true>(v, c, rctl()); break;
                    case kCtl1 + 3: if (on()) apply1<R, 3, 0, true>(v, c, rctl()); break;
                    case kDense2: if (on()) apply2<R, 0, 1, false>(v, c, rctl()); break;
                    case kDense2 + 1: if (on()) apply2<R, 0, 2, false>(v, c, rctl()); break;
                    case kDense2 + 2: if (on()) apply2<R, 0, 3, false>(v, c, rctl()); break;
                    case kDense2 + 3: if (on()) apply2<R, 1, 2, false>(v, c, rctl()); break;
                    case kDense2 + 4: if (on()) apply2<R, 1, 3, false>(v, c, rctl()); break;
                    case kDense2 + 5: if (on()) apply2<R, 2, 3, false>(v, c, rctl()); break;
                    case kSwap2: if (on()) apply2<R, 0, 1, true>(v, c, rctl()); break;
                    case kSwap2 + 1: if (on()) apply2<R, 0, 2, true>(v, c, rctl()); break;
                    case kSwap2 + 2: if (on()) apply2<R, 0, 3, true>(v, c, rctl()); break;
                    case kSwap2 + 3: if (on()) apply2<R, 1, 2, true>(v, c, rctl()); break;
                    case kSwap2 + 4: if (on()) apply2<R, 1, 3, true>(v, c, rctl()); break;
                    case kSwap2 + 5: if (on()) apply2<R, 2, 3, true>(v, c, rctl()); break;
                    case kDiag2: diagonal<R, 0, 1>(v, c, flags(), 0, 0); break;
                    case kDiag2 + 1: diagonal<R, 0, 2>(v, c, flags(), 0, 0); break;
                    case kDiag2 + 2: diagonal<R, 0, 3>(v, c, flags(), 0, 0); break;
                    case kDiag2 + 3: diagonal<R, 1, 2>(v, c, flags(), 0, 0); break;
                    case kDiag2 + 4: diagonal<R, 1, 3>(v, c, flags(), 0, 0); break;
                    case kDiag2 + 5: diagonal<R, 2, 3>(v, c, flags(), 0, 0); break;
                    case kDiag1: diagonal<R, 0, -1>(v, c, flags(), 0, pb()); break;
                    case kDiag1 + 1: diagonal<R, 1, -1>(v, c, flags(), 0, pb()); break;
                    case kDiag1 + 2: diagonal<R, 2, -1>(v, c, flags(), 0, pb()); break;
                    case kDiag1 + 3: diagonal<R, 3, -1>(v, c, flags(), 0, pb()); break;
                    case kDiag0: diagonal<R, -1, -1>(v, c, flags(), pa(), pb()); break;
                    default: break;
                }
            }
#pragma unroll
            for (int j = 0; j < NV; ++j) *slot(j) = v[j];
            __syncthreads();
        }
#pragma unroll
        for (int j = 0; j < NV; ++j) p[joff[j]] = sT[ts ^ swz((uint32_t)(j * THR))];
        __syncthreads();
    }
}

// The swizzle vector of tile bit b (its own value for the low bits): all different in complex64.
template <typename R> uint32_t tile_vec(int b) {
    constexpr uint64_t kVec = sizeof(R) == 4 ? 0xCBA97653ull : 0x34217653ull;
    constexpr int LB = sizeof(R) == 4 ? 4 : 3;
    return b < LB ? 1u << b : (uint32_t)((kVec >> (4 * (b - LB))) & 15);
}

// Rank over GF(2) of a few small vectors.
static int gf2_rank(std::vector<uint32_t> v) {
    int rank = 0;
    for (int bit = 0; bit < 4; ++bit) {
        size_t p = rank;
        while (p < v.size() && !((v[p] >> bit) & 1)) ++p;
        if (p == v.size()) continue;
        std::swap(v[p], v[rank]);
        for (size_t i = 0; i < v.size(); ++i)
            if ((int)i != rank && ((v[i] >> bit) & 1)) v[i] ^= v[rank];
        ++rank;
    }
    return rank;
}

template <typename R>
static void emit_group(const std::vector<TileGate>& g, const std::vector<int>& members, uint64_t set, int n, TileGroup& out) {
    constexpr int B = kBits<R>, TB = kThrBits<R>, LB = sizeof(R) == 4 ? 4 : 3;
    for (int q = 0; q < n && __builtin_popcountll(set) < B; ++q) set |= 1ull << q;  // fill with the lowest qubits
    int pos[64], tb[64];
    int nb = 0;
    for (int q = 0; q < n; ++q)
        if ((set >> q) & 1) { tb[q] = nb; pos[nb++] = q; }
    constexpr int CW = sizeof(R) / 4;
    std::vector<uint64_t> steps, ops, coefs;  // words
    int nops = 0, ncoef = 0;
    std::vector<int> und = members;
    while (!und.empty()) {
        // the step that takes the most operations, grown from any of the first ones that is free to go
        std::vector<int> best;
        uint64_t best_set = 0;
        uint64_t seen = 0;
        for (size_t u = 0; u < und.size() && u < 24; ++u) {
            const TileGate& c = g[und[u]];
            if (u > 0 && (c.diag || (c.all & seen))) { seen |= c.all; continue; }
            seen |= c.all;
            uint64_t s = 0;
            std::vector<int> got = tile_collect(g, und, c.diag ? -1 : und[u], s, kReg, set, ~0ull);
            if (got.size() > best.size()) { best.swap(got); best_set = s; }
        }
        for (int q = n - 1; q >= 0 && __builtin_popcountll(best_set) < kReg; --q) best_set |= set & (1ull << q);
        int rb[64];
        std::vector<int> regs, thr;
        for (int j = 0; j < B; ++j) {
            rb[j] = -1;
            if ((best_set >> pos[j]) & 1) { rb[j] = (int)regs.size(); regs.push_back(j); }
            else thr.push_back(j);
        }
        // thread bits: first LB with independent vectors (conflict-free), then the others
        std::vector<int> order;
        std::vector<uint32_t> vecs;
        for (int j : thr) {
            std::vector<uint32_t> t = vecs;
            t.push_back(tile_vec<R>(j));
            if ((int)order.size() < LB && gf2_rank(t) == (int)t.size()) { order.push_back(j); vecs.swap(t); }
        }
        for (int j : thr)
            if (std::find(order.begin(), order.end(), j) == order.end()) order.push_back(j);
        int tbit[64];
        for (int j = 0; j < B; ++j) tbit[j] = -1;
        Step st;
        std::memset(&st, 0, sizeof(st));
        auto phys = [&](int j) { return ((j < LB ? 0u : 1u << j) ^ tile_vec<R>(j)) * (uint32_t)sizeof(typename Amp<R>::T); };
        for (int i = 0; i < TB; ++i) {
            tbit[order[i]] = i;
            st.pv[i] = phys(order[i]);
        }
        for (int i = 0; i < kReg; ++i) st.pr[i] = phys(regs[i]);
        st.first = (uint32_t)nops;
        st.end = (uint32_t)(nops + (int)best.size());
        uint64_t sw[kStepWords];
        std::memcpy(sw, &st, sizeof(st));
        steps.insert(steps.end(), sw, sw + kStepWords);
        for (int i : best) {
            const TileGate& c = g[i];
            int code = 0, rctl = 0, flags = 0;
            uint64_t tctl = 0, gctl = 0, at = 0, bt = 0, ag = 0, bg = 0;
            std::vector<std::pair<double, double>> cf;
            auto place = [&](int q, uint64_t& tm, uint64_t& gm) {  // a qubit that is not a register bit
                if ((set >> q) & 1) tm |= 1ull << tbit[tb[q]];
                else gm |= 1ull << q;
            };
            auto reg = [&](int q) { return ((set >> q) & 1) ? rb[tb[q]] : -1; };
            if (c.diag) {
                const int ra = reg(c.q[0]), rb2 = c.k > 1 ? reg(c.q[1]) : -1;
                // table index: bit 0 <-> the (lower) register qubit where there is one
                const bool flip = c.k > 1 && (ra < 0 ? rb2 >= 0 : (rb2 >= 0 && rb2 < ra));
                const int qa = flip ? c.q[1] : c.q[0], qb = c.k > 1 ? (flip ? c.q[0] : c.q[1]) : -1;
                const int fa = flip ? rb2 : ra, fb = flip ? ra : rb2;
                code = fa < 0 ? (int)kDiag0 : (fb < 0 ? kDiag1 + fa : kDiag2 + pair_index(fa, fb));
                if (fa < 0) place(qa, at, ag);
                if (qb >= 0 && fb < 0) place(qb, bt, bg);
                bool neg = true;
                for (int m = 0; m < 4; ++m) {
                    const int o = c.k > 1 ? (flip ? ((m & 1) << 1) | (m >> 1) : m) : (m & 1);
                    cf.push_back({c.mat[2 * o], c.mat[2 * o + 1]});
                    if (cf.back() != std::make_pair(1.0, 0.0)) {
                        flags |= 1 << m;
                        neg = neg && cf.back().first == -1.0 && cf.back().second == 0.0;
                    }
                }
                if (neg) flags |= 16;
            } else {
                for (int j = 0; j < c.nc; ++j) {
                    const int r = reg(c.ctl[j]);
                    if (r >= 0) rctl |= 1 << r;
                    else place(c.ctl[j], tctl, gctl);
                }
                const double* m = c.mat.data();
                if (c.k == 1) {
                    const bool real = m[1] == 0 && m[3] == 0 && m[5] == 0 && m[7] == 0;
                    const bool rx = m[1] == 0 && m[7] == 0 && m[2] == 0 && m[4] == 0;
                    code = (rctl || tctl ? kCtl1 : (real ? kReal1 : (rx ? kRx1 : kDense1))) + reg(c.q[0]);
                    for (int x = 0; x < 4; ++x) cf.push_back({m[2 * x], m[2 * x + 1]});
                } else {
                    const int ra = reg(c.q[0]), rb2 = reg(c.q[1]);
                    const bool flip = ra > rb2;
                    auto idx = [&](int x) { return flip ? ((x & 1) << 1) | (x >> 1) : x; };
                    bool swap = true;
                    for (int r = 0; r < 4; ++r)
                        for (int k = 0; k < 4; ++k) {
                            cf.push_back({m[2 * (4 * idx(r) + idx(k))], m[2 * (4 * idx(r) + idx(k)) + 1]});
                            swap = swap && cf.back().second == 0 && cf.back().first == ((r == 0 || r == 3 ? r : 3 - r) == k ? 1.0 : 0.0);
                        }
                    code = (swap ? kSwap2 : kDense2) + pair_index(std::min(ra, rb2), std::max(ra, rb2));
                    if (swap) cf.clear();
                }
            }
            ops.push_back((uint64_t)code | ((uint64_t)rctl << 8) | ((uint64_t)flags << 16) | ((uint64_t)ncoef << 32));
            ops.push_back(tctl | (at << 8) | (bt << 16));
            ops.push_back(gctl);
            ops.push_back(ag);
            ops.push_back(bg);
            ++nops;
            ncoef += (int)cf.size();
            for (const auto& x : cf) {
                R v[2] = {(R)x.first, (R)x.second};
                uint64_t w[2] = {0, 0};
                std::memcpy(w, v, sizeof(v));
                coefs.insert(coefs.end(), w, w + CW);
            }
        }
        std::vector<int> rest;
        for (int i : und)
            if (std::find(best.begin(), best.end(), i) == best.end()) rest.push_back(i);
        und.swap(rest);
    }
    std::memcpy(out.pos, pos, sizeof(int) * B);
    out.steps = (int)(steps.size() / kStepWords);
    out.ops = nops;
    if (ops.size() & 1) ops.push_back(0);  // coefficients start on 16 bytes (a step is 32)
    out.prog = steps;
    out.prog.insert(out.prog.end(), ops.begin(), ops.end());
    out.prog.insert(out.prog.end(), coefs.begin(), coefs.end());
}

}  // namespace tile

bool tile_gate_ok(bool diag, int k, int nc) { return diag ? k + nc <= 2 : k <= 2; }

std::vector<TileGroup> tile_groups(int dtype, int n, const std::vector<TileGate>& g) {
    const int B = dtype == QSIM_C64 ? tile::kBits<float> : tile::kBits<double>;
    const int low = dtype == QSIM_C64 ? tile::kLow<float> : tile::kLow<double>;
    auto words = [&](const TileGate& c) {
        return tile::kStepWords + tile::kOpWords + (dtype == QSIM_C64 ? 1 : 2) * (!c.diag && c.k == 2 ? 16 : 4);
    };
    std::vector<TileGroup> out;
    for (const TileCut& cut : tile_cut(g, B, (1ull << low) - 1, words, tile::kMaxProg - 1, tile::kMaxOps)) {
        TileGroup grp;
        grp.members = cut.members;
        if (grp.members.size() > 1) {
            if (dtype == QSIM_C64) tile::emit_group<float>(g, grp.members, cut.set, n, grp);
            else tile::emit_group<double>(g, grp.members, cut.set, n, grp);
        }
        out.push_back(std::move(grp));
    }
    return out;
}

template <typename R>
static cudaError_t tile_launch(void* psi, int n, const TileGroup& grp, cudaStream_t s, const DevInfo& d) {
    using T = typename Amp<R>::T;
    constexpr int B = tile::kBits<R>;
    if (n < B || grp.steps < 1 || grp.prog.size() > (size_t)tile::kMaxProg) return cudaErrorInvalidValue;
    tile::Args a;
    std::memcpy(a.pos, grp.pos, sizeof(a.pos));
    a.ntiles = 1ull << (n - B);
    a.steps = grp.steps;
    a.ops = grp.ops;
    a.words = (int)grp.prog.size();
    std::memcpy(a.prog, grp.prog.data(), sizeof(uint64_t) * grp.prog.size());
    const size_t smem = (sizeof(T) << B) + sizeof(tile::Rec) * grp.ops + sizeof(uint64_t) * grp.prog.size();
    cudaError_t e = smem_optin(reinterpret_cast<const void*>(tile::k_tile_gates<R>),
                               (int)((sizeof(T) << B) + sizeof(tile::Rec) * tile::kMaxOps + sizeof(uint64_t) * tile::kMaxProg));
    if (e != cudaSuccess) return e;
    const unsigned grid = (unsigned)std::min<uint64_t>(a.ntiles, (uint64_t)d.num_sms * (sizeof(R) == 4 ? 3 : 4));
    tile::k_tile_gates<R><<<grid, tile::kThreads<R>, smem, s>>>(reinterpret_cast<T*>(psi), a);
    return cudaGetLastError();
}

cudaError_t launch_tile_gates(int dtype, void* psi, int n, const TileGroup& grp, cudaStream_t s, const DevInfo& d) {
    return dtype == QSIM_C64 ? tile_launch<float>(psi, n, grp, s, d) : tile_launch<double>(psi, n, grp, s, d);
}

}  // namespace qsim
