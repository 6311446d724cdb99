// k_tcx.cu -- a fused block of up to 5 qubits in the state's own precision (QSIM_PREC_SIMT plans) on the
// tensor cores, by exact integer slices.
//
// Paper Sec. 2.1: a fused block is one small dense matrix applied to every group of 2^k amplitudes. On CUDA
// cores a 5-qubit block is 128 FMAs an amplitude: 3.5 ms at 24 qubits in complex128 (FP64 runs at 1.05 TFLOP/s
// here; moving the state takes 0.08 ms), 0.46 ms at 26 qubits in complex64 (0.16 ms to move it). The tensor
// cores have the rate, so the block is computed as sums of integer products that they add without rounding (the
// error-free splitting of Ozaki, Ogita, Oishi and Rump 2012, on FP16 operands as Mukunoki, Ozaki, Ogita and
// Imamura 2020):
//   * the 64 reals of a row (a group's 32 complex amplitudes) become fixed-point numbers relative to the row's
//     largest exponent E, 2^54 (complex128) or 2^30 (complex64) steps, cut into signed base-256 digits
//     (7 or 4); U likewise. Digits are integers in [-128, 127], exact in FP16.
//   * D_d = sum over digit positions s + t = d of X_s U_t^T accumulates in FP32 tensor memory: at most 7 * 64
//     products of at most 2^14, below 2^24, so every sum is an exact integer. Positions d < 8 (complex128; 34
//     of 49 products) or d < 4 (complex64; 10 of 16) are kept; the first one left out is worth 2^-59
//     (2^-28) of the row's scale.
//   * y = 2^(E') sum_d D_d 2^(-8d): in complex128 summed in a 64-bit integer and rounded once, in complex64 by
//     three FMAs.
// The errors are those of the fixed-point steps, of the positions left out and of the final rounding, all relative to the
// row's largest amplitude: at most 2^-25 (2^-52) of the power of two above it, in rms 2^-27 (2^-54) in the emulated
// digit arithmetic; smaller than the accumulated roundings of 64 FMAs (against 64 bits, 23-qubit brickwork of depth 10: 1.6e-15,
// by FMAs 1.8e-15; 26-qubit random pairs in complex64: 2.3e-7, by FMAs 1.0e-6).
//
// Rows by FMAs. That is an error of the row, and an amplitude that is small beside its row's largest one would lose its
// digits (R_y(2e-4) on five qubits of |0>: the amplitude of two flips, 1e-8, came out with 2 % error in complex64, that of
// three as zero). So the slices take a row only where every result y_i has sum_c |U_ic| |x_c| above 2^-9 of that power of
// two, which bounds its error by 2^-16 (2^-43) of that sum, beside 2^-18 (2^-47) for a chain of 64 FMAs: rows whose amplitudes
// lie within kRange = 8 binades of the largest (the entries of a row of U sum to 1 or more), and rows in which every row
// of U has an entry of at least 2^-7 at an amplitude within 1 binade, or of 2^-4 within 4, or, in complex128, only zeros at
// all amplitudes, for a result that is zero either way (21-qubit random circuit of 8 gates a qubit 0.80 -> 0.44 ms; in complex64
// it cost other circuits 3 to 7 %). The input warps look at U for 0.1 % of the rows of a random state, and few of those
// fail. The others go by FMAs in the state's precision, by the
// output (rows_by_fma): in complex128 the whole row; in complex64, where 64 FMAs lose more than the slices, the results more
// than kLarge = 4 binades below the row's largest amplitude (with whole rows by FMAs the norm of the error of 12 circuits,
// sparse and structured ones among them, was 1.19 times that of the slices alone, at worst 1.56; so it is 0.98, 1.03). Rows
// outside the exponents that the slices take go by FMAs as well; amplitudes that the block joins with an infinity or NaN
// become NaN.
// One pass, complex64 26 qubits / complex128 24 qubits, windows from qubit 8 and from qubit 0: 270, 331 / 240, 273 us, and
// without this 254, 309 / 201, 239; with amplitudes over 30 binades 570 / 710 (CUDA cores 461 / 3457). 16-step TFIM chains of
// small angles, 25 qubits complex64 / 23 complex128: 5.2 -> 10.1 / 4.0 -> 10.2 ms. Measured and left: such rows by three
// more warps, a few of a quadrant or all of them (351 us from qubit 0 in complex64, 850 us at 30 binades); one warp that
// decides for all rows (2.7 ms at 30 binades); rows given away unseen where a quadrant has few (301 us); ROWS = 4 (590 us at
// 30 binades, against 510 with whole rows by FMAs).
//
// Layout. A tile is 128 rows (the 7 lowest index bits outside the block) by 32 columns; blocks of fewer qubits
// take idle qubits as further columns (U x I). Digit plane s of a tile is a K-major operand of 128 x 64 FP16
// (16 KiB, SWIZZLE_128B) in shared memory, digit planes of U are stacked as 64-row operands. Because D_d and
// D_{d+1} are neighbouring 64-column blocks of tensor memory, one MMA of X_s against the stacked rows of
// U_t..U_{t+3} (N = 256) adds to four digit positions at once, at the full rate of the tensor cores (with N = 64
// the reads of A from shared memory would bound it).
//
// Roles, one CTA per SM: input warps load a tile, convert it and write its planes; one warp issues the MMAs;
// output warps sum the positions, convert back and store, and take rows by FMAs. In complex64 (16 input, 8 output warps) planes and
// accumulators are double-buffered, and the next tile's loads are in flight in registers. In complex128 the 8
// positions take all of tensor memory and the planes half of shared memory, so a tile's MMAs commit in four
// groups of planes: as a group retires, the input (8 warps) writes the next tile's planes over it and the output
// (16 warps) adds the positions it finished.
// Bound: complex64 (26 qubits, 270 us, 0.58 of the copy rate) the input's loads and conversion; complex128 (24
// qubits, 240 us, 3457 on CUDA cores) the output: its conversions run on the FP64 units at two a cycle and SM,
// and on the integer pipe about as fast, so they are spread over both; the tensor cores work a quarter of the
// time. Measured and left (against 190 us without the rows by FMAs): one set of warps for input and output (281 us at 24 qubits), 8 output warps (208),
// the next tile staged by cp.async (204), L2 prefetch of the next tile (212), the D_d to integers by F2I (213).
// Every mbarrier wait is bounded (2 s); on expiry the kernel records DEVERR_TIMEOUT, waits once more (bounded)
// for its MMAs, frees its tensor memory and returns.
#include <cuda_fp16.h>

#include <algorithm>
#include <cstring>

#include "common.cuh"
#include "internal.h"
#include "tc_ptx.cuh"

namespace qsim {
namespace tcx {

using namespace qsim::tc;

constexpr int K = 5, D = 1 << K;   // targets (padded), complex columns of a tile
constexpr int NR = 2 * D;          // reals of a row: K and N of one digit product
constexpr int kRowBits = 7;        // 128 rows per tile (MMA M = 128)
constexpr int kPlaneA = 128 * NR * 2;  // bytes of one digit plane of a tile (16 KiB)
constexpr int kPlaneB = NR * NR * 2;   // bytes of one digit plane of U (8 KiB)

template <typename R> struct Cfg;
template <> struct Cfg<float> {
    static constexpr int S = 4, ND = 4;        // digits; digit positions kept
    static constexpr int BUF = 2;              // tiles in flight: A planes and accumulators
    static constexpr int GROUPS = 1;           // commits per tile
    static constexpr int IN = 16, OUT = 8, MMA = 1;  // warps: tile loads and digit planes; accumulators and stores; MMAs
    static constexpr int kStepsU = 30;         // U in 2^-30 steps
    static constexpr int kRange = 8;           // binades below the row's largest amplitude that the slices take
    static constexpr int ROWS = 2;             // rows an output warp takes at a time by FMAs
    static constexpr int U = D;                // columns of U in shared memory, for those rows
    __host__ __device__ static constexpr int group_end(int) { return S; }
};
template <> struct Cfg<double> {
    static constexpr int S = 7, ND = 8;
    static constexpr int BUF = 1;
    static constexpr int GROUPS = 4;           // planes 0-1, 2-3, 4-5, 6
    // Whole warpgroups, so that registers can move between them: launched with 72 a thread (28 warps, 64512 in
    // all), the input takes 96, the output keeps 64, the MMA warpgroup (one warp works) 56: 64512.
    static constexpr int IN = 8, OUT = 16, MMA = 4;
    static constexpr int kRegIn = 96, kRegOut = 64, kRegMma = 56;
    static constexpr int kStepsU = 54;
    static constexpr int kRange = 8;
    static constexpr int ROWS = 1;
    static constexpr int U = 0;                // (stays in global memory: 16 KiB more would take L1 from the loads in flight)
    __host__ __device__ static constexpr int group_end(int g) { return g < 3 ? 2 * g + 2 : S; }
};
template <typename R> constexpr int row_slots() { return Cfg<R>::BUF == 1 ? 4 : 8; }  // tiles whose row exponents are kept
template <typename R> constexpr int threads() { return 32 * (Cfg<R>::IN + Cfg<R>::OUT + Cfg<R>::MMA); }
template <typename R> constexpr int smem_planes() { return Cfg<R>::S * (Cfg<R>::BUF * kPlaneA + kPlaneB); }
template <typename R> constexpr int bars() { return Cfg<R>::BUF * (2 + Cfg<R>::GROUPS) + 9; }
// planes, column offsets, largest and smallest amplitudes of the input's rows [2][IN / 4][128] and which of them are large and
// not zero [2][IN / 4][128], exponents of tiles in flight [row_slots][128], barriers, the TMEM slot, the large entries of U [32][4], U and
// the rows taken by FMAs [OUT][ROWS][32], alignment
template <typename R> constexpr int smem_rows() { return (Cfg<R>::OUT * Cfg<R>::ROWS + Cfg<R>::U) * D * 2 * (int)sizeof(R); }
template <typename R> constexpr size_t smem_bytes() {
    return smem_planes<R>() + smem_rows<R>() + 24 * D + 4 * (4 * (Cfg<R>::IN / 4) + row_slots<R>()) * 128 +
           8 * bars<R>() + 8 + 1024;
}
// With 1 KiB that the system takes, below the 196 KiB that leave 60 KiB of L1: the data of loads in flight lies there
// (complex128, 24 qubits: 201 us a pass; with 28 KiB, 239).
static_assert(smem_bytes<float>() <= 195 * 1024 && smem_bytes<double>() <= 195 * 1024, "");

// How a thread moves its columns: one amplitude per access (lane = row); the columns of qubit 0 (target 0) as
// one vector of two; the columns of qubits 0 and 1 (targets 0 and 1) as one 32-byte vector of four (complex64).
enum Mode { kRows = 0, kPairs = 1, kQuads = 2 };

struct Args {
    int nS;              // 12 index bits covered by a tile
    int spos[12];        // those bit positions, ascending
    int rpos[kRowBits];  // row bit j <-> index bit rpos[j]
    int tpos[K];         // column bit j <-> index bit tpos[j]
    uint64_t ntiles;
    int from_basis;      // the input is |basis>, generated in registers instead of read
    uint64_t basis;
    int k;               // the block's own qubits: column bits 0 .. k - 1
    int digits;          // rows of wide range go by FMAs
    int split;           // 2^split CTAs share a tile: lanes 0 .. 32 / 2^split - 1 of each quadrant are the first one's rows, ...
    int32_t w[4];        // 2^30, 2^22, 2^14, 2^6 (as parameters, so that they stay multiplications)
};

__device__ __forceinline__ void mma_ss(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t hi, uint32_t idesc,
                                       uint32_t acc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 ad, bd;\n\tsetp.ne.b32 p, %5, 0;\n\tmov.b64 ad, {%1, %3};\n\t"
        "mov.b64 bd, {%2, %3};\n\ttcgen05.mma.cta_group::1.kind::f16 [%0], ad, bd, %4, p;\n}"
        :: "r"(d_tmem), "r"(a_lo), "r"(b_lo), "r"(hi), "r"(idesc), "r"(acc) : "memory");
}

// `words` 32-bit words (2, 4 or 8) between registers and global memory, aligned to their size.
template <int N> __device__ __forceinline__ void ld_words(const void* p, uint32_t* w) {
    if constexpr (N == 8)
        asm volatile("ld.global.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                     : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]), "=r"(w[4]), "=r"(w[5]), "=r"(w[6]), "=r"(w[7])
                     : "l"(p) : "memory");
    else if constexpr (N == 4)
        asm volatile("ld.global.v4.b32 {%0,%1,%2,%3}, [%4];"
                     : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]) : "l"(p) : "memory");
    else
        asm volatile("ld.global.v2.b32 {%0,%1}, [%2];" : "=r"(w[0]), "=r"(w[1]) : "l"(p) : "memory");
}
template <int N> __device__ __forceinline__ void st_words(void* p, const uint32_t* w) {
    if constexpr (N == 8)
        asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};"
                     :: "l"(p), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7])
                     : "memory");
    else if constexpr (N == 4)
        asm volatile("st.global.v4.b32 [%0], {%1,%2,%3,%4};"
                     :: "l"(p), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]) : "memory");
    else
        asm volatile("st.global.v2.b32 [%0], {%1,%2};" :: "l"(p), "r"(w[0]), "r"(w[1]) : "memory");
}

// Largest exponents of a row that the slices take: from kLowE on, a zero or subnormal real next to a larger one falls
// below the fixed-point step and needs no case of its own, and results stay normal; up to kHighE (complex128: to_fixed_cvt
// adds 1076 - E to exponents) they do not overflow.
template <typename R> constexpr uint32_t kLowE = sizeof(R) == 8 ? 64 : 32;
template <typename R> constexpr uint32_t kHighE = sizeof(R) == 8 ? 1076 : 247;
// Beside a row's exponent: its small results come from FMAs (complex64; complex128: all), all of them.
constexpr int kByFma = 1 << 20, kAllFma = 1 << 21, kExponent = 0xFFFF;
constexpr int kLarge = 4;  // results within so many binades of the row's largest amplitude come from the slices all the same

// The fixed-point value of a real whose row has largest biased exponent E, plus 128 in every base-256 digit
// (so that the bytes of the result are the digits plus 128). |x| < 2^(E - 1022) maps to 2^54 steps. Two ways that
// give the same value but for ties: shifts on the integer pipe (19 instructions), or a conversion, which the FP64
// units run at two a cycle and SM. The input warps alternate them, so that both units work.
__device__ __forceinline__ void to_fixed_int(uint32_t& lo, uint32_t& hi, uint32_t E) {
    const uint32_t sh = min(E - ((hi >> 20) & 0x7FFu), 63u);
    uint64_t v = (((uint64_t)((hi & 0xFFFFFu) | 0x100000u) << 32) | lo) << 2;  // four times the 53-bit significand
    v = ((v >> sh) + 1) >> 1;                                                  // to nearest
    const uint64_t s = (uint64_t)(int64_t)((int32_t)hi >> 31);
    v = ((v ^ s) - s) + 0x0080808080808080ull;
    lo = (uint32_t)v;
    hi = (uint32_t)(v >> 32);
}
__device__ __forceinline__ void to_fixed_cvt(uint32_t& lo, uint32_t& hi, uint32_t E) {
    // x 2^(1076 - E) by its exponent field; a zero or subnormal becomes a value below 2^-10, which rounds to 0
    const double x = __hiloint2double((int)(hi + ((kHighE<double> - E) << 20)), (int)lo);
    const uint64_t v = (uint64_t)__double2ll_rn(x) + 0x0080808080808080ull;
    lo = (uint32_t)v;
    hi = (uint32_t)(v >> 32);
}

// Y * 2^(E - 1080) to nearest, for kLowE <= E <= 2039, likewise.
__device__ __forceinline__ void to_double_int(int64_t Y, int E, uint32_t& lo, uint32_t& hi) {
    const uint64_t a = (uint64_t)(Y < 0 ? -Y : Y);
    const int lz = __clzll((long long)a);
    const uint64_t t = a << lz;                                           // leading one at bit 63 (a = 0: see below)
    uint64_t r = t >> 11;                                                 // 53 bits; to nearest, ties to even,
    r += (((uint32_t)t & 0x7FFu) + ((uint32_t)r & 1u)) > 0x400u ? 1 : 0;  // which may carry to 2^53
    const uint32_t h = (uint32_t)(r >> 32) + ((uint32_t)(E + 5 - lz) << 20);  // exponent less one: the leading one adds it
    lo = (uint32_t)r;
    hi = a ? h | ((uint32_t)(Y >> 32) & 0x80000000u) : 0u;
}
__device__ __forceinline__ void to_double_cvt(int64_t Y, int E, uint32_t& lo, uint32_t& hi) {
    const double y = __ll2double_rn(Y);
    const uint32_t h = (uint32_t)__double2hiint(y);
    lo = (uint32_t)__double2loint(y);
    hi = h ? h + ((uint32_t)(E - 1080) << 20) : 0u;
}

__device__ __forceinline__ float fmar(float x, float y, float z) { return __fmaf_rn(x, y, z); }
__device__ __forceinline__ double fmar(double x, double y, double z) { return __fma_rn(x, y, z); }

// The rows in `mine` of 32 (`at`: the index of the lane's row) in the state's own arithmetic: sums of FMA chains over
// eight columns each, without the columns that are zero in every row. A warp takes whole rows, NROW at a time, so that it
// has read a row before it is written; a lane is a column of the result, `col` its index bits; xs: room for NROW rows; u: U
// by columns.
template <typename R, int NROW>
__device__ __forceinline__ void rows_by_fma(typename Amp<R>::T* psi, const Args& a, const typename Amp<R>::T* u, typename Amp<R>::T* xs,
                                            uint64_t col, uint32_t mine, uint64_t at) {
    using T = typename Amp<R>::T;
    constexpr bool DBL = sizeof(R) == 8;
    const int lane = threadIdx.x & 31, Du = 1 << a.k, g0 = lane & ~(Du - 1);
    const T* const ucol = u + (lane & (Du - 1));
    while (mine) {
        uint64_t p[NROW];
        uint32_t nz = 0;
        bool has[NROW];
        T x[NROW], y[NROW];
#pragma unroll
        for (int q = 0; q < NROW; ++q) {
            has[q] = mine != 0;
            p[q] = __shfl_sync(0xffffffffu, at, mine ? __ffs(mine) - 1 : 0) + col;
            mine &= mine - 1;
        }
#pragma unroll
        for (int q = 0; q < NROW; ++q) {
            x[q].x = x[q].y = y[q].x = y[q].y = 0;
            if (has[q]) {
                if (a.from_basis) x[q].x = p[q] == a.basis ? (R)1 : (R)0;
                else x[q] = psi[p[q]];
            }
        }
#pragma unroll
        for (int q = 0; q < NROW; ++q) {
            nz |= __ballot_sync(0xffffffffu, x[q].x != 0 || x[q].y != 0);
            xs[q * D + lane] = x[q];
        }
        __syncwarp();
        for (int g = D / 2; g >= Du; g >>= 1) nz |= nz >> g;  // columns of the block
        if (Du < D) nz &= (1u << Du) - 1;
        while (nz) {
            const int c0 = (__ffs(nz) - 1) & 24;
            const uint32_t now = (nz >> c0) & 0xFFu;
            nz &= ~(0xFFu << c0);
            T part[NROW];
#pragma unroll
            for (int q = 0; q < NROW; ++q) part[q].x = part[q].y = 0;
            auto column = [&](T w, int q, T z) {
                part[q].x = fmar(w.x, z.x, part[q].x);
                part[q].x = fmar(-w.y, z.y, part[q].x);
                part[q].y = fmar(w.x, z.y, part[q].y);
                part[q].y = fmar(w.y, z.x, part[q].y);
            };
            if (!DBL && now == 0xFFu) {  // (complex128: FP64 bounds this, not the loads)
#pragma unroll
                for (int c = 0; c < 8; c += 2) {
                    const T w0 = ucol[(c0 + c) * Du], w1 = ucol[(c0 + c + 1) * Du];
#pragma unroll
                    for (int q = 0; q < NROW; ++q) {
                        const uint4 v = *reinterpret_cast<const uint4*>(xs + q * D + g0 + c0 + c);
                        T z0, z1;
                        z0.x = (R)__uint_as_float(v.x); z0.y = (R)__uint_as_float(v.y);
                        z1.x = (R)__uint_as_float(v.z); z1.y = (R)__uint_as_float(v.w);
                        column(w0, q, z0);
                        column(w1, q, z1);
                    }
                }
            } else {
                T ahead = ucol[(c0 + __ffs(now) - 1) * Du];
                for (uint32_t left = now; left; left &= left - 1) {
                    const int c = c0 + __ffs(left) - 1;
                    const T w = ahead;
                    if (left & (left - 1)) ahead = ucol[(c0 + __ffs(left & (left - 1)) - 1) * Du];
#pragma unroll
                    for (int q = 0; q < NROW; ++q) column(w, q, xs[q * D + g0 + c]);
                }
            }
#pragma unroll
            for (int q = 0; q < NROW; ++q) {
                y[q].x += part[q].x;
                y[q].y += part[q].y;
            }
        }
#pragma unroll
        for (int q = 0; q < NROW; ++q) {
            // (read again: a flag a row through the loop above would cost registers that the output's loop has to save)
            const T own = xs[q * D + lane];
            const uint32_t wild = __ballot_sync(0xffffffffu, !isfinite(own.x) || !isfinite(own.y));
            if ((wild >> g0) & (Du < D ? (1u << Du) - 1 : 0xffffffffu)) y[q].x = y[q].y = DBL ? (R)__hiloint2double(0x7FF80000, 0) : (R)__uint_as_float(0x7FC00000u);
            if (has[q]) psi[p[q]] = y[q];
        }
        __syncwarp();  // xs has been read
    }
}
template <typename R, int MODE>
__global__ void __launch_bounds__(threads<R>(), 1)
k_tcx_block(typename Amp<R>::T* __restrict__ psi, const __grid_constant__ Args a, const uint4* __restrict__ bops,
            unsigned* __restrict__ err) {
    using C = Cfg<R>;
    using T = typename Amp<R>::T;
    constexpr bool DBL = sizeof(R) == 8;
    constexpr int S = C::S, ND = C::ND, BUF = C::BUF, GROUPS = C::GROUPS, kIn = C::IN, kOut = C::OUT;
    constexpr int CPI = 128 / kIn, CPO = 128 / kOut;  // complex columns per input and output thread
    constexpr int AW = sizeof(T) / 4;            // words per amplitude
    constexpr int VEC = MODE == kQuads ? 4 : (MODE == kPairs ? 2 : 1);  // amplitudes per access
    constexpr int W = CPI * AW;                  // words of an input thread's share of a tile
    constexpr uint32_t TCOLS = 64 * ND * BUF;
    static_assert(TCOLS == 512 && VEC * AW <= 8, "");

    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* sA = reinterpret_cast<unsigned char*>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    unsigned char* sB = sA + BUF * S * kPlaneA;
    T* sU = reinterpret_cast<T*>(sB + S * kPlaneB);                   // U by columns (complex64)
    T* sX = sU + C::U * D;                                               // [kOut][ROWS][32]
    uint64_t* sCol = reinterpret_cast<uint64_t*>(sX + kOut * C::ROWS * D);
    uint4* sL = reinterpret_cast<uint4*>(sCol + D);                   // of the rows of U, the large entries (and, complex128, those not zero)
    uint32_t* sE = reinterpret_cast<uint32_t*>(sL + D);               // [2][kIn / 4][128]
    uint32_t* sBig = sE + 2 * (kIn / 4) * 128;                        // [2][kIn / 4][128]
    int* sRow = reinterpret_cast<int*>(sBig + 2 * (kIn / 4) * 128);       // [row_slots][128]
    uint64_t* mbar = reinterpret_cast<uint64_t*>(sRow + row_slots<R>() * 128);
    uint32_t* tslot = reinterpret_cast<uint32_t*>(mbar + bars<R>());
    constexpr uint32_t kAll = 0xFFFFFFFFu;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // barriers: per buffer, A stored (full), accumulators read (freed), MMAs of a plane group retired (done); the
    // operand loaded (bbar); per quadrant of 32 rows, the row exponents of its input warps written (rowbar), rows by FMAs
    // stored (fmabar)
    auto full = [&](uint32_t b) { return smem_u32(mbar + b); };
    auto freed = [&](uint32_t b) { return smem_u32(mbar + BUF + b); };
    auto done = [&](uint32_t b, int g) { return smem_u32(mbar + (2 + g) * BUF + b); };
    const uint32_t bbar = smem_u32(mbar + BUF * (2 + GROUPS));
    auto rowbar = [&](int q) { return smem_u32(mbar + BUF * (2 + GROUPS) + 1 + q); };
    [[maybe_unused]] auto fmabar = [&](int q) { return smem_u32(mbar + BUF * (2 + GROUPS) + 5 + q); };
    for (int c = tid; c < D; c += threads<R>()) sCol[c] = deposit((uint64_t)c, a.tpos, K);
    if (tid == 0) {
        for (int j = 0; j < bars<R>(); ++j) {
            const int count = j < BUF ? kIn : (j < 2 * BUF ? kOut : (j <= BUF * (2 + GROUPS) ? 1 : (j < BUF * (2 + GROUPS) + 5 ? kIn / 4 : kOut / 4)));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" :: "r"(smem_u32(mbar + j)), "r"(count) : "memory");
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     :: "r"(smem_u32(tslot)), "r"(TCOLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tbase = *tslot;
    // programmatic dependent launch: the set-up above overlapped the previous kernel's tail
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int* const sums = reinterpret_cast<const int*>(reinterpret_cast<const char*>(bops) + S * kPlaneB);
    const T* const umat = reinterpret_cast<const T*>(sums + NR + 3 * D);  // U by columns
    const uint32_t t0 = blockIdx.x >> a.split, G = gridDim.x >> a.split;  // (fewer than 2^32 tiles: checked by the host)
    const uint32_t m = t0 < a.ntiles ? (uint32_t)((a.ntiles - t0 + G - 1) / G) : 0u;  // tiles of this CTA
    auto tile = [&](uint32_t i) { return (uint64_t)t0 + (uint64_t)i * G; };
    auto buf = [&](uint32_t i) { return i % BUF; };
    auto par = [&](uint32_t i) { return (i / BUF) & 1; };  // phase parity of tile i on its buffer's barriers
    // warp-uniform bounded wait (the TMEM accesses that follow are .sync.aligned)
    auto wait = [&](uint32_t bar, uint32_t p) -> bool {
        const bool ok = !__any_sync(0xffffffffu, !mbar_wait_bounded(bar, p));
        fence_after();
        return ok;
    };
    // input and output warps: thread = row r of the tile, columns c0 ..
    const int quad = warp & 3, r = quad * 32 + lane;
    const bool own = (uint32_t)lane >> (5 - a.split) == (blockIdx.x & ((1u << a.split) - 1));  // the row is this CTA's

    bool bad = false;
    if (warp >= kIn + kOut) {
        // ---- MMA issuer ----
        if constexpr (DBL) asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" :: "n"(Cfg<double>::kRegMma));
        if (warp == kIn + kOut && lane == 0) {
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" :: "r"(bbar), "r"(S * kPlaneB + (C::U > 0 ? (int)sizeof(T) << (2 * a.k) : 0))
                         : "memory");
#pragma unroll 1
            for (int j = 0; j < S; ++j)
                asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                             :: "r"(smem_u32(sB) + j * kPlaneB), "l"(reinterpret_cast<const char*>(bops) + j * kPlaneB),
                                "r"(kPlaneB), "r"(bbar) : "memory");
            if constexpr (C::U > 0)
                asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                             :: "r"(smem_u32(sU)), "l"(umat), "r"((int)sizeof(T) << (2 * a.k)), "r"(bbar) : "memory");
            const uint64_t d0 = sdesc_sw128(smem_u32(sA));
            const uint32_t hi = (uint32_t)(d0 >> 32), alo0 = (uint32_t)d0;
            const uint32_t blo = (uint32_t)sdesc_sw128(smem_u32(sB));
            uint32_t issued = 0;  // tiles issued
            bad = !mbar_wait_bounded(bbar, 0);
            if (bad) mbar_wait_bounded(bbar, 0);  // once more for the copy still in flight
            for (uint32_t i = 0; i < m && !bad; ++i) {
                const uint32_t b = buf(i);
                if (i >= BUF && !mbar_wait_bounded(freed(b), par(i - BUF))) { bad = true; break; }
                if (!mbar_wait_bounded(full(b), par(i))) { bad = true; break; }
                fence_after();
                const uint32_t alo = alo0 + b * ((S * kPlaneA) >> 4), dcol = tbase + b * 64 * ND;
                int g = 0;
#pragma unroll
                for (int s = 0; s < S; ++s) {
                    // plane s against U_0 .. U_{cnt-1}, into D_s .. D_{s+cnt-1}; the digit positions that no plane
                    // before s reached (all of them for s = 0, the last one for s = 1 when ND > S) start here
                    const int cnt = S < ND - s ? S : ND - s;
                    const bool split = s == 1 && ND > S;  // U_{S-1} apart: it starts D_{ND-1}
#pragma unroll
                    for (int u = 0; u < cnt;) {
                        int w = cnt - u < 4 ? cnt - u : 4;
                        if (split && u < cnt - 1 && u + w > cnt - 1) w = cnt - 1 - u;
                        const bool fresh = s == 0 || (split && u == cnt - 1);
                        const uint32_t idesc = (1u << 4) | ((uint32_t)((64 * w) >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
#pragma unroll
                        for (int kk = 0; kk < NR / 16; ++kk)
                            mma_ss(dcol + 64 * (s + u), alo + ((s * kPlaneA + 32 * kk) >> 4), blo + ((u * kPlaneB + 32 * kk) >> 4),
                                   hi, idesc, fresh && kk == 0 ? 0u : 1u);
                        u += w;
                    }
                    if (s + 1 == C::group_end(g)) {
                        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" :: "r"(done(b, g)) : "memory");
                        ++g;
                    }
                }
                issued = i + 1;
            }
            if (bad) {
                atomicOr(err, DEVERR_TIMEOUT);
                if (issued) mbar_wait_bounded(done(buf(issued - 1), GROUPS - 1), par(issued - 1));  // the MMAs already issued
            }
        }
        __syncwarp();
    } else if (warp < kIn) {
        // ---- input: load a tile, convert it to fixed point, write its digit planes ----
        if constexpr (DBL) asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" :: "n"(Cfg<double>::kRegIn));
        const int c0 = CPI * (warp >> 2);
        const volatile uint64_t* vCol = sCol + c0;
        // every warp writes the same words of sL and reads its own writes
        const uint32_t l7 = (uint32_t)sums[NR + lane], l4 = (uint32_t)sums[NR + D + lane];
        if constexpr (DBL) sL[lane] = make_uint4(l7, l4, (uint32_t)sums[NR + 2 * D + lane], 0u);
        else reinterpret_cast<uint2*>(sL)[lane] = make_uint2(l7, l4);
        __syncwarp();
        const T* const prow = psi + deposit((uint64_t)r, a.rpos, kRowBits);
        unsigned char* const arow = sA + (r >> 3) * 1024 + (r & 7) * 128;
        auto load_tile = [&](uint32_t (&X)[W], uint64_t t) {
            const uint64_t b = insert_zeros(t, a.spos, a.nS);
            if (a.from_basis || !own) {
                const uint64_t rb = b + deposit((uint64_t)r, a.rpos, kRowBits);
#pragma unroll
                for (int j = 0; j < CPI; ++j) {
#pragma unroll
                    for (int k = 0; k < AW; ++k) X[AW * j + k] = 0;
                    if (own && rb + vCol[j] == a.basis) X[AW * j + (DBL ? 1 : 0)] = DBL ? 0x3FF00000u : 0x3F800000u;
                }
            } else {
#pragma unroll
                for (int j = 0; j < CPI; j += VEC) ld_words<VEC * AW>(prow + b + vCol[j], X + AW * j);
            }
        };
        // The largest and the smallest magnitude (upper words; an amplitude's is that of its larger part) of the thread's
        // amplitudes: waits for the tile's loads, so that those of the next tile can start.
        // Packed: exponent of the largest (at least 1 unless all are zero) << 16 | 0x7FFF - exponent of the smallest.
        constexpr int EB = DBL ? 20 : 23;  // exponent position in a real's upper word
        auto amplitude = [&](const uint32_t (&X)[W], int j) {
            return max(X[AW * j + (DBL ? 1 : 0)] & 0x7FFFFFFFu, X[AW * j + (DBL ? 3 : 1)] & 0x7FFFFFFFu);
        };
        [[maybe_unused]] auto nonzero = [&](const uint32_t (&X)[W], int j) {
            uint32_t any = 0;
#pragma unroll
            for (int k = 0; k < AW; ++k) any |= DBL && (k & 1) == 0 ? X[AW * j + k] : X[AW * j + k] & 0x7FFFFFFFu;
            return any != 0;
        };
        auto span = [&](const uint32_t (&X)[W]) {
            uint32_t top = 0, low = kAll;
#pragma unroll
            for (int j = 0; j < CPI; ++j) {
                top = max(top, amplitude(X, j));
                low = min(low, amplitude(X, j));
            }
            asm volatile("" : "+r"(top), "+r"(low) :: "memory");  // before any later load is issued (loads share scoreboards)
            return (max(top >> EB, min(top, 1u)) << 16) | (0x7FFFu - (low >> EB));
        };
        // The warps of the quadrant meet at an mbarrier, whose wait ends when one of them has given up (no warp waits at a
        // named barrier: it has no limit).
        uint32_t met = 0;
        auto meet = [&]() -> bool {
            __syncwarp();
            if (lane == 0) mbar_arrive(rowbar(quad));
            return wait(rowbar(quad), met++ & 1);
        };
        // In place: the thread's reals to fixed point relative to the row's largest exponent, which goes to sRow, with kByFma
        // for a row of amplitudes more than kRange binades below its largest, unless every row of U has a large entry at a
        // large amplitude. False if a wait ran out. `planes` is false where no row of the warp needs its digits.
        auto convert = [&](uint32_t (&X)[W], uint32_t i, uint32_t e, bool& planes) -> bool {
            uint32_t* const ex = sE + (i & 1) * (kIn / 4 * 128) + r;
            ex[(warp >> 2) * 128] = e;
            if (!meet()) return false;
#pragma unroll
            for (int k = 0; k < kIn / 4; ++k) e = __vmaxu2(e, ex[k * 128]);
            const uint32_t E0 = e >> 16, low = 0x7FFFu - (e & 0xFFFFu), E = min(max(E0, kLowE<R>), kHighE<R>);
            bool by_fma = E0 != 0 && (E0 != E || (a.digits && E0 - low > (uint32_t)C::kRange));
            uint32_t rows = __ballot_sync(0xffffffffu, by_fma);  // (the same in all warps of the quadrant)
            if (rows) {
                // its columns within 1 and within 4 binades of the largest; has every row of U an entry of 2^-7, or of 2^-4, there
                // (or, complex128, no entry but zeros where the row has amplitudes, for a result that is zero either way)?
                uint32_t big = 0;
                [[maybe_unused]] uint32_t some = 0, bz = 0;
#pragma unroll
                for (int j = 0; j < CPI; ++j) {
                    const uint32_t m = amplitude(X, j) >> EB;
                    if constexpr (DBL) some |= nonzero(X, j) ? 1u << j : 0u;
                    big |= (m + 1 >= E0 ? 1u << j : 0u) | (m + 4 >= E0 ? 0x10000u << j : 0u);
                }
                sBig[(warp >> 2) * 128 + r] = big;
                if constexpr (DBL) sBig[(kIn / 4 + (warp >> 2)) * 128 + r] = some;
                if (!meet()) return false;
                uint32_t b1 = 0, b4 = 0;
#pragma unroll
                for (int k = 0; k < kIn / 4; ++k) {
                    const uint32_t v = sBig[k * 128 + r];
                    b1 |= (v & 0xFFFFu) << (CPI * k);
                    b4 |= (v >> 16) << (CPI * k);
                    if constexpr (DBL) bz |= sBig[(kIn / 4 + k) * 128 + r] << (CPI * k);
                }
                bool held = E0 == E;
                if constexpr (DBL) {
#pragma unroll
                    for (int k = 0; k < D; ++k) {
                        const uint4 l = sL[k];
                        held = held & (((b1 & l.x) | (b4 & l.y)) != 0 || (bz & l.z) == 0);
                    }
                } else {
#pragma unroll 2
                    for (int k = 0; k < D / 2; ++k) {
                        const uint4 l = sL[k];
                        held = held & (((b1 & l.x) | (b4 & l.y)) != 0) & (((b1 & l.z) | (b4 & l.w)) != 0);
                    }
                }
                by_fma = by_fma && !held;
                rows = __ballot_sync(0xffffffffu, by_fma);
            }
            // read by the output warps after this tile's MMAs. The planes of tile i - 1 were stored, so the MMAs of
            // tile i - 1 - BUF have run, for which tile i - 1 - 2 BUF had been read: 2 BUF + 1 slots or more will do
            if (warp < 4) sRow[i % row_slots<R>() * 128 + r] = (int)E | (by_fma ? kByFma | (E0 != E ? kAllFma : 0) : 0);
            planes = !DBL || rows != kAll;
            if (!planes) return true;
            if constexpr (DBL) {
#pragma unroll
                for (int j = 0; j < W; j += 2) {
                    if (j & 6) to_fixed_int(X[j], X[j + 1], E);
                    else to_fixed_cvt(X[j], X[j + 1], E);
                }
            } else {
                const float up = __uint_as_float((283u - E) << 23);  // 2^(156 - E): |x| < 2^(E - 126) to 2^30 steps
#pragma unroll
                for (int j = 0; j < W; ++j) X[j] = (uint32_t)__float2int_rn(__uint_as_float(X[j]) * up) + 0x80808080u;
            }
            return true;
        };
        // Digit plane s of the tile: byte S-1-s of every real, less 128, as FP16 pairs (re, im).
        auto store_plane = [&](const uint32_t (&X)[W], int s, uint32_t b) {
            const int by = (S - 1 - s) & 3, wd = DBL ? (S - 1 - s) >> 2 : 0;
            const uint32_t sel = (uint32_t)by | ((uint32_t)(4 + by) << 8);  // that byte of re to byte 0, of im to byte 2
            unsigned char* const ap = arow + b * (S * kPlaneA) + s * kPlaneA;
#pragma unroll
            for (int q = 0; q < CPI / 4; ++q) {
                uint32_t h[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int j = AW * (4 * q + k);
                    const uint32_t v = (__byte_perm(X[j + wd], X[j + AW / 2 + wd], sel) & 0x00FF00FFu) | 0x64006400u;  // 1024 + byte
                    const __half2 d = __hsub2(*reinterpret_cast<const __half2*>(&v), __half2half2(__ushort_as_half(0x6480)));  // - 1152
                    h[k] = *reinterpret_cast<const uint32_t*>(&d);
                }
                *reinterpret_cast<uint4*>(ap + (((c0 / 4 + q) ^ (r & 7)) << 4)) = make_uint4(h[0], h[1], h[2], h[3]);
            }
        };
        // Tile i: fixed point, then its planes as the planes of tile i - BUF retire.
        auto put = [&](uint32_t (&X)[W], uint32_t i, uint32_t e) -> bool {
            bool planes;
            if (!convert(X, i, e, planes)) return false;
#pragma unroll
            for (int g = 0; g < GROUPS; ++g) {
                if (i >= BUF && !wait(done(buf(i), g), par(i - BUF))) return false;
#pragma unroll
                for (int s = g ? C::group_end(g - 1) : 0; s < C::group_end(g); ++s)
                    if (planes) store_plane(X, s, buf(i));
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(full(buf(i)));
            return true;
        };
        if constexpr (DBL) {
            uint32_t X[W];
            for (uint32_t i = 0; i < m; ++i) {
                load_tile(X, tile(i));
                if (!put(X, i, span(X))) { bad = true; break; }
            }
        } else {  // one tile ahead in registers
            uint32_t XA[W], XB[W];
            if (m > 0) load_tile(XA, tile(0));
            for (uint32_t i = 0; i < m; i += 2) {
                const uint32_t ea = span(XA);
                if (i + 1 < m) load_tile(XB, tile(i + 1));
                if (!put(XA, i, ea)) { bad = true; break; }
                if (i + 1 >= m) break;
                const uint32_t eb = span(XB);
                if (i + 2 < m) load_tile(XA, tile(i + 2));
                if (!put(XB, i + 1, eb)) { bad = true; break; }
            }
        }
        if (bad && lane == 0) atomicOr(err, DEVERR_TIMEOUT);
    } else {
        // ---- output: sum the digit positions, convert back, store ----
        if constexpr (DBL) asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" :: "n"(Cfg<double>::kRegOut));
        const int c0 = CPO * ((warp - kIn) >> 2);
        const volatile uint64_t* vCol = sCol + c0;
        T* const prow = psi + deposit((uint64_t)r, a.rpos, kRowBits);
        const uint32_t trow = tbase + ((uint32_t)(quad * 32) << 16) + 2 * c0;
        // whether every |D_d| <= 2^22: the digits of X are at most 128, so the sum of a row of U's bounds them
        [[maybe_unused]] const bool bounded = !__any_sync(0xffffffffu, max(sums[lane], sums[lane + 32]) > (1 << 15));
        auto finish = [&](uint32_t i) {  // the accumulators have been read
            fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(freed(buf(i)));
        };
        // The rows of the quadrant that the slices do not take, shared out among its warps.
        bool have_u = false;
        [[maybe_unused]] uint32_t met = 0;
        auto quad_rows = [&](uint32_t mask, uint64_t at) -> bool {
            if (mask == 0) return true;
            if (!have_u && !wait(bbar, 0)) return false;
            have_u = true;
            uint32_t mine = 0;
            int rank = 0;
            for (; mask; mask &= mask - 1, ++rank)
                if (rank / C::ROWS % (kOut / 4) == ((warp - kIn) >> 2)) mine |= mask & (0u - mask);
            rows_by_fma<R, C::ROWS>(psi, a, C::U > 0 ? sU : umat, sX + (warp - kIn) * (C::ROWS * D), sCol[lane], mine, at);
            return true;
        };
        for (uint32_t i = 0; i < m; ++i) {
            const uint32_t td = trow + buf(i) * 64 * ND;
            const uint64_t tb = insert_zeros(tile(i), a.spos, a.nS);
            T* const pt = prow + tb;
            if constexpr (DBL) {
                // Y = sum_d D_d 2^(46 - 8d), the last two positions together and rounded; y = Y 2^(E - 1080).
                // The integers come as q + kMagic: the bits of D + 1.5 2^23 where |D| <= 2^22, else by conversion
                // (on the XU unit, which would bound this kernel); Y starts at what that adds.
                constexpr uint32_t kMagic = 0x4B400000u;
                constexpr int64_t kOff = (int64_t)kMagic * ((1ll << 30) + (1ll << 22) + (1ll << 14) + (1ll << 6));
                constexpr uint64_t kY0 = 0ull - (uint64_t)kOff - ((uint64_t)((kMagic << 14) + (kMagic << 6)) << 32);
                int64_t Y[2 * CPO];
                int E = 0;
                uint32_t mask = 0;  // the quadrant's rows that are not in the accumulators
#pragma unroll
                for (int g = 0; g < GROUPS; ++g) {
                    if (!wait(done(buf(i), g), par(i))) { bad = true; break; }
                    if (g == 0) {
                        E = sRow[i % row_slots<R>() * 128 + r];
                        mask = __ballot_sync(0xffffffffu, E & kByFma);
                        E &= ~kAllFma;
                    }
                    if (mask == 0xffffffffu) continue;
#pragma unroll
                    for (int c = 0; c < 2 * CPO; c += 8) {
                        uint32_t v[8], v2[8];
                        tmem_ld<8>(td + 64 * (2 * g) + c, v);
                        tmem_ld<8>(td + 64 * (2 * g + 1) + c, v2);
                        wait_ld();
                        if (bounded) {
#pragma unroll
                            for (int j = 0; j < 8; ++j) {
                                v[j] = __float_as_uint(__fadd_rn(__uint_as_float(v[j]), 12582912.0f));
                                v2[j] = __float_as_uint(__fadd_rn(__uint_as_float(v2[j]), 12582912.0f));
                            }
                        } else {
#pragma unroll
                            for (int j = 0; j < 8; ++j) {
                                v[j] = (uint32_t)__float2int_rn(__uint_as_float(v[j])) + kMagic;
                                v2[j] = (uint32_t)__float2int_rn(__uint_as_float(v2[j])) + kMagic;
                            }
                        }
#pragma unroll
                        for (int j = 0; j < 8; ++j) {
                            if (g == 0) {
                                const uint32_t h = (v[j] << 14) + (v2[j] << 6) + (uint32_t)(kY0 >> 32);
                                Y[c + j] = (int64_t)(((uint64_t)h << 32) | (uint32_t)kY0);
                            } else if (g < 3) {
                                asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(Y[c + j]) : "r"(v[j]), "r"(a.w[2 * g - 2]));
                                asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(Y[c + j]) : "r"(v2[j]), "r"(a.w[2 * g - 1]));
                            } else {
                                Y[c + j] += (int32_t)((v[j] << 8) + v2[j] + (512u - (kMagic << 8) - kMagic)) >> 10;
                            }
                        }
                    }
                }
                if (bad) break;
                finish(i);
#pragma unroll
                for (int j = 0; j < CPO; j += VEC) {
                    uint32_t w[VEC * AW];
#pragma unroll
                    for (int k = 0; k < 2 * VEC; ++k) {
                        if (((2 * j + k) & 3) == 0) to_double_int(Y[2 * j + k], E, w[2 * k], w[2 * k + 1]);
                        else to_double_cvt(Y[2 * j + k], E, w[2 * k], w[2 * k + 1]);
                    }
                    if (E < kByFma && own) st_words<VEC * AW>(pt + vCol[j], w);
                }
                if (!quad_rows(mask, (uint64_t)(pt - psi))) { bad = true; break; }
            } else {
                // y = 2^(E - 138) sum_d D_d 2^(-8d)
                if (!wait(done(buf(i), 0), par(i))) { bad = true; break; }
                const int row = sRow[i % row_slots<R>() * 128 + r], E = row & kExponent;
                const uint32_t mask = __ballot_sync(0xffffffffu, row & kByFma);
                if (mask) {  // by FMAs first: then no warp needs the input of these rows any more
                    bool ok = quad_rows(mask, (uint64_t)(pt - psi));
                    __syncwarp();
                    if (lane == 0) mbar_arrive(fmabar(quad));
                    ok = wait(fmabar(quad), met++ & 1) && ok;
                    if (!ok) { bad = true; break; }
                }
                const float sc = __uint_as_float((uint32_t)(E - 11) << 23);
#pragma unroll
                for (int c = 0; c < 2 * CPO; c += 8) {
                    uint32_t v[4][8], w[8];
#pragma unroll
                    for (int d = 0; d < 4; ++d) tmem_ld<8>(td + 64 * d + c, v[d]);
                    wait_ld();
                    if (c + 8 == 2 * CPO) finish(i);
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        float y = __uint_as_float(v[3][j]);
                        y = __fmaf_rn(y, 0x1p-8f, __uint_as_float(v[2][j]));
                        y = __fmaf_rn(y, 0x1p-8f, __uint_as_float(v[1][j]));
                        y = __fmaf_rn(y, 0x1p-8f, __uint_as_float(v[0][j]));
                        w[j] = __float_as_uint(y * sc);
                    }
                    if (row < kByFma && own) {
#pragma unroll
                        for (int j = 0; j < 4; j += VEC) st_words<VEC * AW>(pt + vCol[c / 2 + j], w + 2 * j);
                    } else if (row < kAllFma && own) {
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            if ((int)(max(w[2 * j] & 0x7FFFFFFFu, w[2 * j + 1] & 0x7FFFFFFFu) >> 23) + kLarge >= E)
                                st_words<AW>(pt + vCol[c / 2 + j], w + 2 * j);
                    }
                }
            }
        }
        if (bad && lane == 0) atomicOr(err, DEVERR_TIMEOUT);
    }
    fence_before();
    __syncthreads();
    if (warp == 0) {
        fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tbase), "r"(TCOLS) : "memory");
    }
}

// The digit planes of U (x I on the padding columns): real form B[2i][2c] = Re U_ic, B[2i][2c+1] = -Im U_ic,
// B[2i+1][2c] = Im U_ic, B[2i+1][2c+1] = Re U_ic in fixed point, plane t = digit t (most significant first).
// After the planes: the sum of |digits| over all planes of each row (64 integers); for each complex row of U x I the columns
// whose entry has a part of at least 2^-7, of at least 2^-4, and other than zero (32 words each); U itself by columns in the state's
// precision. One block per row n.
template <typename R>
__global__ void __launch_bounds__(NR) k_tcx_prepare(const double* __restrict__ U, int k, unsigned char* __restrict__ out) {
    using C = Cfg<R>;
    const int Du = 1 << k, n = blockIdx.x, kk = threadIdx.x, i = n >> 1, c = kk >> 1;
    __shared__ int total[2];
    double v = 0.0;
    if ((i >> k) == (c >> k)) {
        const int e = 2 * ((i & (Du - 1)) * Du + (c & (Du - 1)));
        v = (n & 1) == (kk & 1) ? U[e] : ((n & 1) ? U[e + 1] : -U[e + 1]);
        if (i < Du && c < Du && !(n & 1) && !(kk & 1)) {
            typename Amp<R>::T u;
            u.x = (R)U[e];
            u.y = (R)U[e + 1];
            reinterpret_cast<typename Amp<R>::T*>(out + C::S * kPlaneB + 4 * (NR + 3 * D))[c * Du + i] = u;
        }
    }
    // thread kk of row 2 i has a part of U_ic (c = kk / 2); of the two, the larger counts
    const double part = fmax(fabs(v), fabs(__shfl_xor_sync(0xffffffffu, v, 1)));
    __shared__ uint32_t large[3][2];
    for (int l = 0; l < 3; ++l) {
        const uint32_t b = __ballot_sync(0xffffffffu, l == 2 ? part != 0.0 : part >= (l ? 0x1p-4 : 0x1p-7));
        if ((kk & 31) == 0) large[l][kk >> 5] = b;
    }
    const uint64_t f = (uint64_t)__double2ll_rn(scalbn(v, C::kStepsU)) + (sizeof(R) == 8 ? 0x0080808080808080ull : 0x80808080ull);
    const uint32_t off = sw128_offset(n, kk, NR, 2);
    int sum = 0;
    for (int t = 0; t < C::S; ++t) {
        const int b = (int)((f >> (8 * (C::S - 1 - t))) & 0xFF) - 128;
        sum += b < 0 ? -b : b;
        *reinterpret_cast<__half*>(out + t * kPlaneB + off) = __int2half_rn(b);
    }
    sum = __reduce_add_sync(0xffffffffu, sum);
    if ((kk & 31) == 0) total[kk >> 5] = sum;
    __syncthreads();
    int* const tail = reinterpret_cast<int*>(out + C::S * kPlaneB);
    if (kk == 0) tail[n] = total[0] + total[1];
    if (kk < 3 && !(n & 1)) {
        uint32_t m = 0;
        for (int c = 0; c < D; ++c) m |= (large[kk][c >> 4] >> (2 * (c & 15)) & 1u) << c;
        tail[NR + D * kk + i] = (int)m;
    }
}

}  // namespace tcx

bool tcx_supported(int n, int k) { return k >= 1 && k <= tcx::K && n >= tcx::K + tcx::kRowBits && n <= 43; }

size_t tcx_operand_bytes(int dtype) {
    return (size_t)tcx::kPlaneB * (dtype == QSIM_C64 ? tcx::Cfg<float>::S : tcx::Cfg<double>::S) + sizeof(int) * (tcx::NR + 3 * tcx::D) +
           (size_t)(dtype == QSIM_C64 ? sizeof(float2) : sizeof(double2)) * tcx::D * tcx::D;
}

cudaError_t launch_tcx_prepare(int dtype, const double* dU, int k, void* dB, cudaStream_t s) {
    if (k < 1 || k > tcx::K) return cudaErrorInvalidValue;
    unsigned char* out = static_cast<unsigned char*>(dB);
    if (dtype == QSIM_C64) tcx::k_tcx_prepare<float><<<tcx::NR, tcx::NR, 0, s>>>(dU, k, out);
    else tcx::k_tcx_prepare<double><<<tcx::NR, tcx::NR, 0, s>>>(dU, k, out);
    return cudaGetLastError();
}

cudaError_t launch_tcx_apply(int dtype, void* psi, int n, int k, const int* targets, const void* dB, unsigned* dev_err,
                             cudaStream_t s, const DevInfo& d, const uint64_t* from_basis, bool digits) {
    const uintptr_t addr = reinterpret_cast<uintptr_t>(psi);
    if (!tcx_supported(n, k) || (reinterpret_cast<uintptr_t>(dB) & 15) != 0 || (addr & 15) != 0) return cudaErrorInvalidValue;
    tcx::Args a;
    std::memset(&a, 0, sizeof(a));
    uint64_t tmask = 0;
    for (int j = 0; j < k; ++j) {
        if (targets[j] < 0 || targets[j] >= n || ((tmask >> targets[j]) & 1)) return cudaErrorInvalidValue;
        a.tpos[j] = targets[j];
        tmask |= 1ull << targets[j];
    }
    for (int q = n - 1, j = k; j < tcx::K; --q)  // padding: the highest idle qubits
        if (!((tmask >> q) & 1)) {
            a.tpos[j++] = q;
            tmask |= 1ull << q;
        }
    int nr = 0;
    for (int q = 0; q < n && nr < tcx::kRowBits; ++q)
        if (!((tmask >> q) & 1)) a.rpos[nr++] = q;
    uint64_t smask = tmask;
    for (int j = 0; j < tcx::kRowBits; ++j) smask |= 1ull << a.rpos[j];
    for (int q = 0; q < n; ++q)
        if ((smask >> q) & 1) a.spos[a.nS++] = q;
    a.k = k;
    a.digits = digits;
    a.ntiles = 1ull << (n - a.nS);
    if (a.ntiles >> 32) return cudaErrorInvalidValue;  // 32-bit tile counters in the kernel
    if (from_basis) {
        a.from_basis = 1;
        a.basis = *from_basis;
    }
    for (int j = 0; j < 4; ++j) a.w[j] = 1 << (30 - 8 * j);
    // Fewer tiles than SMs: several CTAs share a tile, each for a part of its rows, so that rows by FMAs are spread (9-step TFIM
    // chains of small angles in complex128, 17 / 18 qubits: 0.83 -> 0.41, 0.97 -> 0.62 ms; random states level).
    while (a.split < 3 && (a.ntiles << (a.split + 1)) <= (uint64_t)d.num_sms) ++a.split;
    auto launch = [&](auto kern, auto* p, int threads, size_t smem) -> cudaError_t {
        cudaError_t e = smem_optin(reinterpret_cast<const void*>(kern), (int)smem);
        if (e != cudaSuccess) return e;
        // programmatic dependent launch, as for the other block kernels (griddepcontrol.wait before any access)
        cudaLaunchConfig_t cfg{};
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.gridDim = dim3((unsigned)std::min<uint64_t>((uint64_t)d.num_sms, a.ntiles) << a.split, 1, 1);
        cfg.blockDim = dim3((unsigned)threads, 1, 1);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = s;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        return cudaLaunchKernelEx(&cfg, kern, p, a, reinterpret_cast<const uint4*>(dB), dev_err);
    };
    using namespace tcx;
    if (dtype == QSIM_C64) {
        float2* p = reinterpret_cast<float2*>(psi);
        constexpr size_t sm = smem_bytes<float>();
        constexpr int th = threads<float>();
        if (a.tpos[0] == 0 && a.tpos[1] == 1 && (addr & 31) == 0) return launch(k_tcx_block<float, kQuads>, p, th, sm);
        if (a.tpos[0] == 0) return launch(k_tcx_block<float, kPairs>, p, th, sm);
        return launch(k_tcx_block<float, kRows>, p, th, sm);
    }
    double2* p = reinterpret_cast<double2*>(psi);
    constexpr size_t sm = smem_bytes<double>();
    constexpr int th = threads<double>();
    if (a.tpos[0] == 0 && (addr & 31) == 0) return launch(k_tcx_block<double, kPairs>, p, th, sm);
    return launch(k_tcx_block<double, kRows>, p, th, sm);
}

}  // namespace qsim
