// FP64-accurate per-mode contraction on the tensor cores: fixed-point bf16
// slices with exact FP32 accumulation (Ozaki's error-free splitting of a dot
// product), for plans with several right-hand sides.
//
// The operation is the one of the other forms (Sec. 3.2, Eqs. 37-38 in the mode
// domain): for every mode k >= 1, pad column a and output component co,
//     U_co(a, n) = sum_{ci, b} M_{co ci}(x_a - x_b) X_ci(b, n),
// n over the x and y' halves of the right-hand sides.  Exactness comes from
// three facts:
//   * every operand value v is scaled by a power of two to |v'| < 1/2 and cut
//     into six slices t_1 .. t_6, t_i an integer of at most 8 bits times
//     2^(-8 i) (round to nearest, so the slices after the first are at most 128
//     units); six slices hold v' to 2^-49;
//   * the product of two slices is exact in FP32 (16 significant bits), and all
//     products t_i s_j with the same i + j = q lie on the grid 2^(-8 q);
//   * an FP32 accumulator that only ever adds values of one grid is exact while
//     the sum stays below 2^24 grid units.  With 192 terms per group (64
//     interface columns x 3 components) and at most q - 1 products of at most
//     2^14 units per term, the diagonals q = 2 .. 5 stay exact in the worst case.
// The 26 slice products with i, j <= 6 and i + j <= 8 are kept.  Diagonals 2, 3,
// 4 and 5 have an accumulator each in tensor memory; 6, 7 and 8 (about 2^-31 of
// the result) share a fifth, whose rounding stays near 2^-54 of the result.  The
// group's five sums are combined in double-float arithmetic, scaled back and
// added to a running double-float sum per output.  What is left out -- slices
// beyond the sixth and products with i + j > 8 -- is about 2^-47 of the largest
// operand product, per term.
//
// Scales: all table entries of a (pad tile, interface tile) pair share 2^E, the
// smallest power of two above twice their largest magnitude over the pair's
// 128 x 64 entries (of the CTA's three reals), so every cell of the pair's table
// sub-box is cut into slices once; the force column n of mode k shares 2^F(k, n),
// found by a reduction before the split.  Row and column scales factor out of the
// GEMM exactly.
//
// A CTA owns 128 pad columns (the GEMM rows, one tensor-memory lane each), one
// output component co, one mode and 32 right-hand sides (N = 64), and walks the
// interface columns tile by tile (64 columns, one accumulation group), in stages
// of 16:
//   * four slicer warps work a tile ahead: they load the CTA's three reals of the
//     tile pair's double-float sub-box into registers, find the pair's scale and
//     cut each cell into 18 bf16 slices in one of two shared-memory buffers;
//   * per stage, two groups of four builder warps in turn gather the slices of the
//     co-th row of M, (M_{co 0}, M_{co 1}, M_{co 2}), and store them into tensor memory
//     one input component at a time (3 x 6 blocks of 128 x 16 bf16), each handed over by
//     its own barrier pair, so the stores of one component overlap the products of
//     the others;
//   * one thread streams the force operand, split once per apply (3 x 6 blocks
//     of 64 x 16 bf16 per stage, 36 KB), with bulk copies into a ring of stages;
//   * one warp (an elected lane) issues the 3 x 26 products (M = 128, N = 64, K = 16) per stage
//     into the five accumulators, neighbouring ones as one tcgen05.mma of N up to 256;
//   * at the start of every tile the builders drain the previous tile's group
//     into their running double-float sums.
// Tensor memory: 5 x 64 accumulator columns and 18 x 8 columns of A: 464 of 512.
// What bounds it: the 312 products of a tile take 9984 SM cycles at the tensor pipe's rate, and the pipe waits at
// the end of a tile for the drain (the accumulators are single), slows for the tensor-memory stores of A and the
// shared-memory traffic of gathers and slicers, and takes about 14000 (ncu: tensor pipe 71 % active, DRAM traffic
// the algorithmic bytes).  4000 x 6000 columns, L = 256, 64 right-hand
// sides: 188 ms with builders that also staged and cut the sub-boxes and products issued one by one from a single
// thread's branch, 144 ms with elected issue, 109 ms in this form.
// The mode k = 0 stays with the double-float kernel, as in the other tensor forms.
//
// Every wait is bounded as in the other tensor-core kernel: pipeline waits give
// up after the plan's wait limit or once another role gave up; the waits for a
// CTA's own bulk copies and products in flight keep the full bound; a stopped CTA
// records the status word, frees its tensor memory and returns.
#include <cuda_bf16.h>

#include <algorithm>

#include "fbc_f32x2.cuh"
#include "fbc_internal.cuh"
#include "fbc_tc.cuh"

namespace fbc {
namespace {

constexpr int kTmemCols = 512;
constexpr int kRows = kTileA;        // GEMM rows (pad columns) per CTA
constexpr int kRhs = 32;             // right-hand sides per CTA
constexpr int kN = 2 * kRhs;         // GEMM columns: (x, y') of each right-hand side
constexpr int kKC = 16;              // interface columns per stage (the bf16 MMA's K)
constexpr int kStages = kTileB / kKC;  // stages per interface tile = per accumulation group
constexpr int kNS = 6;               // slices per operand value
constexpr int kNQ = 5;               // accumulators: diagonals q = 2, 3, 4, 5 and q >= 6 together
constexpr int kNPair = 26;           // slice products with i, j <= 6 and i + j <= 8
constexpr int kBuilderWarps = 8;
constexpr int kSlicerWarp = 8, kSlicers = 4 * 32;  // warps 8 .. 11
constexpr int kMmaWarp = 12, kCopyWarp = 13;        // (14 and 15 fill up their warpgroup)
constexpr int kThreads = 16 * 32;
// Registers per thread: the block is launched with 128 each; the MMA and copy warps' group gives 80 up, the two
// builder groups take 40 more each (256 x 168 + 128 x 128 + 128 x 48 = 512 x 128).
constexpr int kBuilderRegs = 168, kIssueRegs = 48;
constexpr int kSlots = 9;            // force-operand ring at most, in slots of one input component of a stage
constexpr int kMinSlots = 6;
constexpr int kPitchSpan = 16;       // row pitches of a cut sub-box tried, from its width up
constexpr int kMaxCells = 1880;      // largest table sub-box of a tile pair
constexpr uint32_t kAcol = kNQ * kN;                     // first TMEM column of the A blocks (after 5 x 64)
constexpr uint32_t kAcols = 3 * kNS * 8;                 // TMEM columns of the A blocks (18 blocks of 128 x 16 bf16)
static_assert(kAcol + kAcols <= kTmemCols, "tensor memory");
constexpr uint32_t kBBlk = (uint32_t)kN * kKC * 2;       // one (ci, slice) block of a force chunk: 2 KB
constexpr uint32_t kSlot = kNS * kBBlk;                  // one input component of a stage of the force operand: 12 KB
constexpr uint32_t kChunk = 3u * kSlot;                  // one stage: 36 KB
constexpr uint32_t kSBO = (kKC / 8) * 128;               // 8-row group stride of a [rows][16] bf16 block
constexpr uint32_t kSleepNs = 200;  // suspend hint of the copy thread's waits and the MMA thread's force waits
constexpr int kEmin = -120, kEmax = 120;                 // clamp of the scale exponents (2^E a normal float)

// Entry of M(d) in row co, column ci, as (index into the six table reals, sign):
// M = [[A11, A12, -B13], [A12, A22, -B23], [B13, B23, A33]], reals (A11, A12, A22, A33, B13, B23).
__host__ __device__ constexpr int oz_real(int co, int ci) {
    return co == 0 ? (ci == 0 ? 0 : ci == 1 ? 1 : 4) : co == 1 ? (ci == 0 ? 1 : ci == 1 ? 2 : 5) : (ci == 0 ? 4 : ci == 1 ? 5 : 3);
}
__host__ __device__ constexpr bool oz_neg(int co, int ci) { return ci == 2 && co < 2; }

// The slice products, as issued for one input component: instruction p multiplies A slice oz_i(p) with the oz_n(p)
// neighbouring B slices from oz_j(p) on (1-based), 64 GEMM columns each, into the neighbouring accumulators from
// oz_acc(p) on: A slice i times B slices 1 .. 6 - i lands on the diagonals i + 1 .. 6, which lie side by side.
// 17 instructions for the 26 products.  An instruction takes about 33 cycles to issue, a product 32 in the tensor
// pipe, and eight fit its queue: issued one product at a time the pipe ran dry at every hand-over (164 cycles of
// waits a component); the wide ones go last, so the queue covers the next component's waits.
constexpr int kNInst = 17;
__host__ __device__ constexpr int oz_i(int p) {
    constexpr int v[kNInst] = {1, 1, 1, 2, 2, 3, 3, 4, 4, 5, 5, 6, 6, 5, 4, 3, 2};
    return v[p];
}
__host__ __device__ constexpr int oz_j(int p) {
    constexpr int v[kNInst] = {1, 4, 6, 5, 6, 4, 5, 3, 4, 2, 3, 1, 2, 1, 1, 1, 1};
    return v[p];
}
__host__ __device__ constexpr int oz_n(int p) {
    constexpr int v[kNInst] = {3, 2, 1, 1, 1, 1, 1, 1, 1, 1, 1, 1, 1, 1, 2, 3, 4};
    return v[p];
}
__host__ __device__ constexpr int oz_acc(int p) { return (oz_i(p) + oz_j(p) < 6 ? oz_i(p) + oz_j(p) : 6) - 2; }
// every product with i, j <= 6 and i + j <= 8 once, on its own accumulator; the first two overwrite all five
constexpr bool oz_products_ok() {
    int seen[7][7] = {};
    for (int p = 0; p < kNInst; p++)
        for (int u = 0; u < oz_n(p); u++) {
            const int i = oz_i(p), j = oz_j(p) + u, q = i + j;
            if (j > 6 || q > 8 || seen[i][j]++) return false;
            if (oz_acc(p) + u != (q < 6 ? q : 6) - 2) return false;
        }
    int n = 0;
    for (int i = 1; i <= 6; i++)
        for (int j = 1; j <= 6; j++) n += seen[i][j];
    return n == kNPair && oz_acc(0) == 0 && oz_n(0) == oz_acc(1) && oz_acc(1) + oz_n(1) == kNQ;
}
static_assert(oz_products_ok(), "slice products");

// Six fixed-point slices of v' = (hi + lo) s, |v'| < 1/2, s a power of two: t_i is v's remainder
// rounded to the grid 2^(-8 i) (add and subtract 1.5 x 2^(23 - 8 i)).  hi s - t_1 and the later
// remainders are exact; only lo s joins with a rounding, of at most 2^-49.
__device__ __forceinline__ void oz_split(float hi, float lo, float s, float (&t)[kNS]) {
    const float C1 = 49152.0f, C2 = 192.0f, C3 = 0.75f;
    const float C4 = 0.0029296875f, C5 = 1.1444091796875e-05f, C6 = 4.470348358154297e-08f;
    t[0] = __fsub_rn(__fmaf_rn(hi, s, C1), C1);
    float r = __fmaf_rn(hi, s, -t[0]);
    t[1] = __fsub_rn(__fadd_rn(r, C2), C2);
    r = __fsub_rn(r, t[1]);
    t[2] = __fsub_rn(__fadd_rn(r, C3), C3);
    r = __fsub_rn(r, t[2]);
    r = __fmaf_rn(lo, s, r);
    t[3] = __fsub_rn(__fadd_rn(r, C4), C4);
    r = __fsub_rn(r, t[3]);
    t[4] = __fsub_rn(__fadd_rn(r, C5), C5);
    r = __fsub_rn(r, t[4]);
    t[5] = __fsub_rn(__fadd_rn(r, C6), C6);
}

// 2^-E as a float and the exponent E of a magnitude bound m: the smallest power of two above 2 m
// (|v| <= m gives |v 2^-E| < 1/2), clamped to [kEmin, kEmax].
__device__ __forceinline__ int oz_exp_of(float m) {
    const int e = (int)((__float_as_uint(m) >> 23) & 0xffu) - 127;  // floor(log2 m) (m = 0: -127)
    return min(max(e + 2, kEmin), kEmax);
}
__device__ __forceinline__ float oz_pow2(int e) { return __uint_as_float((uint32_t)(127 + e) << 23); }


// ---- force operand: scales and slices (once per apply) ----------------------

// Scale exponent F(k, n) of every force column (right-hand side r, half h) of modes k0 .. k0 + n_modes - 1:
// one block per (mode, rhs), the largest |fh| of the half over the interface columns and its three
// components, compared as the integer bits of the magnitudes.  fexp[(r K + k) 2 + h].
__global__ void __launch_bounds__(256) k_oz_fscale(const double* __restrict__ fh, int K, int NIpad, int k0,
                                                   int* __restrict__ fexp) {
    const int k = k0 + (int)blockIdx.x, r = (int)blockIdx.y;
    const double* src = fh + ((size_t)r * K + k) * NIpad * 6;
    unsigned long long m0 = 0ull, m1 = 0ull;  // halves x (entries 0..2) and y' (3..5)
    for (int i = threadIdx.x; i < NIpad * 3; i += blockDim.x) {  // one double2 per step: entries 2j, 2j + 1
        const double2 v = ((const double2*)src)[i];
        const int j = i % 3;
        const unsigned long long a = (unsigned long long)__double_as_longlong(v.x) & 0x7fffffffffffffffull;
        const unsigned long long b = (unsigned long long)__double_as_longlong(v.y) & 0x7fffffffffffffffull;
        if (j == 0) m0 = max(m0, max(a, b));
        else if (j == 1) m0 = max(m0, a), m1 = max(m1, b);
        else m1 = max(m1, max(a, b));
    }
    const unsigned long long m[2] = {m0, m1};
    __shared__ unsigned long long s_m[2][8];
#pragma unroll
    for (int h = 0; h < 2; h++) {
        unsigned long long v = m[h];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
        if (threadIdx.x % 32 == 0) s_m[h][threadIdx.x / 32] = v;
    }
    __syncthreads();
    if (threadIdx.x < 2) {
        const int h = threadIdx.x;
        unsigned long long v = 0ull;
        for (int w = 0; w < (int)blockDim.x / 32; w++) v = max(v, s_m[h][w]);
        const int e = (int)((v >> 52) & 0x7ffull) - 1023;  // floor(log2 max) (max = 0: -1023)
        fexp[((size_t)r * K + k) * 2 + h] = min(max(e + 2, kEmin), kEmax);
    }
}

// Chunk of the sliced force operand for (k, rhs group g, interface tile tB, stage st).
__host__ __device__ __forceinline__ size_t oz_chunk(int k, int g, int tB, int st, int G, int n_tb) {
    return (((size_t)k * G + g) * n_tb + tB) * kStages + st;
}

// One thread per (mode, rhs group g < Gu, tile, stage, rhs r of the group, core column kc): the eight interface
// columns b0 .. b0 + 7 of both halves and all three components of right-hand side r, each cut into six
// slices at its column's scale, stored as 16-byte core rows of the K-major blocks (ci, slice) of the
// chunk, GEMM column n = 2 r + h.  Right-hand sides at or beyond n_rhs are zero.
__global__ void __launch_bounds__(256) k_oz_prep(const double* __restrict__ fh, const int* __restrict__ fexp, int K,
                                                 int NIpad, int n_tb, int G, int Gu, int n_rhs, int k0, int n_modes,
                                                 unsigned char* __restrict__ out) {
    const size_t total = (size_t)n_modes * Gu * n_tb * kStages * kRhs * 2;
    for (size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (size_t)gridDim.x * blockDim.x) {
        const int kc = (int)(t & 1), rl = (int)((t >> 1) % kRhs);
        size_t q = t / (2 * kRhs);
        const int st = (int)(q % kStages);
        q /= kStages;
        const int tB = (int)(q % n_tb);
        q /= n_tb;
        const int g = (int)(q % Gu);
        const int k = k0 + (int)(q / Gu);
        const int r = g * kRhs + rl;
        const int b0 = tB * kTileB + st * kKC + kc * 8;
        unsigned char* chunk = out + oz_chunk(k, g, tB, st, G, n_tb) * kChunk;
        const double* src = fh + (((size_t)r * K + k) * NIpad + b0) * 6;
#pragma unroll
        for (int h = 0; h < 2; h++) {
            const int n = 2 * rl + h;
            const float s = r < n_rhs ? oz_pow2(-fexp[((size_t)r * K + k) * 2 + h]) : 0.0f;
            const uint32_t off = (uint32_t)(n / 8) * kSBO + (uint32_t)kc * 128u + (uint32_t)(n % 8) * 16u;
#pragma unroll
            for (int ci = 0; ci < 3; ci++) {
                uint32_t w[kNS][4];
#pragma unroll
                for (int i = 0; i < 4; i++) {
                    float t2[2][kNS];
#pragma unroll
                    for (int u = 0; u < 2; u++) {
                        const double x = r < n_rhs ? src[(size_t)(2 * i + u) * 6 + 3 * h + ci] : 0.0;
                        const float hi = d2f_int(x);
                        const float lo = d2f_int(x - f2d_int(hi));
                        oz_split(hi, lo, s, t2[u]);
                    }
#pragma unroll
                    for (int p = 0; p < kNS; p++)
                        asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(w[p][i]) : "f"(t2[1][p]), "f"(t2[0][p]));
                }
#pragma unroll
                for (int p = 0; p < kNS; p++)
                    *(uint4*)(chunk + (size_t)(ci * kNS + p) * kBBlk + off) = make_uint4(w[p][0], w[p][1], w[p][2], w[p][3]);
            }
        }
    }
}

// ---- the contraction --------------------------------------------------------

struct OzArgs {
    ContractArgs A;              // table (double-float), uh, geometry; A.k0 = first mode of the launch
    const unsigned char* bprep;  // sliced force operand, chunks oz_chunk(k, g, tB, st)
    const int* fexp;             // force column scale exponents [rhs][K][2]
    int n_rhs, G;                // rhs applied, rhs groups of the buffer's layout
    int slots;                   // force-operand ring
    const int* off;              // [NIpad] x_b + pitch * y_b of the sorted interface sites
    const int* row;              // [NPpad] pad slot of each GEMM row
    int pitch;                   // cells per row of a cut sub-box
};

struct OzSync {
    uint64_t bfull[kSlots], empty[kSlots], done, drained, afull[3], aempty[3];  // A: one barrier pair per input component
    uint64_t slfull[2], slempty[2];  // the two buffers of cut sub-boxes: slicers -> builders and back
    int E[2];                        // their tile pairs' scale exponents
    uint32_t wmax[4];
    uint32_t tbase;
    volatile int abort;
};

// oz_split on two values at once: (hi, lo) pairs of two values, s a pair of powers of two.
__device__ __forceinline__ void oz_split2(uint64_t hi, uint64_t lo, uint64_t s, uint64_t (&t)[kNS]) {
    const uint64_t C1 = pk2(49152.0f, 49152.0f), C2 = pk2(192.0f, 192.0f), C3 = pk2(0.75f, 0.75f);
    const uint64_t C4 = pk2(0.0029296875f, 0.0029296875f), C5 = pk2(1.1444091796875e-05f, 1.1444091796875e-05f);
    const uint64_t C6 = pk2(4.470348358154297e-08f, 4.470348358154297e-08f);
    const uint64_t m = mul2(hi, s);  // exact: s is a power of two
    t[0] = sub2(add2(m, C1), C1);
    uint64_t r = sub2(m, t[0]);
    t[1] = sub2(add2(r, C2), C2);
    r = sub2(r, t[1]);
    t[2] = sub2(add2(r, C3), C3);
    r = sub2(r, t[2]);
    r = fma2(lo, s, r);
    t[3] = sub2(add2(r, C4), C4);
    r = sub2(r, t[3]);
    t[4] = sub2(add2(r, C5), C5);
    r = sub2(r, t[4]);
    t[5] = sub2(add2(r, C6), C6);
}

__device__ __forceinline__ uint32_t cvt_bf16x2(float hi, float lo) {
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}

// FastTwoSum on pairs: s + e == a + b exactly, per lane, where a is a multiple of b's unit in the last place.
__device__ __forceinline__ void fast_two_sum2(uint64_t a, uint64_t b, uint64_t& s, uint64_t& e) {
    s = add2(a, b);
    e = sub2(b, sub2(s, a));
}

// Running double-float sums of two outputs: (H, L) += the five accumulator sums d[0..4] of a group (pairs:
// diagonals 2, 3, 4, 5 and 6-8), at the group's scale sc.  d2 + d3 + d4 by two-sums: a diagonal's sum is below
// 2^24 units of its grid 2^(-8 q), so its last place is at most the grid of the diagonal before, which the
// running sum is a multiple of, and the three-operation form is exact.  The rest, below 2^-23 of the total,
// joins the low word.  The scale is a power of two: the products s sc in the fused operations are exact.
// 17 packed operations (two cycles each on the FP32 pipe): a drain of 128 x 64 outputs is bound by them.
__device__ __forceinline__ void oz_accumulate2(const uint64_t (&d)[kNQ], uint64_t sc, uint64_t& H, uint64_t& L) {
    uint64_t s, e, s2, e2;
    fast_two_sum2(d[0], d[1], s, e);
    fast_two_sum2(s, d[2], s2, e2);
    const uint64_t l = add2(add2(add2(e, e2), d[3]), d[4]);
    const uint64_t h = fma2(s2, sc, H);  // Knuth's two-sum of H and s2 sc
    const uint64_t nb = sub2(H, h);
    const uint64_t t = add2(sub2(H, add2(h, nb)), fma2(s2, sc, nb));
    H = h;
    L = add2(L, fma2(l, sc, t));
}

// NC: sub-box cells per slicer thread (kSlicers NC >= W H).
template <int NC>
__global__ void __launch_bounds__(kThreads, 1) k_contract_oz(OzArgs O, int wl, int* status) {
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ OzSync sy;
    const ContractArgs& A = O.A;
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const int co = (int)blockIdx.x % 3, tA = (int)blockIdx.x / 3;
    const int k = A.k0 + (int)blockIdx.y, g = (int)blockIdx.z;
    const int n_it = A.n_tb * kStages;
    const int HW = A.H * A.W;
    const int slots = O.slots, HP = A.H * O.pitch;
    unsigned char* sB = smem;                                     // [slots][kSlot]
    int* s_off = (int*)(smem + (size_t)slots * kSlot);            // [2][kTileB]: interface offsets of two tiles
    uint32_t* s_sl = (uint32_t*)(s_off + 2 * kTileB);             // [2][HP][9]: sub-boxes cut into slices
    float* s_me = (float*)(s_sl + (size_t)2 * HP * 9);            // [HP]: largest |hi| of a cell's three reals
    volatile int& s_abort = sy.abort;

    if (threadIdx.x == 0) {
        sy.abort = 0;
        for (int s = 0; s < kSlots; s++) tc::mbar_init(&sy.bfull[s], 1), tc::mbar_init(&sy.empty[s], 1);
        tc::mbar_init(&sy.done, 1);
        tc::mbar_init(&sy.drained, kBuilderWarps);
        for (int c = 0; c < 3; c++) tc::mbar_init(&sy.afull[c], kBuilderWarps / 2), tc::mbar_init(&sy.aempty[c], 1);
        for (int j = 0; j < 2; j++) tc::mbar_init(&sy.slfull[j], kSlicers / 32), tc::mbar_init(&sy.slempty[j], kBuilderWarps);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc::smem_u32(&sy.tbase)),
                     "r"(kTmemCols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    // All 512 columns of the SM are this CTA's: its tensor memory starts at address 0.  The issuing warp's
    // addresses are then constants and its operands stay in uniform registers; taken from the allocation's
    // answer, each product cost about 26 cycles to issue.
    constexpr uint32_t tmem = 0;
    if (threadIdx.x == 0 && sy.tbase != tmem) sy.abort = 1;

    if (warp >= kMmaWarp) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kIssueRegs));
        if (warp == kCopyWarp) {
            // ---- force operand: one bulk copy per input component of a stage ----
            if (lane == 0) {
                const unsigned char* src = O.bprep + oz_chunk(k, g, 0, 0, O.G, A.n_tb) * kChunk;  // the tiles' chunks in a row
                int it = 0, s = 0;
                uint32_t par = 1;
                for (; it < 3 * n_it; it++, src += kSlot) {
                    if (!tc::wait_or_abort_sleep(&sy.empty[s], par, &s_abort, wl, kSleepNs)) {
                        s_abort = 1;
                        break;
                    }
                    tc::mbar_expect_tx(&sy.bfull[s], kSlot);
                    tc::bulk_g2s(sB + (size_t)s * kSlot, src, kSlot, &sy.bfull[s]);
                    if (++s == slots) s = 0, par ^= 1u;
                }
                // copies still in flight land before the CTA may go on or exit: the full bound, whatever the stop flag
                for (int j = max(0, it - slots); j < it; j++) tc::mbar_wait(&sy.bfull[j % slots], (uint32_t)(j / slots) & 1u);
            }
        } else if (warp == kMmaWarp) {
            // ---- tensor-core issue: 3 x 26 products per stage, from the whole warp (one elected lane issues) ----
            const uint32_t el = tc::elect_one();
            const uint64_t dB0 = tc::sdesc(tc::smem_u32(smem), 128, kSBO);
            const uint32_t dBhi = (uint32_t)(dB0 >> 32);
            bool stop = false;
            uint32_t s = 0, par = 0;
            for (int il = 0; il < n_it && !stop; il++) {
                const bool first = (il % kStages) == 0;  // a new group overwrites the accumulators, once they are drained
                // (rolled: the instructions of one component, about 3 KB, are fetched again each time round)
#pragma unroll 1
                for (int ci = 0; ci < 3; ci++) {
                    // the A blocks of input component ci, stored by the builders while the others' products run
                    stop = !__all_sync(0xffffffffu, tc::wait_or_abort(&sy.bfull[s], par, &s_abort, wl) &&
                                                        tc::wait_or_abort(&sy.afull[ci], (uint32_t)il & 1u, &s_abort, wl));
                    if (first && ci == 0 && il > 0)
                        stop = stop || !__all_sync(0xffffffffu, tc::wait_or_abort(&sy.drained, ((uint32_t)(il / kStages) & 1u) ^ 1u,
                                                                                  &s_abort, wl));
                    if (stop) break;
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint32_t dBlo = (uint32_t)dB0 + s * (kSlot >> 4);
#pragma unroll
                    for (int p = 0; p < kNInst; p++)
                        tc::mma_ts<false>((uint32_t)oz_acc(p) * (uint32_t)kN, kAcol + (uint32_t)(ci * kNS + oz_i(p) - 1) * 8u,
                                          tc::desc64(dBlo + (((uint32_t)(oz_j(p) - 1) * kBBlk) >> 4), dBhi),
                                          tc::idesc(1, kRows, oz_n(p) * kN), (first && ci == 0 && p < 2) ? 0u : 1u, el);
                    tc::commit_elected(&sy.aempty[ci], el);
                    tc::commit_elected(&sy.empty[s], el);
                    if (++s == (uint32_t)slots) s = 0, par ^= 1u;
                }
            }
            if (stop) s_abort = 1;
            tc::commit_elected(&sy.done, el);  // also after a stop: fires once the issued products are complete
        }
    } else if (warp >= kSlicerWarp) {
        // ---- slicers: the sub-box of tile tB at the pair's scale, cut into slices, into buffer tB & 1 ----
        const int t = threadIdx.x - kSlicerWarp * 32;  // 0 .. 127; also the pad row of its share of the maximum
        const int2 xa = A.xy_p[O.row[tA * kRows + t]];
        const int4 bA = A.bbox_a[tA];
        const float* tk = A.tabx2 + (size_t)k * A.Dy * A.Dx * 12;
        const int rl0 = oz_real(co, 0), rl1 = oz_real(co, 1), rl2 = oz_real(co, 2);
        const float sg2 = oz_neg(co, 2) ? -1.0f : 1.0f;
        const int dp = O.pitch - A.W;  // cell e = iy W + ix is stored at iy pitch + ix = e + iy dp
        const uint32_t rcpW = 0xffffffffu / (uint32_t)A.W + 1u;  // e / W = umulhi(e, rcpW) for e < 2^16 (W > 1)
        float2 v0[NC], v1[NC], v2[NC];  // (hi, lo) of the three reals of cells t, t + 128, ...
        auto row_of = [&](int e) { return A.W > 1 ? (int)__umulhi((uint32_t)e, rcpW) : e; };
        auto cell_of = [&](int e) { return e + row_of(e) * dp; };
        auto load = [&](int tB) {
            const int4 bB = A.bbox_b[tB];
            const int gx0 = bA.x - bB.y - A.box_x0, gy0 = bA.z - bB.w - A.box_y0;
#pragma unroll
            for (int j = 0; j < NC; j++) {
                const int e = t + kSlicers * j;
                const int iy = row_of(e);
                const int gx = gx0 + e - iy * A.W, gy = gy0 + iy;
                v0[j] = v1[j] = v2[j] = make_float2(0.0f, 0.0f);  // zero outside the box
                if (e < HW && gx < A.Dx && gy < A.Dy) {
                    const float* src = tk + ((size_t)gy * A.Dx + gx) * 12;
                    v0[j] = *(const float2*)(src + 2 * rl0);
                    v1[j] = *(const float2*)(src + 2 * rl1);
                    v2[j] = *(const float2*)(src + 2 * rl2);
                }
            }
        };
        load(0);
        for (int tB = 0; tB < A.n_tb; tB++) {
            const int buf = tB & 1;
            // the builders are done with tile tB - 2; the same stop decision in every slicer
            bool ok = !s_abort && tc::wait_or_abort_sleep(&sy.slempty[buf], ((uint32_t)(tB >> 1) & 1u) ^ 1u, &s_abort, wl, kSleepNs);
            int* off_b = s_off + buf * kTileB;
            if (t < kTileB) off_b[t] = O.off[tB * kTileB + t];
#pragma unroll
            for (int j = 0; j < NC; j++) {
                const int e = t + kSlicers * j;
                if (e < HW) s_me[cell_of(e)] = fmaxf(fabsf(v2[j].x), fmaxf(fabsf(v0[j].x), fabsf(v1[j].x)));
            }
            if (tc::slicers_sync_any<kSlicers>(!ok)) {
                s_abort = 1;
                break;
            }
            // the tile pair's scale: the largest entry over its 128 x 64 pairs (each thread: one row;
            // magnitudes compare as integers)
            const int4 bB = A.bbox_b[tB];
            const int base = (xa.x - (bA.x - bB.y)) + O.pitch * (xa.y - (bA.z - bB.w));
            float m = 0.0f;
#pragma unroll 8
            for (int j = 0; j < kTileB; j++) m = fmaxf(m, s_me[base - off_b[j]]);
            const uint32_t mw = __reduce_max_sync(0xffffffffu, __float_as_uint(m));
            if (lane == 0) sy.wmax[warp - kSlicerWarp] = mw;
            tc::slicers_sync_any<kSlicers>(0);
            const uint32_t mb = max(max(sy.wmax[0], sy.wmax[1]), max(sy.wmax[2], sy.wmax[3]));
            const int E = oz_exp_of(__uint_as_float(mb));
            if (t == 0) sy.E[buf] = E;
            const float s_in = oz_pow2(-E);
            const uint64_t s01 = pk2(s_in, s_in), s22 = pk2(sg2 * s_in, sg2 * s_in);
            // every cell cut once at that scale: 18 bf16 slices (real, slice) in 9 words, two cells at a time
            uint32_t* sl = s_sl + (size_t)buf * HP * 9;
#pragma unroll
            for (int j = 0; j < NC; j += 2) {
                const int e0 = t + kSlicers * j, e1 = e0 + kSlicers;
                if (e0 >= HW) break;
                uint64_t t0[kNS], t1[kNS], t2[kNS];
                oz_split2(pk2(v0[j].x, v1[j].x), pk2(v0[j].y, v1[j].y), s01, t0);
                oz_split2(pk2(v0[j + 1].x, v1[j + 1].x), pk2(v0[j + 1].y, v1[j + 1].y), s01, t1);
                oz_split2(pk2(v2[j].x, v2[j + 1].x), pk2(v2[j].y, v2[j + 1].y), s22, t2);
                uint32_t c0[9], c1[9];
#pragma unroll
                for (int q = 0; q < 3; q++) {  // word q of a real: slices 2q (low half) and 2q + 1
                    float a0, b0, a1, b1, x0, x1, y0, y1;
                    upk2(t0[2 * q], a0, b0);
                    upk2(t0[2 * q + 1], a1, b1);
                    c0[q] = cvt_bf16x2(a1, a0), c0[3 + q] = cvt_bf16x2(b1, b0);
                    upk2(t1[2 * q], a0, b0);
                    upk2(t1[2 * q + 1], a1, b1);
                    c1[q] = cvt_bf16x2(a1, a0), c1[3 + q] = cvt_bf16x2(b1, b0);
                    upk2(t2[2 * q], x0, x1);
                    upk2(t2[2 * q + 1], y0, y1);
                    c0[6 + q] = cvt_bf16x2(y0, x0), c1[6 + q] = cvt_bf16x2(y1, x1);
                }
#pragma unroll
                for (int q = 0; q < 9; q++) sl[9 * cell_of(e0) + q] = c0[q];
                if (e1 < HW)
#pragma unroll
                    for (int q = 0; q < 9; q++) sl[9 * cell_of(e1) + q] = c1[q];
            }
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&sy.slfull[buf]);
            if (tB + 1 < A.n_tb) load(tB + 1);
        }
    } else {
        // ---- builders (warps 0..7): table slices into tensor memory, drains, output ----
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kBuilderRegs));
        const int a_loc = (warp & 3) * 32 + lane;  // TMEM lane = GEMM row
        const int hb = warp >> 2;                  // which items (every other), which 32 of the 64 GEMM columns
        const int a = O.row[tA * kRows + a_loc];
        const int2 xa = A.xy_p[a];
        const int4 bA = A.bbox_a[tA];
        // running double-float sums of this thread's row and GEMM columns hb * 32 .. + 31, as pairs of columns
        uint64_t H[16], L[16];
#pragma unroll
        for (int j = 0; j < 16; j++) H[j] = 0ull, L[j] = 0ull;
        const uint32_t tacc = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(hb * 32);
        auto drain = [&](float sc) {
            const uint64_t sc2 = pk2(sc, sc);
            uint32_t u[2][kNQ][4];  // four columns of the five accumulators; the next four load meanwhile
#pragma unroll
            for (int q = 0; q < kNQ; q++) tc::ld4_nowait(tacc + (uint32_t)(q * kN), u[0][q]);
#pragma unroll
            for (int c = 0; c < 8; c++) {
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                uint32_t v[kNQ][4];
#pragma unroll
                for (int q = 0; q < kNQ; q++)
#pragma unroll
                    for (int j = 0; j < 4; j++) v[q][j] = u[c & 1][q][j];
                if (c < 7)
#pragma unroll
                    for (int q = 0; q < kNQ; q++) tc::ld4_nowait(tacc + (uint32_t)(q * kN + (c + 1) * 4), u[(c + 1) & 1][q]);
#pragma unroll
                for (int j = 0; j < 2; j++) {
                    uint64_t d[kNQ];
#pragma unroll
                    for (int q = 0; q < kNQ; q++) d[q] = pk2(__uint_as_float(v[q][2 * j]), __uint_as_float(v[q][2 * j + 1]));
                    oz_accumulate2(d, sc2, H[c * 2 + j], L[c * 2 + j]);
                }
            }
        };
        const uint32_t trow = tmem + ((uint32_t)((warp & 3) * 32) << 16) + kAcol;
        float sc_prev = 0.0f;  // 2^E of the tile whose group is drained next
        bool ok = true;  // one decision per warp: its stores are warp-wide
        int4 bB = A.bbox_b[0];
        for (int tB = 0; tB < A.n_tb; tB++) {
            const int buf = tB & 1;
            const int base = (xa.x - (bA.x - bB.y)) + O.pitch * (xa.y - (bA.z - bB.w));
            if (tB + 1 < A.n_tb) bB = A.bbox_b[tB + 1];
            ok = __all_sync(0xffffffffu, !s_abort && tc::wait_or_abort(&sy.slfull[buf], (uint32_t)(tB >> 1) & 1u, &s_abort, wl));
            if (!ok) break;
            const int* off_b = s_off + buf * kTileB;
            const uint32_t* sl = s_sl + (size_t)buf * HP * 9;
            const float sc = oz_pow2(sy.E[buf]);
            // A tile's twelve items (stage, input component) alternate between the two builder groups; a warp
            // builds its 32 rows of an item whole, 48 neighbouring tensor-memory columns in two stores (beside
            // running products a store takes about one product's time whatever its width).
            for (int q12 = hb; q12 < 3 * kStages; q12 += 2) {
                const int st = q12 / 3, ci = q12 % 3;
                const uint32_t ph = ((uint32_t)(tB * kStages + st) & 1u) ^ 1u;  // parity of the stage before
                // the six slices of component ci, two columns per 32-bit word (words 3 ci .. 3 ci + 2 of
                // a cell hold its slices 0 .. 5)
                uint32_t w[kNS][8];
                const uint32_t* slc = sl + 3 * ci;
#pragma unroll
                for (int i4 = 0; i4 < 4; i4++) {  // row a_loc, interface columns st * 16 + 4 i4 .. + 3
                    const int4 o4 = *(const int4*)(off_b + st * kKC + 4 * i4);
                    const uint32_t* c0 = slc + 9 * (base - o4.x);
                    const uint32_t* c1 = slc + 9 * (base - o4.y);
                    const uint32_t* c2 = slc + 9 * (base - o4.z);
                    const uint32_t* c3 = slc + 9 * (base - o4.w);
#pragma unroll
                    for (int q = 0; q < 3; q++) {
                        const uint32_t u0 = c0[q], u1 = c1[q], u2 = c2[q], u3 = c3[q];
                        w[2 * q][2 * i4] = __byte_perm(u0, u1, 0x5410);
                        w[2 * q + 1][2 * i4] = __byte_perm(u0, u1, 0x7632);
                        w[2 * q][2 * i4 + 1] = __byte_perm(u2, u3, 0x5410);
                        w[2 * q + 1][2 * i4 + 1] = __byte_perm(u2, u3, 0x7632);
                    }
                }
                if (q12 + 2 >= 3 * kStages) {  // this warp has read all it needs of the buffer
                    __syncwarp();
                    if (lane == 0) tc::mbar_arrive(&sy.slempty[buf]);
                }
                // component ci's blocks are free once the stage before's products of ci are complete
                ok = __all_sync(0xffffffffu, !s_abort && tc::wait_or_abort(&sy.aempty[ci], ph, &s_abort, wl));
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                tc::st32(trow + (uint32_t)(ci * kNS) * 8u, &w[0][0]);
                tc::st16(trow + (uint32_t)(ci * kNS + 4) * 8u, &w[4][0]);
                asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(&sy.afull[ci]);
                // after the tile's first item is in place (its blocks are free before the previous tile's last
                // products): the previous tile's group, once all its products are complete
                if (q12 == hb && tB > 0) {
                    ok = __all_sync(0xffffffffu, !s_abort && tc::wait_or_abort(&sy.aempty[2], 1u, &s_abort, wl));
                    if (!ok) break;
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    drain(sc_prev);
                    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) tc::mbar_arrive(&sy.drained);
                }
            }
            if (!ok) break;
            sc_prev = sc;
        }
        if (!ok) s_abort = 1;
        // every product the MMA thread issued is complete once `done` fires (it commits on every path), so
        // this wait keeps the full bound whatever the stop flag says
        const bool done_ok = tc::mbar_wait(&sy.done, 0u);
        ok = __all_sync(0xffffffffu, done_ok && !s_abort);
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (ok) {
            drain(sc_prev);  // the last tile's group
#pragma unroll
            for (int j = 0; j < 32; j++) {
                const int n = hb * 32 + j, r = g * kRhs + n / 2, h = n & 1;
                if (r < O.n_rhs) {
                    float hv0, hv1, lv0, lv1;
                    upk2(H[j / 2], hv0, hv1);
                    upk2(L[j / 2], lv0, lv1);
                    const float hv = (j & 1) ? hv1 : hv0, lv = (j & 1) ? lv1 : lv0;
                    const float sF = oz_pow2(O.fexp[((size_t)r * A.K + k) * 2 + h]);
                    A.uh[(((size_t)r * A.K + k) * A.NPpad + a) * 6 + 3 * h + co] =
                        f2d_int(__fmul_rn(hv, sF)) + f2d_int(__fmul_rn(lv, sF));
                }
            }
        }
    }
    __syncthreads();
    if (threadIdx.x == 0 && sy.abort) atomicExch(status, FBC_ERR_TIMEOUT);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(sy.tbase), "r"(kTmemCols));
}

// shared memory: the force ring, offsets, two cut sub-boxes of `cells` cells and the cells' magnitudes (dynamic), and the
// static part, which the dynamic one's alignment rounds up to 1024
constexpr size_t kStaticSmem = 1024;
static_assert(sizeof(OzSync) <= kStaticSmem, "the barriers fit");
size_t oz_smem(int cells, int slots) {
    return (size_t)slots * kSlot + 2 * kTileB * 4 + (size_t)cells * (2 * 36 + 4) + kStaticSmem;
}
constexpr size_t kMaxSmem = 227 * 1024;
int oz_ring(int cells) {
    int n = kSlots;
    while (n > kMinSlots && oz_smem(cells, n) > kMaxSmem) n--;
    return n;
}
int oz_groups(const Plan& P) { return (P.opt.max_rhs + kRhs - 1) / kRhs; }
size_t oz_chunk_bytes(const Plan& P) { return (size_t)P.K * oz_groups(P) * P.n_tb * kStages * kChunk; }

}  // namespace

size_t contract_oz_smem(int HW) { return HW > kMaxCells ? kMaxSmem + 1 : oz_smem(HW, oz_ring(HW)); }

// Row order and pitch of the builders' gathers.  The 32 rows (pad sites) of a warp are read at word 9 (x + pitch y) +
// const of a cut sub-box, so rows whose x + pitch y agree modulo 32 share a bank: a read takes as many passes as the
// most frequent residue.  (The products' operand reads, the ring's copies and these reads share the 128 bytes a cycle of
// shared memory.)  A pad tile's 128 sites are dealt to the four warps residue by residue, the surplus of a residue to a
// warp that already repeats one; the pitch is the one with the fewest passes of those that leave room for the ring.
// 4000 x 6000 columns: 2.73 passes in the sites' own order at the sub-box's width 36, 1.32 so at pitch 41.
// rows[NPpad] receives the pad slot of each GEMM row; returns the pitch.
static long long oz_deal(const int2* site, int pitch, int* rows) {
    std::vector<int> by[32];
    std::vector<int> spare;  // padding repeats a site: the same address, any lane
    for (int i = 0; i < kRows; i++) {
        bool dup = false;
        for (int j = 0; j < i && !dup; j++) dup = site[j].x == site[i].x && site[j].y == site[i].y;
        if (dup) spare.push_back(i);
        else by[(unsigned)(site[i].x + pitch * site[i].y) % 32u].push_back(i);
    }
    int order[32], cnt[4][32] = {}, fill[4] = {}, top[4] = {};
    for (int r = 0; r < 32; r++) order[r] = r;
    std::stable_sort(order, order + 32, [&](int a, int b) { return by[a].size() > by[b].size(); });
    auto place = [&](int w, int i) {
        if (rows) rows[w * 32 + fill[w]] = i;
        fill[w]++;
    };
    for (int o = 0; o < 32; o++)
        for (int i : by[order[o]]) {
            const int r = order[o];
            int best = -1;
            auto worse = [&](int a, int b) {  // whether warp a is a worse place than warp b
                const int ra = std::max(cnt[a][r] + 1 - top[a], 0), rb = std::max(cnt[b][r] + 1 - top[b], 0);
                if (ra != rb) return ra > rb;
                const int ua = cnt[a][r] > 0 && cnt[a][r] < top[a] ? top[a] : 0, ub = cnt[b][r] > 0 && cnt[b][r] < top[b] ? top[b] : 0;
                if (ua != ub) return ua < ub;
                if (cnt[a][r] != cnt[b][r]) return cnt[a][r] > cnt[b][r];
                return fill[a] > fill[b];
            };
            for (int w = 0; w < 4; w++)
                if (fill[w] < 32 && (best < 0 || worse(best, w))) best = w;
            top[best] = std::max(top[best], ++cnt[best][r]);
            place(best, i);
        }
    for (int i : spare) {
        int w = 0;
        while (fill[w] == 32) w++;
        place(w, i);
    }
    return top[0] + top[1] + top[2] + top[3];
}
int contract_oz_layout(const Plan& P, int* rows) {
    int best = P.W;
    long long cost = -1;
    for (int p = P.W; p < P.W + kPitchSpan; p++) {
        if (p > P.W && oz_smem(p * P.H, kMinSlots) > kMaxSmem) break;
        long long c = 0;
        for (int t = 0; t < P.n_ta; t++) c += oz_deal(&P.xy_p_sorted[t * kRows], p, nullptr);
        if (cost < 0 || c < cost) cost = c, best = p;
    }
    for (int t = 0; t < P.n_ta; t++) {
        oz_deal(&P.xy_p_sorted[t * kRows], best, rows + t * kRows);
        for (int i = 0; i < kRows; i++) rows[t * kRows + i] += t * kRows;
    }
    return best;
}
int contract_oz_rhs_group() { return kRhs; }

// the sliced force operand of every mode and rhs group, then the scale exponents [max_rhs][K][2]
size_t contract_oz_prep_bytes(const Plan& P) {
    return oz_chunk_bytes(P) + (size_t)P.opt.max_rhs * P.K * 2 * sizeof(int);
}

// Modes A.k0 .. K - 1 (A.k0 >= 1) of an FBC_PREC_BF16X6 plan: scales and slices of the forces, then the
// contraction, one CTA per (pad tile, output component) x mode x group of kRhs right-hand sides.
cudaError_t launch_contract_oz(const ContractArgs& A, const Plan& P, int n_rhs, cudaStream_t st) {
    const int n_modes = P.K - A.k0;
    if (n_modes <= 0 || n_rhs < 1) return cudaSuccess;
    const int HW = P.H * P.W;
    if (HW > kMaxCells || !P.d_off_oz) return cudaErrorInvalidConfiguration;
    const int cells = P.H * P.oz_pitch;
    const size_t smem = oz_smem(cells, oz_ring(cells));
    if (smem > kMaxSmem) return cudaErrorInvalidConfiguration;
    if (!P.d_bprep || P.bprep_prec != FBC_PREC_BF16X6 || P.bprep_bytes < contract_oz_prep_bytes(P) ||
        n_rhs > P.opt.max_rhs || !A.tabx2 || A.tabx2 != P.d_table_x2)
        return cudaErrorInvalidValue;
    OzArgs O;
    O.A = A;
    O.bprep = (const unsigned char*)P.d_bprep;
    O.fexp = (const int*)((const unsigned char*)P.d_bprep + oz_chunk_bytes(P));
    O.n_rhs = n_rhs;
    O.slots = oz_ring(cells);
    O.off = P.d_off_oz, O.row = P.d_off_oz + P.NIpad;
    O.pitch = P.oz_pitch;
    O.G = oz_groups(P);
    k_oz_fscale<<<dim3(n_modes, n_rhs), 256, 0, st>>>(A.fh, P.K, P.NIpad, A.k0, (int*)O.fexp);
    if (cudaError_t e = cudaGetLastError()) return e;
    const int gu = (n_rhs + kRhs - 1) / kRhs;  // rhs groups of this apply
    const size_t total = (size_t)n_modes * gu * P.n_tb * kStages * kRhs * 2;
    const int grid = (int)std::min<size_t>((total + 255) / 256, (size_t)152 * 32);
    k_oz_prep<<<grid, 256, 0, st>>>(A.fh, O.fexp, P.K, P.NIpad, P.n_tb, O.G, gu, n_rhs, A.k0, n_modes,
                                    (unsigned char*)P.d_bprep);
    if (cudaError_t e = cudaGetLastError()) return e;
    const int wl = P.wait_limit > 0 ? P.wait_limit : tc::kWaitLimit;
    const dim3 grid3(3 * P.n_ta, n_modes, gu);
    auto launch = [&](auto kernel) -> cudaError_t {
        if (cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(smem - kStaticSmem))) return e;
        kernel<<<grid3, kThreads, smem - kStaticSmem, st>>>(O, wl, P.d_status);
        return cudaGetLastError();
    };
    // cells in registers: 12 a slicer thread cover the sub-boxes of compact tiles (36 x 42 at 8000 x 12000
    // columns), 16 the largest accepted
    return HW <= 12 * kSlicers ? launch(k_contract_oz<12>) : launch(k_contract_oz<16>);
}

}  // namespace fbc
