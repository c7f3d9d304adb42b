// Per-mode contraction on the 5th-generation tensor cores (tcgen05, FP32
// accumulation in tensor memory), for plans with several right-hand sides.
//
// For one wavenumber k the update is a real GEMM (Sec. 3.2, Eqs. 37-38 in the
// mode domain): with the six-vector form, every pad column a and output
// component c receives
//     U_c(a, :) = sum_{c', b} M_{c c'}(x_a - x_b) X_{c'}(b, :),
// where the columns ':' are the x and y' halves of all right-hand sides and
// M = [[A11, A12, -B13], [A12, A22, -B23], [B13, B23, A33]] comes from the six
// table reals.  A CTA owns 128 pad columns (GEMM rows) at one k and up to 64
// right-hand sides (N = 2 R columns) and walks the interface columns in
// stages of 16, through a ring of shared-memory stages:
//   * a warp stages the table sub-box of each interface tile, a bulk copy per
//     row, a tile ahead where two fit;
//   * twelve builder warps gather the six 128 x 16 blocks A_e(a, b) =
//     T_e(x_a - x_b) from it, a row and two entries a thread, and split them
//     into bf16 pieces (h, m, l) or round them to tf32.  A thread's 32 words are
//     one tcgen05.st into the A operand in tensor memory (TF32, BF16X2: up to
//     four operands of 96 columns above the accumulators, so a stage is built
//     while others are multiplied), or go to shared memory in the K-major
//     no-swizzle canonical layout (BF16X3);
//   * the force operand X_0, X_1, X_2 was split once per apply by k_prep_b
//     into the same layout, one contiguous chunk per (k, rhs group, stage);
//     one thread streams each chunk in with a bulk copy (cp.async.bulk);
//   * one warp (an elected lane) issues the 9 block products per split-product
//     pair as seven tcgen05.mma (M = 128, N = 2 R or 4 R, K = 16 bf16 / 8 tf32)
//     into three TMEM accumulators (one per output component); commits hand the
//     stage back to the builders and the copy thread.
// What bounds it: at 16 right-hand sides the issue of a stage's products (21 of
// some 36 cycles) and the hand-overs around it (a wait on a completed barrier
// takes 100 to 160 cycles); from N = 128 the tensor pipe.  (The gathers' bank
// conflicts are not it: rows dealt to the warps by bank, 3.7 wavefronts a gather
// for 4.5, made it slower, 10.8 ms an update for 10.4.)
// 4502 + 3001 columns, L = 512, 16 right-hand sides, BF16X2: 11.9 ms with eight
// builder warps (12 tcgen05.st a stage each), one A operand and sub-boxes
// copied by the builders, 8.3 ms now; 64 right-hand sides, L = 64: 4.3 and
// 4.2 ms.
// Split products: TF32 (1), BF16X2 (hh + hm + mh), BF16X3 (+ hl + lh + mm),
// pieces h = bf16(x), m = bf16(x - h), l = bf16(x - h - m), all rounded to
// nearest.  The logarithmic k = 0 mode is left to the double-float kernel.
//
// Every wait is bounded.  The pipeline waits (stage hand-offs between the
// roles) give up after the plan's wait limit, or at once when another role has
// given up; on a timeout the CTA records the status word, stops, waits for its
// own bulk copies and tensor-core work -- those two waits ignore the stop and
// keep the full bound, since the CTA may not exit or free its tensor memory
// while either is in flight -- frees its tensor memory and returns.  A warp
// decides to stop as a whole (its tensor-memory accesses take every lane), and
// warps that synchronise on a named barrier leave only right after it, so none
// is left waiting.
#include <cuda_bf16.h>

#include <algorithm>

#include "fbc_f32x2.cuh"
#include "fbc_internal.cuh"
#include "fbc_tc.cuh"

namespace fbc {
namespace {

constexpr int kTmemCols = 512;
constexpr int kRows = kTileA;    // GEMM rows (pad columns) per CTA
constexpr int kRhsPerCta = 64;
constexpr int kNPB = 128;        // force-operand rows per CTA (64 rhs x (x, y'))
constexpr int kKC = 16;          // interface columns per stage
constexpr int kBuilderWarps = 12;
constexpr int kBuilders = kBuilderWarps * 32;
constexpr int kMmaWarp = kBuilderWarps, kCopyWarp = kBuilderWarps + 1, kTabWarp = kBuilderWarps + 2;
constexpr int kThreads = (kBuilderWarps + 3) * 32;
constexpr int kStagesPerTile = kTileB / kKC;
constexpr int kDrainTiles = 16;  // interface tiles per tensor-memory accumulation group
constexpr int kMaxABuf = 4;      // A operands in tensor memory: 96 columns each from the top, 3 NP columns of accumulators below
constexpr int kACols = 96;
__device__ __forceinline__ uint32_t a_col(int j) { return (uint32_t)(kTmemCols - kACols * (j + 1)); }
__device__ __forceinline__ int a_bufs(int NP) { return min(kMaxABuf, (kTmemCols - 3 * NP) / kACols); }

using tc::idesc;
using tc::mbar_expect_tx;
using tc::mbar_init;
using tc::sdesc;
using tc::smem_u32;

template <int PREC>
struct TcCfg;
template <>
struct TcCfg<FBC_PREC_TF32> {
    static constexpr int ES = 4, NS = 1, NPROD = 1, KMMA = 8, FMT = 2, S = 3;
    static constexpr bool ATM = true;  // A operand in tensor memory
};
template <>
struct TcCfg<FBC_PREC_BF16X2> {
    static constexpr int ES = 2, NS = 2, NPROD = 3, KMMA = 16, FMT = 1, S = 3;
    static constexpr bool ATM = true;
};
template <>
struct TcCfg<FBC_PREC_BF16X3> {
    static constexpr int ES = 2, NS = 3, NPROD = 6, KMMA = 16, FMT = 1, S = 1;
    static constexpr bool ATM = false;  // 18 A blocks do not fit beside the accumulators
};

template <int PREC>
struct TcLayout {
    using C = TcCfg<PREC>;
    static constexpr int KPC = 16 / C::ES;                    // K elements per 16-byte core row
    static constexpr uint32_t SBO = (kKC / KPC) * 128;        // bytes per 8-row group of a [rows][16] block
    static constexpr size_t ABLK = (size_t)kRows * kKC * C::ES;
    static constexpr size_t A_STAGE = C::ATM ? 0 : 6 * C::NS * ABLK;  // shared-memory A stage
    static constexpr uint32_t ACOLS = (uint32_t)(kKC * C::ES / 4);         // TMEM columns of one A block
    static_assert(!C::ATM || 6 * C::NS * ACOLS == kACols, "six entries of NS pieces");
    static constexpr size_t B_STAGE = 3 * C::NS * (size_t)kNPB * kKC * C::ES;  // allocated for 128 rows
};

// Products of a stage, in the order in which each accumulator takes them: table entry, force block (X_2 stored
// negated, first in a chunk: [-X_2, X_1, X_0]), accumulator.  M is symmetric up to the sign of its (0, 2) and (1, 2)
// entries, so A12 multiplies X_1 into U_0 and X_0 into U_1, and B23 multiplies -X_2 into U_1 and X_1 into U_2: with the
// blocks and the accumulators in this order each pair is one instruction of 2 NP columns (seven per split product, not
// nine; at NP = 32 an instruction costs its issue, some 33 cycles, whatever its width).  U_2's A33 term negates A.
struct Prod {
    int ent, blk, acc, wide, neg;
};
// Split product pr takes the pieces (kPa[pr], kPb[pr]) of the A and B operands, by decreasing magnitude: hh, hm, mh,
// hl, lh, mm.

// Split x into NS pieces of the operand type; returned as raw bits (bf16 in
// the low 16 bits, or the tf32 bit pattern).  FP32 arithmetic throughout: each
// remainder x - bf16(x) is exact in FP32, and three bf16 pieces hold all 24
// bits of an FP32 value.
template <int PREC>
__device__ __forceinline__ void split(float x, uint32_t (&out)[TcCfg<PREC>::NS]) {
    if (PREC == FBC_PREC_TF32) {
        uint32_t t;
        asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(t) : "f"(x));
        out[0] = t;
    } else {
        float r = x;
#pragma unroll
        for (int s = 0; s < TcCfg<PREC>::NS; s++) {
            const __nv_bfloat16 h = __float2bfloat16_rn(r);
            out[s] = (uint32_t)__bfloat16_as_ushort(h);
            r = __fsub_rn(r, __bfloat162float(h));
        }
    }
}

// 16 bytes of one core-matrix row from KPC elements
template <int ES, int KPC>
__device__ __forceinline__ uint4 pack16(const uint32_t* w) {
    uint4 v;
    if (ES == 2) {
        v.x = w[0] | (w[1] << 16), v.y = w[2] | (w[3] << 16);
        v.z = w[4] | (w[5] << 16), v.w = w[6] | (w[7] << 16);
    } else {
        v.x = w[0], v.y = w[1], v.z = w[2], v.w = w[3];
    }
    return v;
}

using tc::builders_sync_any;
using tc::bulk_g2s;
using tc::cp_async16;
using tc::cp_async8;
using tc::mbar_arrive;
using tc::wait_or_abort;

// Chunk of the split force operand for (k, rhs group g, interface tile tB, stage st).
__host__ __device__ __forceinline__ size_t bchunk_index(int k, int g, int tB, int st, int G, int n_tb) {
    return (((size_t)k * G + g) * n_tb + tB) * kStagesPerTile + st;
}

// Rows of a group's blocks: two per right-hand side, in whole steps of 16 (an instruction's N).
__host__ __device__ __forceinline__ int group_rows(int rpc, int n_rhs, int g) {
    const int RG = rpc < n_rhs - g * rpc ? rpc : n_rhs - g * rpc;
    return RG > 0 ? (2 * RG + 15) / 16 * 16 : 0;
}

// One thread per 16-byte core row (block c, row n, core column kc) of a chunk:
// X_c(b, n = 2 r + h) = fh[g rpc + r][k][b][3 h + c], zero for r beyond the group
// (rpc right-hand sides per group, G groups, chunks of npb >= 2 rpc rows per block).
// A chunk holds, piece by piece, the blocks -X_2, X_1, X_0 of the group's rows.
template <int PREC>
__global__ void k_prep_b(const double* __restrict__ fh, int K, int NIpad, int n_tb, int G, int npb, int rpc,
                         int n_rhs, int k0, int n_modes, unsigned char* __restrict__ out) {
    using C = TcCfg<PREC>;
    using Lt = TcLayout<PREC>;
    constexpr int KPC = Lt::KPC, NKC = kKC / KPC;
    const size_t chunk_bytes = (size_t)3 * C::NS * npb * kKC * C::ES;
    const size_t per_chunk = (size_t)3 * npb * NKC;
    const size_t total = (size_t)n_modes * G * n_tb * kStagesPerTile * per_chunk;
    for (size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (size_t)gridDim.x * blockDim.x) {
        size_t q = t / per_chunk;
        const int rem = (int)(t % per_chunk);
        const int c = rem / (npb * NKC), n = (rem / NKC) % npb, kc = rem % NKC;
        const int st = (int)(q % kStagesPerTile);
        q /= kStagesPerTile;
        const int tB = (int)(q % n_tb);
        q /= n_tb;
        const int g = (int)(q % G);
        const int k = k0 + (int)(q / G);
        const int RG = min(rpc, n_rhs - g * rpc), NP = group_rows(rpc, n_rhs, g);
        if (n >= NP) continue;
        const int r = n >> 1, h = n & 1;
        const int b0 = tB * kTileB + st * kKC + kc * KPC;
        uint32_t w[C::NS][KPC];
#pragma unroll
        for (int i = 0; i < KPC; i++) {
            float v = 0.f;
            if (r < RG) v = (float)fh[(((size_t)(g * rpc + r) * K + k) * NIpad + b0 + i) * 6 + h * 3 + c];
            uint32_t sp[C::NS];
            split<PREC>(c == 2 ? -v : v, sp);
#pragma unroll
            for (int p = 0; p < C::NS; p++) w[p][i] = sp[p];
        }
        unsigned char* base = out + bchunk_index(k, g, tB, st, G, n_tb) * chunk_bytes;
        const uint32_t off = (uint32_t)(n / 8) * Lt::SBO + kc * 128 + (n % 8) * 16;
#pragma unroll
        for (int p = 0; p < C::NS; p++)
            *(uint4*)(base + (size_t)(p * 3 + 2 - c) * NP * kKC * C::ES + off) = pack16<C::ES, KPC>(w[p]);
    }
}

// Shared-memory barriers and flags of the contraction CTA.
template <int S>
struct TcSync {
    uint64_t full[S], bfull[S], empty[S], done, afull[kMaxABuf], aempty[kMaxABuf], tfull[2], tempty[2];
    uint32_t tbase;
    volatile int abort;
};

// The products of one stage.  FIRST: they overwrite the accumulators; accumulator 1's first split product then cannot
// share an instruction with accumulator 0's.
template <int PREC, bool FIRST>
__device__ __forceinline__ void issue_stage(uint32_t tmem, uint32_t ta, uint64_t dAs, uint64_t dBs, uint32_t bblk16, int NP,
                                            uint32_t id, uint32_t idw, uint32_t idn, uint32_t el) {
    using C = TcCfg<PREC>;
    using Lt = TcLayout<PREC>;
#pragma unroll
    for (int q = 0; q < 7; q++)
#pragma unroll
        for (int pr = 0; pr < C::NPROD; pr++)
#pragma unroll
            for (int ks = 0; ks < kKC / C::KMMA; ks++) {
                constexpr int kPa[6] = {0, 0, 1, 0, 2, 1}, kPb[6] = {0, 1, 0, 2, 0, 1};
                constexpr Prod P[7] = {{0, 2, 0, 0, 0}, {1, 1, 0, 1, 0}, {2, 1, 1, 0, 0}, {4, 2, 2, 0, 0},
                                       {4, 0, 0, 0, 0}, {5, 0, 1, 1, 0}, {3, 0, 2, 0, 1}};
                const int ablk = P[q].ent * C::NS + kPa[pr];
                auto mma = [&](int blk, int acc, uint32_t idd, uint32_t en) {
                    const uint64_t db = dBs + (uint64_t)((kPb[pr] * 3 + blk) * bblk16 + 16 * ks);
                    const uint32_t dt = tmem + (uint32_t)(acc * NP);
                    if (C::ATM)  // A from tensor memory: block ablk, K step ks (8 columns per MMA)
                        tc::mma_ts<C::FMT == 2>(dt, ta + (uint32_t)ablk * Lt::ACOLS + 8u * ks, db, idd, en, el);
                    else
                        tc::mma_ss(dt, dAs + (uint64_t)((ablk * Lt::ABLK + 256 * ks) >> 4), db, idd, en, el);
                };
                const bool start = FIRST && pr == 0 && ks == 0;
                if (P[q].wide && !(start && q == 1)) {
                    mma(P[q].blk, P[q].acc, idw, 1u);
                } else if (P[q].wide) {
                    mma(P[q].blk, P[q].acc, id, 1u);
                    mma(P[q].blk + 1, P[q].acc + 1, id, 0u);
                } else {
                    mma(P[q].blk, P[q].acc, P[q].neg ? idn : id, start && (q == 0 || q == 3) ? 0u : 1u);
                }
            }
}

// One work item (job J, mode k = wk.y, pad tile tA = wk.z, rhs group g = wk.w) on the whole CTA.  it_base:
// stages this CTA has run before the item (every role counts alike, so stage s = it % S and the barrier
// phases run on across items); n_done: items run before it (the parity of `done`); aph: the parities of this role's
// next wait on each A buffer (bits 0..3) and table buffer (bits 8, 9), which run on likewise.
template <int PREC>
__device__ __forceinline__ void tc_item(const TcJob& J, const int4 wk, const uint32_t it_base, const uint32_t n_done,
                                        TcSync<TcCfg<PREC>::S>& sy, unsigned char* smem, const int wl, uint32_t& aph) {
    using C = TcCfg<PREC>;
    using Lt = TcLayout<PREC>;
    constexpr int S = C::S;
    uint64_t* full = sy.full;
    uint64_t* bfull = sy.bfull;
    uint64_t* empty = sy.empty;
    uint64_t& done = sy.done;
    uint64_t* afull = sy.afull;
    uint64_t* aempty = sy.aempty;
    uint64_t* tfull = sy.tfull;
    uint64_t* tempty = sy.tempty;
    volatile int& s_abort = sy.abort;
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const ContractArgs& A = J.A;
    {
        const uint32_t tmem = sy.tbase;
        const int HW = A.H * A.W;
        unsigned char* sA = smem;                                   // [S][6][NS][128][16]
        unsigned char* sB = sA + S * Lt::A_STAGE;                   // [S][3][NS][npb][16]
        int* s_off = (int*)(sB + S * Lt::B_STAGE);                  // [nbuf][TB]
        unsigned char* s_tab = (unsigned char*)(s_off + J.nbuf * kTileB);  // [nbuf][tab_bytes]
        const int nbuf = J.nbuf, gs = J.gs;
        const int k = wk.y, tA = wk.z, g = wk.w;
        const int r0 = g * J.rpc;
        const int RG = min(J.rpc, J.n_rhs - r0);
        const int NP = group_rows(J.rpc, J.n_rhs, g);
        const int n_abuf = a_bufs(NP);
        const int n_it = A.n_tb * kStagesPerTile;
        const uint32_t chunk_bytes = (uint32_t)(3 * C::NS * J.npb * kKC * C::ES);
        const uint32_t bblk = (uint32_t)(NP * kKC * C::ES);          // one (block, piece) of a chunk

        if (warp == kCopyWarp) {
            // ---- force operand: one bulk copy per stage ----
            if (lane == 0) {
                int il = 0;
                for (; il < n_it; il++) {
                    const uint32_t it = it_base + il;
                    const int s = it % S;
                    const uint32_t u = it / S;
                    if (!wait_or_abort(&empty[s], (u & 1u) ^ 1u, &s_abort, wl)) {
                        s_abort = 1;
                        break;
                    }
                    const int tB = il / kStagesPerTile, st = il % kStagesPerTile;
                    mbar_expect_tx(&bfull[s], 3 * C::NS * bblk);
                    bulk_g2s(sB + s * Lt::B_STAGE, J.bprep + bchunk_index(k, g, tB, st, J.G, A.n_tb) * chunk_bytes,
                             3 * C::NS * bblk, &bfull[s]);
                }
                // copies still in flight land before the CTA may go on or exit: the full bound, whatever the
                // stop flag says
                for (int j = max(0, il - S); j < il; j++) {
                    const uint32_t it = it_base + j;
                    tc::mbar_wait(&bfull[it % S], (it / S) & 1u);
                }
            }
        } else if (warp == kTabWarp) {
            // ---- table sub-boxes: a bulk copy per row ----
            // A row's 24 W bytes start on an 8-byte boundary, a copy on a 16-byte one: it takes the bytes around them
            // too.  The shared pitch leaves room for them and equals the table's modulo 16, so that the rows stay a
            // pitch apart behind the same offset of 0 or 8.  Cells outside the box are left as they are: nobody reads
            // them (every difference of a pair of tiles lies in it).
            if (J.bulk) {
                const int4 bA = A.bbox_a[tA];
                const unsigned char* tk = (const unsigned char*)(A.tab32 + (size_t)(k - A.kbase) * A.Dy * A.Dx * 6);
                int b = 0;
                uint32_t used = 0;
                for (int tB = 0; tB < A.n_tb; tB++) {
                    const int4 bB = A.bbox_b[tB];
                    const int gx0 = bA.x - bB.y - A.box_x0, gy0 = bA.z - bB.w - A.box_y0;
                    const int rows = min(A.H, A.Dy - gy0), bytes = 24 * min(A.W, A.Dx - gx0);
                    const unsigned char* src = tk + ((size_t)gy0 * A.Dx + gx0) * 24;
                    uint32_t sum = 0;
                    for (int iy = lane; iy < rows; iy += 32) {
                        const size_t p = (size_t)src + (size_t)iy * A.Dx * 24;
                        sum += (uint32_t)(((p + bytes + 15) & ~(size_t)15) - (p & ~(size_t)15));
                    }
                    sum = __reduce_add_sync(0xffffffffu, sum) + kTileB * 4;
                    if (!__all_sync(0xffffffffu, wait_or_abort(&tempty[b], aph >> (8 + b) & 1u, &s_abort, wl))) {
                        s_abort = 1;
                        break;
                    }
                    aph ^= 0x100u << b, used |= 1u << b;
                    if (lane == 0) {
                        mbar_expect_tx(&tfull[b], sum);
                        bulk_g2s(s_off + b * kTileB, J.off + tB * kTileB, kTileB * 4, &tfull[b]);
                    }
                    __syncwarp();
                    unsigned char* dst = s_tab + (size_t)b * J.tab_bytes + ((size_t)src & 15);
                    for (int iy = lane; iy < rows; iy += 32) {
                        const size_t p = (size_t)src + (size_t)iy * A.Dx * 24;
                        bulk_g2s(dst + (size_t)iy * J.pitch - (p & 15), (const void*)(p & ~(size_t)15),
                                 (uint32_t)(((p + bytes + 15) & ~(size_t)15) - (p & ~(size_t)15)), &tfull[b]);
                    }
                    if (++b == J.nbuf) b = 0;
                }
                // copies still in flight land before the CTA may go on or exit: the full bound
                for (b = 0; b < 2; b++)
                    if (used >> b & 1u) tc::mbar_wait(&tfull[b], aph >> (8 + b) & 1u);
            }
        } else if (warp == kMmaWarp) {
            // ---- tensor-core issue, from the whole warp (one elected lane issues) ----
            const uint32_t el = tc::elect_one();
            const uint32_t id = idesc(C::FMT, kRows, NP), idw = idesc(C::FMT, kRows, 2 * NP), idn = id | (1u << 13);  // bit 13: negate A
            // descriptor of B block 0 of stage 0; the others differ by (byte offset >> 4) in the address field
            const uint64_t dB0 = sdesc(smem_u32(sB), 128, Lt::SBO);
            const uint64_t dA0 = sdesc(smem_u32(sA), 128, Lt::SBO);
            const uint32_t bblk16 = bblk >> 4;
            int j = 0;     // A buffer
            int gpos = 0;  // position of the stage in its accumulation group
            bool stop = false;
            for (int il = 0; il < n_it; il++) {
                const uint32_t it = it_base + il;
                const int s = it % S;
                const uint32_t par = (it / S) & 1u;
                uint64_t* af = C::ATM ? &afull[j] : &full[s];
                const uint32_t apar = C::ATM ? (aph >> j & 1u) : par;
                stop = !__all_sync(0xffffffffu, wait_or_abort(af, apar, &s_abort, wl) &&
                                                    wait_or_abort(&bfull[s], par, &s_abort, wl));
                if (stop) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint64_t dBs = dB0 + (uint64_t)((s * Lt::B_STAGE) >> 4);
                const uint64_t dAs = dA0 + (uint64_t)((s * Lt::A_STAGE) >> 4);
                // a new accumulation group starts by overwriting the accumulators
                const bool first = gpos == 0;
                if (++gpos == gs) gpos = 0;
                const uint32_t ta = tmem + a_col(j);
                if (first)
                    issue_stage<PREC, true>(tmem, ta, dAs, dBs, bblk16, NP, id, idw, idn, el);
                else
                    issue_stage<PREC, false>(tmem, ta, dAs, dBs, bblk16, NP, id, idw, idn, el);
                if (C::ATM) {
                    tc::commit_elected(&aempty[j], el);
                    aph ^= 1u << j;
                    if (++j == n_abuf) j = 0;
                }
                tc::commit_elected(&empty[s], el);
            }
            if (stop) s_abort = 1;
            tc::commit_elected(&done, el);  // also after a stop: fires once the issued products are complete
        } else {
            // ---- builders (warps 0..11) ----
            const int tid = threadIdx.x;                  // 0 .. 383
            const int a_loc = (warp & 3) * 32 + lane;     // TMEM lane = GEMM row
            const int pl = warp >> 2;                     // which two of the six entries
            const int a = tA * kRows + a_loc;
            const int2 xa = A.xy_p[a];
            const int4 bA = A.bbox_a[tA];
            const float* tk = A.tab32 + (size_t)(k - A.kbase) * A.Dy * A.Dx * 6;
            // (a table buffer too small for padded rows: the builders copy it themselves)
            const int sy0 = tid / (3 * A.W), sx0 = tid % (3 * A.W), dsy = kBuilders / (3 * A.W), dsx = kBuilders % (3 * A.W);
            // table sub-box and interface offsets of tile tB into buffer buf, by asynchronous copies
            auto stage_async = [&](int buf, int tB) {
                const int4 bB = A.bbox_b[tB];
                const int ox = bA.x - bB.y, oy = bA.z - bB.w;
                const int gx0 = ox - A.box_x0, gy0 = oy - A.box_y0;
                float2* dt = (float2*)(s_tab + (size_t)buf * J.tab_bytes);
                // eight bytes a thread, neighbouring threads neighbouring ones: row iy, 8-byte word cx of it
                const float2* t0 = (const float2*)tk + ((ptrdiff_t)gy0 * A.Dx + gx0) * 3;
                const int cx_in = 3 * (A.Dx - gx0);
                int iy = sy0, cx = sx0;
                for (int e = tid; e < 3 * HW; e += kBuilders) {
                    const bool in = cx < cx_in && gy0 + iy < A.Dy;  // zero fill outside the box
                    cp_async8(dt + e, in ? t0 + ((ptrdiff_t)iy * A.Dx * 3 + cx) : (const float2*)tk, in ? 8 : 0);
                    iy += dsy, cx += dsx;
                    if (cx >= 3 * A.W) cx -= 3 * A.W, iy++;
                }
                if (tid < kTileB / 4) cp_async16(s_off + buf * kTileB + 4 * tid, A.off_i + tB * kTileB + 4 * tid);
                asm volatile("cp.async.commit_group;" ::: "memory");
            };
            // Accumulators -> uh32 (the modes k >= 1 in FP32).  The FP32 accumulation in tensor
            // memory truncates at every step, so the interface sum is split into groups of gs
            // stages whose partial sums are added here with round-to-nearest FP32 adds; the first
            // group writes, the later ones add.  The sums are FP32 values, kept in FP32.
            const uint32_t tacc = tmem + ((uint32_t)((warp & 3) * 32) << 16);
            auto drain = [&](bool add) {
                for (int c0 = pl * 16; c0 < NP; c0 += 48) {
                    float v0[16], v1[16], v2[16];
                    tc::ld16(tacc + (uint32_t)c0, v0);
                    tc::ld16(tacc + (uint32_t)(NP + c0), v1);
                    tc::ld16(tacc + (uint32_t)(2 * NP + c0), v2);
#pragma unroll
                    for (int h = 0; h < 2; h++) {
                        // four right-hand sides at a time: every load issued before any store
                        float2 q[4][3];
                        float2* o[4];
#pragma unroll
                        for (int jj = 0; jj < 4; jj++) {
                            const int r = c0 / 2 + h * 4 + jj;
                            o[jj] = (float2*)(A.uh32 + (((size_t)(r0 + min(r, RG - 1)) * A.K + k) * A.NPpad + a) * 6);
                            if (add && r < RG) q[jj][0] = o[jj][0], q[jj][1] = o[jj][1], q[jj][2] = o[jj][2];
                        }
#pragma unroll
                        for (int jj = 0; jj < 4; jj++) {
                            const int j = h * 4 + jj, r = c0 / 2 + j;
                            if (r >= RG) continue;
                            float w[6] = {v0[2 * j], v1[2 * j], v2[2 * j], v0[2 * j + 1], v1[2 * j + 1], v2[2 * j + 1]};
                            if (add) {
                                w[0] += q[jj][0].x, w[1] += q[jj][0].y, w[2] += q[jj][1].x;
                                w[3] += q[jj][1].y, w[4] += q[jj][2].x, w[5] += q[jj][2].y;
                            }
                            o[jj][0] = make_float2(w[0], w[1]);
                            o[jj][1] = make_float2(w[2], w[3]);
                            o[jj][2] = make_float2(w[4], w[5]);
                        }
                    }
                }
            };
            // A pipeline wait of a builder warp, and its stop decision: one for all lanes, since what follows (tensor-memory
            // loads and stores, __syncwarp) takes the whole warp and lanes that left it would be waited for without a bound.
            // (The stop flag is read among the polls alone: read before every wait as well, an update of 3001 + 4502 columns,
            // L = 512, 16 right-hand sides took 10.46 ms, 10.39 so.)
            auto wait_warp = [&](uint64_t* m, uint32_t parity) {
                const bool go = __all_sync(0xffffffffu, wait_or_abort(m, parity, &s_abort, wl));
                if (!go) s_abort = 1;
                return go;
            };
            int il = 0, gpos = 0;  // stage of the item and its position in the accumulation group
            int j = 0;             // A buffer
            const bool bulk = J.bulk;
            const unsigned pitch = (unsigned)J.pitch, om = bulk ? 1u : 24u;  // bytes of a sub-box row, of a unit of s_off
            if (!bulk && nbuf == 2) stage_async(0, 0);
            for (int tB = 0, buf = 0; tB < A.n_tb; tB++, buf = buf + 1 == nbuf ? 0 : buf + 1) {
                const int4 bB = A.bbox_b[tB];
                if (bulk) {
                    if (!wait_warp(&tfull[buf], aph >> (8 + buf) & 1u)) break;
                    aph ^= 0x100u << buf;
                } else {
                    if (nbuf == 1) {
                        if (builders_sync_any<kBuilders>(s_abort)) break;  // everyone is done with the previous tile
                        stage_async(0, tB);
                    }
                    asm volatile("cp.async.wait_all;" ::: "memory");
                    // this tile's copies are visible to every builder, the previous tile is done;
                    // the same stop decision in every builder
                    if (builders_sync_any<kBuilders>(s_abort)) break;
                    if (nbuf == 2 && tB + 1 < A.n_tb) stage_async(buf ^ 1, tB + 1);
                }
                const unsigned char* tab_b = s_tab + (size_t)buf * J.tab_bytes;
                const int* off_b = s_off + buf * kTileB;
                const int ox = bA.x - bB.y, oy = bA.z - bB.w;
                // byte offset of entries 2 pl of this row's difference to the origin, behind a shift of 0 or 8.  Modulo 2^32,
                // as the columns' offsets: sites may lie so far out that their own offsets wrap, their differences do not.
                const unsigned odd =
                    (((unsigned)(k - A.kbase) * (unsigned)A.Dy + (unsigned)(oy - A.box_y0)) * (unsigned)A.Dx + (unsigned)(ox - A.box_x0)) & 1u;
                const unsigned base = 24u * (unsigned)(xa.x - ox) + pitch * (unsigned)(xa.y - oy) + 8u * (unsigned)pl + (bulk ? 8u * odd : 0u);
                auto entries = [&](int o) { return *(const float2*)(tab_b + (int)(base - om * (unsigned)o)); };
                for (int st = 0; st < kStagesPerTile; st++, il++) {
                    const uint32_t it = it_base + il;
                    const int s = it % S;
                    const uint32_t u = it / S;
                    // (a stop ends the tile; the next one's start ends the item, on the barrier where the builders have one)
                    if (!C::ATM && !wait_warp(&empty[s], (u & 1u) ^ 1u)) break;
                    // At a group boundary, wait for the previous stage's products first (A in tensor
                    // memory: its buffer's release; otherwise the single stage's release above)
                    // and drain the accumulators before gathering, where few registers are live.
                    const bool boundary = il > 0 && gpos == 0;
                    if (++gpos == gs) gpos = 0;
                    if (boundary) {
                        const int jp = j == 0 ? n_abuf - 1 : j - 1;
                        if (C::ATM && !wait_warp(&aempty[jp], aph >> jp & 1u)) break;
                        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                        drain(il > gs);
                        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                    }
                    // row a_loc, the stage's 16 columns: entries 2 pl and 2 pl + 1
                    float2 v[kKC];
#pragma unroll
                    for (int i = 0; i < kKC; i += 4) {
                        const int4 o = *(const int4*)(off_b + st * kKC + i);
                        v[i] = entries(o.x), v[i + 1] = entries(o.y), v[i + 2] = entries(o.z), v[i + 3] = entries(o.w);
                    }
                    // split into NS pieces: w[(entry, piece)][32-bit words of 16 elements], packed round-to-nearest
                    // conversions with exact FP32 remainders (bf16), or one tf32 word per element
                    constexpr int NW = kKC * C::ES / 4;
                    uint32_t w[2 * C::NS * NW];
#pragma unroll
                    for (int p = 0; p < C::NS; p++) {
                        if (C::ES == 2) {
#pragma unroll
                            for (int i = 0; i < kKC; i += 2) {
                                uint32_t h0, h1;
                                asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(h0) : "f"(v[i + 1].x), "f"(v[i].x));
                                asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(h1) : "f"(v[i + 1].y), "f"(v[i].y));
                                w[p * NW + i / 2] = h0, w[(C::NS + p) * NW + i / 2] = h1;
                                if (p + 1 < C::NS) {  // exact remainders, of a column's two entries at a time
                                    upk2(sub2(pk2(v[i].x, v[i].y), pk2(__uint_as_float(h0 << 16), __uint_as_float(h1 << 16))),
                                         v[i].x, v[i].y);
                                    upk2(sub2(pk2(v[i + 1].x, v[i + 1].y), pk2(__uint_as_float(h0 & 0xffff0000u),
                                                                               __uint_as_float(h1 & 0xffff0000u))),
                                         v[i + 1].x, v[i + 1].y);
                                }
                            }
                        } else {
#pragma unroll
                            for (int i = 0; i < kKC; i++) {
                                asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(w[i]) : "f"(v[i].x));
                                asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(w[NW + i]) : "f"(v[i].y));
                            }
                        }
                    }
                    if (C::ATM) {
                        // free once the products of the stage that had the buffer before are complete
                        if (!wait_warp(&aempty[j], aph >> j & 1u)) break;
                        aph ^= 1u << j;
                        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                        // lane = row a_loc; this warp's entries and pieces: 32 columns in a row
                        tc::st32(tmem + ((uint32_t)((warp & 3) * 32) << 16) + a_col(j) + 32u * pl, w);
                        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&afull[j]);
                        if (++j == n_abuf) j = 0;
                    } else {
                        unsigned char* dstA = sA + s * Lt::A_STAGE + (size_t)(a_loc / 8) * Lt::SBO + (a_loc % 8) * 16;
#pragma unroll
                        for (int q = 0; q < 2 * C::NS; q++)
#pragma unroll
                            for (int i = 0; i < NW; i += 4)
                                *(uint4*)(dstA + (size_t)(2 * pl * C::NS + q) * Lt::ABLK + 32 * i) =
                                    make_uint4(w[q * NW + i], w[q * NW + i + 1], w[q * NW + i + 2], w[q * NW + i + 3]);
                        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&full[s]);
                    }
                }
                __syncwarp();
                if (bulk && lane == 0) mbar_arrive(&tempty[buf]);
            }
            asm volatile("cp.async.wait_all;" ::: "memory");  // a prefetch still in flight after a stop
            // ---- epilogue: accumulators -> uh (FP64) ----
            // the MMA thread commits `done` once per item on every path, also after a stop; every product it
            // issued is complete once `done` fires, so this wait keeps the full bound whatever the stop flag says
            const bool done_ok = tc::mbar_wait(&done, n_done & 1u);
            const bool ok = __all_sync(0xffffffffu, done_ok && !s_abort);
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            if (ok) drain(n_it > gs);  // the last group; earlier groups were drained in the loop
        }
    }
}

// a filling role's first wait on a buffer passes, a reading role's does not
__device__ __forceinline__ uint32_t first_parities() {
    const int warp = threadIdx.x / 32;
    return warp < kBuilderWarps ? 0xfu : warp == kTabWarp ? 0x300u : 0u;
}

template <int PREC>
__device__ __forceinline__ void tc_setup(TcSync<TcCfg<PREC>::S>& sy) {
    constexpr int S = TcCfg<PREC>::S;
    if (threadIdx.x == 0) {
        sy.abort = 0;
        for (int s = 0; s < S; s++) mbar_init(&sy.full[s], kBuilderWarps), mbar_init(&sy.bfull[s], 1), mbar_init(&sy.empty[s], 1);
        mbar_init(&sy.done, 1);
        for (int j = 0; j < kMaxABuf; j++) mbar_init(&sy.afull[j], kBuilderWarps), mbar_init(&sy.aempty[j], 1);
        for (int j = 0; j < 2; j++) mbar_init(&sy.tfull[j], 1), mbar_init(&sy.tempty[j], kBuilderWarps);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (threadIdx.x / 32 == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&sy.tbase)),
                     "r"(kTmemCols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

template <int PREC>
__device__ __forceinline__ void tc_teardown(TcSync<TcCfg<PREC>::S>& sy, int* status) {
    __syncthreads();
    if (threadIdx.x == 0 && sy.abort) atomicExch(status, FBC_ERR_TIMEOUT);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (threadIdx.x / 32 == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(sy.tbase), "r"(kTmemCols));
}

// One plan: one item per CTA from its grid position (pad tile, mode k0 + y, rhs group).
template <int PREC>
__global__ void __launch_bounds__(kThreads, 1) k_contract_tc(TcJob J, int wl, int* status) {
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ TcSync<TcCfg<PREC>::S> sy;
    tc_setup<PREC>(sy);
    uint32_t aph = first_parities();
    tc_item<PREC>(J, make_int4(0, J.A.k0 + (int)blockIdx.y, (int)blockIdx.x, (int)blockIdx.z), 0u, 0u, sy, smem, wl, aph);
    tc_teardown<PREC>(sy, status);
}

// A batch of plans: persistent CTAs take items (job, k, pad tile, rhs group) from a queue with atomicAdd; no
// CTA waits for another.  The stage counters and barrier phases run on across items, so no barrier is
// re-initialised while a tensor-core commit could still arrive on it; the CTA-wide barrier between items
// orders the drain of one item's accumulators before the next item's first products.
template <int PREC>
__global__ void __launch_bounds__(kThreads, 1)
    k_contract_tc_queue(const TcJob* __restrict__ jobs, const int4* __restrict__ items, int n_items,
                        int* __restrict__ counter, int wl, int* status) {
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ TcSync<TcCfg<PREC>::S> sy;
    __shared__ int s_item;
    __shared__ int4 s_wk;
    __shared__ TcJob s_job;  // the current item's job
    tc_setup<PREC>(sy);
    uint32_t it_base = 0, n_done = 0, aph = first_parities();
    for (;;) {
        if (threadIdx.x == 0) {
            const int ii = atomicAdd(counter, 1);
            s_item = ii;
            if (ii < n_items) s_wk = items[ii], s_job = jobs[s_wk.x];
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (s_item >= n_items || sy.abort) break;
        tc_item<PREC>(s_job, s_wk, it_base, n_done, sy, smem, wl, aph);
        it_base += (uint32_t)(s_job.A.n_tb * kStagesPerTile);
        n_done++;
        // a table buffer that the builders filled themselves may be the next item's target of bulk copies: their writes
        // come before those of the other proxy
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();  // every role is done with s_job and s_wk before thread 0 overwrites them
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    }
    tc_teardown<PREC>(sy, status);
}

// with the static part, which the dynamic one's alignment rounds up to 1024
constexpr size_t kStaticSmem = 1024;
static_assert(sizeof(TcSync<3>) + sizeof(TcJob) + 32 <= kStaticSmem, "the barriers and the queue's job fit");
template <int PREC>
size_t tc_smem(size_t tab_bytes, int nbuf) {
    using Lt = TcLayout<PREC>;
    return TcCfg<PREC>::S * (Lt::A_STAGE + Lt::B_STAGE) + nbuf * (tab_bytes + (size_t)kTileB * 4) + kStaticSmem;
}
// How a plan's table sub-boxes are staged: two buffers (the next tile prefetched) when they fit, else one; rows by bulk
// copies with the pitch these need, unless that costs a buffer or does not fit: then the builders copy them with
// cp.async, in 8-byte pieces without padding (4502 + 3001 columns, BF16X2, 16 right-hand sides: 11.3 ms, of which the
// builders spent 40 % issuing these, against 8.3 ms by bulk copies).
struct TcStaging {
    int nbuf, bulk, pitch;
    size_t tab_bytes, smem;
};
template <int PREC>
TcStaging tc_staging(const Plan& P) {
    const size_t flat = ((size_t)24 * P.W * P.H + 15) / 16 * 16, rows = ((size_t)contract_tc_pitch(P) * P.H + 47) / 16 * 16;
    TcStaging t;
    t.nbuf = tc_smem<PREC>(flat, 2) <= 227 * 1024 ? 2 : 1;
    t.bulk = tc_smem<PREC>(rows, t.nbuf) <= 227 * 1024;
    t.pitch = t.bulk ? contract_tc_pitch(P) : 24 * P.W;
    t.tab_bytes = t.bulk ? rows : flat;
    t.smem = tc_smem<PREC>(t.tab_bytes, t.nbuf);
    return t;
}

int prep_groups(const Plan& P) { return (P.opt.max_rhs + kRhsPerCta - 1) / kRhsPerCta; }
int prep_rows(const Plan& P) { return ((2 * std::min(kRhsPerCta, P.opt.max_rhs) + 15) / 16) * 16; }
int rows_for(int rpc) { return ((2 * rpc + 15) / 16) * 16; }

template <int PREC>
size_t prep_bytes(const Plan& P) {
    using C = TcCfg<PREC>;
    return (size_t)P.K * prep_groups(P) * P.n_tb * kStagesPerTile * 3 * C::NS * prep_rows(P) * kKC * C::ES;
}

// Split the force operand of modes k0 .. k0 + n_modes - 1 into the plan's buffer, rpc right-hand sides per group.
template <int PREC>
cudaError_t prep_tc(const Plan& P, const double* fh, int rpc, int n_rhs, int k0, int n_modes, cudaStream_t st) {
    using Lt = TcLayout<PREC>;
    const int G = (P.opt.max_rhs + rpc - 1) / rpc, npb = rows_for(rpc);
    const size_t total = (size_t)n_modes * G * P.n_tb * kStagesPerTile * 3 * npb * (kKC / Lt::KPC);
    const int grid = (int)std::min<size_t>((total + 255) / 256, (size_t)152 * 32);
    k_prep_b<PREC><<<grid, 256, 0, st>>>(fh, P.K, P.NIpad, P.n_tb, G, npb, rpc, n_rhs, k0, n_modes,
                                         (unsigned char*)P.d_bprep);
    return cudaGetLastError();
}

template <int PREC>
TcJob make_job(const ContractArgs& A, const Plan& P, int n_rhs, int rpc) {
    const TcStaging t = tc_staging<PREC>(P);
    TcJob J;
    J.A = A;
    J.bprep = (const unsigned char*)P.d_bprep;
    J.n_rhs = n_rhs;
    J.rpc = rpc;
    J.G = (P.opt.max_rhs + rpc - 1) / rpc;
    J.npb = rows_for(rpc);
    // accumulation groups of kDrainTiles interface tiles (1024 columns), or one group
    const int n_it = P.n_tb * kStagesPerTile;
    J.gs = (P.opt.flags & FBC_PLAN_TC_FAST_ACCUMULATE) ? n_it : std::min(n_it, kDrainTiles * kStagesPerTile);
    J.nbuf = t.nbuf, J.bulk = t.bulk, J.pitch = t.pitch, J.tab_bytes = (int)t.tab_bytes;
    J.off = P.d_off_tc;
    return J;
}

template <int PREC>
cudaError_t launch_tc(const ContractArgs& A, const Plan& P, int n_rhs, cudaStream_t st, int n_modes) {
    const size_t all = tc_staging<PREC>(P).smem, smem = all - kStaticSmem;
    if (all > 227 * 1024 || !P.d_off_tc) return cudaErrorInvalidConfiguration;
    if (!P.d_bprep || P.bprep_prec != PREC || n_rhs > P.opt.max_rhs) return cudaErrorInvalidValue;
    const int rpc = std::min(kRhsPerCta, P.opt.max_rhs);
    if (cudaError_t e = prep_tc<PREC>(P, A.fh, rpc, n_rhs, A.k0, n_modes, st)) return e;
    cudaError_t e = cudaFuncSetAttribute(k_contract_tc<PREC>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e) return e;
    const TcJob J = make_job<PREC>(A, P, n_rhs, rpc);
    dim3 grid(P.n_ta, n_modes, (n_rhs + rpc - 1) / rpc);
    const int wl = P.wait_limit > 0 ? P.wait_limit : tc::kWaitLimit;
    k_contract_tc<PREC><<<grid, kThreads, smem, st>>>(J, wl, P.d_status);
    return cudaGetLastError();
}

template <int PREC>
cudaError_t launch_tc_batch(const TcJob* d_jobs, const int4* d_items, int n_items, int* d_counter, int grid,
                            size_t all, int wl, int* status, cudaStream_t st) {
    const size_t smem = all - kStaticSmem;
    cudaError_t e =
        cudaFuncSetAttribute(k_contract_tc_queue<PREC>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e) return e;
    k_contract_tc_queue<PREC><<<grid, kThreads, smem, st>>>(d_jobs, d_items, n_items, d_counter, wl, status);
    return cudaGetLastError();
}

}  // namespace

size_t contract_tc_smem(int precision, const Plan& P) {
    if (precision == FBC_PREC_TF32) return tc_staging<FBC_PREC_TF32>(P).smem;
    if (precision == FBC_PREC_BF16X2) return tc_staging<FBC_PREC_BF16X2>(P).smem;
    return tc_staging<FBC_PREC_BF16X3>(P).smem;
}
// Bytes from row to row of a sub-box staged by bulk copies: room for 8 bytes on either side of a row's 24 W, and the
// table's own pitch modulo 16.
int contract_tc_pitch(const Plan& P) {
    int p = 24 * P.W + 16;
    if ((p & 15) != 8 * (P.Dx & 1)) p += 8;
    return p;
}

size_t contract_tc_prep_bytes(const Plan& P, int precision) {
    if (precision == FBC_PREC_TF32) return prep_bytes<FBC_PREC_TF32>(P);
    if (precision == FBC_PREC_BF16X2) return prep_bytes<FBC_PREC_BF16X2>(P);
    return prep_bytes<FBC_PREC_BF16X3>(P);
}

// Largest rhs group a plan's force-operand buffer holds (right-hand sides per CTA), and whether rpc fits it:
// the buffer holds G x npb rows per (mode, stage) for the plan's own group size.
int contract_tc_max_rpc(const Plan& P) { return std::min(kRhsPerCta, P.opt.max_rhs); }
bool contract_tc_rpc_fits(const Plan& P, int rpc) {
    if (rpc < 1 || rpc > contract_tc_max_rpc(P)) return false;
    const long long want = (long long)((P.opt.max_rhs + rpc - 1) / rpc) * rows_for(rpc);
    return want <= (long long)prep_groups(P) * prep_rows(P);
}

cudaError_t contract_tc_prep(const Plan& P, const double* fh, int rpc, int n_rhs, int k0, int n_modes, cudaStream_t st) {
    if (!P.d_bprep || P.bprep_prec != P.precision || !contract_tc_rpc_fits(P, rpc)) return cudaErrorInvalidValue;
    if (P.precision == FBC_PREC_TF32) return prep_tc<FBC_PREC_TF32>(P, fh, rpc, n_rhs, k0, n_modes, st);
    if (P.precision == FBC_PREC_BF16X2) return prep_tc<FBC_PREC_BF16X2>(P, fh, rpc, n_rhs, k0, n_modes, st);
    if (P.precision == FBC_PREC_BF16X3) return prep_tc<FBC_PREC_BF16X3>(P, fh, rpc, n_rhs, k0, n_modes, st);
    return cudaErrorInvalidValue;
}

TcJob contract_tc_job(const Plan& P, int n_rhs, int rpc) {
    const ContractArgs A = make_contract_args(P);
    if (P.precision == FBC_PREC_TF32) return make_job<FBC_PREC_TF32>(A, P, n_rhs, rpc);
    if (P.precision == FBC_PREC_BF16X2) return make_job<FBC_PREC_BF16X2>(A, P, n_rhs, rpc);
    return make_job<FBC_PREC_BF16X3>(A, P, n_rhs, rpc);
}

cudaError_t launch_contract_tc_batch(int precision, const TcJob* d_jobs, const int4* d_items, int n_items,
                                     int* d_counter, int grid, size_t smem, int wl, int* status, cudaStream_t st) {
    if (n_items == 0) return cudaSuccess;
    if (precision == FBC_PREC_TF32)
        return launch_tc_batch<FBC_PREC_TF32>(d_jobs, d_items, n_items, d_counter, grid, smem, wl, status, st);
    if (precision == FBC_PREC_BF16X2)
        return launch_tc_batch<FBC_PREC_BF16X2>(d_jobs, d_items, n_items, d_counter, grid, smem, wl, status, st);
    if (precision == FBC_PREC_BF16X3)
        return launch_tc_batch<FBC_PREC_BF16X3>(d_jobs, d_items, n_items, d_counter, grid, smem, wl, status, st);
    return cudaErrorInvalidValue;
}

// Modes A.k0 .. A.k0 + n_modes - 1 (default: through K - 1) on the tensor cores (A.k0 >= 1).
cudaError_t launch_contract_tc(const ContractArgs& A, const Plan& P, int n_rhs, cudaStream_t st, int n_modes) {
    if (n_modes < 0) n_modes = P.K - A.k0;
    if (P.precision == FBC_PREC_TF32) return launch_tc<FBC_PREC_TF32>(A, P, n_rhs, st, n_modes);
    if (P.precision == FBC_PREC_BF16X2) return launch_tc<FBC_PREC_BF16X2>(A, P, n_rhs, st, n_modes);
    if (P.precision == FBC_PREC_BF16X3) return launch_tc<FBC_PREC_BF16X3>(A, P, n_rhs, st, n_modes);
    return cudaErrorInvalidValue;
}

}  // namespace fbc
