// Fused inference of the mode-table surrogate on the tensor cores (tcgen05).
//
// Tiles of 128 rows pass through the whole network 4 -> H -> H -> H -> 6 without
// leaving the SM.  A CTA keeps two tiles in flight, each with eight epilogue
// warps and a warp that issues its products:
//   * the row features (computed from the difference and the mode, or read)
//     are split into three bf16 pieces side by side in one [128][16] A operand,
//     the first layer's weights repeated along K to match; three more columns
//     hold ones, against which B operands of the biases' three bf16 pieces (24
//     bits) start the accumulators;
//   * each layer is one or two passes of tcgen05.mma (M = 128, N = H or 16,
//     K = 16 per instruction) over the activation pieces, against the layer's
//     BF16 weights held in shared memory for the kernel's lifetime, with the
//     FP32 accumulator in tensor memory, in two buffers by turns: a layer's
//     products start as soon as 16 columns of its operand are there;
//   * the epilogue reads the accumulator (tcgen05.ld), applies SiLU and splits
//     the activation into hi + lo bf16 pieces for the next layer (warps w and
//     w + 4 share a TMEM lane quadrant and take one half of the columns each),
//     16 columns to a hand-over;
//   * the last layer's six outputs are written as rows, or multiplied by the
//     decay s(q, r) and written straight into the mode slice of the difference.
// Weights are exact in bf16 and activations carry about 16 mantissa bits
// (inputs 24), so the result matches an FP32 evaluation with BF16 weights to
// a few units in 1e-5.
//
// What bounds it: the epilogues, 3 H SiLU a row.  Their special-function
// instructions (two a value would be 20 us more than the pair's three) and the
// rest, about 9 issue slots a value, take 61 % of the issue slots; the tensor pipe
// runs 39 % of the time.  10^6 rows, H = 128: 1.18 ms with one tile in flight,
// barriers of the whole CTA, expf and a rounded reciprocal; 0.24 ms with two
// tiles, 0.17 ms with the products started by column chunks of 16 (0.19 of 32)
// and the biases in the products.  Against 64 bits the outputs of 2 * 10^5 rows
// differ by 3.5e-6 to 5.3e-6 at H = 32 to 128, 0.1 to 3 % less than before.
//
// Every wait on an mbarrier is bounded; on a timeout the CTA records the
// status word, stops, waits once more (bounded) for its own tensor-core work,
// frees its tensor memory and returns.
#include <cuda_bf16.h>

#include "fbc_f32x2.cuh"
#include "fbc_internal.cuh"
#include "fbc_tc.cuh"

namespace fbc {
namespace {

constexpr int kRows = 128;
constexpr int kMaxH = 128;
constexpr int kTiles = 2;                       // tile slots (tiles in flight) per CTA
constexpr int kEpiWarps = 8;                    // epilogue warps of a tile
constexpr int kThreads = (kTiles * kEpiWarps + 4) * 32;  // with a warpgroup of which one warp a slot issues its products
constexpr int kRegsLaunch = 96, kRegsEpi = 104, kRegsMma = 64;  // registers a thread
constexpr int kXPieces = 3, kActPieces = 2;
constexpr int kXBytes = kRows * 16 * 2;         // the input operand [128][16]
constexpr int kTmemCols = 512;                  // two accumulators of 128 columns per slot
static_assert(kXPieces * kSurIn <= 16 && kSurOut <= 8, "input pieces share one K = 16 step, outputs one read");

using tc::canon_bf16;
using tc::sdesc;
using tc::smem_u32;

constexpr size_t smem_bytes(int H) {
    return 3 * (size_t)H * 16 * 2 + 2 * (size_t)H * H * 2 + (size_t)16 * H * 2 + 16 * 4 +
           kTiles * (kXBytes + (size_t)kActPieces * kRows * H * 2);
}

__device__ __forceinline__ uint32_t bf16_bits(float x) { return (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(x)); }
__device__ __forceinline__ uint32_t bf16_pair(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}

// SiLU of z0 and z1, z / (1 + 2^(-z log2 e)), split into bf16 pieces hi + lo.  One reciprocal serves both: each z is held at
// -41.5 from below (a NaN stays one), so that the product of the two denominators stays below 2^120; there and beyond the
// result is -4e-17 where |SiLU| is at most that.  The factors that multiply z are at most 1: a large z passes through
// whatever its neighbour is.  The approximate instructions are good to about 2^-22, the pieces to 2^-17.
__device__ __forceinline__ void silu_split2(float z0, float z1, uint32_t& hi, uint32_t& lo) {
    float t0, t1, e0, e1, a0, a1, r, v0, v1;
    asm("max.NaN.f32 %0, %1, %2;" : "=f"(z0) : "f"(z0), "f"(-41.5f));
    asm("max.NaN.f32 %0, %1, %2;" : "=f"(z1) : "f"(z1), "f"(-41.5f));
    const uint64_t z = pk2(z0, z1);
    upk2(mul2(z, pk2(-1.4426950408889634f, -1.4426950408889634f)), t0, t1);
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e0) : "f"(t0));
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e1) : "f"(t1));
    upk2(add2(pk2(e0, e1), pk2(1.f, 1.f)), a0, a1);
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a0 * a1));
    const uint64_t v = mul2(z, mul2(pk2(a1, a0), pk2(r, r)));
    upk2(v, v0, v1);
    hi = bf16_pair(v0, v1);
    upk2(sub2(v, pk2(__uint_as_float(hi << 16), __uint_as_float(hi & 0xffff0000u))), v0, v1);
    lo = bf16_pair(v0, v1);
}

// the weights of a layer as B operand [N][K] (element (n, k) = W[k][n]), eight k of a column at a time
__device__ __forceinline__ void load_weights(unsigned char* dst, const float* __restrict__ W, int K, int N, int n_w) {
    const uint32_t sbo = (uint32_t)K * 16;
    for (int e = threadIdx.x; e < N * (K / 8); e += kThreads) {
        const int kg = e / N, n = e % N;
        uint32_t w[4];
#pragma unroll
        for (int j = 0; j < 4; j++) {
            const float* p = W + (size_t)(8 * kg + 2 * j) * n_w + n;
            w[j] = n < n_w ? bf16_bits(p[0]) | bf16_bits(p[n_w]) << 16 : 0u;
        }
        *(uint4*)(dst + canon_bf16(n, 8 * kg, sbo)) = make_uint4(w[0], w[1], w[2], w[3]);
    }
}

constexpr __host__ __device__ uint32_t idesc(int N) {  // bf16 operands, FP32 accumulator, M = 128
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(kRows >> 4) << 24);
}

static_assert(kTiles * kEpiWarps * 32 * kRegsEpi + 128 * kRegsMma <= kThreads * kRegsLaunch, "the shares fit in the launch's");

template <int H, bool SLICE>
__global__ void __launch_bounds__(kThreads, 1) k_mlp_tc(MlpArgs a) {
    extern __shared__ __align__(1024) unsigned char smem[];
    constexpr int CH = 16;       // columns of one read and one hand-over, one K step of the next layer
    constexpr int NCH = H / CH;  // chunk q: columns (q & 1) H / 2 + (q >> 1) CH, of one half of the warps
    __shared__ uint64_t bar_x[kTiles], bar_act[kTiles][NCH], bar_acc[kTiles], bar_out[kTiles], bar_drain[kTiles];
    __shared__ uint32_t tbase;
    __shared__ int s_abort;
    constexpr uint32_t sboH = (uint32_t)H * 16;       // 8-row group stride of a K = H operand
    constexpr size_t actPiece = (size_t)kRows * H * 2;
    unsigned char* sW1 = smem;                        // 3 x [H][16]: layer 1's weights and bias, layer 2's and 3's bias
    unsigned char* sW2 = sW1 + 3 * (size_t)H * 16 * 2;  // [H][H]
    unsigned char* sW3 = sW2 + (size_t)H * H * 2;     // [H][H]
    unsigned char* sW4 = sW3 + (size_t)H * H * 2;     // [16][H]
    unsigned char* sX0 = sW4 + (size_t)16 * H * 2;    // per tile [128][16]
    unsigned char* sAct0 = sX0 + kTiles * kXBytes;    // per tile 2 x [128][H]
    float* sB4 = (float*)(sAct0 + kTiles * kActPieces * actPiece);  // [16]
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;

    {
        const float* P = a.params;
        for (int e = threadIdx.x; e < 3 * H; e += kThreads) {
            const int l = e / H, n = e % H;
            uint32_t w[8] = {};  // K = 16: the four inputs' weights once per piece (layer 1), the bias' three pieces, 0
            if (l == 0)
#pragma unroll
                for (int p = 0; p < 2 * kXPieces; p++) {
                    const float* W = P + a.off[0] + 2 * (p & 1) * H + n;
                    w[p] = bf16_bits(W[0]) | bf16_bits(W[H]) << 16;
                }
            float b = P[a.off[1 + 2 * l] + n];
            uint32_t q[3];
#pragma unroll
            for (int p = 0; p < 3; p++) {
                q[p] = bf16_bits(b);
                b = __fsub_rn(b, __uint_as_float(q[p] << 16));
            }
            w[6] = q[0] | q[1] << 16, w[7] = q[2];
            unsigned char* o = sW1 + (size_t)l * H * 16 * 2;
            *(uint4*)(o + canon_bf16(n, 0, 256)) = make_uint4(w[0], w[1], w[2], w[3]);
            *(uint4*)(o + canon_bf16(n, 8, 256)) = make_uint4(w[4], w[5], w[6], w[7]);
        }
        load_weights(sW2, P + a.off[2], H, H, H);
        load_weights(sW3, P + a.off[4], H, H, H);
        load_weights(sW4, P + a.off[6], H, 16, kSurOut);
        for (int e = threadIdx.x; e < 16; e += kThreads) sB4[e] = e < kSurOut ? P[a.off[7] + e] : 0.f;
    }
    if (threadIdx.x == 0) {
        s_abort = 0;
        for (int t = 0; t < kTiles; t++) {
            tc::mbar_init(&bar_x[t], kEpiWarps / 2);
            for (int q = 0; q < NCH; q++) tc::mbar_init(&bar_act[t][q], kEpiWarps / 2);
            tc::mbar_init(&bar_acc[t], 1);
            tc::mbar_init(&bar_out[t], 1);
            tc::mbar_init(&bar_drain[t], 1);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tbase)),
                     "r"(kTmemCols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tbase;
    volatile int* abort = &s_abort;

    const int tiles_per_mode = (a.n + kRows - 1) / kRows;
    const int n_tiles = tiles_per_mode * (SLICE ? a.n_modes : 1);
    const int step = kTiles * gridDim.x;

    auto wait = [&](uint64_t* m, uint32_t parity) {
        const bool ok = __all_sync(0xffffffffu, tc::wait_or_abort(m, parity, abort, tc::kWaitLimit));
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        return ok;
    };

    if (warp >= kTiles * kEpiWarps) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsMma));
        const int t = warp - kTiles * kEpiWarps;  // the tile slot whose products this warp issues
        if (t < kTiles) {
            const uint32_t el = tc::elect_one();
            const uint64_t dX = sdesc(smem_u32(sX0 + t * kXBytes), 128, 256), dW1 = sdesc(smem_u32(sW1), 128, 256);
            const uint64_t dA = sdesc(smem_u32(sAct0 + t * kActPieces * actPiece), 128, sboH);
            const uint64_t dW2 = sdesc(smem_u32(sW2), 128, sboH), dW4 = sdesc(smem_u32(sW4), 128, sboH);
            const uint32_t acc = tmem + 256 * t;
            uint32_t px = 0, pa = 0;
            bool ok = true;
            for (int tile = t * gridDim.x + blockIdx.x; ok && tile < n_tiles; tile += step) {
                if (!(ok = wait(&bar_x[t], px))) break;
                px ^= 1u;
                tc::mma_ss(acc, dX, dW1, idesc(H), 0u, el);
                tc::commit_elected(&bar_acc[t], el);
                for (int l = 1; l < 4; l++, pa ^= 1u) {
                    const uint64_t dB = l == 3 ? dW4 : dW2 + (uint64_t)(l - 1) * (H * H * 2 / 16);
                    const uint32_t d = acc + 128 * (l & 1), id = l == 3 ? idesc(16) : idesc(H);
                    // (chunks 0 and 1 first: all eight warps have passed one of them, so they are done with the accumulator
                    // of layer l - 2)
                    if (!(ok = wait(&bar_act[t][0], pa))) break;
#pragma unroll
                    for (int q = 0; q < NCH; q++) {
                        if (q != 1 && !(ok = wait(&bar_act[t][q ? q : 1], pa))) break;
                        if (q == 0 && l < 3)  // the bias: the input operand's ones
                            tc::mma_ss(d, dX, dW1 + l * (H * 16 * 2 / 16), id, 0u, el);
#pragma unroll
                        for (int p = 0; p < kActPieces; p++)
#pragma unroll
                            for (int k = 0; k < CH / 16; k++) {
                                const int s = ((q & 1) * (H / 2) + (q >> 1) * CH) / 16 + k;
                                tc::mma_ss(d, dA + p * (actPiece / 16) + 16 * s, dB + 16 * s, id, (q | p | k) || l < 3 ? 1u : 0u,
                                           el);
                            }
                    }
                    if (!ok) break;
                    tc::commit_elected(l == 3 ? &bar_out[t] : &bar_acc[t], el);
                }
            }
            if (!ok) {  // a second and last bounded wait, for this warp's own tensor-core work
                *abort = 1;
                tc::commit_elected(&bar_drain[t], el);
                tc::mbar_wait(&bar_drain[t], 0);
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            }
        }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsEpi));
        const int t = warp / kEpiWarps;                         // the CTA's tile slot
        const int quad = warp & 3, half = (warp >> 2) & 1;
        const int row = quad * 32 + lane;                       // TMEM lane = row of the tile
        const uint32_t acc = tmem + 256 * t + ((uint32_t)(quad * 32) << 16);
        unsigned char* sX = sX0 + t * kXBytes;
        unsigned char* sAct = sAct0 + t * kActPieces * actPiece;
        uint32_t pc = 0, po = 0;
        // The first half of the warps writes a tile's input operand from what it has fetched before, the second half the
        // tile's outputs.
        float x[kSurIn];
        int2 d = make_int2(1, 0);
        auto fetch = [&](int tile) {
            const int i = (tile % tiles_per_mode) * kRows + row;
            if (SLICE) {
                if (i < a.n) d = a.far[i];
            } else if (half == 0) {
#pragma unroll
                for (int j = 0; j < kSurIn; j++) x[j] = i < a.n ? a.X[(size_t)i * kSurIn + j] : 0.f;
            }
        };
        auto put_x = [&](int tile) {
            if (SLICE) surrogate_features(d.x, d.y, a.k0 + tile / tiles_per_mode, a.L, a.c, x);
            uint32_t w[8] = {0, 0, 0, 0, 0, 0, 0x3f803f80u, 0x3f80u};  // three ones for the bias
#pragma unroll
            for (int p = 0; p < kXPieces; p++)
#pragma unroll
                for (int j = 0; j < kSurIn; j += 2) {
                    const uint32_t h = bf16_pair(x[j], x[j + 1]);
                    w[(p * kSurIn + j) / 2] = h;
                    x[j] = __fsub_rn(x[j], __uint_as_float(h << 16));
                    x[j + 1] = __fsub_rn(x[j + 1], __uint_as_float(h & 0xffff0000u));
                }
            *(uint4*)(sX + canon_bf16(row, 0, 256)) = make_uint4(w[0], w[1], w[2], w[3]);
            *(uint4*)(sX + canon_bf16(row, 8, 256)) = make_uint4(w[4], w[5], w[6], w[7]);
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&bar_x[t]);
        };

        int tile = t * gridDim.x + blockIdx.x;
        bool ok = true;
        if (tile < n_tiles) {
            fetch(tile);
            if (half == 0) put_x(tile);
        }
        for (; ok && tile < n_tiles; tile += step) {
            if (half == 0 && tile + step < n_tiles) fetch(tile + step);
            for (int l = 0; ok && l < 3; l++) {
                if (!(ok = wait(&bar_acc[t], pc))) break;
                pc ^= 1u;
#pragma unroll
                for (int c = 0; c < H / 2; c += CH) {
                    float v[CH];
                    tc::ld16(acc + 128 * (l & 1) + (uint32_t)(half * (H / 2) + c), v);
                    unsigned char* o = sAct + canon_bf16(row, half * (H / 2) + c, sboH);
#pragma unroll
                    for (int j = 0; j < CH; j += 8) {
                        uint32_t hi[4], lo[4];
#pragma unroll
                        for (int q = 0; q < 4; q++) silu_split2(v[j + 2 * q], v[j + 2 * q + 1], hi[q], lo[q]);
                        *(uint4*)(o + 16 * j) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
                        *(uint4*)(o + 16 * j + actPiece) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
                    }
                    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) tc::mbar_arrive(&bar_act[t][2 * (c / CH) + half]);
                }
            }
            if (!ok) break;
            if (half == 0) {
                if (tile + step < n_tiles) put_x(tile + step);  // (the products that read this tile's input are done)
                continue;
            }
            double sc = 0.0;
            size_t cell = 0;
            if (SLICE) {
                sc = surrogate_scale(surrogate_qr(d.x, d.y, a.k0 + tile / tiles_per_mode, a.L, a.c), a.c);
                cell = (size_t)(d.y - a.box_y0) * a.Dx + (d.x - a.box_x0);
            }
            if (!(ok = wait(&bar_out[t], po))) break;
            po ^= 1u;
            uint32_t u[8];
            tc::ld8_nowait(acc + 128, u);
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
            const int i = (tile % tiles_per_mode) * kRows + row;
            if (i < a.n) {
                float* o = SLICE ? a.slice + (size_t)(tile / tiles_per_mode) * a.slice_floats + cell * kSurOut
                                 : a.Y + (size_t)i * kSurOut;
#pragma unroll
                for (int j = 0; j < kSurOut; j++) {
                    const float y = __uint_as_float(u[j]) + sB4[j];
                    o[j] = SLICE ? (float)((double)y * sc) : y;
                }
            }
            if (tile + step < n_tiles) fetch(tile + step);
        }
        if (!ok) *abort = 1;
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (threadIdx.x == 0 && s_abort) atomicExch(a.status, FBC_ERR_TIMEOUT);
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols));
}

template <int H>
cudaError_t launch_width(const MlpArgs& a, int grid, cudaStream_t st) {
    constexpr size_t smem = smem_bytes(H);
    const auto k = a.slice ? k_mlp_tc<H, true> : k_mlp_tc<H, false>;
    if (cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) return e;
    k<<<grid, kThreads, smem, st>>>(a);
    return cudaGetLastError();
}

int sm_count() {
    static int n = 0;
    if (!n) {
        int dev = 0;
        cudaGetDevice(&dev);
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1) n = 1;
    }
    return n;
}

}  // namespace

// the epilogue gives each half of the CTA H / 2 columns in steps of 16
bool mlp_tc_supported(int H) { return H >= 32 && H <= kMaxH && H % 32 == 0; }

cudaError_t launch_mlp_tc(const MlpArgs& a, cudaStream_t st) {
    if (!mlp_tc_supported(a.H) || a.n < 1 || !a.status) return cudaErrorInvalidValue;
    if (a.slice ? !a.far || a.n_modes < 1 : !a.X || !a.Y) return cudaErrorInvalidValue;
    const int tiles = ((a.n + kRows - 1) / kRows) * (a.slice ? a.n_modes : 1);
    const int grid = std::min(tiles, sm_count());
    switch (a.H) {
        case 32: return launch_width<32>(a, grid, st);
        case 64: return launch_width<64>(a, grid, st);
        case 96: return launch_width<96>(a, grid, st);
        default: return launch_width<128>(a, grid, st);
    }
}

}  // namespace fbc
