// conv.cu -- 3x3x3 convolutions with zero padding as implicit GEMMs on the tcgen05 tensor
// cores:
//   Y[m][co] = sum_{tap, ci} X[m shifted by tap][ci] * W[co][tap * cin + ci]
// for activations X [B][n][n][n][cin] (BF16, channels last, voxel m = ((b n + z) n + y) n + x)
// and W [cout][Kp] (K index tap * cin + ci, tap = (kz 3 + ky) 3 + kx reading the input at
// (z + kz - 1, y + ky - 1, x + kx - 1)).  No im2col matrix goes through HBM: the A operand of
// the K block (tap, channel chunk) is loaded straight from X by one 5D TMA box
//   {BKC channels, bx, by, bz, bb} at (c0, x0 + kx - 1, y0 + ky - 1, z0 + kz - 1, b0),
// the 128 voxels of the M tile (bx by bz bb = 128, whole x-rows) seen through the tap's
// shift; the box's out-of-range part -- the zero padding -- arrives as zeros (TMA fill).
// The box lands in shared memory exactly as the 2D box of an im2col matrix would (rows of
// BKC channels, 128-byte swizzle for 64 channels, 64-byte swizzle for 32).  Three kernels:
//   conv_bf16_kernel    one tap at a time, the MMA side the GEMM's: one CTA of 128 threads per
//                       128 x BN tile, warp 0 producing into a 4-stage mbarrier ring, warp 1
//                       issuing tcgen05.mma into TMEM (an elected lane of each issues), all
//                       four warps draining the accumulator (grids below 16^3, and 256^3);
//   conv_x3_kernel      three kx taps side by side in the MMA's N, persistent, 320 threads, up to
//                       eight stages, epilogue warps of their own (16^3 to 128^3);
//   conv_wgrad_kernel, conv_wgrad9_kernel   the weight gradient, below.
// Epilogues: bias + ReLU + BF16 (the forward pass) or FP32 (the input gradient, the convolution
// of the output gradient with the mirrored weights).  Every wait is bounded as in gemm.cu.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <mutex>

#include "nn.h"
#include "tc.cuh"
#include "wgrad_plan.h"

namespace lbm {
namespace nn {

namespace {

constexpr int CBM = 128, CSTAGES = 4;

template <int BN, int BKC>
struct ConvSmem {
    static constexpr int A_BYTES = CBM * BKC * 2;
    static constexpr int B_BYTES = BN * BKC * 2;
    static constexpr int STAGE = A_BYTES + B_BYTES;
    static constexpr int BYTES = 1024 + CSTAGES * STAGE + 256;
    static constexpr uint32_t TMEM_COLS = BN < 32 ? 32 : BN;
};

struct ConvArgs {
    int M, N;               // output rows (B n^3) and columns (cout)
    int n;                  // grid edge
    int chunks;             // channel chunks of BKC per tap (cin / BKC)
    int bx, by, bz;         // the M tile as a box of the grid (with bb = 128 / (bx by bz))
    int mode;               // CONV_BIAS_RELU_BF16 or CONV_F32
    void* C;                // output [M][N]
    const float* bias;      // bias[N] (CONV_BIAS_RELU_BF16)
    int* err;
};

__device__ __forceinline__ uint64_t sdesc(uint32_t saddr, int bkc) {
    return bkc == 64 ? sdesc_k_sw128(saddr) : sdesc_k_sw64(saddr);
}

// Epilogue of 16 output channels col0.. of one voxel: bias + ReLU + BF16, or FP32.
__device__ __forceinline__ void conv_store16(void* out, int N, int mode, const float* __restrict__ bias,
                                             int row, int col0, float (&v)[16]) {
    if (col0 >= N) return;
    const bool whole = (N % 8) == 0;  // 16-byte stores of 8 (BF16) or 4 columns: none is cut
    if (mode == CONV_BIAS_RELU_BF16) {
        __nv_bfloat16* C = static_cast<__nv_bfloat16*>(out) + (int64_t)row * N;
#pragma unroll
        for (int j = 0; j < 16; ++j) v[j] = fmaxf(v[j] + (col0 + j < N ? bias[col0 + j] : 0.f), 0.f);
        if (whole) {
            uint4 pk[2];
            __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(pk);
#pragma unroll
            for (int j = 0; j < 8; ++j) h[j] = __floats2bfloat162_rn(v[2 * j], v[2 * j + 1]);
            reinterpret_cast<uint4*>(C + col0)[0] = pk[0];
            if (col0 + 8 < N) reinterpret_cast<uint4*>(C + col0)[1] = pk[1];
        } else {
#pragma unroll
            for (int j = 0; j < 16; ++j)
                if (col0 + j < N) C[col0 + j] = __float2bfloat16_rn(v[j]);
        }
    } else {
        float* C = static_cast<float*>(out) + (int64_t)row * N;
        if (whole) {
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (col0 + 4 * j < N)
                    reinterpret_cast<float4*>(C + col0)[j] =
                        make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
        } else {
#pragma unroll
            for (int j = 0; j < 16; ++j)
                if (col0 + j < N) C[col0 + j] = v[j];
        }
    }
}

template <int BN, int BKC>
__global__ void __launch_bounds__(128, 1)
    conv_bf16_kernel(const __grid_constant__ CUtensorMap tmX,
                     const __grid_constant__ CUtensorMap tmW, ConvArgs args) {
    using L = ConvSmem<BN, BKC>;
    extern __shared__ uint8_t conv_smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>(
        (reinterpret_cast<uintptr_t>(conv_smem_raw) + 1023) & ~uintptr_t(1023));
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + CSTAGES * L::STAGE);
    uint64_t* empty = full + CSTAGES;
    uint64_t* done = empty + CSTAGES;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
    __shared__ volatile int failed;

    if (*static_cast<volatile int*>(args.err) != 0) return;  // another CTA timed out
    const int warp = warp_index(), lane = threadIdx.x & 31;
    const int m0 = blockIdx.x * CBM, n0 = blockIdx.y * BN;
    const int nkb = 27 * args.chunks;

    if (threadIdx.x == 0) {
        failed = 0;
        for (int s = 0; s < CSTAGES; ++s) {
            mbar_init(full + s, 1);
            mbar_init(empty + s, 1);
        }
        mbar_init(done, 1);
        mbar_fence_init();
    }
    if (warp == 0) tmem_alloc(tmem_slot, L::TMEM_COLS);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    int issued = 0;
    if (warp == 0) {
        const bool elected = elect_lane();
        // the tile's first voxel (its x0 is 0 unless a row holds several tiles)
        const int n = args.n;
        const int x0 = m0 % n, y0 = (m0 / n) % n, z0 = (m0 / (n * n)) % n, b0 = m0 / (n * n * n);
        int tap = 0, chunk = 0;
        for (int i = 0; i < nkb; ++i) {
            const int s = i % CSTAGES;
            const uint32_t ph = (uint32_t)(i / CSTAGES) & 1u;
            if (i >= CSTAGES && !mbar_wait_warp(empty + s, ph ^ 1u, args.err, 1, &failed)) {
                failed = 1;
                break;
            }
            uint8_t* a = smem + s * L::STAGE;
            const int kz = tap / 9, ky = (tap / 3) % 3, kx = tap % 3;
            if (elected) {
                mbar_expect_tx(full + s, L::STAGE);
                tma_load_5d(a, &tmX, full + s, chunk * BKC, x0 + kx - 1, y0 + ky - 1, z0 + kz - 1, b0);
                tma_load_2d(a + L::A_BYTES, &tmW, full + s, i * BKC, n0);
            }
            ++issued;
            if (++chunk == args.chunks) {
                chunk = 0;
                ++tap;
            }
        }
    } else if (warp == 1) {
        const bool elected = elect_lane();
        const uint32_t idesc = idesc_bf16_f32(CBM, BN), dhi = (uint32_t)(sdesc(0, BKC) >> 32);
        for (int i = 0; i < nkb; ++i) {
            const int s = i % CSTAGES;
            const uint32_t ph = (uint32_t)(i / CSTAGES) & 1u;
            if (!mbar_wait_warp(full + s, ph, args.err, 2, &failed)) {
                failed = 1;
                break;
            }
            tc_fence_after();
            const uint32_t a = (uint32_t)sdesc(smem_u32(smem + s * L::STAGE), BKC), b = a + (L::A_BYTES >> 4);
            if (elected) {
#pragma unroll
                for (int kk = 0; kk < BKC / 16; ++kk)
                    mma_bf16(tmem, a + kk * 2, dhi, b + kk * 2, dhi, idesc, (i > 0 || kk > 0) ? 1u : 0u);
                mma_commit(empty + s);
            }
        }
        if (elected) mma_commit(done);  // also when stopped early: every issued MMA drains before dealloc
    }
    __syncwarp();
    if (!mbar_wait(done, 0, args.err, 3)) failed = 1;
    __syncthreads();
    const bool ok = !failed;
    if (warp == 0 && lane == 0 && failed) {  // let every started copy land
        for (int i = max(0, issued - CSTAGES); i < issued; ++i)
            mbar_wait(full + (i % CSTAGES), (uint32_t)(i / CSTAGES) & 1u, args.err, 4);
    }
    tc_fence_after();
    if (ok) {
        const int row = m0 + warp * 32 + lane;
#pragma unroll 1
        for (int c = 0; c < BN; c += 16) {
            float v[16];
            tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c, v);
            if (row < args.M) conv_store16(args.C, args.N, args.mode, args.bias, row, n0 + c, v);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, L::TMEM_COLS);
}

// 32 bytes to a 32-byte boundary.
__device__ __forceinline__ void store32(void* p, const uint32_t (&h)[8]) {
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(h[0]), "r"(h[1]), "r"(h[2]),
                 "r"(h[3]), "r"(h[4]), "r"(h[5]), "r"(h[6]), "r"(h[7])
                 : "memory");
}

// ---------------------------------------------------------------------------------
// The same convolution with the three kx taps side by side in the MMA's N (16 <= n <= 128; the
// kernel above takes the grids below and beyond).
// An MMA of M = 128 voxels reads 4 KB of A from shared memory per 16 input channels whatever
// its N, so at N = 32 output channels the operand reads (40 cycles) and not the 16 cycles of
// tensor math bound the kernels above.  Here B holds the weights of kx = 0, 1, 2 of a (kz, ky)
// row as 3 BN columns, and A is the UNSHIFTED x-row: the accumulator column kx BN + c of voxel
// x is P_kx[x] = sum over (kz, ky, ci) of X[x] W[c][kz, ky, kx], and the epilogue adds
//   Y[x] = P_0[x - 1] + P_1[x] + P_2[x + 1]
// (P outside the row is the zero padding), the neighbours' values coming by warp shuffles and,
// where an x-row spans several warps (n > 32), through shared memory.  A third of the A reads
// and MMAs, each three times as wide.  A stage holds, of one kz and 32 input channels, the x-rows
// of MT tiles plus one on either side (one 5D box, zero-filled outside the grid), and the tile of
// tap ky is the 128-row window starting at row (t by + ky) n of that box: whole x-rows, so every
// window starts on a swizzle atom, and each loaded row serves three ky taps.
// ---------------------------------------------------------------------------------
struct X3Args {
    int N, n, chunks, cin;  // chunks of 32 input channels
    int ntiles, items;      // tiles of BN output channels; (group of MT tiles, channel tile) pairs
    int mt;                 // tiles per item
    int a_bytes;            // one stage's input box: (mt by + 2) n 64 bytes, by x-rows per 128-voxel tile
    int stage_bytes;        // a_bytes + 9 BN 64
    int stages;
    int mode;
    void* C;
    const float* bias;
    int wide;  // rows of C start on 32 bytes and hold whole 16-column chunks
    int* err;
};
constexpr int kX3Threads = 320;  // producer, MMA, two sets of four epilogue warps

constexpr int kX3Bias = 256;  // output channels in whole tiles, at most: 4 of 64, 5 of 48

// The store of 16 output channels of a row, bias and ReLU applied.  In 32-byte pieces where the
// rows allow it: a lane's row is a sector of its own, which two 16-byte stores write twice.
__device__ __forceinline__ void x3_store16(const X3Args& a, int row, int col0, const float (&v)[16]) {
    if (col0 >= a.N) return;
    if (a.mode == CONV_BIAS_RELU_BF16) {
        __nv_bfloat16* C = static_cast<__nv_bfloat16*>(a.C) + (int64_t)row * a.N + col0;
        uint32_t h[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const __nv_bfloat162 b = __floats2bfloat162_rn(v[2 * j], v[2 * j + 1]);
            h[j] = *reinterpret_cast<const uint32_t*>(&b);
        }
        if (a.wide) {
            store32(C, h);
        } else if (a.N % 8 == 0) {
            reinterpret_cast<uint4*>(C)[0] = make_uint4(h[0], h[1], h[2], h[3]);
            if (col0 + 8 < a.N) reinterpret_cast<uint4*>(C)[1] = make_uint4(h[4], h[5], h[6], h[7]);
        } else {
#pragma unroll
            for (int j = 0; j < 16; ++j)
                if (col0 + j < a.N) C[j] = __float2bfloat16_rn(v[j]);
        }
    } else {
        float* C = static_cast<float*>(a.C) + (int64_t)row * a.N + col0;
        if (a.wide) {
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                uint32_t h[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) h[j] = __float_as_uint(v[8 * q + j]);
                store32(C + 8 * q, h);
            }
        } else if (a.N % 8 == 0) {
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (col0 + 4 * j < a.N)
                    reinterpret_cast<float4*>(C)[j] = make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
        } else {
#pragma unroll
            for (int j = 0; j < 16; ++j)
                if (col0 + j < a.N) C[j] = v[j];
        }
    }
}

// One item's place: first row, grid position, output channels, the kz planes inside the grid.
struct X3Item {
    int m0, n0, y0, z0, b0, kz0, kz1;
    __device__ X3Item(const X3Args& a, int item, int bn) {
        const int mg = item / a.ntiles, n = a.n;
        n0 = (item - mg * a.ntiles) * bn;
        m0 = mg * a.mt * CBM;
        y0 = (m0 / n) % n, z0 = (m0 / (n * n)) % n, b0 = m0 / (n * n * n);
        kz0 = z0 == 0 ? 1 : 0, kz1 = z0 == n - 1 ? 2 : 3;
    }
};

// Persistent: a CTA per SM takes items by stride.  The producer warp keeps the stage ring full
// across items, the MMA warp fills one of two accumulator sets while the epilogue warps drain
// the other.  (With a CTA per item, two on an SM, the 64^3 96 -> 32 layer, batch 2, spent 25 of
// 87 us in 2048 CTAs' set-up and 22 in epilogues.)  Per call with the host wait, that form / this
// one: that layer 110 / 92 us, 64^3 32 -> 32 77 / 64, 32^3 64 -> 192 in FP32 80 / 68, 128^3
// 32 -> 32 234 / 169, 16^3 128 -> 128 (an item per CTA) 35 / 35.  A 96 -> 32 item takes 66 cycles per
// MMA of 96 columns (48 of math); leaving out either the weights' or the input's loads changes
// that little.  With 32 input channels the epilogue is the longer part: the rows' ends go between
// warps as quadruples that every lane reads, the bias comes from shared memory, and a lane's channels
// are stored as whole 32-byte sectors.  Before / after those: 64^3 batch 2 32 -> 32 63 / 59 us and
// in FP32 73 / 68, 128^3 FP32 233 / 203, 32^3 64 -> 192 FP32 67 / 62.
template <int BN>
__global__ void __launch_bounds__(kX3Threads, 1)
    conv_x3_kernel(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmW,
                   X3Args args) {
    extern __shared__ uint8_t x3_smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>(
        (reinterpret_cast<uintptr_t>(x3_smem_raw) + 1023) & ~uintptr_t(1023));
    const int S = args.stages;
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + S * args.stage_bytes);
    uint64_t* empty = full + S;
    uint64_t* acc_full = empty + S;   // [2]
    uint64_t* acc_empty = acc_full + 2;
    uint64_t* done = acc_empty + 2;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
    __shared__ volatile int failed;
    __shared__ float4 edge[2][2][4][2][4];  // of each epilogue set: P_0 of a warp's last row, P_2 of its first
    constexpr int W = 3 * BN, B_TILE = BN * 64;

    __shared__ float4 bias[kX3Bias / 4];

    if (*static_cast<volatile int*>(args.err) != 0) return;  // another CTA timed out
    const int warp = warp_index(), lane = threadIdx.x & 31;
    const int MT = args.mt, n = args.n;
    if (args.mode == CONV_BIAS_RELU_BF16)
        for (int c = threadIdx.x; c < kX3Bias; c += kX3Threads)
            reinterpret_cast<float*>(bias)[c] = c < args.N ? args.bias[c] : 0.f;

    if (threadIdx.x == 0) {
        failed = 0;
        for (int s = 0; s < S; ++s) {
            mbar_init(full + s, 1);
            mbar_init(empty + s, 1);
        }
        for (int s = 0; s < 2; ++s) {
            mbar_init(acc_full + s, 1);
            mbar_init(acc_empty + s, 8);  // a lane of every epilogue warp
        }
        mbar_init(done, 1);
        mbar_fence_init();
    }
    if (warp == 0) tmem_alloc(tmem_slot, 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    int issued = 0;
    if (warp == 0) {
        const bool elected = elect_lane();
        int s = 0;
        uint32_t ph = 1;  // parity of the slot's last release
        bool ok = true;
        for (int item = blockIdx.x; ok && item < args.items; item += gridDim.x) {
            const X3Item it(args, item, BN);
            for (int kz = it.kz0; ok && kz < it.kz1; ++kz)
                for (int chunk = 0; chunk < args.chunks; ++chunk) {
                    if (issued >= S && !mbar_wait_warp(empty + s, ph, args.err, 1, &failed)) {
                        failed = 1;
                        ok = false;
                        break;
                    }
                    uint8_t* a = smem + s * args.stage_bytes;
                    if (elected) {
                        mbar_expect_tx(full + s, (uint32_t)(args.a_bytes + 9 * B_TILE));
                        tma_load_5d(a, &tmX, full + s, chunk * 32, 0, it.y0 - 1, it.z0 + kz - 1, it.b0);
#pragma unroll
                        for (int t = 0; t < 9; ++t)  // (ky, kx) of this kz
                            tma_load_2d(a + args.a_bytes + t * B_TILE, &tmW, full + s,
                                        (kz * 9 + t) * args.cin + chunk * 32, it.n0);
                    }
                    ++issued;
                    if (++s == S) s = 0, ph ^= 1u;
                }
        }
    } else if (warp == 1) {
        const bool elected = elect_lane();
        const uint32_t idesc = idesc_bf16_f32(CBM, W), dhi = (uint32_t)(sdesc_k_sw64(0) >> 32);
        const uint32_t window = (uint32_t)(n * 64 >> 4);
        int s = 0, k = 0;
        uint32_t ph = 0;
        bool ok = true;
        for (int item = blockIdx.x; ok && item < args.items; item += gridDim.x, ++k) {
            const X3Item it(args, item, BN);
            const uint32_t acc = tmem + (uint32_t)((k & 1) * 256);
            if (k >= 2 && !mbar_wait_warp(acc_empty + (k & 1), (uint32_t)(k / 2 + 1) & 1u, args.err, 5, &failed)) {
                failed = 1;
                break;
            }
            const int nkb = (it.kz1 - it.kz0) * args.chunks;
            for (int i = 0; i < nkb; ++i) {
                if (!mbar_wait_warp(full + s, ph, args.err, 2, &failed)) {
                    failed = 1;
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint32_t stage = smem_u32(smem + s * args.stage_bytes);
                const uint32_t alo = (uint32_t)sdesc_k_sw64(stage);
                const uint32_t blo = (uint32_t)sdesc_k_sw64(stage + (uint32_t)args.a_bytes);
                if (elected) {
                    for (int t = 0; t < MT; ++t) {
#pragma unroll
                        for (int ky = 0; ky < 3; ++ky) {  // the window of tap ky: 128 t + n ky rows of 64 bytes on
                            const uint32_t at = alo + (uint32_t)(t * (CBM * 64 >> 4)) + (uint32_t)ky * window;
                            const uint32_t bt = blo + (uint32_t)(ky * (3 * B_TILE >> 4));
#pragma unroll
                            for (int kk = 0; kk < 2; ++kk)
                                mma_bf16(acc + (uint32_t)(t * W), at + kk * 2, dhi, bt + kk * 2, dhi, idesc,
                                         (i > 0 || ky > 0 || kk > 0) ? 1u : 0u);
                        }
                    }
                    mma_commit(empty + s);
                }
                if (++s == S) s = 0, ph ^= 1u;
            }
            if (elected && ok) mma_commit(acc_full + (k & 1));
        }
        if (elected) mma_commit(done);  // also when stopped early: every issued MMA drains before dealloc
    } else {
        const int quarter = warp & 3, set = (warp - 2) >> 2;  // a warp reads the TMEM lanes of its index mod 4
        const int x = (quarter * 32 + lane) & (n - 1);
        const bool first = x == 0, last = x == n - 1;
        int k = 0, par = 0;
        for (int item = blockIdx.x; item < args.items; item += gridDim.x, ++k) {
            const X3Item it(args, item, BN);
            // the four warps of a set give up together: they meet at its barrier below
            const bool there = mbar_wait_warp(acc_full + (k & 1), (uint32_t)(k / 2) & 1u, args.err, 3, &failed);
            if (!bar_all(1 + set, 128, there)) {
                failed = 1;
                break;
            }
            tc_fence_after();
            const uint32_t acc = tmem + (uint32_t)((k & 1) * 256) + ((uint32_t)(quarter * 32) << 16);
            // the item's MT BN / 16 chunks of 16 channels go to the two sets in turn
            for (int q = set; q < MT * (BN / 16); q += 2, par ^= 1) {
                const int t = q / (BN / 16), c = (q - t * (BN / 16)) * 16;
                const uint32_t base = acc + (uint32_t)(t * W + c);
                float p0[16], v[16], p2[16];
                tmem_ld16_issue(base, p0);
                tmem_ld16_issue(base + (uint32_t)BN, v);
                tmem_ld16_issue(base + (uint32_t)(2 * BN), p2);
                tmem_wait_ld();
                tmem_landed(p0);
                tmem_landed(v);
                tmem_landed(p2);
                float l[16], r[16];
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    l[j] = __shfl_up_sync(0xffffffffu, p0[j], 1);
                    r[j] = __shfl_down_sync(0xffffffffu, p2[j], 1);
                }
                if (n > 32) {  // block-uniform: an x-row spans warps
                    float4(&e)[4][2][4] = edge[set][par];
                    if (lane == 31) {
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            e[quarter][0][j] = make_float4(p0[4 * j], p0[4 * j + 1], p0[4 * j + 2], p0[4 * j + 3]);
                    }
                    if (lane == 0) {
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            e[quarter][1][j] = make_float4(p2[4 * j], p2[4 * j + 1], p2[4 * j + 2], p2[4 * j + 3]);
                    }
                    bar_sync(1 + set, 128);
                    // every lane reads (one address per warp) and the lanes at the warp's ends take it
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const float4 el = e[(quarter + 3) & 3][0][j], er = e[(quarter + 1) & 3][1][j];
                        l[4 * j] = lane == 0 ? el.x : l[4 * j];
                        l[4 * j + 1] = lane == 0 ? el.y : l[4 * j + 1];
                        l[4 * j + 2] = lane == 0 ? el.z : l[4 * j + 2];
                        l[4 * j + 3] = lane == 0 ? el.w : l[4 * j + 3];
                        r[4 * j] = lane == 31 ? er.x : r[4 * j];
                        r[4 * j + 1] = lane == 31 ? er.y : r[4 * j + 1];
                        r[4 * j + 2] = lane == 31 ? er.z : r[4 * j + 2];
                        r[4 * j + 3] = lane == 31 ? er.w : r[4 * j + 3];
                    }
                }
#pragma unroll
                for (int j = 0; j < 16; ++j) v[j] += (first ? 0.f : l[j]) + (last ? 0.f : r[j]);
                const int row = it.m0 + t * CBM + quarter * 32 + lane, col0 = it.n0 + c;
                if (args.mode == CONV_BIAS_RELU_BF16) {
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const float4 bj = bias[(col0 >> 2) + j];
                        v[4 * j] = fmaxf(v[4 * j] + bj.x, 0.f);
                        v[4 * j + 1] = fmaxf(v[4 * j + 1] + bj.y, 0.f);
                        v[4 * j + 2] = fmaxf(v[4 * j + 2] + bj.z, 0.f);
                        v[4 * j + 3] = fmaxf(v[4 * j + 3] + bj.w, 0.f);
                    }
                }
                x3_store16(args, row, col0, v);
            }
            tc_fence_before();
            if (lane == 0) mbar_arrive(acc_empty + (k & 1));
        }
    }
    __syncwarp();
    if (!mbar_wait(done, 0, args.err, 3)) failed = 1;
    if (warp == 0 && lane == 0 && failed) {  // let every started copy land
        for (int i = max(0, issued - S); i < issued; ++i)
            mbar_wait(full + (i % S), (uint32_t)(i / S) & 1u, args.err, 4);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0) tmem_dealloc(tmem, 512);
}

using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                   const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                   const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                   CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                             &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    });
    return fn;
}

// X [B][n][n][n][cin] as a 5D tensor (innermost first) read in boxes of
// {bkc, bx, by, bz, bb}; out-of-range elements read as zeros.
bool make_x_map(CUtensorMap* map, const void* X, int B, int n, int cin, int bkc, int bx, int by,
                int bz, int bb) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    const cuuint64_t dims[5] = {(cuuint64_t)cin, (cuuint64_t)n, (cuuint64_t)n, (cuuint64_t)n,
                                (cuuint64_t)B};
    const cuuint64_t row = (cuuint64_t)cin * 2;
    const cuuint64_t strides[4] = {row, row * n, row * n * n, row * n * n * n};
    const cuuint32_t box[5] = {(cuuint32_t)bkc, (cuuint32_t)bx, (cuuint32_t)by, (cuuint32_t)bz,
                               (cuuint32_t)bb};
    const cuuint32_t estr[5] = {1, 1, 1, 1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void*>(X), dims, strides, box,
              estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
              bkc == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B,
              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// W [N][Kp] (row stride ld) read in boxes of bkc x box_rows.
bool make_w_map(CUtensorMap* map, const void* W, int N, int K, long long ld, int bkc, int box_rows) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    const cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)N};
    const cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
    const cuuint32_t box[2] = {(cuuint32_t)bkc, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(W), dims, strides, box,
              estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
              bkc == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B,
              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// ---------------------------------------------------------------------------------
// Weight gradient as an implicit GEMM on both operands in their natural layouts:
//   dW^T[r][co] = sum over voxels v of X[v + shift(tap)][ci] dZ[v][co],  r = tap cin + ci,
// a contraction over the voxels, so both operands are MN-major for the tensor core (the
// row index r of A and the column index co of B are the contiguous ones in memory) and
// neither X nor dZ is transposed or expanded.  K block = 64 consecutive voxels, the box
// {bx, by, bz, bb} of the grid with bx by bz bb = 64 (x-row segments for n >= 64, whole
// rows, planes or samples below).  A operand of the M tile (128 rows = four (tap,
// 32-channel) groups): four 5D TMA boxes {32 channels, bx, by, bz, bb} of X at
// (ci0, x0 + kx - 1, y0 + ky - 1, z0 + kz - 1, b0) with the 64-byte swizzle, each landing
// as 64 K rows of 32 channels (64 bytes): the canonical MN-major tile, swizzle atoms of 8
// K rows 512 bytes apart, the four channel groups 4 KB apart.  The tap's shift and the
// zero padding come from the box coordinates and TMA's zero fill; the innermost
// coordinate stays a multiple of 32 channels.  B operand: dZ [voxels][cout] in boxes
// {BB channels, 64 voxels} (BB = 64 with the 128-byte swizzle, 32 with the 64-byte one
// when BN = 32), BN / BB of them B_GROUP bytes apart.  Split K over the voxels: split z
// stores its partial tile in slice z of the workspace; the slices are added in order
// afterwards.
// ---------------------------------------------------------------------------------
constexpr int WG_STAGES = 4;

template <int BN>
struct WgradSmem {
    static constexpr int A_BYTES = CBM * 64 * 2, B_BYTES = BN * 64 * 2;
    static constexpr int STAGE = A_BYTES + B_BYTES;
    // 2 KB past the ring: the operand reads of the last stage stay inside the allocation
    // under either assignment of the two descriptor strides
    static constexpr int BYTES = 1024 + WG_STAGES * STAGE + 2048 + 256;
    static constexpr uint32_t TMEM_COLS = BN < 32 ? 32 : BN;
    static constexpr int BB = BN < 64 ? BN : 64;         // output channels per B box
    static constexpr uint32_t B_GROUP = BB * 2 * 64;     // bytes of one B box (64 K rows)
    static constexpr uint32_t B_ATOM = BB * 2 * 8;       // bytes of 8 K rows of it
    static constexpr uint32_t B_LAYOUT = BB == 64 ? 2u : 4u;
};

struct WgradArgs {
    int rows;            // 27 cin (rows beyond it, up to the padded count, read as zeros)
    int N;               // cout
    int cin, ln;         // input channels, log2 of the grid edge
    int kblocks;         // 64-voxel blocks in all (ceil(B n^3 / 64))
    int kb_per_split;
    int Mrows;           // rows of a workspace slice (the padded 27 cin)
    float* ws;           // [splits][Mrows][N]
    int* err;
};

template <int BN>
__global__ void __launch_bounds__(128, 1)
    conv_wgrad_kernel(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmB,
                      WgradArgs args) {
    using L = WgradSmem<BN>;
    extern __shared__ uint8_t wg_smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>(
        (reinterpret_cast<uintptr_t>(wg_smem_raw) + 1023) & ~uintptr_t(1023));
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + WG_STAGES * L::STAGE + 2048);
    uint64_t* empty = full + WG_STAGES;
    uint64_t* done = empty + WG_STAGES;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
    __shared__ volatile int failed;

    if (*static_cast<volatile int*>(args.err) != 0) return;  // another CTA timed out
    const int warp = warp_index(), lane = threadIdx.x & 31;
    const int m0 = blockIdx.x * CBM, n0 = blockIdx.y * BN;
    const int kb0 = blockIdx.z * args.kb_per_split;
    const int nkb = min(args.kb_per_split, args.kblocks - kb0);

    if (threadIdx.x == 0) {
        failed = 0;
        for (int s = 0; s < WG_STAGES; ++s) {
            mbar_init(full + s, 1);
            mbar_init(empty + s, 1);
        }
        mbar_init(done, 1);
        mbar_fence_init();
    }
    if (warp == 0) tmem_alloc(tmem_slot, L::TMEM_COLS);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    int issued = 0;
    if (nkb > 0 && warp == 0) {
        const bool elected = elect_lane();
        const int ln = args.ln, mask = (1 << ln) - 1;
        // the (tap, channel) groups of the M tile do not change along K
        int gx[4], gy[4], gz[4], gc[4];
#pragma unroll
        for (int g = 0; g < 4; ++g) {
            const int r = m0 + 32 * g;
            gx[g] = 0, gy[g] = 0, gz[g] = 0, gc[g] = args.cin;  // padding rows: past the channels
            if (r < args.rows) {
                const int tap = r / args.cin;
                gc[g] = r - tap * args.cin;
                gx[g] = tap % 3 - 1;
                gy[g] = (tap / 3) % 3 - 1;
                gz[g] = tap / 9 - 1;
            }
        }
        for (int i = 0; i < nkb; ++i) {
            const int s = i % WG_STAGES;
            const uint32_t ph = (uint32_t)(i / WG_STAGES) & 1u;
            if (i >= WG_STAGES && !mbar_wait_warp(empty + s, ph ^ 1u, args.err, 1, &failed)) {
                failed = 1;
                break;
            }
            uint8_t* a = smem + s * L::STAGE;
            const int v0 = (kb0 + i) << 6;
            const int x0 = v0 & mask, y0 = (v0 >> ln) & mask, z0 = (v0 >> (2 * ln)) & mask, b0 = v0 >> (3 * ln);
            if (elected) {
                mbar_expect_tx(full + s, L::STAGE);
#pragma unroll
                for (int g = 0; g < 4; ++g)
                    tma_load_5d(a + g * 4096, &tmX, full + s, gc[g], x0 + gx[g], y0 + gy[g], z0 + gz[g], b0);
#pragma unroll
                for (int j = 0; j < BN / L::BB; ++j)
                    tma_load_2d(a + L::A_BYTES + j * L::B_GROUP, &tmB, full + s, n0 + j * L::BB, v0);
            }
            ++issued;
        }
    } else if (nkb > 0 && warp == 1) {
        const bool elected = elect_lane();
        const uint32_t idesc = idesc_bf16_f32_mn(CBM, BN);
        // with one B box the leading offset is never used: give it the K stride too
        constexpr uint32_t b_lbo = BN / L::BB > 1 ? L::B_GROUP : L::B_ATOM;
        for (int i = 0; i < nkb; ++i) {
            const int s = i % WG_STAGES;
            const uint32_t ph = (uint32_t)(i / WG_STAGES) & 1u;
            if (!mbar_wait_warp(full + s, ph, args.err, 2, &failed)) {
                failed = 1;
                break;
            }
            tc_fence_after();
            const uint32_t a = smem_u32(smem + s * L::STAGE);
            const uint64_t ad = sdesc_mn(a, 4096, 512, 4);
            const uint64_t bd = sdesc_mn(a + L::A_BYTES, b_lbo, L::B_ATOM, L::B_LAYOUT);
            if (elected) {
#pragma unroll
                for (int kk = 0; kk < 4; ++kk)  // K = 16 per MMA: two atoms of 8 K rows
                    mma_bf16(tmem, (uint32_t)ad + kk * 64, (uint32_t)(ad >> 32),
                                    (uint32_t)bd + kk * (2 * L::B_ATOM >> 4), (uint32_t)(bd >> 32), idesc,
                                    (i > 0 || kk > 0) ? 1u : 0u);
                mma_commit(empty + s);
            }
        }
        if (elected) mma_commit(done);  // also when stopped early: every issued MMA drains before dealloc
    }
    __syncwarp();
    if (nkb > 0 && !mbar_wait(done, 0, args.err, 3)) failed = 1;
    __syncthreads();
    const bool ok = nkb > 0 && !failed;
    if (warp == 0 && lane == 0 && failed) {  // let every started copy land
        for (int i = max(0, issued - WG_STAGES); i < issued; ++i)
            mbar_wait(full + (i % WG_STAGES), (uint32_t)(i / WG_STAGES) & 1u, args.err, 4);
    }
    tc_fence_after();
    if (ok) {
        const int row = m0 + warp * 32 + lane;
        float* C = args.ws + ((int64_t)blockIdx.z * args.Mrows + row) * args.N;
#pragma unroll 1
        for (int c = 0; c < BN; c += 16) {
            float v[16];
            tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c, v);
            const int col0 = n0 + c;
            if (row >= args.Mrows || col0 >= args.N) continue;
            if (col0 + 16 <= args.N && (args.N % 4) == 0) {
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    reinterpret_cast<float4*>(C + col0)[j] = make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
            } else {
#pragma unroll
                for (int j = 0; j < 16; ++j)
                    if (col0 + j < args.N) C[col0 + j] = v[j];
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, L::TMEM_COLS);
}

// ---------------------------------------------------------------------------------
// The weight gradient with the nine (ky, kx) taps side by side in N (n >= 16, up to 64 output
// channels).  With the tap's shift on the other operand,
//   dW^T[kz, ky, kx][ci][co] = sum over u of X[u + kz][ci] dZ[u - (ky, kx)][co],
// one A operand -- 64 voxels of X, four chunks of (kz, 32 channels) as the M tile's rows --
// serves nine taps: for each ky one MMA of M = 128, N = 96 (kx, 32 output channels).  The kernel
// above reads 4 KB of A from shared memory per MMA of N = 32, and every A byte from L2 once per
// tap.  The kx shifts of dZ are three TMA boxes (zero-filled outside the grid); the ky shifts
// come from the neighbouring x-rows: a slot of the ring holds the X rows y0 .. y0 + RB - 1 of a
// block of 64 voxels and the dZ rows one further on, y0 + 1 .. y0 + RB, and the MMAs take the dZ
// rows y0 - 1 .. y0 + RB from this slot and the one or two before it, so that each dZ row is
// loaded once per kx.  A run of blocks that starts (at a plane's or the range's first block)
// is led in by slots with dZ rows only.
// Operand reads and fills of shared memory bound the kernel, not the tensor pipe: per 16 voxels
// three MMAs read 3 (4 + 3) KB and the fill adds 7, 219 cycles at 128 bytes a cycle against 144
// of math.  The dZ rows lie one after another in their ring, [row][kx], so the rows of two ky taps
// are one operand of N = 192 and the A tile is read twice, not three times.  Calls with the host
// wait, three MMAs / two: 64^3 batch 2, 96 -> 32 channels 187 / 163 us, batch 4 535 / 437, 128^3
// 32 -> 32 370 / 304, 64^3 64 -> 64 118 / 105, 32^3 batch 4, 96 -> 64 125 / 117,
// batch 2, 192 -> 64 103 / 97.
// Padding is by zeros of dZ along x and y, of X along z: a non-finite X at an x or y face also reaches
// the taps that point outward there (times zero), as a non-finite dZ does in the kernel above.
// The accumulators fill 288 tensor-memory columns: a CTA holds one M tile of 32 output
// channels and a range of the blocks; where that leaves SMs idle, two CTAs of a cluster share a
// range and the second adds its sums to the first's through distributed shared memory (a fixed
// order).
// ---------------------------------------------------------------------------------
constexpr int W9_N = 96;                    // columns of one ky: 3 kx of 32 output channels
constexpr int W9_ROWS = 64 * 64;            // bytes of 64 voxels of 32 channels
constexpr int W9_X = 4 * W9_ROWS;           // a ring slot's four chunks of X
constexpr int W9_Z = 3 * W9_ROWS;           // and its dZ rows, three copies each
constexpr int W9_SLOTS = 7;
constexpr int W9_RING = W9_SLOTS * (W9_X + W9_Z);  // the X slots, then the dZ slots
constexpr int W9_SUM = 128 * 3 * W9_N * 4;  // bytes of one CTA's accumulators
static_assert(W9_RING >= W9_SUM, "the pair's sums go where the ring was");

struct Wgrad9Args {
    int N, cin, n;       // output channels, input channels, grid edge
    int segs, run;       // 64-voxel segments of an x-row, blocks of a run (the rows of one
                         // segment of one plane)
    int total, per;      // blocks (64 voxels each) in all and per CTA
    int Mrows;           // rows of a workspace slice (the padded 27 cin)
    int pair;            // two CTAs of a cluster share a slice
    float* ws;           // [slices][Mrows][N]
    int* err;
};

// Walks a CTA's ring slots: `lead` slots before the first block of the range and of every run,
// then the blocks, each at (b, z, seg, y): sample, plane, x-segment and block of its run.
struct W9Walk {
    int count, run, lead, segs, n;  // count: blocks still to come
    int b, z, seg, y, left;         // left: lead-in slots still to come before this block
    __device__ W9Walk(int first, int count_, int run_, int lead_, int segs_, int n_)
        : count(count_), run(run_), lead(lead_), segs(segs_), n(n_), left(lead_) {
        const int r = first / run, pl = r / segs;
        y = first - r * run;
        seg = r - pl * segs;
        b = pl / n;
        z = pl - b * n;
    }
    __device__ bool more() const { return count > 0; }
    __device__ bool data() const { return left == 0; }  // a block's slot, not a lead-in
    __device__ void next() {
        if (left > 0) {
            --left;
            return;
        }
        --count;
        if (++y < run) return;
        y = 0, left = lead;
        if (++seg < segs) return;
        seg = 0;
        if (++z == n) z = 0, ++b;
    }
};

// RB: x-rows of a 64-voxel block: 64 / n, or 1.
template <int RB>
__global__ void __launch_bounds__(128, 1)
    conv_wgrad9_kernel(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmZ,
                       Wgrad9Args args) {
    constexpr int S = W9_SLOTS;
    extern __shared__ uint8_t w9_smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>(
        (reinterpret_cast<uintptr_t>(w9_smem_raw) + 1023) & ~uintptr_t(1023));
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + W9_RING);
    uint64_t* empty = full + S;
    uint64_t* done = empty + S;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
    __shared__ volatile int failed;

    const int warp = warp_index(), lane = threadIdx.x & 31;
    const int slice = args.pair ? blockIdx.x >> 1 : blockIdx.x;
    const uint32_t rank = args.pair ? cluster_rank() : 0u;
    const int mt = blockIdx.y, n0 = blockIdx.z * 32, n = args.n;
    const int first = blockIdx.x * args.per;  // the pair's CTAs take consecutive ranges
    const int nst = max(0, min(args.per, args.total - first));
    constexpr int lead = RB == 1 ? 2 : 1;
    constexpr int line = W9_ROWS / RB;        // bytes of an x-row of the block
    const int gpt = args.cin >> 5;            // channel groups per kz

    if (threadIdx.x == 0) {
        // another CTA timed out: nothing is stored (the loads and MMAs go on until a wait sees it), and
        // the pair's barriers are kept
        failed = *static_cast<volatile int*>(args.err) != 0;
        for (int s = 0; s < S; ++s) {
            mbar_init(full + s, 1);
            mbar_init(empty + s, 1);
        }
        mbar_init(done, 1);
        mbar_fence_init();
    }
    if (warp == 0) tmem_alloc(tmem_slot, 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    int issued = 0;
    if (warp == 0) {
        const bool elected = elect_lane();
        int gz[4], gc[4];  // kz - 1 and first channel of the M tile's chunks
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int c = mt * 4 + q, kz = c / gpt;
            gz[q] = kz < 3 ? kz - 1 : 0;
            gc[q] = kz < 3 ? (c - kz * gpt) * 32 : args.cin;  // past the last chunk: zeros
        }
        W9Walk w(first, nst, args.run, lead, args.segs, n);
        int s = 0;
        uint32_t ph = 1;  // parity of the slot's last release
        for (int i = 0; w.more(); ++i, w.next()) {
            if (i >= S && !mbar_wait_warp(empty + s, ph, args.err, 1, &failed)) {
                failed = 1;
                break;
            }
            uint8_t* a = smem + s * W9_X;
            uint8_t* z = smem + S * W9_X + s * W9_Z;
            const int x0 = w.seg * 64, y0 = w.y * RB, yz = y0 + 1 - w.left * RB;  // dZ rows yz .. yz + RB - 1
            if (elected) {
                mbar_expect_tx(full + s, (w.data() ? 7 : 3) * W9_ROWS);
                if (w.data()) {
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        tma_load_5d(a + q * W9_ROWS, &tmX, full + s, gc[q], x0, y0, w.z + gz[q], w.b);
                }
#pragma unroll
                for (int q = 0; q < 3 * RB; ++q)
                    tma_load_5d(z + q * line, &tmZ, full + s, n0, x0 + 1 - q % 3, yz + q / 3, w.z, w.b);
            }
            ++issued;
            if (++s == S) s = 0, ph ^= 1u;
        }
    } else if (nst > 0 && warp == 1) {
        const bool elected = elect_lane();
        const uint32_t idesc = idesc_bf16_f32_mn(CBM, W9_N), idesc2 = idesc_bf16_f32_mn(CBM, 2 * W9_N);
        const uint32_t ahi = (uint32_t)(sdesc_mn(0, W9_ROWS, 512, 4) >> 32);
        const uint32_t xring = (uint32_t)sdesc_mn(smem_u32(smem), W9_ROWS, 512, 4);
        // dZ: a ring of x-rows, [row][kx][voxel]
        const uint32_t zring = (uint32_t)sdesc_mn(smem_u32(smem + S * W9_X), line, 512, 4);
        constexpr int ROWS = S * RB;
        uint32_t acc = 0;
        W9Walk w(first, nst, args.run, lead, args.segs, n);
        int s = 0, s1 = S - 1, s2 = S - 2;  // this slot and the ones before
        uint32_t ph = 0;
        for (int i = 0; w.more(); ++i, w.next()) {
            if (!mbar_wait_warp(full + s, ph, args.err, 2, &failed)) {
                failed = 1;
                break;
            }
            const uint32_t a = xring + (uint32_t)(s * (W9_X >> 4));
            // RB = 1: the dZ of this slot, of the one before and of two before
            const uint32_t zs[3] = {zring + (uint32_t)(s * (W9_Z >> 4)), zring + (uint32_t)(s1 * (W9_Z >> 4)),
                                    zring + (uint32_t)(s2 * (W9_Z >> 4))};
            tc_fence_after();
            if (elected && w.data()) {
                // tap ky takes the dZ row ky rows before this one into the columns (2 - ky) 96; two rows
                // that don't straddle the ring's end are one operand of six 32-channel groups
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) {  // K = 16 per MMA: two atoms of 8 voxels
                    const int row = s * RB + kk * RB / 4;
                    const auto z = [&](int ky) {
                        if constexpr (RB == 1) return zs[ky] + kk * 64;
                        const int at = row >= ky ? row - ky : row - ky + ROWS;
                        return zring + (uint32_t)((at * 3 * line + kk % (4 / RB) * 1024) >> 4);
                    };
                    const bool old = RB == 1 ? s1 != 0 : row != 1;  // the older two together, else the newer two
                    mma_bf16(tmem + (old ? 0u : (uint32_t)W9_N), a + kk * 64, ahi, z(old ? 2 : 1), ahi, idesc2, acc);
                    mma_bf16(tmem + (old ? 2u * W9_N : 0u), a + kk * 64, ahi, z(old ? 0 : 2), ahi, idesc, acc);
                    acc = 1;
                }
            }
            if (elected && i >= lead) mma_commit(empty + (lead == 2 ? s2 : s1));  // its dZ rows are used up
            s2 = s1, s1 = s;
            if (++s == S) s = 0, ph ^= 1u;
        }
        if (elected) mma_commit(done);  // also when stopped early: every issued MMA drains before dealloc
    }
    __syncwarp();
    if (nst > 0 && !mbar_wait(done, 0, args.err, 3)) failed = 1;
    __syncthreads();
    if (warp == 0 && lane == 0 && failed) {  // let every started copy land
        for (int i = max(0, issued - S); i < issued; ++i)
            mbar_wait(full + (i % S), (uint32_t)(i / S) & 1u, args.err, 4);
    }
    __syncwarp();
    tc_fence_after();
    const uint32_t lanes = tmem + ((uint32_t)(warp * 32) << 16);
    float4* sum = reinterpret_cast<float4*>(smem);  // [column / 4][128 rows]
    if (args.pair) {
        cluster_sync();  // both pipelines are done with their shared memory
        if (rank == 1 && !failed) {
            const uint32_t peer = cluster_map(smem_u32(smem), 0);
#pragma unroll 1
            for (int c = 0; c < 3 * W9_N; c += 16) {
                float v[16];
                tmem_ld16(lanes + (uint32_t)c, v);
                if (nst == 0) {  // nothing accumulated
#pragma unroll
                    for (int j = 0; j < 16; ++j) v[j] = 0.f;
                }
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    cluster_store4(peer + (uint32_t)((((c >> 2) + j) * 128 + threadIdx.x) * 16),
                                   make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]));
            }
        }
        cluster_sync();
    }
    const bool ok = rank == 0 && nst > 0 && !failed && *static_cast<volatile int*>(args.err) == 0;
    const int chunk = mt * 4 + warp, kz = chunk / gpt;  // this warp's rows: one chunk
    if (ok && kz < 3) {
        const int ci = (chunk - kz * gpt) * 32 + lane;
        float* slab = args.ws + (int64_t)slice * args.Mrows * args.N;
#pragma unroll 1
        for (int c = 0; c < 3 * W9_N; c += 16) {
            float v[16];
            tmem_ld16(lanes + (uint32_t)c, v);
            if (args.pair) {
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float4 w = sum[((c >> 2) + j) * 128 + threadIdx.x];
                    v[4 * j] += w.x;
                    v[4 * j + 1] += w.y;
                    v[4 * j + 2] += w.z;
                    v[4 * j + 3] += w.w;
                }
            }
            const int g = c >> 5, t = (2 - g / 3) * 3 + g % 3, col0 = n0 + (c & 31);  // t: tap (ky, kx) within kz
            float* C = slab + (int64_t)((kz * 9 + t) * args.cin + ci) * args.N + col0;
#pragma unroll
            for (int j = 0; j < 4; ++j)  // N is a multiple of 8: whole quadruples
                if (col0 + 4 * j < args.N)
                    reinterpret_cast<float4*>(C)[j] = make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
        }
    }
    if (ok && mt == 0) {  // the padding rows
        float* pad = args.ws + ((int64_t)slice * args.Mrows + 27 * args.cin) * args.N;
        for (int e = threadIdx.x; e < (args.Mrows - 27 * args.cin) * 32; e += 128)
            if (n0 + (e & 31) < args.N) pad[(int64_t)(e >> 5) * args.N + n0 + (e & 31)] = 0.f;
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, 512);
}

template <int BN, int BKC>
cudaError_t launch_conv(const CUtensorMap& tx, const CUtensorMap& tw, const ConvArgs& a,
                        cudaStream_t st) {
    using L = ConvSmem<BN, BKC>;
    static std::once_flag once;
    static cudaError_t attr = cudaSuccess;
    std::call_once(once, [] {
        attr = cudaFuncSetAttribute(conv_bf16_kernel<BN, BKC>,
                                    cudaFuncAttributeMaxDynamicSharedMemorySize, L::BYTES);
    });
    if (attr != cudaSuccess) return attr;
    const dim3 grid((a.M + CBM - 1) / CBM, (a.N + BN - 1) / BN, 1);
    conv_bf16_kernel<BN, BKC><<<grid, 128, L::BYTES, st>>>(tx, tw, a);
    return cudaGetLastError();
}

constexpr int kX3Smem = 216 * 1024;  // stages of a CTA
constexpr int kSMs = 152;

template <int BN>
cudaError_t launch_x3(const CUtensorMap& tx, const CUtensorMap& tw, const X3Args& a, cudaStream_t st) {
    static std::once_flag once;
    static cudaError_t attr = cudaSuccess;
    std::call_once(once, [] {
        attr = cudaFuncSetAttribute(conv_x3_kernel<BN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    1024 + kX3Smem + 256);
    });
    if (attr != cudaSuccess) return attr;
    // the whole budget whatever the stages take: one CTA per SM owns the tensor memory
    conv_x3_kernel<BN><<<std::min(a.items, kSMs), kX3Threads, 1024 + kX3Smem + 256, st>>>(tx, tw, a);
    return cudaGetLastError();
}

template <int BKC>
cudaError_t launch_conv_bkc(const CUtensorMap& tx, const CUtensorMap& tw, const ConvArgs& a,
                            int BN, cudaStream_t st) {
    switch (BN) {
    case 32: return launch_conv<32, BKC>(tx, tw, a, st);
    case 64: return launch_conv<64, BKC>(tx, tw, a, st);
    case 128: return launch_conv<128, BKC>(tx, tw, a, st);
    default: return launch_conv<256, BKC>(tx, tw, a, st);
    }
}

template <int BN>
cudaError_t launch_wgrad(const CUtensorMap& tx, const CUtensorMap& tb, const WgradArgs& a, int mtiles, int splits,
                         cudaStream_t st) {
    using L = WgradSmem<BN>;
    static std::once_flag once;
    static cudaError_t attr = cudaSuccess;
    std::call_once(once, [] {
        attr = cudaFuncSetAttribute(conv_wgrad_kernel<BN>, cudaFuncAttributeMaxDynamicSharedMemorySize, L::BYTES);
    });
    if (attr != cudaSuccess) return attr;
    const dim3 grid(mtiles, (a.N + BN - 1) / BN, splits);
    conv_wgrad_kernel<BN><<<grid, 128, L::BYTES, st>>>(tx, tb, a);
    return cudaGetLastError();
}

}  // namespace

// Rows are 32-bit in the kernels, up to the end of the last 128-row tile.
bool conv_rows_supported(int B, int n) {
    return B >= 1 && (int64_t)B * n * n * n <= (int64_t(1) << 31) - CBM;
}

// Operands that TMA reads start on 16 bytes, and so does an output written in 16-byte pieces
// (conv_store16, x3_store16: rows of a multiple of 8 values); else it is aligned to its elements.
bool conv_bases_supported(const void* X, const void* W, const float* bias, const void* out, int cout, int mode) {
    const uintptr_t o = cout % 8 == 0 ? 15 : mode == CONV_F32 ? 3 : 1, b = mode == CONV_F32 ? 0 : 3;
    return !((uintptr_t)X & 15) && !((uintptr_t)W & 15) && !((uintptr_t)bias & b) && !((uintptr_t)out & o);
}

bool conv_implicit_supported(int n, int cin, int cout) {
    return cin % 32 == 0 && n >= 2 && n <= 256 && (n & (n - 1)) == 0 && cout >= 1 && cout <= 256;
}

cudaError_t conv_implicit(const __nv_bfloat16* X, int B, int n, int cin, const __nv_bfloat16* W,
                          long long ldw, int cout, const float* bias, void* out, int mode, int* err,
                          cudaStream_t st) {
    if (!conv_implicit_supported(n, cin, cout) || !conv_rows_supported(B, n) ||
        !conv_bases_supported(X, W, bias, out, cout, mode) || (ldw % 8) || ldw < 27LL * cin || (mode == CONV_BIAS_RELU_BF16 && !bias) ||
        (mode != CONV_BIAS_RELU_BF16 && mode != CONV_F32))
        return cudaErrorInvalidValue;
    const int bkc = cin % 64 == 0 ? 64 : 32;
    // the 128-voxel M tile as a box: whole x-rows, then y, z and samples
    const int bx = n < 128 ? n : 128;
    const int by = 128 / bx < n ? 128 / bx : n;
    const int bz = 128 / (bx * by) < n ? 128 / (bx * by) : n;
    const int bb = 128 / (bx * by * bz);
    if (bx * by * bz * bb != 128) return cudaErrorInvalidValue;
    const int BN = cout <= 32 ? 32 : cout <= 64 ? 64 : cout <= 128 ? 128 : 256;
    if (n >= 16 && n <= 128) {
        // output channels per CTA: one tile up to 64, else tiles of 48 or 64 with less padding
        const int bn = cout <= 16 ? 16 : cout <= 32 ? 32 : cout <= 48 ? 48 : cout <= 64 ? 64
                     : (cout + 47) / 48 * 48 < (cout + 63) / 64 * 64 ? 48 : 64;
        const int ntiles = (cout + bn - 1) / bn;
        const int by1 = 128 / n, b_bytes = 9 * bn * 64;
        const int64_t tiles = (int64_t)B * n * n * n / CBM;
        auto stage_of = [&](int mt) { return (mt * by1 + 2) * n * 64 + b_bytes; };
        // as many tiles per item as two sets of accumulators of 256 columns and four stages allow
        // (they share the weights and the halo rows), and as leave every SM an item
        int mt = 4;
        while (mt > 1 && (mt * 3 * bn > 256 || mt * by1 > n || 4 * stage_of(mt) > kX3Smem ||
                          tiles / mt * ntiles < kSMs))
            mt >>= 1;
        const int stage = stage_of(mt);
        CUtensorMap tx, tw;
        if (!make_x_map(&tx, X, B, n, cin, 32, n, mt * by1 + 2, 1, 1) ||
            !make_w_map(&tw, W, cout, 27 * cin, ldw, 32, bn))
            return cudaErrorInvalidValue;
        X3Args a{cout, n, cin / 32, cin, ntiles, (int)(tiles / mt) * ntiles, mt, (mt * by1 + 2) * n * 64, stage,
                 std::min(8, kX3Smem / stage), mode, out, bias, cout % 16 == 0 && !((uintptr_t)out & 31), err};
        switch (bn) {
        case 16: return launch_x3<16>(tx, tw, a, st);
        case 32: return launch_x3<32>(tx, tw, a, st);
        case 48: return launch_x3<48>(tx, tw, a, st);
        default: return launch_x3<64>(tx, tw, a, st);
        }
    }
    CUtensorMap tx, tw;
    if (!make_x_map(&tx, X, B, n, cin, bkc, bx, by, bz, bb) ||
        !make_w_map(&tw, W, cout, 27 * cin, ldw, bkc, BN))
        return cudaErrorInvalidValue;
    ConvArgs a{B * n * n * n, cout, n, cin / bkc, bx, by, bz, mode, out, bias, err};
    return bkc == 64 ? launch_conv_bkc<64>(tx, tw, a, BN, st) : launch_conv_bkc<32>(tx, tw, a, BN, st);
}

// The nine-tap weight gradient into *slices <= max_slices slices of ws (plan_wgrad9).
cudaError_t launch_wgrad9(const __nv_bfloat16* X, int B, int n, int cin, const __nv_bfloat16* dZ, int cout, int Kp,
                          float* ws, int max_slices, int* slices, int* err, cudaStream_t st) {
    const int total = (int)((int64_t)B * n * n * n / 64);
    const int mtiles = (3 * (cin / 32) + 3) / 4, ntiles = (cout + 31) / 32;
    const Wgrad9Plan plan = plan_wgrad9(total, cin, cout, max_slices);
    *slices = plan.slices;
    constexpr int smem = 1024 + W9_RING + 256;
    const auto kernel = n == 16 ? conv_wgrad9_kernel<4> : n == 32 ? conv_wgrad9_kernel<2> : conv_wgrad9_kernel<1>;
    static std::once_flag once;
    static cudaError_t attr = cudaSuccess;
    std::call_once(once, [] {
        for (const auto k : {conv_wgrad9_kernel<4>, conv_wgrad9_kernel<2>, conv_wgrad9_kernel<1>})
            if (attr == cudaSuccess) attr = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    });
    if (attr != cudaSuccess) return attr;
    const int bx = n < 64 ? n : 64, RB = 64 / bx, segs = n / bx;
    CUtensorMap tx, tz;
    if (!make_x_map(&tx, X, B, n, cin, 32, bx, RB, 1, 1) || !make_x_map(&tz, dZ, B, n, cout, 32, bx, 1, 1, 1))
        return cudaErrorInvalidValue;
    const Wgrad9Args a{cout, cin, n, segs, n / RB, total, plan.per, Kp, plan.ctas == 2, ws, err};
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(plan.slices * plan.ctas), (unsigned)mtiles, (unsigned)ntiles);
    cfg.blockDim = dim3(128);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)plan.ctas;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = plan.ctas == 2 ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, tx, tz, a);
}

bool conv_wgrad_implicit_supported(int B, int n, int cin, int cout) {
    const int64_t M = (int64_t)B * n * n * n;
    return n >= 2 && n <= 256 && (n & (n - 1)) == 0 && cin % 32 == 0 && cout >= 8 && cout <= 256 &&
           cout % 8 == 0 && B >= 1 && M < (int64_t(1) << 31) - 64;
}

// As conv_bases_supported; the slices of ws are written in 16-byte pieces but for the one-tap form
// of 8 output channels.
bool conv_wgrad_bases_supported(const void* X, const void* dZ, const float* ws, const float* dWT, int cout) {
    return !((uintptr_t)X & 15) && !((uintptr_t)dZ & 15) && !((uintptr_t)ws & (cout > 8 ? 15 : 3)) &&
           !((uintptr_t)dWT & 3);
}

cudaError_t conv_wgrad_implicit(const __nv_bfloat16* X, int B, int n, int cin, const __nv_bfloat16* dZ, int cout,
                                int Kp, float* ws, size_t ws_floats, int splits, float* dWT, int accumulate,
                                int* err, cudaStream_t st) {
    if (!conv_wgrad_implicit_supported(B, n, cin, cout) || Kp < 27 * cin || splits < 1 ||
        !conv_wgrad_bases_supported(X, dZ, ws, dWT, cout))
        return cudaErrorInvalidValue;
    const int64_t M = (int64_t)B * n * n * n;
    const int kblocks = (int)((M + 63) / 64);
    const int per = (kblocks + splits - 1) / splits;
    const int used = (kblocks + per - 1) / per;
    const int mtiles = (Kp + CBM - 1) / CBM;
    if ((size_t)used * Kp * cout > ws_floats) return cudaErrorInvalidValue;
    // The nine-tap form where it has less to do on the busiest SM (nine_taps_pay).  More than 64 output
    // channels fill the one-tap form's MMAs.
    if (n >= 16 && cout <= 64 && !((uintptr_t)ws & 15) && nine_taps_pay(M, cin, cout, Kp, used, per)) {
        int slices = 0;
        const cudaError_t e = launch_wgrad9(X, B, n, cin, dZ, cout, Kp, ws, used, &slices, err, st);
        if (e != cudaSuccess) return e;
        return add_splits(ws, slices, Kp, cout, cout, dWT, accumulate, st);
    }
    // the 64-voxel K block as a box of the grid: x-row segments, whole rows, planes, samples
    const int bx = n < 64 ? n : 64;
    const int by = 64 / bx < n ? 64 / bx : n;
    const int bz = 64 / (bx * by) < n ? 64 / (bx * by) : n;
    const int bb = 64 / (bx * by * bz);
    if (bx * by * bz * bb != 64) return cudaErrorInvalidValue;
    const int BN = cout <= 32 ? 32 : cout <= 64 ? 64 : cout <= 128 ? 128 : 256;
    CUtensorMap tx, tb;
    if (!make_x_map(&tx, X, B, n, cin, 32, bx, by, bz, bb) ||
        !make_w_map(&tb, dZ, (int)M, cout, cout, BN < 64 ? BN : 64, 64))
        return cudaErrorInvalidValue;
    int ln = 0;
    while ((1 << ln) < n) ++ln;
    WgradArgs a{27 * cin, cout, cin, ln, kblocks, per, Kp, ws, err};
    cudaError_t e;
    switch (BN) {
    case 32: e = launch_wgrad<32>(tx, tb, a, mtiles, used, st); break;
    case 64: e = launch_wgrad<64>(tx, tb, a, mtiles, used, st); break;
    case 128: e = launch_wgrad<128>(tx, tb, a, mtiles, used, st); break;
    default: e = launch_wgrad<256>(tx, tb, a, mtiles, used, st); break;
    }
    if (e != cudaSuccess) return e;
    return add_splits(ws, used, Kp, cout, cout, dWT, accumulate, st);
}

}  // namespace nn
}  // namespace lbm
