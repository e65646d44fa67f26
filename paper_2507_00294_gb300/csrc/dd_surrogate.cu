// dd_surrogate.cu -- kernels of the learned surrogate of the field map (no counterpart
// in the paper): six 3x3 convolutions, NHWC BF16 activations, FP32 accumulation on the
// tensor cores (tcgen05.mma with TMEM accumulators for rows of 128 pixels, mma.sync
// m16n8k16 for other rows and the weight gradient), FP32 master weights with Adam.
//
// Layers: 16 -> 32 -> 32 -> 32 -> 32 -> 32 -> 16 channels (the first layer's input has 4
// real planes padded to 16, the last layer's output 1 real channel padded to 16), ReLU
// after the first five.  Weights are [Cout][tap = ky*3+kx][Cin] BF16; the data gradient
// uses the flipped, transposed copy [Cin][8 - tap][Cout] so that it is the same forward
// kernel.  Every convolution is an implicit GEMM: M = pixels, N = Cout, K = 9 Cin for
// the forward and data gradient; M = Cout, N = 9 Cin, K = pixels for the weight gradient
// (split over CTAs by image rows, partials reduced in a fixed order).
#include <cuda_bf16.h>

#include <algorithm>
#include <atomic>
#include <cstdint>

#include "dd_internal.h"
#include "dd_umma.cuh"

namespace ddk {

typedef __nv_bfloat16 bf16;

__device__ __forceinline__ void ldsm_x4(uint32_t addr, uint32_t &r0, uint32_t &r1, uint32_t &r2, uint32_t &r3) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];\n"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(addr));
}
__device__ __forceinline__ void ldsm_x4_t(uint32_t addr, uint32_t &r0, uint32_t &r1, uint32_t &r2, uint32_t &r3) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];\n"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(addr));
}
__device__ __forceinline__ void ldsm_x2_t(uint32_t addr, uint32_t &r0, uint32_t &r1) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0, %1}, [%2];\n"
                 : "=r"(r0), "=r"(r1) : "r"(addr));
}
// D = A (16x16, row) * B (16x8, col) + D, BF16 inputs, FP32 accumulators.
__device__ __forceinline__ void mma_bf16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                         uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

enum { kEpiReluBf16 = 0, kEpiLinearF32 = 1, kEpiMaskBf16 = 2 };
constexpr int kTW = 64;   // pixels of one image row per CTA
constexpr int kMaxDil = 32;

// out = conv3x3(in, w) with the epilogue EPI:
//   kEpiReluBf16:  bf16(max(z + bias, 0))                   [B,H,W,CO]
//   kEpiLinearF32: float(z + bias), channel 0 only            [B,H,W]
//   kEpiMaskBf16:  bf16(z * (mask > 0)), mask [B,H,W,CO]      (data gradient through ReLU)
template <int CI, int CO, int EPI>
__global__ void __launch_bounds__(128)
conv3x3_kernel(const bf16 *__restrict__ in, const bf16 *__restrict__ w, const float *__restrict__ bias,
               const bf16 *__restrict__ mask, void *__restrict__ out, int H, int W, int dil) {
    constexpr int CIP = CI + 8;          // padded rows: ldmatrix rows land in distinct banks
    constexpr int KW = 9 * CI + 8;
    // dynamic shared memory: weights [CO][KW], then input rows [3][kTW + 2 dil][CIP]
    extern __shared__ __align__(16) unsigned char smem_raw[];
    bf16 (*s_w)[KW] = reinterpret_cast<bf16 (*)[KW]>(smem_raw);
    bf16 *s_in = reinterpret_cast<bf16 *>(smem_raw + sizeof(bf16) * CO * KW);
    const int cols = kTW + 2 * dil;
    auto IN = [&](int ky, int px) -> bf16 * { return s_in + ((size_t)ky * cols + px) * CIP; };
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int tiles_per_row = W / kTW;
    const int x0 = (blockIdx.x % tiles_per_row) * kTW;
    const int row = blockIdx.x / tiles_per_row;          // b * H + y
    const int y = row % H;
    const int64_t img0 = (int64_t)(row - y) * W;         // first pixel of image b

    for (int v = tid; v < CO * 9 * CI / 8; v += 128) {
        const int co = v / (9 * CI / 8), r = v - co * (9 * CI / 8);
        *reinterpret_cast<uint4 *>(&s_w[co][r * 8]) = *reinterpret_cast<const uint4 *>(w + (int64_t)co * 9 * CI + r * 8);
    }
    // tap (ky, kx) of output pixel x reads input (y + (ky-1) dil, x + (kx-1) dil); staged
    // column px holds input x0 - dil + px
    for (int v = tid; v < 3 * cols * (CI / 8); v += 128) {
        const int ky = v / (cols * (CI / 8));
        const int rem = v - ky * cols * (CI / 8);
        const int px = rem / (CI / 8), c8 = rem - px * (CI / 8);
        const int yy = y + (ky - 1) * dil, xx = x0 + px - dil;
        uint4 val = make_uint4(0, 0, 0, 0);
        if (yy >= 0 && yy < H && xx >= 0 && xx < W)
            val = *reinterpret_cast<const uint4 *>(in + (img0 + (int64_t)yy * W + xx) * CI + c8 * 8);
        *reinterpret_cast<uint4 *>(IN(ky, px) + c8 * 8) = val;
    }
    __syncthreads();

    const int m0 = warp * 16;
    float acc[CO / 8][4];
#pragma unroll
    for (int n = 0; n < CO / 8; ++n) acc[n][0] = acc[n][1] = acc[n][2] = acc[n][3] = 0.f;
#pragma unroll
    for (int tap = 0; tap < 9; ++tap) {
        const int ky = tap / 3, kx = tap % 3;
#pragma unroll
        for (int c0 = 0; c0 < CI; c0 += 16) {
            uint32_t a0, a1, a2, a3;
            ldsm_x4(smem_u32(IN(ky, m0 + (lane & 7) + 8 * ((lane >> 3) & 1) + kx * dil) + c0 + 8 * (lane >> 4)),
                    a0, a1, a2, a3);
#pragma unroll
            for (int n = 0; n < CO / 8; n += 2) {
                uint32_t b0, b1, b2, b3;
                ldsm_x4(smem_u32(&s_w[n * 8 + (lane & 7) + 8 * (lane >> 4)][tap * CI + c0 + 8 * ((lane >> 3) & 1)]),
                        b0, b1, b2, b3);
                mma_bf16(acc[n], a0, a1, a2, a3, b0, b1);
                mma_bf16(acc[n + 1], a0, a1, a2, a3, b2, b3);
            }
        }
    }
    const int g = lane >> 2, t2 = 2 * (lane & 3);
#pragma unroll
    for (int n = 0; n < CO / 8; ++n) {
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            const int64_t pix = img0 + (int64_t)y * W + x0 + m0 + g + 8 * half;
            const int ch = n * 8 + t2;
            float v0 = acc[n][2 * half], v1 = acc[n][2 * half + 1];
            if (EPI == kEpiReluBf16) {
                v0 = fmaxf(v0 + bias[ch], 0.f);
                v1 = fmaxf(v1 + bias[ch + 1], 0.f);
                *reinterpret_cast<__nv_bfloat162 *>(static_cast<bf16 *>(out) + pix * CO + ch) = __floats2bfloat162_rn(v0, v1);
            } else if (EPI == kEpiLinearF32) {
                if (ch == 0) static_cast<float *>(out)[pix] = v0 + bias[0];
            } else {
                const __nv_bfloat162 m = *reinterpret_cast<const __nv_bfloat162 *>(mask + pix * CO + ch);
                v0 = __bfloat162float(m.x) > 0.f ? v0 : 0.f;
                v1 = __bfloat162float(m.y) > 0.f ? v1 : 0.f;
                *reinterpret_cast<__nv_bfloat162 *>(static_cast<bf16 *>(out) + pix * CO + ch) = __floats2bfloat162_rn(v0, v1);
            }
        }
    }
}

// ---- the forward / data-gradient convolution on the 5th-generation tensor cores ------
//
// An output row tile is M = 128 pixels x N = Cout, computed with tcgen05.mma (kind::f16,
// BF16 operands, FP32 accumulator in tensor memory): 9 taps x Cin/16 MMAs of K = 16,
// issued by one thread; the accumulator is read back with tcgen05.ld (warp w reads TMEM
// lanes 32w..32w+31, i.e. its 32 pixels) for the epilogue.  Operands are staged in the
// canonical K-major layout without swizzle: "core matrices" of 8 rows x 16 bytes.
//   input row [c8][px][8]: pixel rows 16 bytes apart, so the 128 pixels of any tap
//          (shifted by kx*dil columns) form 16 core matrices 128 bytes apart (SBO), and
//          the next 8 channels sit one channel-group plane further (LBO = plane*16 bytes);
//   weight [tap][c8][co][8]: SBO 128 bytes (next 8 outputs), LBO Cout*16 bytes.
constexpr int kTW5 = 128;
static __device__ int g_tc_timeout;       // set when an MMA completion wait gives up

// Pixels per channel-group plane of a staged row: the row's, padded to 2 mod 8, so that the copies of
// a pixel's channel groups (consecutive threads, whole sectors of global memory) land in
// different banks.
__host__ __device__ constexpr int conv_plane(int dil) { return kTW5 + 2 * dil + (2 - (kTW5 + 2 * dil) % 8 + 8) % 8; }

// 32 bytes in one access (a whole sector; the address a multiple of 32), else in two
__device__ __forceinline__ void store32(void *p, uint4 a, uint4 b, bool wide) {
    if (wide) {
        asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
                     :: "l"(p), "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b.x), "r"(b.y), "r"(b.z), "r"(b.w) : "memory");
    } else {
        reinterpret_cast<uint4 *>(p)[0] = a;
        reinterpret_cast<uint4 *>(p)[1] = b;
    }
}
__device__ __forceinline__ void load32(const void *p, uint4 &a, uint4 &b, bool wide) {
    if (wide) {
        asm volatile("ld.global.nc.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                     : "=r"(a.x), "=r"(a.y), "=r"(a.z), "=r"(a.w), "=r"(b.x), "=r"(b.y), "=r"(b.z), "=r"(b.w) : "l"(p));
    } else {
        a = reinterpret_cast<const uint4 *>(p)[0];
        b = reinterpret_cast<const uint4 *>(p)[1];
    }
}

// 16-byte global -> shared copy that completes asynchronously; src_bytes 0 writes zeros.
__device__ __forceinline__ void cp_async16_zfill(void *smem, const void *gmem, int src_bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(smem)), "l"(gmem), "r"(src_bytes)
                 : "memory");
}

// Persistent CTAs of three roles over work items.  An item is a segment of at most kSeg output
// rows of one 128-pixel column strip, taken with stride dil (rows y0, y0 + dil, ...).  Input row i
// of that chain takes part in output rows i - 1, i and i + 1, so its MMAs, one per tap column and
// 16 channels, carry the weights of all three rows side by side (N = 3 CO): a third of the
// MMAs and of the shared-memory reads of the pixels that one output row at a time takes.  The
// output rows of an item are neighbouring blocks of CO columns of tensor memory; an input row
// starts the block of row i + 1 with an MMA of its own (no accumulate).
//   warps 0-3: epilogue (blocks are given back as soon as they are in registers);
//   warps 4-7: copies (cp.async) into a ring of input rows;
//   warp 8: one thread issues the MMAs.
// The roles hand over two rows at a time: the waits, commits and fences of a row took longer than
// its work (2000 clocks per row and role one row at a time).  Step k of an item brings the input
// rows j0 - 1 + 2 k and j0 + 2 k, starts output rows j0 + 2 k and the next, and completes the two
// before.  Every wait is bounded; a wait that gives up stops the CTA's roles and sets the timeout
// flag.  Two CTAs per SM (256 TMEM columns each).
// A 32 -> 32 layer on 256 maps (537 MB) takes 115 to 132 us over the dilations, 4.1 to 4.7 TB/s: bound
// by memory beside the hand-overs (58 us with no copies, MMAs or stores, 90 without the stores).
// One input row at a time took 122 to 142 us, one output row at a time, each with its nine taps,
// 152 on average.  Eight epilogue warps or two steps ahead gave nothing.
constexpr int kSeg = 8;
constexpr int kConvAhead = 1, kConvMaxSlots = 5, kConvThreads = 288;     // slots of two rows
static_assert(kConvMaxSlots > kConvAhead + 1 && kSeg % 4 == 0, "a slot is refilled after its rows have been handed over");

struct ConvItem {
    int64_t img0;
    int x0, rho, j0, j1, J;         // output rows rho + j dil, j0 <= j < j1; input rows 0 <= j < J
};

template <int CI, int CO, int EPI>
__global__ void __launch_bounds__(kConvThreads, 2)
conv3x3_tc_kernel(const bf16 *__restrict__ in, const bf16 *__restrict__ w, const float *__restrict__ bias,
                  const bf16 *__restrict__ mask, void *__restrict__ out, int H, int W, int dil, int seg,
                  int items_per_strip, int n_items, int n_slots, int withhold_mma, bool wide) {
    constexpr int C8 = CI / 8, N = 3 * CO, kCols = kSeg * CO;
    static_assert(CI % 16 == 0 && (CO == 16 || CO == 32), "K steps of 16; 16 or 32 accumulator columns");
    // dynamic shared memory: weights [kx][C8][2 - ky][CO][8], the ring of input rows [slot][2][C8][plane][8]
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t s_full[kConvMaxSlots], s_empty[kConvMaxSlots], s_done[kSeg / 2], s_free[kSeg / 2], s_end;
    __shared__ __align__(16) float s_bias[CO];
    __shared__ uint32_t s_tmem;
    __shared__ int s_fail;
    bf16 *s_w = reinterpret_cast<bf16 *>(smem_raw);
    const int cols = kTW5 + 2 * dil, plane = conv_plane(dil), row_elems = C8 * plane * 8;
    bf16 *s_ring = s_w + 3 * C8 * N * 8;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int tiles_per_row = W / kTW5;
    const int long_rows = H / dil + 1, long_segs = (long_rows + seg - 1) / seg, short_segs = (long_rows - 1 + seg - 1) / seg;

    if (EPI == kEpiReluBf16 && tid < CO) s_bias[tid] = bias[tid];
    for (int v = tid; v < 3 * C8 * N; v += kConvThreads) {
        const int n = v % N, c8 = (v / N) % C8, kx = v / (N * C8), ky = 2 - n / CO, co = n % CO;
        cp_async16_zfill(s_w + (size_t)v * 8, w + ((int64_t)co * 9 + ky * 3 + kx) * CI + c8 * 8, 16);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     :: "r"(smem_u32(&s_tmem)), "n"(kCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        for (int k = 0; k < kConvMaxSlots; ++k) {
            mbar_init(s_full + k, 4);
            mbar_init(s_empty + k, 1);
        }
        for (int k = 0; k < kSeg / 2; ++k) {
            mbar_init(s_done + k, 1);
            mbar_init(s_free + k, 4);
        }
        mbar_init(&s_end, 1);
        s_fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    fence_proxy_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;

    // at most 2^18 tries of at most 1 us each (the suspend-time hint): a quarter second
    auto wait = [&](uint64_t *bar, uint32_t parity) -> bool {
        uint32_t done = 0;
        for (int it = 0; it < (1 << 18); ++it) {
            asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, 1000;\n"
                         " selp.u32 %0, 1, 0, p;\n}\n"
                         : "=r"(done) : "r"(smem_u32(bar)), "r"(parity) : "memory");
            if (done) return true;
            if (*(volatile int *)&s_fail) return false;
        }
        *(volatile int *)&s_fail = 1;
        return false;
    };
    // by every lane: one lane's wait and a shuffle were slower
    auto warp_wait = [&](uint64_t *bar, uint32_t parity) -> bool { return __all_sync(0xffffffffu, wait(bar, parity)); };
    auto arrive = [&](uint64_t *bar) {
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" :: "r"(smem_u32(bar)) : "memory");
    };
    // item q: strip (image, column tile), then the segment within the strip
    auto decode = [&](int q) -> ConvItem {
        ConvItem I;
        const int strip = q / items_per_strip;
        int r = q - strip * items_per_strip;
        const int bimg = strip / tiles_per_row;
        I.x0 = (strip - bimg * tiles_per_row) * kTW5;
        I.img0 = (int64_t)bimg * H * W;
        // chains rho < H mod dil have long_rows rows, the others one less
        const int n_long = (H - (long_rows - 1) * dil) * long_segs;
        const bool is_long = r < n_long;
        const int ns = is_long ? long_segs : short_segs, rest = is_long ? r : r - n_long, c = rest / ns;
        I.J = is_long ? long_rows : long_rows - 1;
        I.rho = is_long ? c : c + H - (long_rows - 1) * dil;
        I.j0 = (rest - c * ns) * seg;
        I.j1 = min(I.J, I.j0 + seg);
        return I;
    };
    // first block of an item after one at `base`: items of at most half the blocks alternate
    auto next_base = [&](int base, const ConvItem &I) { return 2 * (I.j1 - I.j0) <= kSeg && base == 0 ? kSeg / 2 : 0; };

    if (warp < 4) {                                              // epilogue
        uint32_t phase = 0;                                      // bit: parity of the pair's use
        int base = 0;
        bool ok = true;
        for (int q = blockIdx.x; q < n_items && ok; q += gridDim.x) {
            const ConvItem I = decode(q);
            base = next_base(base, I);
            for (int j = I.j0; j < I.j1; j += 2) {
                const int pair = (base + j - I.j0) / 2, n_out = min(2, I.j1 - j);
                int64_t pix[2];
                uint4 mk[2][CO / 8];            // the pixels' mask, in flight while the MMAs run
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    pix[r] = I.img0 + (int64_t)(I.rho + (j + r) * dil) * W + I.x0 + 32 * warp + lane;
                    if (EPI == kEpiMaskBf16 && r < n_out) {
#pragma unroll
                        for (int qq = 0; qq < CO / 8; qq += 2) load32(mask + pix[r] * CO + 8 * qq, mk[r][qq], mk[r][qq + 1], wide);
                    }
                }
                if (!(ok = warp_wait(s_done + pair, (phase >> pair) & 1u))) break;
                phase ^= 1u << pair;
                tc_fence_after();
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    if (r >= n_out) break;
                    uint32_t v[CO];
                    tmem_ld_32x32b<CO>(tmem + (uint32_t)(CO * (2 * pair + r)) + ((uint32_t)(32 * warp) << 16), v);
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                    if (r == n_out - 1) {
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) arrive(s_free + pair);
                    }
                    if (EPI == kEpiLinearF32) {
                        static_cast<float *>(out)[pix[r]] = __uint_as_float(v[0]) + bias[0];
                    } else {
                        uint4 o[CO / 8];
#pragma unroll
                        for (int qq = 0; qq < CO / 8; ++qq) {
                            uint32_t packed[4];
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                const int ch = 8 * qq + 2 * e;
                                float v0 = __uint_as_float(v[ch]), v1 = __uint_as_float(v[ch + 1]);
                                if (EPI == kEpiReluBf16) {
                                    v0 = fmaxf(v0 + s_bias[ch], 0.f);
                                    v1 = fmaxf(v1 + s_bias[ch + 1], 0.f);
                                } else {
                                    const uint32_t mw = e == 0 ? mk[r][qq].x : e == 1 ? mk[r][qq].y : e == 2 ? mk[r][qq].z : mk[r][qq].w;
                                    const __nv_bfloat162 m2 = *reinterpret_cast<const __nv_bfloat162 *>(&mw);
                                    v0 = __bfloat162float(m2.x) > 0.f ? v0 : 0.f;
                                    v1 = __bfloat162float(m2.y) > 0.f ? v1 : 0.f;
                                }
                                const __nv_bfloat162 h2 = __floats2bfloat162_rn(v0, v1);
                                packed[e] = *reinterpret_cast<const uint32_t *>(&h2);
                            }
                            o[qq] = make_uint4(packed[0], packed[1], packed[2], packed[3]);
                        }
#pragma unroll
                        for (int qq = 0; qq < CO / 8; qq += 2) store32(static_cast<bf16 *>(out) + pix[r] * CO + 8 * qq, o[qq], o[qq + 1], wide);
                    }
                }
            }
        }
        if (!ok && lane == 0) atomicExch(&g_tc_timeout, 1);
    } else if (warp < 8) {                                       // copies
        // thread: channel group c8 of the pixels px0, px0 + kStep, ..
        constexpr int kStep = 128 / C8;
        const int t = tid - 128, c8 = t % C8, px0 = t / C8;
        int n = 0, slot = 0, given = 0;                          // steps issued, the next one's slot; the next to hand over
        uint32_t parity = 1;                                     // of the slots' last release (none yet: passes)
        bool ok = true;
        for (int q = blockIdx.x; q < n_items && ok; q += gridDim.x) {
            const ConvItem I = decode(q);
            for (int i = I.j0 - 1; i <= I.j1; i += 2) {
                if (!(ok = warp_wait(s_empty + slot, parity))) break;
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    if (i + r < 0 || i + r > I.j1 || i + r >= I.J) continue;
                    int xx = I.x0 + px0 - dil;
                    const bf16 *src = in + (I.img0 + (int64_t)(I.rho + (i + r) * dil) * W + xx) * CI + c8 * 8;
                    bf16 *dst = s_ring + (2 * slot + r) * row_elems + (c8 * plane + px0) * 8;
#pragma unroll 3
                    for (int px = px0; px < cols; px += kStep) {
                        const bool inside = (unsigned)xx < (unsigned)W;          // zeros beside the image
                        cp_async16_zfill(dst, inside ? src : in, inside ? 16 : 0);
                        xx += kStep;
                        src += kStep * CI;
                        dst += kStep * 8;
                    }
                }
                asm volatile("cp.async.commit_group;" ::: "memory");
                if (++slot == n_slots) { slot = 0; parity ^= 1u; }
                if (++n > kConvAhead) {                          // the step kConvAhead back has landed
                    asm volatile("cp.async.wait_group %0;" :: "n"(kConvAhead) : "memory");
                    fence_proxy_async_smem();
                    __syncwarp();
                    if (lane == 0) arrive(s_full + given);
                    if (++given == n_slots) given = 0;
                }
            }
        }
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        fence_proxy_async_smem();
        __syncwarp();
        for (int k = min(n, kConvAhead); k > 0; --k) {
            if (lane == 0) arrive(s_full + given);
            if (++given == n_slots) given = 0;
        }
        // the MMAs' releases of the last steps arrive before the CTA ends
        for (int b = min(n, n_slots); b > 0 && ok; --b) {
            const int s = slot - b;                              // step n - b; < 0: of the round before
            ok = warp_wait(s_empty + (s < 0 ? s + n_slots : s), s < 0 ? parity : parity ^ 1u);
        }
        if (!ok && t == 0) atomicExch(&g_tc_timeout, 1);
    } else if (lane == 0 && !withhold_mma) {                     // MMAs
        int slot = 0, base = 0;
        uint32_t parity = 0, phase = 0xFFFFFFFFu;                // phase: parity of the pair's last release
        const uint64_t w0 = umma_smem_desc(smem_u32(s_w), N * 16u, 128u);
        bool ok = true;
        for (int q = blockIdx.x; q < n_items && ok; q += gridDim.x) {
            const ConvItem I = decode(q);
            base = next_base(base, I);
            const int i0 = max(I.j0 - 1, 0), i1 = min(I.j1, I.J - 1);
            for (int i = I.j0 - 1; i <= I.j1; i += 2) {
                const int pair = (base + i + 1 - I.j0) / 2;      // the output rows this step starts
                if (i + 1 < I.j1) {
                    if (!(ok = wait(s_free + pair, (phase >> pair) & 1u))) break;
                    phase ^= 1u << pair;
                }
                if (!(ok = wait(s_full + slot, parity))) break;
                tc_fence_after();
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    const int ii = i + r;
                    if (ii < i0 || ii > i1) continue;
                    const int lo = max(I.j0, ii - 1), hi = min(I.j1 - 1, ii + 1);
                    const int fresh = ii == i0 ? lo : ii + 1;    // blocks from here on start with this row
                    const uint64_t a = umma_smem_desc(smem_u32(s_ring + (2 * slot + r) * row_elems), (uint32_t)plane * 16u, 128u);
                    auto mma = [&](int kx, int c0, int ja, int jb, int accumulate) {
                        umma_bf16(tmem + (uint32_t)(CO * (base + ja - I.j0)), a + (uint32_t)((c0 / 8) * plane + kx * dil),
                                  w0 + (uint32_t)((kx * C8 + c0 / 8) * N + (ja - ii + 1) * CO),
                                  umma_idesc_bf16(kTW5, (jb - ja + 1) * CO), accumulate);
                    };
#pragma unroll
                    for (int kx = 0; kx < 3; ++kx) {
#pragma unroll
                        for (int c0 = 0; c0 < CI; c0 += 16) {
                            if (kx == 0 && c0 == 0) {
                                if (fresh > lo) mma(0, 0, lo, min(hi, fresh - 1), 1);
                                if (fresh <= hi) mma(0, 0, fresh, hi, 0);
                            } else {
                                mma(kx, c0, lo, hi, 1);
                            }
                        }
                    }
                }
                umma_commit(s_empty + slot);
                if (++slot == n_slots) { slot = 0; parity ^= 1u; }
                if (i >= I.j0) umma_commit(s_done + pair - 1);   // the two before are complete
            }
        }
        umma_commit(&s_end);                                     // none in flight when the memory is given back
        mbar_wait_bounded(&s_end, 0, 1 << 18);
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem), "n"(kCols) : "memory");
}

// Weight gradient partials: CTA c sums rows [c*rows, (c+1)*rows) of the B*H image rows, 64 pixels
// at a time.
//   part[c][co*9*CI + tap*CI + ci] = sum_p dz[p][co] * x[p + offset(tap)][ci]
//   part[c][CO*9*CI + co]          = sum_p dz[p][co]
// The next 64 pixels' three input rows and dz come in by cp.async while these run (two shared
// buffers of the dilation's size, padded rows: no bank conflicts of ldmatrix).  Bound by the
// shared-memory reads of the operands (ldmatrix) and mma.sync.  32 maps of 128 x 128, 32 -> 32
// channels: 100 -> 54 us with the reduction below (20 of the gain the reduction's).
template <int CI, int CO>
struct WgradSmem {
    static constexpr int CIP = CI + 8, COP = CO + 8;
    static __host__ __device__ int x_elems(int dil) { return 3 * (kTW + 2 * dil) * CIP; }
    static __host__ __device__ int elems(int dil) { return x_elems(dil) + kTW * COP; }
};
template <int CI, int CO>
__global__ void __launch_bounds__(128, 4)
conv3x3_wgrad_kernel(const bf16 *__restrict__ x, const bf16 *__restrict__ dz, int H, int W, int rows_total,
                     int rows_per_cta, int dil, float *__restrict__ part) {
    using S = WgradSmem<CI, CO>;
    constexpr int CIP = S::CIP, COP = S::COP;
    constexpr int NT = 9 * CI / 8;                 // n-tiles of 8 (tap, ci) columns
    constexpr int MT = CO / 16;                    // m-tiles of 16 output channels
    constexpr int NTW = (NT + 3) / 4;              // n-tiles per warp (round robin)
    constexpr int DBP = 128 / CO;                  // threads per channel of the bias gradient
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ float s_db[128];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int cols = kTW + 2 * dil, per_row = W / kTW;
    auto bx = [&](int b) { return reinterpret_cast<bf16 *>(smem_raw) + b * S::elems(dil); };
    auto bdz = [&](int b) { return bx(b) + S::x_elems(dil); };
    auto stage = [&](int t, int b) {
        const int row = t / per_row, x0 = (t - row * per_row) * kTW, y = row % H;
        const int64_t img0 = (int64_t)(row - y) * W;
        bf16 *const sx = bx(b), *const sd = bdz(b);
#pragma unroll
        for (int ky = 0; ky < 3; ++ky) {
            const int yy = y + (ky - 1) * dil;
            const bool row_in = yy >= 0 && yy < H;
            for (int v = tid; v < cols * (CI / 8); v += 128) {
                const int px = v / (CI / 8), c8 = v % (CI / 8), xx = x0 + px - dil;
                const bool in = row_in && xx >= 0 && xx < W;
                cp_async16_zfill(sx + (ky * cols + px) * CIP + c8 * 8,
                                 in ? x + (img0 + (int64_t)yy * W + xx) * CI + c8 * 8 : x, in ? 16 : 0);
            }
        }
        const bf16 *const src = dz + (img0 + (int64_t)y * W + x0) * CO;
        for (int v = tid; v < kTW * CO / 8; v += 128) {
            const int px = v / (CO / 8), c8 = v % (CO / 8);
            cp_async16_zfill(sd + px * COP + c8 * 8, src + px * CO + c8 * 8, 16);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    float acc[MT][NTW][4];
#pragma unroll
    for (int m = 0; m < MT; ++m)
#pragma unroll
        for (int n = 0; n < NTW; ++n) acc[m][n][0] = acc[m][n][1] = acc[m][n][2] = acc[m][n][3] = 0.f;
    float db = 0.f;
    const int t0 = blockIdx.x * rows_per_cta * per_row;
    const int t1 = min(rows_total, (blockIdx.x + 1) * rows_per_cta) * per_row;
    if (t0 < t1) stage(t0, 0);
    for (int t = t0; t < t1; ++t) {
        const int b = (t - t0) & 1;
        if (t + 1 < t1) {
            stage(t + 1, b ^ 1);
            asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        __syncthreads();
        const bf16 *const sx = bx(b), *const sd = bdz(b);
        {
            const int co = tid % CO;
#pragma unroll
            for (int px = tid / CO; px < kTW; px += DBP) db += __bfloat162float(sd[px * COP + co]);
        }
#pragma unroll
        for (int p0 = 0; p0 < kTW; p0 += 16) {
            uint32_t a[MT][4];
#pragma unroll
            for (int m = 0; m < MT; ++m)
                ldsm_x4_t(smem_u32(sd + (p0 + (lane & 7) + 8 * (lane >> 4)) * COP + m * 16 + 8 * ((lane >> 3) & 1)),
                          a[m][0], a[m][1], a[m][2], a[m][3]);
#pragma unroll
            for (int j = 0; j < NTW; ++j) {
                const int nt = warp + 4 * j;
                if (nt < NT) {
                    const int tap = (nt * 8) / CI, ci0 = (nt * 8) % CI;
                    const int ky = tap / 3, kx = tap % 3;
                    uint32_t b0, b1;
                    ldsm_x2_t(smem_u32(sx + (ky * cols + p0 + (lane & 7) + 8 * ((lane >> 3) & 1) + kx * dil) * CIP + ci0), b0, b1);
#pragma unroll
                    for (int m = 0; m < MT; ++m) mma_bf16(acc[m][j], a[m][0], a[m][1], a[m][2], a[m][3], b0, b1);
                }
            }
        }
        __syncthreads();                           // this buffer is staged again next
    }
    float *dst = part + (int64_t)blockIdx.x * (CO * 9 * CI + CO);
    const int g = lane >> 2, t2 = 2 * (lane & 3);
#pragma unroll
    for (int m = 0; m < MT; ++m)
#pragma unroll
        for (int j = 0; j < NTW; ++j) {
            const int nt = warp + 4 * j;
            if (nt >= NT) continue;
            const int n = nt * 8 + t2;
            const int co = m * 16 + g;
            dst[co * 9 * CI + n] = acc[m][j][0];
            dst[co * 9 * CI + n + 1] = acc[m][j][1];
            dst[(co + 8) * 9 * CI + n] = acc[m][j][2];
            dst[(co + 8) * 9 * CI + n + 1] = acc[m][j][3];
        }
    s_db[tid] = db;
    __syncthreads();
    if (tid < CO) {
        float v = 0.f;
#pragma unroll
        for (int k = 0; k < DBP; ++k) v += s_db[k * CO + tid];
        dst[CO * 9 * CI + tid] = v;
    }
}

// out[i] = sum over the parts in a fixed order: 32 consecutive outputs per CTA, the parts dealt out
// to its eight warps (each with eight loads in flight), then the eight sums in warp order.  One
// thread per output over all 608 parts left 37 CTAs waiting on one another's loads.
__global__ void __launch_bounds__(256) reduce_partials_kernel(const float *__restrict__ part, int n_parts, int len,
                                                             float *__restrict__ out) {
    __shared__ float s_sum[8][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int i = blockIdx.x * 32 + lane;
    float s = 0.f;
    if (i < len) {
#pragma unroll 8
        for (int c = warp; c < n_parts; c += 8) s += part[(int64_t)c * len + i];
    }
    s_sum[warp][lane] = s;
    __syncthreads();
    if (warp == 0 && i < len) {
        float t = 0.f;
#pragma unroll
        for (int k = 0; k < 8; ++k) t += s_sum[k][lane];
        out[i] = t;
    }
}

// dz[p][0] = 2 w[p] (pred[p] - target[p]) / n, dz[p][1..15] = 0; per-block sums of
// w[p] (pred[p] - target[p])^2 (w = 1 when weight is NULL).
__global__ void mse_kernel(const float *__restrict__ pred, const float *__restrict__ target,
                           const float *__restrict__ weight, int64_t n, bf16 *__restrict__ dz,
                           double *__restrict__ block_sums) {
    __shared__ double s[256];
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    double e = 0.0;
    if (p < n) {
        const float d = pred[p] - target[p];
        const float wp = weight ? weight[p] : 1.0f;
        e = (double)wp * d * d;
        uint4 z = make_uint4(0, 0, 0, 0);
        __nv_bfloat162 g = __floats2bfloat162_rn(2.0f * wp * d / (float)n, 0.0f);
        z.x = *reinterpret_cast<uint32_t *>(&g);
        uint4 *o = reinterpret_cast<uint4 *>(dz + p * 16);
        o[0] = z;
        o[1] = make_uint4(0, 0, 0, 0);
    }
    s[threadIdx.x] = e;
    __syncthreads();
    for (int k = 128; k > 0; k >>= 1) {
        if (threadIdx.x < k) s[threadIdx.x] += s[threadIdx.x + k];
        __syncthreads();
    }
    if (threadIdx.x == 0) block_sums[blockIdx.x] = s[0];
}

__global__ void sum_doubles_kernel(const double *__restrict__ v, int n, double *__restrict__ out) {
    __shared__ double s[256];
    double a = 0.0;
    for (int i = threadIdx.x; i < n; i += 256) a += v[i];
    s[threadIdx.x] = a;
    __syncthreads();
    for (int k = 128; k > 0; k >>= 1) {
        if (threadIdx.x < k) s[threadIdx.x] += s[threadIdx.x + k];
        __syncthreads();
    }
    if (threadIdx.x == 0) *out = s[0];
}

// Adam on FP32 master weights [co][tap][ci] (+ separate bias array handled the same way),
// writing the BF16 copy and the flipped copy [ci][8 - tap][co] used by the data gradient.
__global__ void adam_kernel(float *__restrict__ p, const float *__restrict__ g, float *__restrict__ m,
                            float *__restrict__ v, int n, float lr, float b1, float b2, float eps, float c1, float c2,
                            bf16 *__restrict__ wb, bf16 *__restrict__ wflip, int ci_n, int co_n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float pi = p[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    p[i] = pi;
    if (wb) {
        wb[i] = __float2bfloat16_rn(pi);
        const int ci = i % ci_n, tap = (i / ci_n) % 9, co = i / (9 * ci_n);
        wflip[((int64_t)ci * 9 + (8 - tap)) * co_n + co] = __float2bfloat16_rn(pi);
    }
}

// Input planes [B,H,W,16]: the time map value where visited (its encoding is the caller's), visited mask,
// standardised log D and log dwell; channels 4..15 zero.  tmap < 0 marks unvisited.
__global__ void planes_kernel(const float *__restrict__ tmap, const float *__restrict__ scal, int HW, int64_t n,
                              bf16 *__restrict__ x) {
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    const int b = (int)(p / HW);
    const float t = tmap[p];
    __nv_bfloat162 c01 = __floats2bfloat162_rn(t >= 0.f ? t : 0.f, t >= 0.f ? 1.f : 0.f);
    __nv_bfloat162 c23 = __floats2bfloat162_rn(scal[2 * b], scal[2 * b + 1]);
    uint4 z = make_uint4(0, 0, 0, 0);
    z.x = *reinterpret_cast<uint32_t *>(&c01);
    z.y = *reinterpret_cast<uint32_t *>(&c23);
    uint4 *o = reinterpret_cast<uint4 *>(x + p * 16);
    o[0] = z;
    o[1] = make_uint4(0, 0, 0, 0);
}

// The planes of planes_kernel, plus channel 4: each background visit's own term at its
// position (a visit older than k_exact dwells at the end of the scan: ln(w1/w0) of Eq. 3/4,
// w1 = 2 s + 4 kappa age, w0 = 2 s + 4 kappa (age - 1), as the normalised log10 of the
// target), and channel 5: the background mask.  scal3[b] = (standardised log D,
// standardised log dwell, kappa = D dwell / pitch^2).
__global__ void planes_bg_kernel(const float *__restrict__ tmap, const float *__restrict__ scal3, float s_dim,
                                 float k_exact, float mu, float inv_sigma, int HW, int64_t n, bf16 *__restrict__ x) {
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    const int b = (int)(p / HW);
    const float t = tmap[p];
    float own = 0.f, bg = 0.f;
    if (t > 0.f) {
        const float age = 1.0f / t;                      // 1 for the last visit
        if (age > k_exact + 0.5f) {
            const float kap = scal3[3 * b + 2];
            const float v = log1pf(4.0f * kap / (2.0f * s_dim + 4.0f * kap * (age - 1.0f)));
            own = (log10f(v) - mu) * inv_sigma;
            bg = 1.f;
        }
    }
    __nv_bfloat162 c01 = __floats2bfloat162_rn(t >= 0.f ? t : 0.f, t >= 0.f ? 1.f : 0.f);
    __nv_bfloat162 c23 = __floats2bfloat162_rn(scal3[3 * b], scal3[3 * b + 1]);
    __nv_bfloat162 c45 = __floats2bfloat162_rn(own, bg);
    uint4 z = make_uint4(0, 0, 0, 0);
    z.x = *reinterpret_cast<uint32_t *>(&c01);
    z.y = *reinterpret_cast<uint32_t *>(&c23);
    z.z = *reinterpret_cast<uint32_t *>(&c45);
    uint4 *o = reinterpret_cast<uint4 *>(x + p * 16);
    o[0] = z;
    o[1] = make_uint4(0, 0, 0, 0);
}

// One CTA per map: peak = max_p psi[m][p] * scale[m], then
// target[m][p] = (log10(max(psi[m][p] * scale[m], peak * 10^floor_rel)) - mu) * inv_sigma
__global__ void targets_kernel(const double *__restrict__ psi, const double *__restrict__ scale, int64_t hw,
                               double floor_rel, float mu, float inv_sigma, float *__restrict__ out) {
    __shared__ double s[256];
    const int64_t m = blockIdx.x;
    const double sc = scale[m];
    double mx = 0.0;
    for (int64_t p = threadIdx.x; p < hw; p += blockDim.x) mx = fmax(mx, psi[m * hw + p] * sc);
    s[threadIdx.x] = mx;
    __syncthreads();
    for (int k = 128; k > 0; k >>= 1) {
        if (threadIdx.x < k) s[threadIdx.x] = fmax(s[threadIdx.x], s[threadIdx.x + k]);
        __syncthreads();
    }
    const double lo = fmax(s[0] * pow(10.0, floor_rel), 1e-300);
    for (int64_t p = threadIdx.x; p < hw; p += blockDim.x)
        out[m * hw + p] = (float)((log10(fmax(psi[m * hw + p] * sc, lo)) - (double)mu) * (double)inv_sigma);
}

// Per-pixel loss weights of one map per CTA, from its normalised log targets:
//   f_p = 10^(target_p sigma + mu),  w_p = alpha hw f_p^2 / sum_q f_q^2 + (1 - alpha).
// With alpha = 1 the weighted squared log error sum_p w_p (log10 error_p)^2 / hw is, to
// first order, (relative L2 error of the linear map / ln 10)^2: a pixel weighs as much as
// its share of the map's squared norm; 1 - alpha keeps every pixel in the loss.
__global__ void weights_kernel(const float *__restrict__ target, int64_t hw, float mu, float sigma, float alpha,
                               float *__restrict__ w) {
    __shared__ double s[256];
    const int64_t m = blockIdx.x;
    const float *t = target + m * hw;
    double acc = 0.0;
    for (int64_t p = threadIdx.x; p < hw; p += blockDim.x) {
        const double f = pow(10.0, (double)t[p] * sigma + mu);
        acc += f * f;
    }
    s[threadIdx.x] = acc;
    __syncthreads();
    for (int k = 128; k > 0; k >>= 1) {
        if (threadIdx.x < k) s[threadIdx.x] += s[threadIdx.x + k];
        __syncthreads();
    }
    const double norm = s[0] > 0.0 ? (double)alpha * (double)hw / s[0] : 0.0;
    for (int64_t p = threadIdx.x; p < hw; p += blockDim.x) {
        const double f = pow(10.0, (double)t[p] * sigma + mu);
        w[m * hw + p] = (float)(norm * f * f + (1.0 - (double)alpha));
    }
}

// psi[m][p] = 10^(pred[m][p] * sigma + mu) / scale[m]  (back to u/m^2)
__global__ void fields_kernel(const float *__restrict__ pred, const double *__restrict__ scale, int64_t hw,
                              int64_t n, float mu, float sigma, double *__restrict__ psi) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    psi[i] = pow(10.0, (double)pred[i] * sigma + mu) / scale[i / hw];
}

// err[m] = || psi_pred(spots) + add(spots) - exact ||_2 / || exact ||_2 over the k spot
// points of map m (add: an exactly computed part of the field, or NULL)
__global__ void spot_error_kernel(const float *__restrict__ pred, const int32_t *__restrict__ idx,
                                  const double *__restrict__ exact, const double *__restrict__ scale,
                                  const double *__restrict__ add, int hw, int k, float mu, float sigma,
                                  double *__restrict__ err) {
    const int m = blockIdx.x;
    __shared__ double sn[128], sd[128];
    double num = 0.0, den = 0.0;
    for (int j = threadIdx.x; j < k; j += blockDim.x) {
        const int p = idx[(int64_t)m * k + j];
        const double e = exact[(int64_t)m * k + j];
        const double v = pow(10.0, (double)pred[(int64_t)m * hw + p] * sigma + mu) / scale[m] +
                         (add ? add[(int64_t)m * hw + p] : 0.0);
        num += (v - e) * (v - e);
        den += e * e;
    }
    sn[threadIdx.x] = num;
    sd[threadIdx.x] = den;
    __syncthreads();
    for (int s = 64; s > 0; s >>= 1) {
        if (threadIdx.x < s) { sn[threadIdx.x] += sn[threadIdx.x + s]; sd[threadIdx.x] += sd[threadIdx.x + s]; }
        __syncthreads();
    }
    if (threadIdx.x == 0) err[m] = sd[0] > 0.0 ? sqrt(sn[0] / sd[0]) : (sn[0] > 0.0 ? INFINITY : 0.0);
}

}  // namespace ddk

namespace {

template <int CI, int CO, int EPI>
cudaError_t launch_conv(const void *in, const void *w, const float *bias, const void *mask, void *out, int B,
                        int H, int W, int dil, cudaStream_t st) {
    constexpr int KW = 9 * CI + 8, CIP = CI + 8;
    const size_t smem = sizeof(ddk::bf16) * ((size_t)CO * KW + (size_t)3 * (ddk::kTW + 2 * dil) * CIP);
    static bool configured = false;     // allow the largest dilation's staging area once
    if (!configured) {
        const size_t most = sizeof(ddk::bf16) * ((size_t)CO * KW + (size_t)3 * (ddk::kTW + 2 * ddk::kMaxDil) * CIP);
        cudaError_t err = cudaFuncSetAttribute(ddk::conv3x3_kernel<CI, CO, EPI>,
                                               cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
        if (err != cudaSuccess) return err;
        configured = true;
    }
    const unsigned grid = (unsigned)(B * H * (W / ddk::kTW));
    ddk::conv3x3_kernel<CI, CO, EPI><<<grid, 128, smem, st>>>((const ddk::bf16 *)in, (const ddk::bf16 *)w, bias,
                                                               (const ddk::bf16 *)mask, out, H, W, dil);
    return cudaGetLastError();
}

// The tensor-memory variant (W a multiple of 128): persistent CTAs over segments of
// dilation-strided row chains.  Each CTA holds at most 256 TMEM columns and asks for more than a
// third of an SM's shared memory, so that at most two share an SM and an allocation never waits.
template <int CI, int CO, int EPI>
cudaError_t launch_conv_tc(const void *in, const void *w, const float *bias, const void *mask, void *out, int B,
                           int H, int W, int dil, cudaStream_t st) {
    constexpr size_t kLeast = 77 * 1024, kMost = 112 * 1024;
    const size_t w_bytes = sizeof(ddk::bf16) * 9 * CI * CO, slot = 2 * sizeof(ddk::bf16) * CI * ddk::conv_plane(dil);
    const int n_slots = std::min<int>(ddk::kConvMaxSlots, (int)((kMost - w_bytes) / slot));
    static_assert((kMost - sizeof(ddk::bf16) * 9 * CI * CO) / (2 * sizeof(ddk::bf16) * CI * ddk::conv_plane(ddk::kMaxDil)) > ddk::kConvAhead + 1,
                  "slots at the largest dilation");
    const size_t bytes = std::max(kLeast, w_bytes + n_slots * slot);
    static std::atomic<uint64_t> configured{0};    // per device: the attributes are set
    int dev = 0, sms = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err == cudaSuccess) err = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (err != cudaSuccess) return err;
    if (dev >= 64 || !(configured.load() & (uint64_t(1) << dev))) {
        err = cudaFuncSetAttribute(ddk::conv3x3_tc_kernel<CI, CO, EPI>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMost);
        if (err == cudaSuccess)
            err = cudaFuncSetAttribute(ddk::conv3x3_tc_kernel<CI, CO, EPI>,
                                       cudaFuncAttributePreferredSharedMemoryCarveout,
                                       (int)cudaSharedmemCarveoutMaxShared);
        if (err != cudaSuccess) return err;
        if (dev < 64) configured.fetch_or(uint64_t(1) << dev);
    }
    // Rows per item: the length at which the CTA with the most items has the least to do; an item
    // also reads two rows beside it (most of them from L2)
    int seg = ddk::kSeg, per_strip = 0;
    int64_t best = INT64_MAX;
    for (int s = ddk::kSeg; s >= 3; --s) {
        int items = 0;                             // per (image, column tile): the segments of every chain rho < dil
        for (int rho = 0; rho < dil; ++rho) items += ((H - rho + dil - 1) / dil + s - 1) / s;
        const int64_t n = (int64_t)B * (W / ddk::kTW5) * items, cost = (n + 2 * sms - 1) / (2 * sms) * (s + 1);
        if (s == ddk::kSeg || (cost < best && n <= INT32_MAX)) {
            best = cost;
            seg = s;
            per_strip = items;
        }
    }
    const int n_items = B * (W / ddk::kTW5) * per_strip;
    const int grid = std::max(1, std::min(n_items, 2 * sms));
    // DD_FAULT=tc_wait (tests): no MMA is issued, so every completion wait runs out and the
    // timeout path (flag, no output, TMEM released) is exercised without a GPU fault
    const int withhold = dd::fault_injected("tc_wait") ? 1 : 0;
    // 32-byte accesses of the output and the mask (a multiple of 32 bytes per pixel) where both start
    // on one
    const bool wide = ((reinterpret_cast<uintptr_t>(out) | reinterpret_cast<uintptr_t>(mask)) & 31) == 0;
    ddk::conv3x3_tc_kernel<CI, CO, EPI><<<grid, ddk::kConvThreads, bytes, st>>>(
        (const ddk::bf16 *)in, (const ddk::bf16 *)w, bias, (const ddk::bf16 *)mask, out, H, W, dil, seg, per_strip,
        n_items, n_slots, withhold, wide);
    return cudaGetLastError();
}

template <int CI, int CO>
cudaError_t launch_wgrad(int n_cta, const ddk::bf16 *x, const ddk::bf16 *dz, int H, int W, int rows_total, int rows_per,
                         int dil, float *part, cudaStream_t st) {
    auto bytes = [](int d) { return (int)(2 * sizeof(ddk::bf16)) * ddk::WgradSmem<CI, CO>::elems(d); };
    static std::atomic<uint64_t> done{0};          // per device: the attributes are set
    int dev = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess || dev >= 64) return err != cudaSuccess ? err : cudaErrorInvalidDevice;
    if (!(done.load() & (uint64_t(1) << dev))) {
        err = cudaFuncSetAttribute(ddk::conv3x3_wgrad_kernel<CI, CO>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   bytes(ddk::kMaxDil));
        if (err == cudaSuccess)
            err = cudaFuncSetAttribute(ddk::conv3x3_wgrad_kernel<CI, CO>, cudaFuncAttributePreferredSharedMemoryCarveout,
                                       (int)cudaSharedmemCarveoutMaxShared);
        if (err != cudaSuccess) return err;
        done.fetch_or(uint64_t(1) << dev);
    }
    ddk::conv3x3_wgrad_kernel<CI, CO><<<n_cta, 128, bytes(dil), st>>>(x, dz, H, W, rows_total, rows_per, dil, part);
    return cudaGetLastError();
}

bool conv_shape_ok(int cin, int cout) {
    return (cin == 16 && cout == 32) || (cin == 32 && cout == 32) || (cin == 32 && cout == 16) ||
           (cin == 16 && cout == 16);
}

}  // namespace

extern "C" {

dd_status dd_sur_conv3x3(const void *in, const void *w, const float *bias, const void *mask, void *out,
                         int32_t B, int32_t H, int32_t W, int32_t cin, int32_t cout, int32_t dilation,
                         int32_t epilogue, void *cuda_stream) {
    dd::clear_error();
    if (!in || !w || !out || B < 1 || H < 1 || W < ddk::kTW || W % ddk::kTW)
        return dd::fail(DD_EINVAL, "dd_sur_conv3x3: bad buffers or shape (W must be a multiple of 64)");
    if (!conv_shape_ok(cin, cout)) return dd::fail(DD_EINVAL, "dd_sur_conv3x3: unsupported (cin, cout)");
    if (dilation < 1 || dilation > ddk::kMaxDil) return dd::fail(DD_EINVAL, "dd_sur_conv3x3: dilation must be 1..32");
    if (epilogue < 0 || epilogue > 2 || (epilogue != 2 && !bias) || (epilogue == 2 && !mask))
        return dd::fail(DD_EINVAL, "dd_sur_conv3x3: bad epilogue arguments");
    cudaStream_t st = (cudaStream_t)cuda_stream;
    const char *name = epilogue == 2 ? "conv3x3_dgrad" : "conv3x3_fwd";
    dd::ProfScope ps(name, st);
    cudaError_t err = cudaSuccess;
    // rows of 128 pixels: tcgen05 MMA tiles of 128 pixels; otherwise 64-pixel tiles on mma.sync
    const bool tc = W % ddk::kTW5 == 0;
#define DD_CONV(CI, CO)                                                                                   \
    if (cin == CI && cout == CO) {                                                                        \
        if (tc) {                                                                                         \
            if (epilogue == 0) err = launch_conv_tc<CI, CO, ddk::kEpiReluBf16>(in, w, bias, mask, out, B, H, W, dilation, st);  \
            else if (epilogue == 1) err = launch_conv_tc<CI, CO, ddk::kEpiLinearF32>(in, w, bias, mask, out, B, H, W, dilation, st); \
            else err = launch_conv_tc<CI, CO, ddk::kEpiMaskBf16>(in, w, bias, mask, out, B, H, W, dilation, st);  \
        } else {                                                                                          \
            if (epilogue == 0) err = launch_conv<CI, CO, ddk::kEpiReluBf16>(in, w, bias, mask, out, B, H, W, dilation, st);  \
            else if (epilogue == 1) err = launch_conv<CI, CO, ddk::kEpiLinearF32>(in, w, bias, mask, out, B, H, W, dilation, st); \
            else err = launch_conv<CI, CO, ddk::kEpiMaskBf16>(in, w, bias, mask, out, B, H, W, dilation, st);  \
        }                                                                                                 \
    }
    DD_CONV(16, 32)
    DD_CONV(32, 32)
    DD_CONV(32, 16)
    DD_CONV(16, 16)
#undef DD_CONV
    if (err != cudaSuccess) return dd::fail_cuda(err, "dd_sur_conv3x3 launch");
    return DD_OK;
}

dd_status dd_sur_check(void) {
    dd::clear_error();
    DD_CUDA_TRY(cudaDeviceSynchronize());
    int flag = 0;
    DD_CUDA_TRY(cudaMemcpyFromSymbol(&flag, ddk::g_tc_timeout, sizeof(int)));
    if (!flag) return DD_OK;
    const int zero = 0;
    DD_CUDA_TRY(cudaMemcpyToSymbol(ddk::g_tc_timeout, &zero, sizeof(int)));
    return dd::fail(DD_ETIMEOUT, "dd_sur_check: a tensor-core convolution gave up waiting for its MMAs");
}

dd_status dd_sur_wgrad(const void *x, const void *dz, int32_t B, int32_t H, int32_t W, int32_t cin, int32_t cout,
                       int32_t dilation, float *part, int64_t part_floats, float *grad, void *cuda_stream) {
    dd::clear_error();
    if (!x || !dz || !part || !grad || B < 1 || H < 1 || W < ddk::kTW || W % ddk::kTW)
        return dd::fail(DD_EINVAL, "dd_sur_wgrad: bad buffers or shape");
    if (!conv_shape_ok(cin, cout) || cout % 16) return dd::fail(DD_EINVAL, "dd_sur_wgrad: unsupported (cin, cout)");
    if (dilation < 1 || dilation > ddk::kMaxDil) return dd::fail(DD_EINVAL, "dd_sur_wgrad: dilation must be 1..32");
    const int rows_total = B * H;
    const int len = cout * 9 * cin + cout;
    int n_cta = 4 * 152;
    if (n_cta > rows_total) n_cta = rows_total;
    const int rows_per = (rows_total + n_cta - 1) / n_cta;
    n_cta = (rows_total + rows_per - 1) / rows_per;
    if ((int64_t)n_cta * len > part_floats) return dd::fail(DD_EINVAL, "dd_sur_wgrad: partial buffer too small");
    cudaStream_t st = (cudaStream_t)cuda_stream;
    dd::ProfScope ps("conv3x3_wgrad", st);
    const ddk::bf16 *xb = (const ddk::bf16 *)x, *db = (const ddk::bf16 *)dz;
    const int d = dilation;
    cudaError_t err = cudaSuccess;
    if (cin == 16 && cout == 32) err = launch_wgrad<16, 32>(n_cta, xb, db, H, W, rows_total, rows_per, d, part, st);
    else if (cin == 32 && cout == 32) err = launch_wgrad<32, 32>(n_cta, xb, db, H, W, rows_total, rows_per, d, part, st);
    else if (cin == 32 && cout == 16) err = launch_wgrad<32, 16>(n_cta, xb, db, H, W, rows_total, rows_per, d, part, st);
    else err = launch_wgrad<16, 16>(n_cta, xb, db, H, W, rows_total, rows_per, d, part, st);
    if (err != cudaSuccess) return dd::fail_cuda(err, "dd_sur_wgrad launch");
    ddk::reduce_partials_kernel<<<(len + 31) / 32, 256, 0, st>>>(part, n_cta, len, grad);
    DD_CUDA_TRY(cudaGetLastError());
    return DD_OK;
}

dd_status dd_sur_mse(const float *pred, const float *target, int64_t n, void *dz, double *block_sums,
                     double *loss_sum, void *cuda_stream) {
    dd::clear_error();
    if (!pred || !target || !dz || !block_sums || !loss_sum || n < 1) return dd::fail(DD_EINVAL, "dd_sur_mse: bad arguments");
    cudaStream_t st = (cudaStream_t)cuda_stream;
    const int nb = (int)((n + 255) / 256);
    ddk::mse_kernel<<<nb, 256, 0, st>>>(pred, target, nullptr, n, (ddk::bf16 *)dz, block_sums);
    ddk::sum_doubles_kernel<<<1, 256, 0, st>>>(block_sums, nb, loss_sum);
    DD_CUDA_TRY(cudaGetLastError());
    return DD_OK;
}

dd_status dd_sur_wmse(const float *pred, const float *target, const float *weight, int64_t n, void *dz,
                      double *block_sums, double *loss_sum, void *cuda_stream) {
    dd::clear_error();
    if (!pred || !target || !weight || !dz || !block_sums || !loss_sum || n < 1)
        return dd::fail(DD_EINVAL, "dd_sur_wmse: bad arguments");
    cudaStream_t st = (cudaStream_t)cuda_stream;
    const int nb = (int)((n + 255) / 256);
    ddk::mse_kernel<<<nb, 256, 0, st>>>(pred, target, weight, n, (ddk::bf16 *)dz, block_sums);
    ddk::sum_doubles_kernel<<<1, 256, 0, st>>>(block_sums, nb, loss_sum);
    DD_CUDA_TRY(cudaGetLastError());
    return DD_OK;
}

dd_status dd_sur_weights(const float *target, int64_t n_maps, int64_t hw, float mu, float sigma, float alpha,
                         float *w, void *cuda_stream) {
    dd::clear_error();
    if (!target || !w || n_maps < 1 || hw < 1 || !(alpha >= 0.f && alpha <= 1.f))
        return dd::fail(DD_EINVAL, "dd_sur_weights: bad arguments");
    ddk::weights_kernel<<<(unsigned)n_maps, 256, 0, (cudaStream_t)cuda_stream>>>(target, hw, mu, sigma, alpha, w);
    DD_CUDA_TRY(cudaGetLastError());
    return DD_OK;
}

dd_status dd_sur_adam(float *param, const float *grad, float *m, float *v, int64_t n, float lr, float beta1,
                      float beta2, float eps, int32_t step, void *w_bf16, void *w_flip_bf16, int32_t cin,
                      int32_t cout, void *cuda_stream) {
    dd::clear_error();
    if (!param || !grad || !m || !v || n < 1 || step < 1) return dd::fail(DD_EINVAL, "dd_sur_adam: bad arguments");
    if (w_bf16 && (!w_flip_bf16 || (int64_t)cin * cout * 9 != n)) return dd::fail(DD_EINVAL, "dd_sur_adam: bad weight shape");
    const float c1 = 1.f - powf(beta1, (float)step), c2 = 1.f - powf(beta2, (float)step);
    cudaStream_t st = (cudaStream_t)cuda_stream;
    ddk::adam_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(param, grad, m, v, (int)n, lr, beta1, beta2, eps, c1, c2,
                                                                 (ddk::bf16 *)w_bf16, (ddk::bf16 *)w_flip_bf16, cin, cout);
    DD_CUDA_TRY(cudaGetLastError());
    return DD_OK;
}

dd_status dd_sur_planes(const float *tmap, const float *scal, int32_t B, int32_t H, int32_t W, void *x, void *cuda_stream) {
    dd::clear_error();
    if (!tmap || !scal || !x || B < 1 || H < 1 || W < 1) return dd::fail(DD_EINVAL, "dd_sur_planes: bad arguments");
    const int64_t n = (int64_t)B * H * W;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    ddk::planes_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(tmap, scal, H * W, n, (ddk::bf16 *)x);
    DD_CUDA_TRY(cudaGetLastError());
    return DD_OK;
}

dd_status dd_sur_planes_bg(const float *tmap, const float *scal3, float s_dim, int32_t k_exact, float mu, float sigma,
                           int32_t B, int32_t H, int32_t W, void *x, void *cuda_stream) {
    dd::clear_error();
    if (!tmap || !scal3 || !x || B < 1 || H < 1 || W < 1 || !(s_dim > 0.f) || k_exact < 0 || !(sigma > 0.f))
        return dd::fail(DD_EINVAL, "dd_sur_planes_bg: bad arguments");
    const int64_t n = (int64_t)B * H * W;
    ddk::planes_bg_kernel<<<(unsigned)((n + 255) / 256), 256, 0, (cudaStream_t)cuda_stream>>>(
        tmap, scal3, s_dim, (float)k_exact, mu, 1.0f / sigma, H * W, n, (ddk::bf16 *)x);
    DD_CUDA_TRY(cudaGetLastError());
    return DD_OK;
}

dd_status dd_sur_targets(const double *psi, const double *scale, int64_t n_maps, int64_t hw, double floor_rel_log10,
                         float mu, float sigma, float *out, void *cuda_stream) {
    dd::clear_error();
    if (!psi || !scale || !out || n_maps < 1 || hw < 1 || !(sigma > 0.f) || !(floor_rel_log10 < 0.0))
        return dd::fail(DD_EINVAL, "dd_sur_targets: bad arguments");
    ddk::targets_kernel<<<(unsigned)n_maps, 256, 0, (cudaStream_t)cuda_stream>>>(psi, scale, hw, floor_rel_log10, mu,
                                                                               1.0f / sigma, out);
    DD_CUDA_TRY(cudaGetLastError());
    return DD_OK;
}

dd_status dd_sur_fields(const float *pred, const double *scale, int64_t n_maps, int64_t hw, float mu, float sigma,
                        double *psi, void *cuda_stream) {
    dd::clear_error();
    if (!pred || !scale || !psi || n_maps < 1 || hw < 1) return dd::fail(DD_EINVAL, "dd_sur_fields: bad arguments");
    const int64_t n = n_maps * hw;
    ddk::fields_kernel<<<(unsigned)((n + 255) / 256), 256, 0, (cudaStream_t)cuda_stream>>>(pred, scale, hw, n, mu,
                                                                                          sigma, psi);
    DD_CUDA_TRY(cudaGetLastError());
    return DD_OK;
}

dd_status dd_sur_spot_error(const float *pred, const int32_t *idx, const double *exact, const double *scale,
                            const double *add, int32_t n_maps, int32_t hw, int32_t k, float mu, float sigma,
                            double *err, void *cuda_stream) {
    dd::clear_error();
    if (!pred || !idx || !exact || !scale || !err || n_maps < 1 || hw < 1 || k < 1)
        return dd::fail(DD_EINVAL, "dd_sur_spot_error: bad arguments");
    ddk::spot_error_kernel<<<n_maps, 128, 0, (cudaStream_t)cuda_stream>>>(pred, idx, exact, scale, add, hw, k, mu,
                                                                          sigma, err);
    DD_CUDA_TRY(cudaGetLastError());
    return DD_OK;
}

}  // extern "C"
