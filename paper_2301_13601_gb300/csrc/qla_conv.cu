// 3x3 convolution with circular padding on BF16 NHWC activations, as an
// implicit GEMM on the tcgen05 tensor cores with FP32 accumulation in TMEM.
//
// Activations hold nimg images of H x W stacked ([nimg][H][W][C]); each image
// is periodic on its own. One tile = 128 consecutive pixels of one image row
// (M = 128), all output channels, K = 9 taps x input channels. Input rows
// (130 pixels with the x halo, CIN channels) are staged once each, so the three
// x taps are shifted windows of the same row. 64 channels: a pixel is one
// 128-byte line of the 128-byte swizzled K-major layout, loaded by TMA, and a
// window starts on any line. 16 channels: the interleaved K-major layout
// without swizzle (any 16-byte aligned start is a valid operand). Each
// staged input row is multiplied once per (x tap, 16-channel slice) against
// the weights of all three y taps at once (N = 3 NOUT), accumulating into the
// TMEM accumulators of the three output rows it feeds. All 9 taps of the
// packed weights stay resident in shared memory. One thread issues the MMAs;
// the epilogue warps (32 TMEM lanes each) run the fused epilogue:
//   EPI_GELU      z = acc + b;  act = GELU(z) (+ residual);  stores act and, if asked, z (BF16)
//   EPI_LINEAR    out = acc + b (FP32, NOUT channels)
//   EPI_DGRAD     g = acc + g_in (FP32);  dz = BF16(g * GELU'(z_prev))
//   EPI_QUPDATE   q_out[c] = q_in[c] + scale * (acc + b)[c], c < 6, FP32 planes [nimg][6][H][W]
// GELU is the tanh form 0.5 x (1 + tanh(sqrt(2/pi) (x + 0.044715 x^3))).
#include <cuda_bf16.h>
#include <math.h>
#include <string.h>

#include "../../include/qla_surrogate.h"
#include "qla_internal.h"
#include "qla_pack.cuh"
#include "qla_tc.cuh"
#include "qla_tma.h"

namespace qla {

enum ConvEpi { EPI_GELU = QLA_EPI_GELU, EPI_LINEAR = QLA_EPI_LINEAR, EPI_DGRAD = QLA_EPI_DGRAD, EPI_QUPDATE = QLA_EPI_QUPDATE };


// GELU (tanh form) with the hardware tanh approximation (tanh.approx.f32,
// relative error about 2^-11, below the BF16 resolution of the outputs).
__device__ __forceinline__ float tanh_fast(float x) {
    float y;
    asm("tanh.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ float gelu_grad(float x) {
    const float k0 = 0.7978845608028654f, k1 = 0.7978845608028654f * 0.044715f;
    const float x2 = x * x;
    const float t = tanh_fast(x * fmaf(k1, x2, k0));
    // d/dx [0.5 x (1 + t)] = 0.5 (1 + t) + 0.5 x (1 - t^2) (k0 + 3 k1 x^2)
    return fmaf(0.5f * x * fmaf(-t, t, 1.0f), fmaf(3.0f * k1, x2, k0), 0.5f * (1.0f + t));
}

__device__ __forceinline__ void cp_async16(void *dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(tc::smem_addr(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_0() { asm volatile("cp.async.wait_group 0;\n" ::: "memory"); }

// Two channels per operation (the same roundings as one by one): the epilogues
// are bound by their instruction issue.
struct F2 {
    unsigned long long v;
};
__device__ __forceinline__ F2 f2(float a, float b) {
    F2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void f2_get(F2 a, float &x, float &y) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(a.v));
}
__device__ __forceinline__ F2 f2_fma(F2 a, F2 b, F2 c) {
    F2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}
__device__ __forceinline__ F2 f2_mul(F2 a, F2 b) {
    F2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 f2_add(F2 a, F2 b) {
    F2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 gelu_f2(F2 x) {  // GELU, tanh form; k0 = sqrt(2/pi), k1 = 0.044715 k0
    const float k0 = 0.7978845608028654f, k1 = 0.7978845608028654f * 0.044715f;
    const F2 arg = f2_mul(x, f2_fma(f2(k1, k1), f2_mul(x, x), f2(k0, k0)));
    float a, b;
    f2_get(arg, a, b);
    const F2 t = f2(tanh_fast(a), tanh_fast(b)), hx = f2_mul(x, f2(0.5f, 0.5f));
    return f2_fma(hx, t, hx);
}

__device__ __forceinline__ uint32_t bf2(float a, float b) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t *>(&h);
}

// Shared memory: a ring of NS halo rows, As[c][slot][130 px][16 B] (c = 8-channel
// chunk), then the packed weights of all nine taps, Bs[kx][c][ky][n][16 B]
// (the three y taps consecutive along N), then one staging buffer per epilogue
// warp for its BF16 output rows (32 pixels x one column half).
template <int CCH, int NOUT>
struct ConvLayout {
    static constexpr int HALO_PX = 130;
    // Ring depth; even, so that a slot is always released by the same epilogue group.
    static constexpr int NS = CCH >= 8 && NOUT >= 64 ? 8 : (CCH >= 8 ? 6 : 8);
    static_assert(NS % 2 == 0, "ring slots alternate between the two epilogue groups");
    // SWZ: the ring is NS * 130 lines of 128 bytes, line = slot * 130 + pixel;
    // the swizzle (16-byte chunk ^ line mod 8) goes by absolute line, for TMA and
    // MMA alike, so slots need no alignment of their own. One lane loads a row
    // in three boxes where a warp's cp.async took about 35 instructions per lane.
    // Last layer at 1024^2 94 -> 72 us, hidden layers 96 -> 95 (bound by the MMA
    // issue, see mma_bf16_leader, and their stores).
    static constexpr bool SWZ = CCH == 8;
    static constexpr int A_BYTES = CCH * NS * HALO_PX * 16;
    static constexpr int B_BYTES = 9 * CCH * NOUT * 16;
    static constexpr int A_OFF = 0;
    static constexpr int B_OFF = ((A_BYTES + 1023) / 1024) * 1024;
    static constexpr int STG_OFF = B_OFF + B_BYTES;
    static constexpr int STG_STRIDE = (NOUT < 32 ? NOUT : 32) * 2 + 16;  // bytes per pixel: an odd number of 16 B units
    static constexpr int STG_BYTES = 8 * 32 * STG_STRIDE;
    static constexpr int SMEM = STG_OFF + STG_BYTES;
    // At least half of an SM's shared memory, so one CTA per SM owns all of TMEM.
    static constexpr int SMEM_LAUNCH = SMEM > 116 * 1024 ? SMEM : 116 * 1024;
    static constexpr int TMEM_COLS = 512;
    static constexpr int NB = TMEM_COLS / NOUT;  // output-row accumulators (NOUT columns each)
};

// 16-byte chunk c of the pixel at `line` in the swizzled ring (byte offset).
__device__ __forceinline__ int conv_swz(int line, int c) { return line * 128 + ((c ^ (line & 7)) << 4); }

// Tensor maps of the swizzled form's input [nimg * H][W][64]: boxes of 128
// pixels and of one (the halo pixels, which wrap around the image).
struct ConvMaps {
    CUtensorMap px128, px1;
};

__device__ __forceinline__ void conv_tma(uint32_t dst, const CUtensorMap *map, int x, int row, uint64_t *bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], "
        "[%5];\n" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(0), "r"(x), "r"(row), "r"(tc::smem_addr(bar))
        : "memory");
}

constexpr int CONV_EPI_WARPS = 8;
constexpr int CONV_MMA_WARP = 8;
constexpr int CONV_LOAD_WARP = 9;
constexpr int CONV_THREADS = 320;
constexpr uint32_t CONV_WAIT_TRIES = 1u << 22;

__device__ __forceinline__ void cp_async_arrive_noinc(uint64_t *bar) {
    asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];\n" ::"r"(tc::smem_addr(bar)) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
    asm volatile("{\n.reg .b64 st;\nmbarrier.arrive.shared::cta.b64 st, [%0];\n}\n" ::"r"(tc::smem_addr(bar))
                 : "memory");
}

// Stores BF16 outputs of one column half of a warp's 32 pixels: vals[c] holds
// channels cb0 + 8c .. cb0 + 8c + 7 of this lane's pixel p_w0 + lane. The
// values pass through the warp's staging buffer so that the global stores are
// runs of NC * 2 bytes per pixel (whole sectors) instead of 16-byte pieces of
// 32 different pixels per instruction.
template <int NC, int NOUT, int STRIDE>
__device__ __forceinline__ void store_half_bf16(uint8_t *stg, const uint4 (&vals)[NC / 8], __nv_bfloat16 *out,
                                                size_t p_w0, int cb0, int lane) {
    constexpr int CH = NC / 8;  // 16-byte chunks per pixel
#pragma unroll
    for (int c = 0; c < CH; ++c) *reinterpret_cast<uint4 *>(stg + lane * STRIDE + c * 16) = vals[c];
    __syncwarp();
#pragma unroll
    for (int k = 0; k < CH; ++k) {
        const int idx = 32 * k + lane, pp = idx / CH, cc = idx % CH;
        const uint4 w = *reinterpret_cast<const uint4 *>(stg + pp * STRIDE + cc * 16);
        *reinterpret_cast<uint4 *>(out + (p_w0 + pp) * NOUT + cb0 + 8 * cc) = w;
    }
    __syncwarp();
}

// Segment walker shared by all roles: the CTA's rows, ordered (image, column
// block, row), split into runs of consecutive rows of one column block.
struct ConvSeg {
    int img, x0, y_s, len;
};
__host__ __device__ __forceinline__ ConvSeg conv_segment(long long u0, long long u_end, int H, int TPR) {
    ConvSeg g;
    g.y_s = int(u0 % H);
    const long long t2 = u0 / H;
    g.x0 = int(t2 % TPR) * 128;
    g.img = int(t2 / TPR);
    const long long end = (u0 - g.y_s + H) < u_end ? (u0 - g.y_s + H) : u_end;
    g.len = int(end - u0);
    return g;
}

// ---------------------------------------------------------------------------
// The MMA issue schedule, shared by the kernel's MMA warp and by the host-side
// enumeration (qla_conv_schedule) that tests/test_conv_schedule.py checks.
// Input row j of a run of `len` output rows (ring row r) feeds output rows
// j - ky (ky = 0..2); output row `on` = o_run + j owns accumulator block
// b0 = (-on) mod NB of the TMEM ring, so the rows it feeds are consecutive
// blocks and one MMA covers them (split in two where the ring wraps).
// ---------------------------------------------------------------------------
struct ConvMma {
    int kx, k2;      // x tap, 16-channel slice
    int ka, kb;      // y taps ka..kb in one MMA (N = (kb - ka + 1) NOUT)
    int blk;         // accumulator block of y tap ka
    int acc;         // 0: the first MMA of a new accumulator (accumulation off)
    uint32_t a_off;  // A descriptor start, 16-byte units from the row's ring slot
    uint32_t b_off;  // B descriptor start, 16-byte units from the weights
};

__host__ __device__ __forceinline__ int conv_block(long long on, int NB) { return int((NB - on % NB) % NB); }

// The MMAs of input row j: the y taps whose output row lies inside the run,
// split where the block ring wraps, the first MMA of a new accumulator (x tap
// 0, first slice, ky = 0) alone with accumulation off.
template <int CCH, int NOUT, int NS, int HP, class F>
__host__ __device__ __forceinline__ void conv_row_mmas(int j, int len, int b0, F &&emit) {
    constexpr int NB = 512 / NOUT;
    const int k_lo = j - len + 1 > 0 ? j - len + 1 : 0;
    const int k_hi = j < 2 ? j : 2;
    const int wrap = NB - b0;  // first ky whose block wraps to 0
    if (k_lo == 0 && k_hi == 2 && wrap > 2) {
        // a row inside the run whose three blocks do not wrap (most of them): a
        // list of constants
#pragma unroll
        for (int kx = 0; kx < 3; ++kx) {
#pragma unroll
            for (int k2 = 0; k2 < CCH / 2; ++k2) {
                const uint32_t ao = uint32_t((2 * k2) * NS * HP + kx), bo = uint32_t((kx * CCH + 2 * k2) * 3 * NOUT);
                if (kx == 0 && k2 == 0) {
                    emit(ConvMma{kx, k2, 0, 0, b0, 0, ao, bo});
                    emit(ConvMma{kx, k2, 1, 2, b0 + 1, 1, ao, bo + NOUT});
                } else {
                    emit(ConvMma{kx, k2, 0, 2, b0, 1, ao, bo});
                }
            }
        }
        return;
    }
#pragma unroll 1
    for (int kx = 0; kx < 3; ++kx) {
#pragma unroll 1
        for (int k2 = 0; k2 < CCH / 2; ++k2) {
            const bool first = kx == 0 && k2 == 0;
            for (int ka = k_lo; ka <= k_hi;) {
                int kb = k_hi;
                if (ka < wrap && wrap <= kb) kb = wrap - 1;
                if (first && ka == 0) kb = 0;
                const int blk = b0 + ka < NB ? b0 + ka : b0 + ka - NB;
                emit(ConvMma{kx, k2, ka, kb, blk, (first && ka == 0) ? 0 : 1, uint32_t((2 * k2) * NS * HP + kx),
                             uint32_t((kx * CCH + 2 * k2) * 3 * NOUT + ka * NOUT)});
                ka = kb + 1;
            }
        }
    }
}

// Before the MMAs of input row j: a new accumulator (j < len) reuses the block
// of output row on - NB, so the MMA warp waits for that row's epilogue on
// acc_empty[b0], phase parity (on / NB + 1) & 1. Returns false if no wait.
__host__ __device__ __forceinline__ bool conv_row_acc_wait(int j, int len, long long on, int NB, uint32_t *parity) {
    *parity = uint32_t(((on / NB) + 1) & 1);
    return j < len && on >= NB;
}

// After the MMAs of input row j: output row on - 2 has all its taps; its
// block is committed to acc_full (-1: none yet).
__host__ __device__ __forceinline__ int conv_row_done_block(int j, long long on, int NB) {
    return j >= 2 ? conv_block(on - 2, NB) : -1;
}

// Walks the CTA's rows in the order of every role: for each run, input rows
// j = 0 .. len + 1 (ring row g + j, output row o + j); row(sg, j, r, on)
// returns false to stop.
template <class F>
__host__ __device__ __forceinline__ void conv_walk_rows(long long u_begin, long long u_end, int H, int TPR, F &&row) {
    long long g = 0, o = 0;
    for (long long u0 = u_begin; u0 < u_end;) {
        const ConvSeg sg = conv_segment(u0, u_end, H, TPR);
        for (int j = 0; j < sg.len + 2; ++j)
            if (!row(sg, j, g + j, o + j)) return;
        g += sg.len + 2;
        o += sg.len;
        u0 += sg.len;
    }
}

// Persistent, warp-specialised conv kernel (320 threads = 10 warps). Work =
// rows of 128-pixel column blocks, ordered (image, column block, row); each CTA
// takes a contiguous range and walks down its column blocks with a ring of
// halo rows in shared memory, so every input row is loaded once per block.
//   warp 9 (loader)   copies each halo row into the ring (64 channels: three TMA
//                     boxes by one lane; 16: cp.async), which complete on
//                     full[slot]; waits on empty[slot]
//   warp 8 (MMA)      per input row, one lane issues the 3 x CCH/2 MMAs (x tap,
//                     16-channel slice) whose N = 3 NOUT columns are the
//                     accumulators of the three output rows the row feeds,
//                     then releases the row (empty[slot]) and commits acc_full
//                     of the output row it completes
//   warps 0-7 (epilogue) wait acc_full, tcgen05.ld, fused epilogue, stores;
//                     arrive on acc_empty, and on empty[slot] of the centre
//                     row (a residual equal to the input is read from the
//                     ring), so a row is free after its MMAs and its
//                     epilogue (edge rows of a run get their arrival at the
//                     run's start and end)
// TMEM holds NB = 512 / NOUT accumulators in a ring; output row o (counted
// over the CTA's runs) owns block (-o) mod NB, so the rows j, j-1, j-2 that
// input row j feeds are consecutive blocks and one MMA covers them (split in
// two where the ring wraps). Every wait is bounded; a timeout sets the error
// flag and the role stops, and the others time out in turn, so the kernel
// always ends.
// DG: the input-gradient epilogue (a kernel of its own: the registers of its
// prefetched rows cost the others 10%).
template <int CCH, int NOUT, bool DG>
__global__ void __launch_bounds__(CONV_THREADS, 1) conv3x3_tc_kernel(const ConvArgs a, const __grid_constant__ ConvMaps maps) {
    using L = ConvLayout<CCH, NOUT>;
    constexpr int CIN = 8 * CCH;
    constexpr int NS = L::NS;
    constexpr int HP = L::HALO_PX;
    extern __shared__ __align__(1024) unsigned char smem[];
    constexpr int NB = L::NB;
    __shared__ uint64_t full_bar[NS], empty_bar[NS], accf_bar[NB], acce_bar[NB], done_bar;
    __shared__ uint32_t tmem_base_s;
    __shared__ __align__(16) float bias_s[64];
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int H = a.H, W = a.W;
    const int TPR = W / 128;
    const long long T = (long long)a.nimg * TPR * H;
    const long long u_begin = T * blockIdx.x / gridDim.x;
    const long long u_end = T * (blockIdx.x + 1) / gridDim.x;
    uint8_t *As = smem + L::A_OFF;
    uint8_t *Bs = smem + L::B_OFF;

    {
        const uint4 *src = static_cast<const uint4 *>(a.w);
        for (int i = tid; i < 9 * CCH * NOUT; i += CONV_THREADS) {  // [t][c][n] -> [kx][c][ky][n]
            const int n = i % NOUT, c = (i / NOUT) % CCH, t = i / (NOUT * CCH);
            const int ky = t / 3, kx = t - 3 * ky;
            cp_async16(Bs + (((kx * CCH + c) * 3 + ky) * NOUT + n) * 16, src + i);
        }
        cp_async_commit();
        if (tid < 64) bias_s[tid] = (a.bias && tid < NOUT && a.epi != EPI_DGRAD) ? a.bias[tid] : 0.0f;
    }
    if (warp == CONV_MMA_WARP) tc::tmem_alloc(&tmem_base_s, L::TMEM_COLS);
    if (tid == 0) {
        for (int s = 0; s < NS; ++s) {
            tc::mbar_init(&full_bar[s], L::SWZ ? 1 : 32);
            tc::mbar_init(&empty_bar[s], 1 + CONV_EPI_WARPS / 2);
        }
        for (int b = 0; b < NB; ++b) {
            tc::mbar_init(&accf_bar[b], 1);
            tc::mbar_init(&acce_bar[b], CONV_EPI_WARPS / 2);
        }
        tc::mbar_init(&done_bar, 1);
        tc::fence_mbar_init();
    }
    cp_async_wait_0();
    tc::fence_proxy_async();
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = tmem_base_s;

    if (warp == CONV_LOAD_WARP) {
        // ---------------- loader ----------------
        const __nv_bfloat16 *xg = static_cast<const __nv_bfloat16 *>(a.x);
        long long g = 0;  // running row counter (ring position)
        bool ok = true;
        for (long long u0 = u_begin; u0 < u_end && ok;) {
            const ConvSeg sg = conv_segment(u0, u_end, H, TPR);
            const __nv_bfloat16 *ximg = xg + (size_t)sg.img * H * W * CIN;
            for (int j = 0; j < sg.len + 2 && ok; ++j, ++g) {
                const int slot = int(g % NS);
                if (g >= NS && !tc::mbar_wait(&empty_bar[slot], uint32_t((g / NS - 1) & 1), CONV_WAIT_TRIES)) {
                    ok = false;
                    break;
                }
                int yy = (sg.y_s - 1 + j) % H;
                yy = yy < 0 ? yy + H : yy;
                if constexpr (L::SWZ) {
                    if (lane == 0) {
                        const int row = sg.img * H + yy;
                        const uint32_t dst = tc::smem_addr(As) + uint32_t(slot * HP * 128);
                        tc::mbar_arrive_expect_tx(&full_bar[slot], HP * 128);
                        conv_tma(dst, &maps.px1, sg.x0 == 0 ? W - 1 : sg.x0 - 1, row, &full_bar[slot]);
                        conv_tma(dst + 128, &maps.px128, sg.x0, row, &full_bar[slot]);
                        conv_tma(dst + 129 * 128, &maps.px1, sg.x0 + 128 == W ? 0 : sg.x0 + 128, row, &full_bar[slot]);
                    }
                    __syncwarp();
                    continue;
                }
                const __nv_bfloat16 *row = ximg + (size_t)yy * W * CIN;
                for (int i = lane; i < CCH * HP; i += 32) {
                    const int c = i % CCH, px = i / CCH;
                    int xx = sg.x0 + px - 1;
                    xx = xx < 0 ? xx + W : (xx >= W ? xx - W : xx);
                    cp_async16(As + ((c * NS + slot) * HP + px) * 16, row + (size_t)xx * CIN + 8 * c);
                }
                cp_async_arrive_noinc(&full_bar[slot]);
            }
            u0 += sg.len;
        }
        cp_async_wait_0();
        if constexpr (L::SWZ) {  // no copy outlives the CTA, also when a role gave up
            for (long long r = g > NS ? g - NS : 0; r < g; ++r)
                if (!tc::mbar_wait(&full_bar[r % NS], uint32_t((r / NS) & 1), CONV_WAIT_TRIES)) ok = false;
        }
        if (!ok && lane == 0) atomicExch(a.error, 1);
    } else if (warp == CONV_MMA_WARP) {
        // ---------------- MMA issuer ----------------
        // Input row j of a run feeds output rows j - ky (ky = 0..2) through
        // the weights of y tap ky; those rows' accumulators are the blocks
        // b0, b0 + 1, b0 + 2 (mod NB), b0 = block of output row j. The first
        // MMA of a new accumulator (x tap 0, first slice, ky = 0) runs alone
        // with accumulation off; the rest add to what is there.
        constexpr uint32_t IDESC1 = tc::make_idesc_bf16(128, NOUT);
        constexpr uint32_t IDESC2 = tc::make_idesc_bf16(128, 2 * NOUT);
        constexpr uint32_t IDESC3 = tc::make_idesc_bf16(128, 3 * NOUT);
        constexpr uint32_t A_LBO = NS * HP * 16, A_SBO = 128;
        constexpr uint32_t B_LBO = 3 * NOUT * 16, B_SBO = 128;
        const uint64_t ad0 = L::SWZ ? tc::make_desc_sw128(tc::smem_addr(As), 1024)
                                    : tc::make_desc(tc::smem_addr(As), A_LBO, A_SBO);
        const uint64_t bd0 = tc::make_desc(tc::smem_addr(Bs), B_LBO, B_SBO);
        const uint32_t a_lo0 = uint32_t(ad0), a_hi = uint32_t(ad0 >> 32);
        const uint32_t b_lo0 = uint32_t(bd0), b_hi = uint32_t(bd0 >> 32);
        const uint32_t leader = tc::elect_one();
        bool ok = true;
        conv_walk_rows(u_begin, u_end, H, TPR, [&](const ConvSeg &sg, int j, long long r, long long on) {
            const int b0 = conv_block(on, NB);
            if (!tc::mbar_wait(&full_bar[r % NS], uint32_t((r / NS) & 1), CONV_WAIT_TRIES)) ok = false;
            uint32_t par = 0;
            if (ok && conv_row_acc_wait(j, sg.len, on, NB, &par) && !tc::mbar_wait(&acce_bar[b0], par, CONV_WAIT_TRIES))
                ok = false;
            if (!ok) return false;
            // Rows copied by cp.async are generic-proxy writes; the barrier orders
            // them before this thread, the fence before the tensor cores' reads.
            if constexpr (!L::SWZ) tc::fence_proxy_async();
            tc::fence_after_sync();
            {
                // (slot * HP * line bytes) >> 4
                const uint32_t a_row = a_lo0 + uint32_t(int(r % NS) * HP * (L::SWZ ? 8 : 1));
                conv_row_mmas<CCH, NOUT, NS, HP>(j, sg.len, b0, [&](const ConvMma &m) {
                    const uint32_t idesc = m.kb == m.ka ? IDESC1 : (m.kb == m.ka + 1 ? IDESC2 : IDESC3);
                    // swizzled: a pixel is 8 units of 16 bytes, a 16-channel slice 2
                    const uint32_t a_off = L::SWZ ? uint32_t(8 * m.kx + 2 * m.k2) : m.a_off;
                    tc::mma_bf16_leader(leader, tmem + uint32_t(m.blk * NOUT), a_row + a_off, a_hi, b_lo0 + m.b_off,
                                        b_hi, idesc, uint32_t(m.acc));
                });
                tc::mma_commit_leader(leader, &empty_bar[r % NS]);  // the tensor cores are done with row r
                const int bd = conv_row_done_block(j, on, NB);
                if (bd >= 0) tc::mma_commit_leader(leader, &accf_bar[bd]);  // output row on - 2
            }
            return true;
        });
        tc::mma_commit_leader(leader, &done_bar);  // tracks every MMA issued above
        if (!tc::mbar_wait(&done_bar, 0u, CONV_WAIT_TRIES)) ok = false;
        if (!ok && lane == 0) atomicExch(a.error, 1);
    } else {
        // ---------------- epilogue ----------------
        // Two groups of four warps (grp = warp / 4) take alternate output rows
        // (o mod 2), so the epilogues of two rows overlap; each warp covers its
        // TMEM lane quarter and all NOUT columns. Ring rows are released by the
        // group of the output row they are the centre of (edge rows: the group
        // of the neighbouring output row), so a slot is always released by the
        // same group and its arrivals come in order.
        const int q = warp & 3, grp = warp >> 2;
        const int m = 32 * q + lane;
        uint8_t *stg = smem + L::STG_OFF + warp * 32 * L::STG_STRIDE;  // this warp's staging buffer
        constexpr int NC = NOUT < 32 ? NOUT : 32;
        constexpr int NCB = NOUT >= 64 ? 2 : 1;
        const bool res_smem = a.epi == EPI_GELU && a.aux0 != nullptr && a.aux0 == a.x && CIN == NOUT;
        long long o = 0, g = 0;
        bool ok = true;
        for (long long u0 = u_begin; u0 < u_end && ok;) {
            const ConvSeg sg = conv_segment(u0, u_end, H, TPR);
            const long long o_seg = o;
            __syncwarp();
            if (lane == 0 && int((o_seg - 1) & 1) == grp) mbar_arrive(&empty_bar[g % NS]);  // first halo row
            // q update (the surrogate's last layer, NOUT = 16): the FP32 input
            // state of this group's rows is loaded one of its rows ahead, before
            // the wait for the row's accumulator, so that the load latency overlaps
            // the wait and the previous row's epilogue (issued after the wait it was
            // exposed once per row). Other widths load it after the wait.
            constexpr bool QPRE = NOUT == 16;
            constexpr int NQ = QPRE ? 6 : 1;
            const size_t qP = (size_t)H * W;
            bool qup = false;
            const float *qi = nullptr;
            float qv[NQ];
            auto qload = [&](int i, float (&dst)[NQ]) {
                const size_t pix = (size_t)(sg.y_s + i) * W + sg.x0 + m;
#pragma unroll
                for (int c = 0; c < NQ; ++c) dst[c] = qi[c * qP + pix];
            };
            if constexpr (QPRE) {
                qup = a.epi == EPI_QUPDATE;
                if (qup) {
                    qi = static_cast<const float *>(a.aux0) + (size_t)sg.img * 6 * qP;
                    const int i_first = int(((long long)grp - o_seg) & 1);  // first i with (o_seg + i) mod 2 == grp
                    if (i_first < sg.len) qload(i_first, qv);
                }
            }
            // input gradient (64 channels out): the incoming gradient and the
            // pre-activation of the next 32 channels are loaded as soon as the last
            // ones are used, before their accumulator is waited for
            constexpr bool DPRE = DG && NOUT == 64;
            constexpr int NGQ = DPRE ? 8 : 1, NZQ = DPRE ? 4 : 1;
            float4 gq[NGQ];
            uint4 zq[NZQ];
            const size_t dstep = a.tiled ? 128 : 1;  // 16-byte pieces of a pixel
            auto dpix = [&](int i, int cb0, int per) {  // in units of `per` channels (16 bytes)
                const size_t row = (size_t)sg.img * H + sg.y_s + i;
                return a.tiled ? (row * TPR + (sg.x0 >> 7)) * (NOUT / per * 128) + cb0 / per * 128 + m
                               : ((row * W + sg.x0 + m) * NOUT + cb0) / per;
            };
            auto dload = [&](int i, int cb0) {
                if (a.aux0) {
                    const float4 *const gin = static_cast<const float4 *>(a.aux0) + dpix(i, cb0, 4);
#pragma unroll
                    for (int k = 0; k < NGQ; ++k) gq[k] = gin[k * dstep];
                } else {
#pragma unroll
                    for (int k = 0; k < NGQ; ++k) gq[k] = make_float4(0.f, 0.f, 0.f, 0.f);
                }
                const uint4 *const zp = static_cast<const uint4 *>(a.zprev) + dpix(i, cb0, 8);
#pragma unroll
                for (int k = 0; k < NZQ; ++k) zq[k] = zp[k * dstep];
            };
            if constexpr (DPRE) {
                const int i_first = int(((long long)grp - o_seg) & 1);
                if (i_first < sg.len) dload(i_first, 0);
            }
            for (int i = 0; i < sg.len; ++i, ++o) {
                if (int(o & 1) != grp) continue;
                float qn[NQ];
                bool q_more = false;
                if constexpr (QPRE) {
                    q_more = qup && i + 2 < sg.len;
                    if (q_more) qload(i + 2, qn);
                }
                const int b = int((NB - o % NB) % NB);
                if (!tc::mbar_wait(&accf_bar[b], uint32_t((o / NB) & 1), CONV_WAIT_TRIES)) {
                    ok = false;
                    break;
                }
                tc::fence_after_sync();
                if constexpr (L::SWZ) {
                    // the centre row, which TMA wrote and this warp may read as the
                    // residual, is released only below, so this phase is the row's
                    if (res_smem && !tc::mbar_wait(&full_bar[(g + i + 1) % NS], uint32_t(((g + i + 1) / NS) & 1),
                                                   CONV_WAIT_TRIES)) {
                        ok = false;
                        break;
                    }
                }
#pragma unroll 1
                for (int cbi = 0; cbi < NCB; ++cbi) {
                    const int cb0 = 32 * cbi;
                    const int y = sg.y_s + i;
                    const size_t p = ((size_t)sg.img * H + y) * W + sg.x0 + m;
                    const size_t tile = ((size_t)sg.img * H + y) * TPR + (sg.x0 >> 7);  // ConvArgs::tiled
                    float v[32];
                    const uint32_t ta = tmem + uint32_t(b * NOUT + cb0) + (uint32_t(32 * q) << 16);
                    if constexpr (NC == 32) tc::tmem_ld32(ta, v);
                    else tc::tmem_ld16(ta, v);
                    if constexpr (!DG) {
#pragma unroll
                        for (int k = 0; k < NC; k += 4) {
                            const float4 bb = *reinterpret_cast<const float4 *>(bias_s + cb0 + k);
                            f2_get(f2_add(f2(v[k], v[k + 1]), f2(bb.x, bb.y)), v[k], v[k + 1]);
                            f2_get(f2_add(f2(v[k + 2], v[k + 3]), f2(bb.z, bb.w)), v[k + 2], v[k + 3]);
                        }
                    }
                    if (!DG && a.epi == EPI_GELU) {
                        const bool res = a.aux0 != nullptr;
                        const uint4 *const rp =
                            reinterpret_cast<const uint4 *>(static_cast<const __nv_bfloat16 *>(a.aux0) + p * NOUT + cb0);
                        const int line = int((g + i + 1) % NS) * HP + m + 1;  // the centre pixel in the ring
                        uint4 av[NC / 8], zv[NC / 8];
#pragma unroll
                        for (int c4 = 0; c4 < NC / 8; ++c4) {
                            float g8[8];
#pragma unroll
                            for (int k = 0; k < 8; k += 2)
                                f2_get(gelu_f2(f2(v[8 * c4 + k], v[8 * c4 + k + 1])), g8[k], g8[k + 1]);
                            if (res) {
                                const uint4 w4 =
                                    res_smem ? *reinterpret_cast<const uint4 *>(
                                                   L::SWZ ? As + conv_swz(line, cb0 / 8 + c4)
                                                          : As + (((cb0 / 8 + c4) * NS + int((g + i + 1) % NS)) * HP +
                                                                  m + 1) * 16)
                                             : rp[c4];
                                const uint32_t ww[4] = {w4.x, w4.y, w4.z, w4.w};
#pragma unroll
                                for (int k = 0; k < 4; ++k)
                                    f2_get(f2_add(f2(g8[2 * k], g8[2 * k + 1]),
                                                  f2(__uint_as_float(ww[k] << 16),
                                                     __uint_as_float(ww[k] & 0xffff0000u))),
                                           g8[2 * k], g8[2 * k + 1]);
                            }
                            av[c4] = make_uint4(bf2(g8[0], g8[1]), bf2(g8[2], g8[3]), bf2(g8[4], g8[5]),
                                                bf2(g8[6], g8[7]));
                            const float *z = v + 8 * c4;
                            zv[c4] = make_uint4(bf2(z[0], z[1]), bf2(z[2], z[3]), bf2(z[4], z[5]), bf2(z[6], z[7]));
                        }
                        // Staged stores: hidden layer at 1024^2 69.3 us against 75.3 with a
                        // lane storing its own pixel's 16-byte pieces.
                        store_half_bf16<NC, NOUT, L::STG_STRIDE>(stg, av, static_cast<__nv_bfloat16 *>(a.out1),
                                                                 p - lane, cb0, lane);
                        if (a.out0 && a.tiled) {
                            uint4 *const zo = static_cast<uint4 *>(a.out0) + tile * (NOUT / 8 * 128) + cb0 / 8 * 128 + m;
#pragma unroll
                            for (int c4 = 0; c4 < NC / 8; ++c4) zo[c4 * 128] = zv[c4];
                        } else if (a.out0) {
                            store_half_bf16<NC, NOUT, L::STG_STRIDE>(stg, zv, static_cast<__nv_bfloat16 *>(a.out0),
                                                                     p - lane, cb0, lane);
                        }
                    } else if (!DG && a.epi == EPI_LINEAR) {
                        float4 *op = reinterpret_cast<float4 *>(static_cast<float *>(a.out0) + p * NOUT + cb0);
#pragma unroll
                        for (int k = 0; k < NC / 4; ++k)
                            op[k] = make_float4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
                    } else if constexpr (DG) {
                        if constexpr (DPRE) {
                            float4 *const go = static_cast<float4 *>(a.out0) + dpix(i, cb0, 4);
                            uint4 dzv[NC / 8], zc[NC / 8];
#pragma unroll
                            for (int c4 = 0; c4 < NC / 8; ++c4) {
                                const float4 ga = gq[2 * c4], gb = gq[2 * c4 + 1];
                                float *const g8 = v + 8 * c4;
                                if (a.aux0) {
                                    g8[0] += ga.x; g8[1] += ga.y; g8[2] += ga.z; g8[3] += ga.w;
                                    g8[4] += gb.x; g8[5] += gb.y; g8[6] += gb.z; g8[7] += gb.w;
                                }
                                zc[c4] = zq[c4];
                            }
                            if (cb0 == 0) dload(i, 32);
                            else if (i + 2 < sg.len) dload(i + 2, 0);
#pragma unroll
                            for (int c4 = 0; c4 < NC / 8; ++c4) {
                                const float *const g8 = v + 8 * c4;
                                go[2 * c4 * dstep] = make_float4(g8[0], g8[1], g8[2], g8[3]);
                                go[(2 * c4 + 1) * dstep] = make_float4(g8[4], g8[5], g8[6], g8[7]);
                                const uint32_t zz[4] = {zc[c4].x, zc[c4].y, zc[c4].z, zc[c4].w};
                                float d[8];
#pragma unroll
                                for (int k = 0; k < 4; ++k) {
                                    d[2 * k] = g8[2 * k] * gelu_grad(__uint_as_float(zz[k] << 16));
                                    d[2 * k + 1] = g8[2 * k + 1] * gelu_grad(__uint_as_float(zz[k] & 0xffff0000u));
                                }
                                dzv[c4] = make_uint4(bf2(d[0], d[1]), bf2(d[2], d[3]), bf2(d[4], d[5]), bf2(d[6], d[7]));
                            }
                            store_half_bf16<NC, NOUT, L::STG_STRIDE>(
                                stg, dzv, static_cast<__nv_bfloat16 *>(a.out1), p - lane, cb0, lane);
                        } else {
                            const float4 *const gin =
                                a.aux0 ? static_cast<const float4 *>(a.aux0) + p * NOUT / 4 : nullptr;
                            float4 *const go = static_cast<float4 *>(a.out0) + p * NOUT / 4;
                            const uint4 *const zp = static_cast<const uint4 *>(a.zprev) + p * NOUT / 8;
                            uint4 dzv[NC / 8];
#pragma unroll
                            for (int c4 = 0; c4 < NC / 8; ++c4) {
                                float *const g8 = v + 8 * c4;
                                if (gin) {
                                    const float4 ga = gin[2 * c4], gb = gin[2 * c4 + 1];
                                    g8[0] += ga.x; g8[1] += ga.y; g8[2] += ga.z; g8[3] += ga.w;
                                    g8[4] += gb.x; g8[5] += gb.y; g8[6] += gb.z; g8[7] += gb.w;
                                }
                                go[2 * c4] = make_float4(g8[0], g8[1], g8[2], g8[3]);
                                go[2 * c4 + 1] = make_float4(g8[4], g8[5], g8[6], g8[7]);
                                const uint4 z4 = zp[c4];
                                const uint32_t zz[4] = {z4.x, z4.y, z4.z, z4.w};
                                float d[8];
#pragma unroll
                                for (int k = 0; k < 4; ++k) {
                                    d[2 * k] = g8[2 * k] * gelu_grad(__uint_as_float(zz[k] << 16));
                                    d[2 * k + 1] = g8[2 * k + 1] * gelu_grad(__uint_as_float(zz[k] & 0xffff0000u));
                                }
                                dzv[c4] = make_uint4(bf2(d[0], d[1]), bf2(d[2], d[3]), bf2(d[4], d[5]), bf2(d[6], d[7]));
                            }
                            store_half_bf16<NC, NOUT, L::STG_STRIDE>(
                                stg, dzv, static_cast<__nv_bfloat16 *>(a.out1), p - lane, cb0, lane);
                        }
                    } else if (cb0 == 0) {  // EPI_QUPDATE: channels 0..5
                        const size_t pix = (size_t)y * W + sg.x0 + m;
                        float *qo = static_cast<float *>(a.out0) + (size_t)sg.img * 6 * qP;
                        if constexpr (QPRE) {
#pragma unroll
                            for (int c = 0; c < 6; ++c) qo[c * qP + pix] = qv[c] + a.scale * v[c];
                        } else {
                            const float *qin = static_cast<const float *>(a.aux0) + (size_t)sg.img * 6 * qP;
#pragma unroll
                            for (int c = 0; c < 6; ++c) qo[c * qP + pix] = qin[c * qP + pix] + a.scale * v[c];
                        }
                    }
                }
                if (q_more) {
#pragma unroll
                    for (int c = 0; c < NQ; ++c) qv[c] = qn[c];
                }
                tc::fence_before_sync();
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive(&acce_bar[b]);
                    mbar_arrive(&empty_bar[(g + i + 1) % NS]);  // centre row of output row i
                }
            }
            if (!ok) break;
            __syncwarp();
            if (lane == 0 && int((o_seg + sg.len) & 1) == grp)
                mbar_arrive(&empty_bar[(g + sg.len + 1) % NS]);  // last halo row
            g += sg.len + 2;
            u0 += sg.len;
        }
        if (!ok && lane == 0) atomicExch(a.error, 1);
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    if (warp == CONV_MMA_WARP) tc::tmem_dealloc(tmem, L::TMEM_COLS);
}

// Tensor map of rows of W 64-channel pixels, boxes of n pixels in swizzled lines.
cudaError_t pixel_map(CUtensorMap *map, const void *base, int W, long long rows, unsigned n) {
    const EncodeTiledFn fn = encode_tiled_fn();
    if (!fn) return cudaErrorNotSupported;
    const cuuint64_t dim[3] = {64, cuuint64_t(W), cuuint64_t(rows)};
    const cuuint64_t str[2] = {128, cuuint64_t(W) * 128};
    const cuuint32_t one[3] = {1, 1, 1}, box[3] = {64, n, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(base), dim, str, box, one,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS
               ? cudaSuccess
               : cudaErrorInvalidValue;
}

template <int CCH, int NOUT, bool DG>
cudaError_t launch_conv_t(const ConvArgs &a, cudaStream_t st) {
    using L = ConvLayout<CCH, NOUT>;
    cudaError_t e = cudaFuncSetAttribute(conv3x3_tc_kernel<CCH, NOUT, DG>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         L::SMEM_LAUNCH);
    if (e != cudaSuccess) return e;
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const long long rows = (long long)a.nimg * a.H * (a.W / 128);
    const int grid = rows < sms ? int(rows) : sms;
    ConvMaps maps;
    memset(&maps, 0, sizeof(maps));
    if (L::SWZ) {
        const long long img_rows = (long long)a.nimg * a.H;
        if ((e = pixel_map(&maps.px128, a.x, a.W, img_rows, 128)) != cudaSuccess) return e;
        if ((e = pixel_map(&maps.px1, a.x, a.W, img_rows, 1)) != cudaSuccess) return e;
    }
    conv3x3_tc_kernel<CCH, NOUT, DG><<<grid, CONV_THREADS, L::SMEM_LAUNCH, st>>>(a, maps);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Weight gradient on the tensor cores:
//   dW[n][c][ky][kx] = sum_p g[p][n] x[p + (ky-1, kx-1)][c]
// as D[m][n] = sum_k A[m][k] B[n][k] with K = the 128 pixels of a tile of x and
// both operands MN-major. A rows are (ky, c) for two consecutive rows of x stacked
// in M = 128 (ky = 0, 1 in one tile; ky = 2 and an unused half in the other); B
// columns are (kx, n): g[p + (0, 1 - kx)] for the three kx side by side, N = 3 NT,
// so that an A tile is read from shared memory once for the three of them (one
// MMA of N = 64 per kx read 6 KB for 32 cycles of arithmetic, and, with kx as a
// shift of A, across lines: 80 cycles each). The tile's edges need g's halo pixels,
// not x's. With 64 channels a pixel of g is a swizzled line, and the next kx is
// the operand that starts one line earlier: no copies. At 4 x 256 x 512 the
// 64 -> 64 layers take 36 us (54 before), of which 20 are their DRAM traffic
// (134 MB) and 22 their MMAs; 16 -> 64 35 (48), 64 -> 16 25 (42).
// Two accumulator tiles (the row pairs) stay in TMEM for all of a CTA's rows; at
// the end each CTA writes its partial sums [9][NT][64] (FP32), reduced over CTAs
// in a fixed order later, and those of the bias gradient [NT], summed by warps
// that the tensor cores leave idle (a kernel of its own read g once more, 22 us
// per layer).
// The x ring has one mirror slot after the last, a copy of slot 0, so that two
// consecutive rows are always adjacent in memory. Source x may have 16 or 64
// channels (16: the other chunks stay zero).
// ---------------------------------------------------------------------------
constexpr int WG_SUM_WARPS = 4;  // warps that sum the bias gradient
// The load warp and the epilogue warps that sum nothing copy 16-channel rows.
constexpr int WG_LOADERS = 1 + CONV_EPI_WARPS - WG_SUM_WARPS;

template <int CS, int NT>
struct WgradLayout {
    // 64-channel operands lie in swizzled lines of one pixel each, brought by TMA;
    // 16-channel ones in planes of 8-channel chunks, copied by WG_LOADERS warps.
    static constexpr bool SWX = CS == 64, SWG = NT == 64;
    static constexpr int NSX = 6;
    static constexpr int XSLOT = 128 * 128;
    static constexpr int X_BYTES = (NSX + 1) * XSLOT;
    static constexpr int NSG = 4;
    static constexpr int GSLOT = SWG ? 130 * 128 : 3 * NT * 128 * 2;  // halo pixels, or three shifted copies
    static constexpr int G_OFF = X_BYTES;
    static constexpr int SMEM = G_OFF + NSG * GSLOT;
    static constexpr int TMEM_COLS = NT == 64 ? 512 : 128;  // 2 tiles x 3 NT columns
};

struct WgradMaps {
    CUtensorMap x128, g128, g1;
};

template <int CS, int NT>
__global__ void __launch_bounds__(CONV_THREADS, 1) wgrad_tc_kernel(const WgradArgs a,
                                                                   const __grid_constant__ WgradMaps maps) {
    using L = WgradLayout<CS, NT>;
    constexpr int NSX = L::NSX, NSG = L::NSG;
    constexpr bool SWX = L::SWX, SWG = L::SWG;
    constexpr int CCS = CS / 8, CCT = NT / 8;  // chunks per pixel
    // A warp copies 4 (or 2) chunks of 8 (or 16) pixels at a time: whole lines of
    // shared memory, half lines of global memory.
    constexpr int XB = CCS < 4 ? CCS : 4, GB = CCT < 4 ? CCT : 4;
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ uint64_t xf_bar[NSX], xe_bar[NSX], gf_bar[NSG], ge_bar[NSG], done_bar;
    __shared__ uint32_t tmem_base_s;
    __shared__ float bias_s[WG_SUM_WARPS][NT];
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int H = a.H, W = a.W;
    const int TPR = W / 128;
    const long long T = (long long)a.nimg * TPR * H;
    const long long u_begin = T * blockIdx.x / gridDim.x;
    const long long u_end = T * (blockIdx.x + 1) / gridDim.x;
    uint8_t *Xs = smem;
    uint8_t *Gs = smem + L::G_OFF;

    if constexpr (!SWX)  // the other chunks stay zero
        for (int i = tid; i < L::X_BYTES / 16; i += CONV_THREADS)
            reinterpret_cast<uint4 *>(Xs)[i] = make_uint4(0, 0, 0, 0);
    if (warp == CONV_MMA_WARP) tc::tmem_alloc(&tmem_base_s, L::TMEM_COLS);
    if (tid == 0) {
        for (int s = 0; s < NSX; ++s) {
            tc::mbar_init(&xf_bar[s], SWX ? 1 : 32 * WG_LOADERS);
            tc::mbar_init(&xe_bar[s], 1);
        }
        for (int s = 0; s < NSG; ++s) {
            tc::mbar_init(&gf_bar[s], SWG ? 1 : 32 * WG_LOADERS);
            tc::mbar_init(&ge_bar[s], 1 + WG_SUM_WARPS);
        }
        tc::mbar_init(&done_bar, 1);
        tc::fence_mbar_init();
    }
    tc::fence_proxy_async();
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = tmem_base_s;

    if (warp == CONV_LOAD_WARP || (!(SWX && SWG) && warp >= WG_SUM_WARPS && warp < CONV_EPI_WARPS)) {
        const bool tma = warp == CONV_LOAD_WARP && lane == 0;
        const int loader = 32 * (warp == CONV_LOAD_WARP ? 0 : warp - WG_SUM_WARPS + 1) + lane;
        const __nv_bfloat16 *xg = static_cast<const __nv_bfloat16 *>(a.x);
        const __nv_bfloat16 *gg = static_cast<const __nv_bfloat16 *>(a.g);
        long long gx = 0, gn = 0;
        bool ok = true;
        auto load_x = [&](const ConvSeg &sg, int j) -> bool {
            const int slot = int(gx % NSX);
            if (gx >= NSX && !tc::mbar_wait(&xe_bar[slot], uint32_t((gx / NSX - 1) & 1), CONV_WAIT_TRIES)) return false;
            int yy = (sg.y_s - 1 + j) % H;
            yy = yy < 0 ? yy + H : yy;
            const int row = sg.img * H + yy;
            if constexpr (SWX) {
                if (tma) {
                    const uint32_t dst = tc::smem_addr(Xs) + uint32_t(slot * L::XSLOT);
                    tc::mbar_arrive_expect_tx(&xf_bar[slot], (slot == 0 ? 2 : 1) * L::XSLOT);
                    conv_tma(dst, &maps.x128, sg.x0, row, &xf_bar[slot]);
                    if (slot == 0) conv_tma(dst + NSX * L::XSLOT, &maps.x128, sg.x0, row, &xf_bar[slot]);
                }
                __syncwarp();
            } else {
                const __nv_bfloat16 *src = xg + ((size_t)row * W + sg.x0) * CS;
                for (int i = loader; i < CCS * 128; i += 32 * WG_LOADERS) {
                    const int c = i % XB + i / (XB * 128) * XB, px = i / XB % 128;
                    cp_async16(Xs + ((slot * 8 + c) * 128 + px) * 16, src + px * CS + 8 * c);
                    if (slot == 0) cp_async16(Xs + ((NSX * 8 + c) * 128 + px) * 16, src + px * CS + 8 * c);
                }
                cp_async_arrive_noinc(&xf_bar[slot]);
            }
            ++gx;
            return true;
        };
        auto load_g = [&](const ConvSeg &sg, int i) -> bool {
            const int slot = int(gn % NSG);
            if (gn >= NSG && !tc::mbar_wait(&ge_bar[slot], uint32_t((gn / NSG - 1) & 1), CONV_WAIT_TRIES)) return false;
            const int row = sg.img * H + sg.y_s + i;
            if constexpr (SWG) {
                if (tma) {
                    const uint32_t dst = tc::smem_addr(Gs) + uint32_t(slot * L::GSLOT);
                    tc::mbar_arrive_expect_tx(&gf_bar[slot], L::GSLOT);
                    conv_tma(dst, &maps.g1, sg.x0 == 0 ? W - 1 : sg.x0 - 1, row, &gf_bar[slot]);
                    conv_tma(dst + 128, &maps.g128, sg.x0, row, &gf_bar[slot]);
                    conv_tma(dst + 129 * 128, &maps.g1, sg.x0 + 128 == W ? 0 : sg.x0 + 128, row, &gf_bar[slot]);
                }
                __syncwarp();
            } else {
                const __nv_bfloat16 *src = gg + (size_t)row * W * NT;
                for (int k = loader; k < CCT * 128; k += 32 * WG_LOADERS) {
                    const int c = k % GB + k / (GB * 128) * GB, px = k / GB % 128;
#pragma unroll
                    for (int s = 0; s < 3; ++s) {
                        int xx = sg.x0 + px - 1 + s;
                        xx = xx < 0 ? xx + W : (xx >= W ? xx - W : xx);
                        cp_async16(Gs + slot * L::GSLOT + ((s * CCT + c) * 128 + px) * 16, src + (size_t)xx * NT + 8 * c);
                    }
                }
                cp_async_arrive_noinc(&gf_bar[slot]);
            }
            ++gn;
            return true;
        };
        for (long long u0 = u_begin; u0 < u_end && ok;) {
            const ConvSeg sg = conv_segment(u0, u_end, H, TPR);
            ok = load_x(sg, 0) && load_x(sg, 1);
            for (int i = 0; i < sg.len && ok; ++i) ok = load_x(sg, i + 2) && load_g(sg, i);
            u0 += sg.len;
        }
        cp_async_wait_0();
        // no copy outlives the CTA, also when a role gave up
        if constexpr (SWX)
            for (long long r = gx > NSX ? gx - NSX : 0; r < gx; ++r)
                if (!tc::mbar_wait(&xf_bar[r % NSX], uint32_t((r / NSX) & 1), CONV_WAIT_TRIES)) ok = false;
        if constexpr (SWG)
            for (long long r = gn > NSG ? gn - NSG : 0; r < gn; ++r)
                if (!tc::mbar_wait(&gf_bar[r % NSG], uint32_t((r / NSG) & 1), CONV_WAIT_TRIES)) ok = false;
        if (!ok && lane == 0) atomicExch(a.error, 1);
    } else if (warp == CONV_MMA_WARP) {
        constexpr uint32_t IDESC = tc::make_idesc_bf16(128, 3 * NT) | (1u << 15) | (1u << 16);  // A, B MN-major
        const uint32_t x_base = tc::smem_addr(Xs), g_base = tc::smem_addr(Gs);
        // MN-major, swizzled: an atom is 8 pixels (lines) x 64 channels; the leading
        // byte offset steps along M/N (the next row of x; the g shifted by one
        // pixel more: the next line), the stride byte offset along K (the next 8
        // lines). Without swizzle a core matrix is 8 pixels x 8 channels; the
        // leading byte offset steps along K, the stride byte offset along M/N.
        const uint64_t ad0 = SWX ? tc::make_desc_sw128(x_base, 1024, L::XSLOT) : tc::make_desc(x_base, 128, 128 * 16);
        const uint64_t bd0 = SWG ? tc::make_desc_sw128(g_base, 1024, 128) : tc::make_desc(g_base, 128, 128 * 16);
        constexpr uint32_t A_K = SWX ? 128 : 16, B_K = SWG ? 128 : 16;  // 16 pixels on, in 16 bytes
        const uint32_t a_lo0 = uint32_t(ad0), a_hi = uint32_t(ad0 >> 32);
        const uint32_t b_lo0 = uint32_t(bd0), b_hi = uint32_t(bd0 >> 32);
        const uint32_t leader = tc::elect_one();
        long long gx = 0, gn = 0;
        bool ok = true, first = true;
        for (long long u0 = u_begin; u0 < u_end && ok;) {
            const ConvSeg sg = conv_segment(u0, u_end, H, TPR);
            for (int i = 0; i < sg.len && ok; ++i, ++gn) {
                for (int j = (i == 0 ? 0 : 2); j < 3; ++j) {
                    const long long r = gx + i + j;
                    if (!tc::mbar_wait(&xf_bar[r % NSX], uint32_t((r / NSX) & 1), CONV_WAIT_TRIES)) ok = false;
                }
                if (!tc::mbar_wait(&gf_bar[gn % NSG], uint32_t((gn / NSG) & 1), CONV_WAIT_TRIES)) ok = false;
                if (!ok) break;
                // as in conv3x3_tc_kernel: rows copied by cp.async, before the tensor cores read them
                if constexpr (!(SWX && SWG)) tc::fence_proxy_async();
                tc::fence_after_sync();
                const uint32_t s0 = uint32_t((gx + i) % NSX), s2 = uint32_t((gx + i + 2) % NSX);
                const uint32_t g_lo = b_lo0 + uint32_t(gn % NSG) * (L::GSLOT >> 4);
                const uint32_t a0_lo = a_lo0 + s0 * (L::XSLOT >> 4), a1_lo = a_lo0 + s2 * (L::XSLOT >> 4);
                const uint32_t acc0 = first ? 0u : 1u;
#pragma unroll
                for (int kk = 0; kk < 8; ++kk) {
                    const uint32_t acc = kk == 0 ? acc0 : 1u;
                    tc::mma_bf16_leader(leader, tmem, a0_lo + A_K * kk, a_hi, g_lo + B_K * kk, b_hi, IDESC, acc);
                    tc::mma_bf16_leader(leader, tmem + 3 * NT, a1_lo + A_K * kk, a_hi, g_lo + B_K * kk, b_hi, IDESC, acc);
                }
                tc::mma_commit_leader(leader, &ge_bar[gn % NSG]);
                tc::mma_commit_leader(leader, &xe_bar[(gx + i) % NSX]);
                if (i == sg.len - 1) {
                    tc::mma_commit_leader(leader, &xe_bar[(gx + i + 1) % NSX]);
                    tc::mma_commit_leader(leader, &xe_bar[(gx + i + 2) % NSX]);
                }
                first = false;
            }
            gx += sg.len + 2;
            u0 += sg.len;
        }
        tc::mma_commit_leader(leader, &done_bar);
        if (!ok && lane == 0) atomicExch(a.error, 1);
    }
    if (warp < WG_SUM_WARPS) {
        // bias gradient: the column sums of g, from the staged rows, while the
        // tensor cores work. Lane = pixel (32 of the row's 128 per warp); its sums
        // of all NT channels stay in registers until the CTA's rows are done.
        float sum[NT];
#pragma unroll
        for (int k = 0; k < NT; ++k) sum[k] = 0.0f;
        const long long rows = u_end - u_begin;
        bool ok = true;
        for (long long r = 0; r < rows; ++r) {
            const int slot = int(r % NSG);
            if (!tc::mbar_wait(&gf_bar[slot], uint32_t((r / NSG) & 1), CONV_WAIT_TRIES)) {
                ok = false;
                break;
            }
            const int px = 32 * warp + lane;
            const uint8_t *const line = Gs + slot * L::GSLOT + (px + 1) * 128;
            const uint32_t swz = (tc::smem_addr(line) >> 7) & 7;
#pragma unroll
            for (int c = 0; c < NT / 8; ++c) {
                const uint4 v = *reinterpret_cast<const uint4 *>(
                    SWG ? line + ((c ^ swz) << 4) : Gs + slot * L::GSLOT + ((CCT + c) * 128 + px) * 16);
                const uint32_t vv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    f2_get(f2_add(f2(sum[8 * c + 2 * k], sum[8 * c + 2 * k + 1]),
                                  f2(__uint_as_float(vv[k] << 16), __uint_as_float(vv[k] & 0xffff0000u))),
                           sum[8 * c + 2 * k], sum[8 * c + 2 * k + 1]);
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&ge_bar[slot]);
        }
        if (!ok && lane == 0) atomicExch(a.error, 1);
#pragma unroll
        for (int k = 0; k < NT; ++k) {
            float v = sum[k];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if (lane == k % 32) bias_s[warp][k] = v;
        }
    }
    if (warp < CONV_EPI_WARPS) {
        // epilogue: partial sums of this CTA
        const bool ok = tc::mbar_wait(&done_bar, 0u, CONV_WAIT_TRIES);
        if (!ok && lane == 0) atomicExch(a.error, 1);
        tc::fence_after_sync();
        const int q = warp & 3, half = warp >> 2;
        const int m = 32 * q + lane;
        const int c = m & 63;
        float *part = a.part + (size_t)blockIdx.x * 9 * NT * 64;
        if (ok && (NT == 64 || half == 0)) {
            for (int pr = 0; pr < 2; ++pr) {
                const int ky = 2 * pr + (m >> 6);
                for (int kx = 0; kx < 3; ++kx) {
                    float v[32];
                    if (NT == 64) {
                        tc::tmem_ld32(tmem + (pr * 3 + kx) * NT + 32 * half + (uint32_t(32 * q) << 16), v);
                        if (ky <= 2) {
                            float *o = part + ((size_t)(ky * 3 + 2 - kx) * NT + 32 * half) * 64 + c;
#pragma unroll
                            for (int k = 0; k < 32; ++k) o[k * 64] = v[k];
                        }
                    } else {
                        tc::tmem_ld32(tmem + (pr * 3 + kx) * NT + (uint32_t(32 * q) << 16), v);  // 16 used
                        if (ky <= 2) {
                            float *o = part + ((size_t)(ky * 3 + 2 - kx) * NT) * 64 + c;
#pragma unroll
                            for (int k = 0; k < 16; ++k) o[k * 64] = v[k];
                        }
                    }
                }
            }
        }
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    if (tid < NT) {
        float v = bias_s[0][tid];
        for (int w = 1; w < WG_SUM_WARPS; ++w) v += bias_s[w][tid];
        a.bpart[(size_t)blockIdx.x * NT + tid] = v;
    }
    if (warp == CONV_MMA_WARP) tc::tmem_dealloc(tmem, L::TMEM_COLS);
}

template <int CS, int NT>
cudaError_t launch_wgrad_t(const WgradArgs &a, int grid, cudaStream_t st) {
    using L = WgradLayout<CS, NT>;
    cudaError_t e = cudaFuncSetAttribute(wgrad_tc_kernel<CS, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         L::SMEM);
    if (e != cudaSuccess) return e;
    WgradMaps maps;
    memset(&maps, 0, sizeof(maps));
    const long long rows = (long long)a.nimg * a.H;
    if (L::SWX && (e = pixel_map(&maps.x128, a.x, a.W, rows, 128)) != cudaSuccess) return e;
    if (L::SWG && (e = pixel_map(&maps.g128, a.g, a.W, rows, 128)) != cudaSuccess) return e;
    if (L::SWG && (e = pixel_map(&maps.g1, a.g, a.W, rows, 1)) != cudaSuccess) return e;
    wgrad_tc_kernel<CS, NT><<<grid, CONV_THREADS, L::SMEM, st>>>(a, maps);
    return cudaGetLastError();
}

int wgrad_grid(const WgradArgs &a) {
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const long long rows = (long long)a.nimg * a.H * (a.W / 128);
    return rows < sms ? int(rows) : sms;
}

cudaError_t launch_wgrad_tc(const WgradArgs &a, int *grid_out, cudaStream_t st) {
    const int grid = wgrad_grid(a);
    if (grid_out) *grid_out = grid;
    if (a.cs == 64 && a.nt == 64) return launch_wgrad_t<64, 64>(a, grid, st);
    if (a.cs == 16 && a.nt == 64) return launch_wgrad_t<16, 64>(a, grid, st);
    if (a.cs == 64 && a.nt == 16) return launch_wgrad_t<64, 16>(a, grid, st);
    return cudaErrorInvalidValue;
}

bool conv_supported(int cin, int nout) {
    return (cin == 16 && nout == 64) || (cin == 64 && nout == 64) || (cin == 64 && nout == 16);
}

cudaError_t launch_conv(int cin, int nout, const ConvArgs &a, cudaStream_t st) {
    const bool dg = a.epi == EPI_DGRAD;
    if (cin == 16 && nout == 64) return dg ? launch_conv_t<2, 64, true>(a, st) : launch_conv_t<2, 64, false>(a, st);
    if (cin == 64 && nout == 64) return dg ? launch_conv_t<8, 64, true>(a, st) : launch_conv_t<8, 64, false>(a, st);
    if (cin == 64 && nout == 16) return dg ? launch_conv_t<8, 16, true>(a, st) : launch_conv_t<8, 16, false>(a, st);
    return cudaErrorInvalidValue;
}

}  // namespace qla

extern "C" qla_status qla_conv3x3_bf16(const void *x, int nimg, int H, int W, int cin, const void *w_packed,
                                       const float *bias, int nout, int epilogue, const void *aux0, const void *zprev,
                                       void *out0, void *out1, float scale, int *error_flag, void *stream) {
    if (!x || !w_packed || !error_flag || nimg < 1 || H < 1 || W < 128 || W % 128 != 0) return QLA_EINVAL;
    if ((long long)nimg * H * W > (1LL << 31) - 1) return QLA_EINVAL;
    if (!qla::conv_supported(cin, nout)) return QLA_EUNSUPPORTED;
    if (epilogue < 0 || epilogue > 3) return QLA_EINVAL;
    if (epilogue != qla::EPI_GELU && !out0) return QLA_EINVAL;
    if ((epilogue == qla::EPI_GELU || epilogue == qla::EPI_DGRAD) && !out1) return QLA_EINVAL;
    if (epilogue == qla::EPI_DGRAD && !zprev) return QLA_EINVAL;
    if (epilogue == qla::EPI_QUPDATE && (!aux0 || nout < 6)) return QLA_EINVAL;
    qla::ConvArgs a;
    a.x = x;
    a.w = w_packed;
    a.bias = bias;
    a.nimg = nimg;
    a.H = H;
    a.W = W;
    a.epi = epilogue;
    a.aux0 = aux0;
    a.zprev = zprev;
    a.out0 = out0;
    a.out1 = out1;
    a.scale = scale;
    a.error = error_flag;
    a.tiled = 0;
    const cudaError_t e = qla::launch_conv(cin, nout, a, static_cast<cudaStream_t>(stream));
    return e == cudaSuccess ? QLA_OK : QLA_ECUDA;
}

namespace qla {

__global__ void pack_conv_weights_kernel(const float *__restrict__ w, int nout, int cin, int nout_pad, int cin_pad,
                                         int mode, __nv_bfloat16 *__restrict__ out) {
    pack_conv_weights_elements(w, nout, cin, nout_pad, cin_pad, mode, out);
}

cudaError_t launch_pack_weights(const float *w, int nout, int cin, int nout_pad, int cin_pad, int mode,
                                void *packed, cudaStream_t st) {
    const int total = 9 * cin_pad * nout_pad;
    pack_conv_weights_kernel<<<(total + 255) / 256, 256, 0, st>>>(w, nout, cin, nout_pad, cin_pad, mode,
                                                                  static_cast<__nv_bfloat16 *>(packed));
    return cudaGetLastError();
}

}  // namespace qla

extern "C" qla_status qla_pack_conv_weights(const float *w, int nout, int cin, int nout_pad, int cin_pad,
                                            int transpose_flip, void *packed, void *stream) {
    if (!w || !packed || nout < 1 || cin < 1 || cin_pad % 8 != 0 || nout_pad % 8 != 0) return QLA_EINVAL;
    if (!transpose_flip && (nout > nout_pad || cin > cin_pad)) return QLA_EINVAL;
    if (transpose_flip && (cin > nout_pad || nout > cin_pad)) return QLA_EINVAL;
    const cudaError_t e = qla::launch_pack_weights(w, nout, cin, nout_pad, cin_pad,
                                                   transpose_flip ? qla::PACK_ADJOINT : qla::PACK_PLAIN, packed,
                                                   static_cast<cudaStream_t>(stream));
    return e == cudaSuccess ? QLA_OK : QLA_ECUDA;
}

namespace qla {
namespace {

// Host-side walk of one CTA's MMA warp (the same helpers the kernel calls).
template <int CCH, int NOUT>
long long conv_schedule_t(int nimg, int H, int W, int grid, int cta, int *rec, long long cap) {
    using L = ConvLayout<CCH, NOUT>;
    constexpr int NB = L::NB, NS = L::NS, HP = L::HALO_PX;
    const int TPR = W / 128;
    const long long T = (long long)nimg * TPR * H;
    const long long u_begin = T * cta / grid, u_end = T * (cta + 1) / grid;
    long long n = 0;
    auto put = [&](int type, long long r, long long on, int j, int len, int a, int b, int c, int d, int e, int f,
                   uint32_t g, uint32_t h) {
        if (n < cap) {
            int *p = rec + n * QLA_CONV_SCHEDULE_FIELDS;
            const int v[QLA_CONV_SCHEDULE_FIELDS] = {type, int(r), int(on), j, len, a, b, c, d, e, f, int(g), int(h), 0};
            for (int k = 0; k < QLA_CONV_SCHEDULE_FIELDS; ++k) p[k] = v[k];
        }
        ++n;
    };
    conv_walk_rows(u_begin, u_end, H, TPR, [&](const ConvSeg &sg, int j, long long r, long long on) {
        const int b0 = conv_block(on, NB);
        uint32_t par = 0;
        if (conv_row_acc_wait(j, sg.len, on, NB, &par)) put(2, r, on, j, sg.len, b0, int(par), 0, 0, 0, 0, 0, 0);
        conv_row_mmas<CCH, NOUT, NS, HP>(j, sg.len, b0, [&](const ConvMma &m) {
            put(0, r, on, j, sg.len, m.kx, m.k2, m.ka, m.kb, m.blk, m.acc, m.a_off, m.b_off);
        });
        put(3, r, on, j, sg.len, int(r % NS), 0, 0, 0, 0, 0, 0, 0);
        const int bd = conv_row_done_block(j, on, NB);
        if (bd >= 0) put(1, r, on, j, sg.len, bd, 0, 0, 0, 0, 0, 0, 0);
        return true;
    });
    return n;
}

}  // namespace
}  // namespace qla

extern "C" qla_status qla_conv_schedule(int cin, int nout, int nimg, int H, int W, int grid, int cta, int *records,
                                        long long capacity, long long *count) {
    if (!count || nimg < 1 || H < 1 || W < 128 || W % 128 != 0 || grid < 1 || cta < 0 || cta >= grid ||
        capacity < 0 || (capacity > 0 && !records) || (long long)nimg * H * (W / 128) > (1LL << 30))
        return QLA_EINVAL;
    long long n;
    if (cin == 16 && nout == 64) n = qla::conv_schedule_t<2, 64>(nimg, H, W, grid, cta, records, capacity);
    else if (cin == 64 && nout == 64) n = qla::conv_schedule_t<8, 64>(nimg, H, W, grid, cta, records, capacity);
    else if (cin == 64 && nout == 16) n = qla::conv_schedule_t<8, 16>(nimg, H, W, grid, cta, records, capacity);
    else return QLA_EUNSUPPORTED;
    *count = n;
    return QLA_OK;
}
