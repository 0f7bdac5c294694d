// Forward convolutions of the warm-start network on the 5th-generation tensor cores
// (tcgen05.mma, accumulators in tensor memory), fed by TMA.
//
// A convolution out[p][co] = sum_{t, ci} in[p + d_t][ci] w[co][t][ci] is an implicit GEMM with
// M = pixels, N = output channels, K = taps x input channels.  A block computes tiles of
// 16 x 8 output pixels (M = 128, GEMM row m = 8 y + x) times N output channels:
//
//   * the input tile plus a one-pixel halo (3x3 taps), 18 x 10 pixels, is loaded by TMA once per
//     block of CB = 32 or 16 input channels, as rows of one pixel's channels swizzled over 64 or 32
//     bytes (zero fill outside the image is the convolution's zero padding).  Every tap (dy, dx) is
//     then the same shared-memory matrix at another start address, (dy + 1) * 10 + (dx + 1) pixels
//     on: the swizzle is a function of the address, so it follows.  No input pixel is copied more
//     than once per channel block.  (Unswizzled, the operand's core matrices are 16 bytes wide, the
//     copies had rows of 16 bytes and a pixel's channel block took two of them.)
//   * the weights of that channel block are a prepacked [tap][8-channel half][N][8] BF16 slab
//     (one bulk copy), the K-major canonical layout of the MMA's B operand.
//   * one MMA per tap (K = 16) accumulates into one of two TMEM accumulators of N FP32
//     columns, so the epilogue of one tile overlaps the MMAs of the next.
//
// Warp roles (192 threads): warp 4 issues the TMA copies into an S-stage mbarrier ring, one
// thread of warp 5 issues the MMAs and their commits, warps 0-3 (one TMEM lane quarter each)
// read the accumulators back (tcgen05.ld), add the bias, apply the activation and store BF16
// NHWC.  Optional fused epilogues: 2x2 average pooling, nearest upsampling plus a skip tensor
// (the decoder's 1x1 reductions), and the 1x1 FP32 head.  Every mbarrier wait is bounded; a
// wait that runs out raises the error flag and the block finishes without further copies.
//
// The weight gradient of training, dw[co][t][ci] = sum_p g[p][co] in[p + d_t][ci], is a GEMM
// with M = output channels, N = input channels and K = pixels, per tap (k_tc_wgrad).  Both
// operands come straight from the NHWC tensors as MN-major matrices: a pixel's 32 channels are 64
// contiguous bytes, a row of a swizzle atom, and a tile of pixels is loaded by one 5-D TMA copy per
// operand (channel in block, x, y, image, channel block) with zero fill outside the image for the tap
// shift.  One accumulator of N FP32 columns per tap and block covers a chunk of pixel tiles; the
// epilogue writes it to a partial-sum buffer that a second kernel reduces in a fixed order.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <stdint.h>

#include "gabp_nn.h"
#include "gabp_per_device.h"

namespace gabp {
namespace nn {

namespace {

constexpr int TC_THREADS = 192;
constexpr int TILE_Y = 16, TILE_X = 8;          // output pixels per tile (M = 128)
// the staged input of T taps and CB channels: pixels, bytes copied, stage bytes (a multiple of 1024,
// so that every stage starts a swizzle pattern)
template <int T, int CB> struct InTile {
    static constexpr int X = TILE_X + (T == 9 ? 2 : 0), Y = TILE_Y + (T == 9 ? 2 : 0);
    static constexpr uint32_t ROW = CB * 2, BYTES = X * Y * ROW, PITCH = (BYTES + 1023) & ~1023u;
};

__device__ __forceinline__ uint32_t saddr(const void *p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// bounded wait for the phase with the given parity; false if it did not complete in time
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
    const long long t0 = clock64();
    for (;;) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(bar), "r"(parity)
            : "memory");
        if (ok) return true;
        if (clock64() - t0 > (1LL << 32)) return false;
    }
}

__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap *map, int c0, int c1, int c2, int c3,
                                            uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(bar)
        : "memory");
}
__device__ __forceinline__ void bulk_load(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}

// Shared-memory matrix descriptor of tcgen05 (no swizzle, K-major canonical layout): start
// address, leading-dimension byte offset (between the 8-element K chunks), stride byte offset
// (between 8-row groups), descriptor version 1.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
    return (uint64_t)((addr & 0x3FFFF) >> 4) | ((uint64_t)((lbo >> 4) & 0x3FFF) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFF) << 32) | ((uint64_t)1 << 46);
}
// the same with a 64-byte (CB = 32) or 32-byte (CB = 16) swizzle
template <int CB> __device__ __forceinline__ uint64_t smem_desc_sw(uint32_t addr, uint32_t lbo, uint32_t sbo) {
    return smem_desc(addr, lbo, sbo) | ((uint64_t)(CB == 32 ? 4 : 6) << 61);
}
__device__ __forceinline__ void tma_load_5d(uint32_t dst, const CUtensorMap *map, int c0, int c1, int c2, int c3, int c4,
                                            uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.5d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4, %5, %6}], [%7];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4), "r"(bar)
        : "memory");
}

// Instruction descriptor, kind::f16: D FP32, A and B BF16, both MN-major (transpose bits 15
// and 16), M = 64 or 128, N.
__device__ __forceinline__ uint32_t instr_desc_mn(int M, int N) {
    return (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) | ((uint32_t)(N >> 3) << 17) |
           ((uint32_t)(M >> 4) << 24);
}

// Instruction descriptor, kind::f16: D FP32, A and B BF16, both K-major, M = 128, N.
template <int N> __device__ __forceinline__ uint32_t instr_desc() {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
}

__device__ __forceinline__ void umma(uint32_t tmem_d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
        "l"(a), "l"(b), "r"(idesc), "r"(acc)
        : "memory");
}
// One lane of the (converged) warp.  The MMA loops run on the whole warp with warp-uniform
// descriptors and only the instruction itself on the elected lane: issued from a loop of one
// divergent lane, with the descriptors formed per MMA, an MMA takes 71 cycles however small it is;
// this way 40 (M = 128, N = 32: the shared-memory reads of its operands) to 128 (N = 256).
__device__ __forceinline__ bool elect_lane() {
    uint32_t e;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(e));
    return e != 0;
}
__device__ __forceinline__ void umma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// BF16 pairs in one register (low half first)
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    const __nv_bfloat162 p = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t *>(&p);
}
__device__ __forceinline__ float bf_lo(uint32_t v) { return __uint_as_float(v << 16); }
__device__ __forceinline__ float bf_hi(uint32_t v) { return __uint_as_float(v & 0xffff0000u); }
__device__ __forceinline__ uint32_t relu_bf16(uint32_t v) {   // max(., 0); rounding and max commute
    const __nv_bfloat162 m = __hmax2(*reinterpret_cast<const __nv_bfloat162 *>(&v), __nv_bfloat162(__float2bfloat16(0.f), __float2bfloat16(0.f)));
    return *reinterpret_cast<const uint32_t *>(&m);
}
__device__ __forceinline__ uint32_t positive_mask(uint32_t v) {   // all ones in the halves above zero
    return __hgt2_mask(*reinterpret_cast<const __nv_bfloat162 *>(&v), __nv_bfloat162(__float2bfloat16(0.f), __float2bfloat16(0.f)));
}
// 16 channels of a pixel (32 bytes, aligned) in one 256-bit access: a whole sector per lane (two
// 128-bit stores made two partial writes of each: 85 -> 72 us for 32 x 32 x 9 over 2.1 M pixels,
// 112 -> 98 us with the loads too for 64 x 32 x 1 with upsampling, 0.5 M to 2.1 M)
__device__ __forceinline__ void store16_bf16(__nv_bfloat16 *dst, const uint32_t (&v)[8]) {
    asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(dst), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]),
                 "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
                 : "memory");
}
__device__ __forceinline__ void load16_bf16(const __nv_bfloat16 *src, uint32_t (&v)[8]) {
    asm volatile("ld.global.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
                 : "l"(src));
}
template <int N, int T, int CB>
__global__ void __launch_bounds__(TC_THREADS, 4) k_tc_conv(const __grid_constant__ CUtensorMap in_map, TcConvArgs a) {
    using IN = InTile<T, CB>;
    constexpr bool UP = T == 1;   // the epilogues: 1x1 convolutions may upsample, 3x3 ones may pool or have the head
    constexpr uint32_t WBYTES = (uint32_t)T * 2 * CB * N;      // weight slab of one channel block
    extern __shared__ __align__(1024) unsigned char smem[];
    const int S = a.stages;
    const int nkb = a.Cin / CB;
    // resident weights: all nkb slabs stay in shared memory and the ring carries halos only;
    // otherwise every stage carries a halo and its weight slab
    const bool resident = a.resident != 0;
    const uint32_t wres = resident ? (uint32_t)nkb * WBYTES : 0u;   // resident weight bytes
    const uint32_t STAGE = resident ? IN::PITCH : IN::PITCH + WBYTES;   // multiples of 1024
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + wres + (size_t)S * STAGE);
    // full[S], empty[S], acc_full[2], acc_empty[2], weights
    uint32_t *tslot = reinterpret_cast<uint32_t *>(bars + 2 * S + 5);
    volatile int *fail = reinterpret_cast<volatile int *>(tslot + 1);
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const uint32_t sbase = saddr(smem);
    auto full = [&](int s) { return saddr(&bars[s]); };
    auto empty = [&](int s) { return saddr(&bars[S + s]); };
    auto accf = [&](int i) { return saddr(&bars[2 * S + i]); };
    auto acce = [&](int i) { return saddr(&bars[2 * S + 2 + i]); };
    const uint32_t wbar = saddr(&bars[2 * S + 4]);
    const uint32_t ring = sbase + wres;

    if (tid == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(full(s), 1);
            mbar_init(empty(s), 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(accf(i), 1);
            mbar_init(acce(i), 4);
        }
        mbar_init(wbar, 1);
        *fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(saddr(tslot)),
                     "r"(2 * N));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tslot;

    const int64_t ntiles = a.ntiles;
    auto tile_coords = [&](int64_t tile, int &b, int &y0, int &x0, int &nb) {
        uint32_t r = (uint32_t)tile / (uint32_t)a.nblocks;   // fewer than 2^31 tiles (checked on the host)
        nb = (int)((uint32_t)tile - r * (uint32_t)a.nblocks);
        const uint32_t q = r / (uint32_t)a.tiles_x;
        const int tx = (int)(r - q * (uint32_t)a.tiles_x);
        b = (int)(q / (uint32_t)a.tiles_y);
        const int ty = (int)(q - (uint32_t)b * (uint32_t)a.tiles_y);
        y0 = ty * TILE_Y;
        x0 = tx * TILE_X;
    };

    if (warp == 4) {
        // ---- TMA producer ----
        if (lane == 0) {
            if (resident) {   // one output-channel block: load all its weight slabs once
                mbar_expect_tx(wbar, wres);
                for (int kb = 0; kb < nkb; ++kb)
                    bulk_load(sbase + (uint32_t)kb * WBYTES, a.wpk + (int64_t)kb * (WBYTES / 2), WBYTES, wbar);
            }
            int64_t it = 0;
            for (int64_t tile = blockIdx.x; tile < ntiles && !*fail; tile += gridDim.x) {
                int b, y0, x0, nb;
                tile_coords(tile, b, y0, x0, nb);
                for (int kb = 0; kb < nkb; ++kb, ++it) {
                    const int s = (int)(it % S);
                    const uint32_t use = (uint32_t)(it / S);
                    if (!mbar_wait(empty(s), (use & 1) ^ 1)) {
                        *fail = 1;
                        break;
                    }
                    const uint32_t st = ring + (uint32_t)s * STAGE;
                    mbar_expect_tx(full(s), IN::BYTES + (resident ? 0u : WBYTES));
                    tma_load_4d(st, &in_map, CB * kb, x0 - (T == 9), y0 - (T == 9), b, full(s));
                    if (!resident)
                        bulk_load(st + IN::PITCH, a.wpk + ((int64_t)nb * nkb + kb) * (WBYTES / 2), WBYTES, full(s));
                }
            }
        }
    } else if (warp == 5) {
        // ---- MMA issuer ----
        const uint32_t idesc = instr_desc<N>();
        const bool one = elect_lane();
        const uint64_t ad0 = smem_desc_sw<CB>(0, 16, IN::X * IN::ROW), bd0 = smem_desc(0, N * 16, 128);
        uint32_t it = 0;
        int lt = 0;
        bool ok = !resident || mbar_wait(wbar, 0);
        if (__any_sync(0xffffffffu, !ok)) *fail = 1;
        __syncwarp();
        for (int64_t tile = blockIdx.x; tile < ntiles && !*fail; tile += gridDim.x, ++lt) {
            const int acc = lt & 1;
            ok = mbar_wait(acce(acc), (((uint32_t)lt >> 1) & 1) ^ 1);
            if (__any_sync(0xffffffffu, !ok)) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t d = tmem + (uint32_t)(acc * N);
            int kb = 0;
            for (; kb < nkb; ++kb, ++it) {
                const uint32_t s = it % (uint32_t)S;
                ok = mbar_wait(full(s), (it / (uint32_t)S) & 1);
                if (__any_sync(0xffffffffu, !ok)) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t st = ring + s * STAGE;
                const uint64_t ad = ad0 + (st >> 4), bd = bd0 + ((resident ? sbase + (uint32_t)kb * WBYTES : st + IN::PITCH) >> 4);
                if (one) {
#pragma unroll
                    for (int j = 0; j < CB / 16; ++j)   // 16 channels: one MMA per tap
#pragma unroll
                        for (int t = 0; t < T; ++t)
                            umma(d, ad + (uint64_t)((t / 3 * IN::X + t % 3) * (int)(IN::ROW / 16) + 2 * j),
                                 bd + (uint64_t)((j * T + t) * 2 * N), idesc, (kb > 0 || j > 0 || t > 0) ? 1u : 0u);
                    umma_commit(empty(s));   // the stage is free once these MMAs have read it
                }
                __syncwarp();
            }
            if (kb < nkb) break;   // a wait ran out
            if (one) umma_commit(accf(acc));   // accumulator complete
            __syncwarp();
        }
        if (__any_sync(0xffffffffu, !ok)) *fail = 1;
    } else {
        // ---- epilogue: warps 0-3, TMEM lanes 32 w .. 32 w + 31 = tile pixels ----
        const int m = 32 * warp + lane;
        const int yy = m >> 3, xx = m & 7;
        int lt = 0;
        for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ++lt) {
            const int acc = lt & 1;
            int b, y0, x0, nb;
            tile_coords(tile, b, y0, x0, nb);
            const int gy = y0 + yy, gx = x0 + xx;
            const bool valid = gy < a.H && gx < a.W;
            const int co0 = nb * N;
            const int64_t pix = ((int64_t)b * a.H + gy) * a.W + gx;
            auto fine = [&](int q) {   // pixel q of the 2 x 2 above this one on the twice as fine grid
                return (((int64_t)b * (2 * a.H) + 2 * gy + (q >> 1)) * (2 * a.W) + 2 * gx + (q & 1)) * a.Cout;
            };
            // what the epilogue reads, towards L2 while the accumulator is made (a tile earlier, by the
            // producer, 80 MB in flight ran each other out of L2: the skip tensor was read twice)
            if (UP && a.up_out && valid)
#pragma unroll
                for (int q = 0; q < 4; q += N == 32 ? 2 : 1)
#pragma unroll
                    for (int c = 0; c < N; c += 64) asm volatile("prefetch.global.L2 [%0];" ::"l"(a.up_skip + fine(q) + co0 + c));
            if (a.mask && valid)
#pragma unroll
                for (int c = 0; c < N; c += 64) asm volatile("prefetch.global.L2 [%0];" ::"l"(a.mask + pix * a.Cout + co0 + c));
            const bool ok = mbar_wait(accf(acc), ((uint32_t)lt >> 1) & 1);
            if (!ok) *fail = 1;
            if (__any_sync(0xffffffffu, !ok) || *fail) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            float h0 = 0.f, h1 = 0.f;
            if (!UP && a.head_w) {
                h0 = a.head_b[0];
                h1 = a.head_b[1];
            }
#pragma unroll 1
            for (int c = 0; c < N; c += 16) {
                uint32_t r[16], v[8];   // 16 channels: FP32 sums, BF16 pairs
                // the mask and the skip tensor first: all their loads in flight at once
                uint32_t mk[8], sv[4][8];
                if (a.mask && valid) load16_bf16(a.mask + pix * a.Cout + co0 + c, mk);
                if (UP && a.up_out && valid)
#pragma unroll
                    for (int q = 0; q < 4; ++q) load16_bf16(a.up_skip + fine(q) + co0 + c, sv[q]);
                tmem_ld16(tmem + ((uint32_t)(32 * warp) << 16) + (uint32_t)(acc * N + c), r);
                const float4 *bias4 = reinterpret_cast<const float4 *>(a.bias + co0 + c);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float4 bv = bias4[j];
                    v[2 * j] = pack_bf16(__uint_as_float(r[4 * j]) + bv.x, __uint_as_float(r[4 * j + 1]) + bv.y);
                    v[2 * j + 1] = pack_bf16(__uint_as_float(r[4 * j + 2]) + bv.z, __uint_as_float(r[4 * j + 3]) + bv.w);
                }
                if (a.relu)
#pragma unroll
                    for (int j = 0; j < 8; ++j) v[j] = relu_bf16(v[j]);
                if (a.mask && valid)   // the ReLU's backward: zero where its output was not positive
#pragma unroll
                    for (int j = 0; j < 8; ++j) v[j] &= positive_mask(mk[j]);
                if (a.out && valid) store16_bf16(a.out + pix * a.Cout + co0 + c, v);
                if (!UP && a.pool_out) {
                    // 2x2 sum, scaled: (y, x), (y, x+1), (y+1, x), (y+1, x+1) are lanes +0, +1, +8, +9
                    uint32_t pv[8];
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const uint32_t v1 = __shfl_down_sync(0xffffffffu, v[j], 1), v8 = __shfl_down_sync(0xffffffffu, v[j], 8);
                        const uint32_t v9 = __shfl_down_sync(0xffffffffu, v[j], 9);
                        pv[j] = pack_bf16(a.pool_scale * (((bf_lo(v[j]) + bf_lo(v1)) + bf_lo(v8)) + bf_lo(v9)),
                                          a.pool_scale * (((bf_hi(v[j]) + bf_hi(v1)) + bf_hi(v8)) + bf_hi(v9)));
                    }
                    if (valid && !(xx & 1) && !(yy & 1)) {
                        const int64_t q = ((int64_t)b * (a.H / 2) + gy / 2) * (a.W / 2) + gx / 2;
                        store16_bf16(a.pool_out + q * a.Cout + co0 + c, pv);
                    }
                }
                if (UP && a.up_out && valid) {
                    // nearest upsampling to (2H, 2W) plus the skip tensor there
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        uint32_t u[8];
#pragma unroll
                        for (int j = 0; j < 8; ++j)
                            u[j] = pack_bf16(bf_lo(v[j]) + bf_lo(sv[q][j]), bf_hi(v[j]) + bf_hi(sv[q][j]));
                        store16_bf16(a.up_out + fine(q) + co0 + c, u);
                    }
                }
                if (!UP && a.head_w) {
#pragma unroll
                    for (int j = 0; j < 16; ++j) {
                        const float f = j & 1 ? bf_hi(v[j >> 1]) : bf_lo(v[j >> 1]);
                        h0 = fmaf(a.head_w[c + j], f, h0);
                        h1 = fmaf(a.head_w[a.Cout + c + j], f, h1);
                    }
                }
            }
            if (!UP && a.head_w && valid) {
                a.head_out[2 * pix] = h0;
                a.head_out[2 * pix + 1] = h1;
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(acce(acc));
        }
    }

    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (*fail && tid == 0) atomicExch(a.err, 1);
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * N));
    }
}

// ---- weight gradient ----
constexpr int WG_THREADS = 192;
constexpr int WG_KX = 16;                               // pixels per tile row (one MMA, K = 16)

// bytes of a stage: the copied operands, and no less than an A operand of M rows reaches
__host__ __device__ inline uint32_t wg_stage_bytes(int M, int ga, int N, int ky, int h) {
    const uint32_t ag = (uint32_t)(WG_KX * ky) * 64;
    const uint32_t both = (uint32_t)ga * ag + (uint32_t)(N * (WG_KX + 2 * h) * (ky + 2 * h)) * 2;
    const uint32_t reach = (uint32_t)(M / 32) * ag;
    return ((both > reach ? both : reach) + 1023u) & ~1023u;
}
// the same with taps stacked: the input (and a pixel past it, which the fourth tap reaches), then g
__host__ __device__ inline uint32_t wg_stacked_x_bytes(int cin, int ky) {
    return ((uint32_t)((WG_KX + 2) * (ky + 2) + 1) * (uint32_t)cin * 2 + 1023u) & ~1023u;
}

// Block: a group of taps [t0, t0 + tpc), output-channel block mb (of M), input-channel block nb (N),
// pixel-tile chunk.  A tile is 16 x KY pixels.  Shared memory per stage, in blocks of 32 channels (the
// input's 16 where it has only 16) whose pixels are rows of 64 (32) bytes, swizzled:
//   A [channel block][KY][16]: g at the tile's pixels;
//   B [channel block][KY + 2 h][16 + 2 h]: the input at the tile's pixels plus a one-pixel halo (h = 1
//     for 3x3 taps), so that every tap (dy, dx) of a tile row is the same matrix at another start
//     address, (row + h + dy) (16 + 2 h) + h + dx pixels on (the swizzle is a function of the address).
// MN-major: 8 pixels x one channel block are a swizzle atom, the K-direction atoms follow each other
// (SBO), channel blocks are one block apart (LBO).  One MMA per tile row and tap accumulates into that
// tap's N TMEM columns.  With fewer output channels than M the A operand runs on into the stage's B:
// those accumulator rows are not read.  (As [8-channel group][pixel] tiles without a swizzle the copies
// had 16-byte rows, of which the TMA unit moves one per 2.4 cycles: 75 -> 42 us for 128 x 128 x 9 over
// 131 k pixels, 101 -> 54 us for 256 x 256 x 9 over 33 k.)
//
// STACK (3x3 taps of 16 or 32 input channels, at most 64 output channels): the operands exchange roles,
// and A is the input with the taps of a row as its channel blocks, one pixel apart: M = 4 blocks
// (dx = -1, 0, 1 and one that is not read) x Cin, N = Cout.  An MMA is bound by reading its operands
// from shared memory (M = 64, N = 32: 24 cycles; this one: 64) and does the work of three; all nine
// taps take 3 Cout TMEM columns, so no tile is loaded twice.  32 x 32 x 9 over 2.1 M pixels: 88 us (51 of
// them by the operand reads alone; memory: 40), and a training step's four layers of this kind 432 ->
// 259 us.  (Keeping g as A, M = 64, and three taps in N = 96: 313.)
template <bool STACK>
__global__ void __launch_bounds__(WG_THREADS) k_tc_wgrad(const __grid_constant__ CUtensorMap gmap,
                                                         const __grid_constant__ CUtensorMap xmap, TcWgradArgs a) {
    extern __shared__ __align__(1024) unsigned char smem[];
    const int S = a.stages, N = a.N, KY = a.ky, h = a.T == 9 ? 1 : 0;
    const int HX = WG_KX + 2 * h, HY = KY + 2 * h;
    const uint32_t AROW = 64, BROW = (uint32_t)a.cbx * 2;   // bytes of a pixel's channel block
    const uint32_t AG = (uint32_t)(WG_KX * KY) * AROW, BG = (uint32_t)(HX * HY) * BROW;
    const int NBX = STACK ? 1 : N / a.cbx;
    const uint32_t ABYTES = (uint32_t)a.ga * AG;
    const uint32_t GOFF = STACK ? (uint32_t)a.xbytes : 0, XOFF = STACK ? 0 : ABYTES;   // g and the input in a stage
    const uint32_t STAGE = (uint32_t)a.stage;
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + (size_t)S * STAGE);   // full[S], empty[S], acc
    uint32_t *tslot = reinterpret_cast<uint32_t *>(bars + 2 * S + 1);
    volatile int *fail = reinterpret_cast<volatile int *>(tslot + 1);
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const uint32_t sbase = saddr(smem);
    auto full = [&](int s) { return saddr(&bars[s]); };
    auto empty = [&](int s) { return saddr(&bars[S + s]); };
    const uint32_t accb = saddr(&bars[2 * S]);
    const uint32_t need = (uint32_t)((STACK ? 3 : a.tpc) * N);
    const uint32_t tcols = need <= 32 ? 32u : (need <= 64 ? 64u : (need <= 128 ? 128u : (need <= 256 ? 256u : 512u)));

    // block -> (chunk, tap group, mb, nb)
    int64_t r = blockIdx.x;
    const int nb = (int)(r % a.nbn);
    r /= a.nbn;
    const int mb = (int)(r % a.nbm);
    r /= a.nbm;
    const int tg = (int)(r % a.ngroups);
    const int chunk = (int)(r / a.ngroups);
    const int t0 = tg * a.tpc;
    const int ntap = a.T - t0 < a.tpc ? a.T - t0 : a.tpc;
    const int64_t kt0 = (int64_t)chunk * a.per_chunk;
    const int64_t kt1 = kt0 + a.per_chunk < a.ktiles ? kt0 + a.per_chunk : a.ktiles;
    const int nk = (int)(kt1 > kt0 ? kt1 - kt0 : 0);
    const bool bias = tg == 0 && nb == 0;   // this block also sums g over its pixels

    if (tid == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(full(s), 1);
            mbar_init(empty(s), bias ? 5 : 1);   // the MMAs, and the four warps that sum the bias gradient
        }
        mbar_init(accb, 1);
        *fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(saddr(tslot)),
                     "r"(tcols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tslot;

    if (warp == 4) {
        // ---- TMA producer: tile k = (image, tile row, tile column) ----
        if (lane == 0) {
            for (int i = 0; i < nk && !*fail; ++i) {
                const int s = i % S;
                if (!mbar_wait(empty(s), ((uint32_t)(i / S) & 1) ^ 1)) {
                    *fail = 1;
                    break;
                }
                const int64_t k = kt0 + i;
                const int tx = (int)(k % a.tiles_x);
                const int64_t q = k / a.tiles_x;
                const int ty = (int)(q % a.tiles_y);
                const int b = (int)(q / a.tiles_y);
                const int x0 = tx * WG_KX, y0 = ty * KY;
                const uint32_t st = sbase + (uint32_t)s * STAGE;
                mbar_expect_tx(full(s), ABYTES + (uint32_t)NBX * BG);
                tma_load_5d(st + GOFF, &gmap, 0, x0, y0, b, (a.M / 32) * mb, full(s));
                tma_load_5d(st + XOFF, &xmap, 0, x0 - h, y0 - h, b, nb * NBX, full(s));
            }
        }
    } else if (warp == 5) {
        // ---- MMA issuer: one MMA (K = 16) per tile row and tap ----
        const uint32_t idesc = instr_desc_mn(a.M, N);
        const bool one = elect_lane();
        const uint32_t xg = STACK ? BROW : BG;   // between the input's blocks: one pixel, one channel block
        const uint64_t ad0 = smem_desc_sw<32>(0, AG, 8 * AROW);
        const uint64_t bd0 = a.cbx == 32 ? smem_desc_sw<32>(0, xg, 8 * BROW) : smem_desc_sw<16>(0, xg, 8 * BROW);
        const uint32_t bunit = BROW / 16;   // a pixel in descriptor units
        const uint64_t brow = (uint64_t)((uint32_t)HX * bunit);   // a row of the input tile
        bool ok = true;
        for (int i = 0; i < nk && !*fail; ++i) {
            const uint32_t s = (uint32_t)i % (uint32_t)S;
            ok = mbar_wait(full(s), ((uint32_t)i / (uint32_t)S) & 1);
            if (__any_sync(0xffffffffu, !ok)) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t st = sbase + s * STAGE;
            const uint64_t ad = ad0 + ((st + GOFF) >> 4), bd = bd0 + ((st + XOFF) >> 4);
            // loops and descriptors outside the elected lane's branch: inside it they would not be
            // computed in uniform registers (44 cycles per MMA against 27)
            for (int j = 0; !STACK && j < ntap; ++j) {
                const int t = t0 + j, dy = h ? t / 3 - 1 : 0, dx = h ? t % 3 - 1 : 0;
                uint64_t bt = bd + (uint64_t)((uint32_t)((h + dy) * HX + h + dx) * bunit), at = ad;
                const uint32_t d = tmem + (uint32_t)(j * N);
                for (int k4 = 0; k4 < KY; k4 += 4) {   // KY is 4 or 8
                    const uint64_t b1 = bt + brow, b2 = b1 + brow, b3 = b2 + brow;
                    const uint32_t first = i > 0 || k4 > 0 ? 1u : 0u;
                    if (one) {
                        umma(d, at, bt, idesc, first);
                        umma(d, at + WG_KX * 4, b1, idesc, 1u);
                        umma(d, at + 2 * WG_KX * 4, b2, idesc, 1u);
                        umma(d, at + 3 * WG_KX * 4, b3, idesc, 1u);
                    }
                    __syncwarp();
                    bt = b3 + brow;
                    at += 4 * WG_KX * 4;
                }
            }
            // (consecutive MMAs into different accumulators)
            if (STACK)
                for (int k = 0; k < KY; ++k) {
                    const uint64_t x0 = bd + (uint64_t)k * brow, x1 = x0 + brow, x2 = x1 + brow, g = ad + (uint64_t)(k * WG_KX * 4);
                    const uint32_t acc = i > 0 || k > 0 ? 1u : 0u;
                    if (one) {
                        umma(tmem, x0, g, idesc, acc);
                        umma(tmem + (uint32_t)N, x1, g, idesc, acc);
                        umma(tmem + (uint32_t)(2 * N), x2, g, idesc, acc);
                    }
                    __syncwarp();
                }
            if (one) {
                umma_commit(empty(s));   // the stage is free once these MMAs have read it
            }
            __syncwarp();
        }
        if (__any_sync(0xffffffffu, !ok)) *fail = 1;
        if (one) umma_commit(accb);   // also after a failure, so that the epilogue does not wait out
    } else {
        // ---- epilogue: warps 0-3.  M = 128: TMEM lane 32 w + lane = output channel 128 mb + 32 w +
        // lane; M = 64: the accumulator's rows 16 w .. 16 w + 15 are the first 16 lanes of warp w ----
        // The bias gradient first, from the staged g while the MMAs run: thread = 8 channels (16 bytes
        // of a pixel's row) of every R-th pixel.  (A kernel of its own read g once more: 290 us of a
        // training step of 8 512^2 grids, which took 3.13 ms; with this and one packing launch 2.74.)
        const int C8 = 4 * a.ga, R = 128 / C8, ch = tid % C8, pr = tid / C8;   // 4, 8 or 16 groups of channels
        float bs[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        if (bias)
            for (int i = 0; i < nk; ++i) {
                const int s = i % S;
                const bool got = mbar_wait(full(s), (uint32_t)(i / S) & 1);
                if (__any_sync(0xffffffffu, !got)) {
                    *fail = 1;
                    break;
                }
                const unsigned char *A = smem + (size_t)s * STAGE + GOFF + (size_t)(ch >> 2) * AG;
                for (int q = pr; q < WG_KX * KY; q += R) {
                    // the 64-byte swizzle: address bits 4, 5 exclusive-or bits 7, 8
                    const uint4 v = *reinterpret_cast<const uint4 *>(A + q * 64 + (((ch & 3) ^ ((q >> 1) & 3)) << 4));
                    const uint32_t w4[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        bs[2 * e] += bf_lo(w4[e]);
                        bs[2 * e + 1] += bf_hi(w4[e]);
                    }
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(empty(s));
            }
        const bool ok = mbar_wait(accb, 0);
        if (!ok) *fail = 1;
        // warp-uniform decision: tcgen05.ld is a whole-warp instruction
        const bool go = __all_sync(0xffffffffu, ok && !*fail);
        if (STACK && go) {
            // accumulator row = (tap of the row: this warp, input channel), column = output channel
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const bool mine = warp < 3 && lane < a.Cin;
#pragma unroll 1
            for (int j = 0; j < 3; ++j)
#pragma unroll 1
                for (int c = 0; c < N; c += 16) {
                    uint32_t v[16] = {};
                    if (nk > 0) tmem_ld16(tmem + ((uint32_t)(32 * warp) << 16) + (uint32_t)(j * N + c), v);
                    float *dst = a.part + (((int64_t)chunk * a.Cout + c) * 9 + 3 * j + warp) * a.Cin + lane;
                    if (mine) {
#pragma unroll
                        for (int e = 0; e < 16; ++e) dst[(int64_t)e * 9 * a.Cin] = __uint_as_float(v[e]);
                    }
                }
        }
        const int co = a.M == 128 ? 128 * mb + 32 * warp + lane : (lane < 16 ? 16 * warp + lane : a.Cout);
        if (!STACK && go && nk > 0) {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll 1
            for (int j = 0; j < ntap; ++j) {
                float *dst = a.part + (((int64_t)chunk * a.Cout + co) * a.T + t0 + j) * a.Cin + nb * N;
#pragma unroll 1
                for (int c = 0; c < N; c += 16) {
                    uint32_t v[16];
                    tmem_ld16(tmem + ((uint32_t)(32 * warp) << 16) + (uint32_t)(j * N + c), v);
                    if (co < a.Cout) {
#pragma unroll
                        for (int e = 0; e < 16; e += 4)
                            *reinterpret_cast<float4 *>(dst + c + e) =
                                make_float4(__uint_as_float(v[e]), __uint_as_float(v[e + 1]),
                                            __uint_as_float(v[e + 2]), __uint_as_float(v[e + 3]));
                    }
                }
            }
        } else if (!STACK && go && co < a.Cout) {   // an empty chunk: zero partial sums
            for (int j = 0; j < ntap; ++j) {
                float *dst = a.part + (((int64_t)chunk * a.Cout + co) * a.T + t0 + j) * a.Cin + nb * N;
                for (int c = 0; c < N; ++c) dst[c] = 0.f;
            }
        }
        if (bias) {   // the R pixel groups' sums in order; every MMA has read the stages
            float *sc = reinterpret_cast<float *>(smem);
            asm volatile("bar.sync 1, 128;" ::: "memory");   // and every warp of the sums
#pragma unroll
            for (int e = 0; e < 8; ++e) sc[pr * 32 * a.ga + 8 * ch + e] = bs[e];
            asm volatile("bar.sync 1, 128;" ::: "memory");
            const int c0 = STACK ? tid : a.M * mb + tid;
            if (tid < 32 * a.ga && c0 < a.Cout) {
                float t = 0.f;
                for (int q = 0; q < R; ++q) t += sc[q * 32 * a.ga + tid];
                a.part[(int64_t)a.chunks * a.Cout * a.T * a.Cin + (int64_t)chunk * a.Cout + c0] = t;
            }
        }
    }

    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (*fail && tid == 0) atomicExch(a.err, 1);
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(tcols));
    }
}

// Packed weights of every layer in one launch, layer l at the same offset as in w.  Forward:
// packed[nb][kb][t][h][n][e] = w[nb * N + n][t][16 kb + 8 h + e].  FLIP, the convolution of the input
// gradient: the same of the weights flipped in space with Cin and Cout exchanged.
template <bool FLIP> __global__ void k_tc_pack(const __nv_bfloat16 *w, TcPackLayers p, __nv_bfloat16 *out) {
    int l = 0;
    while (l + 1 < p.n && (int)blockIdx.x >= p.block0[l + 1]) ++l;
    const int T = p.taps[l], Cin = p.cin[l], Cout = p.cout[l];
    const int i = ((int)blockIdx.x - p.block0[l]) * 256 + (int)threadIdx.x;
    if (i >= Cout * T * Cin) return;
    const int K = FLIP ? Cout : Cin, R = FLIP ? Cin : Cout, N = R < 128 ? R : 128;   // contraction, rows, rows per block
    int r = i >> 3;
    const int n = r % N;
    r /= N;
    const int h = r & 1;
    r >>= 1;
    const int t = r % T;
    r /= T;
    const int kb = r % (K / 16), nb = r / (K / 16);
    const int row = nb * N + n, k = 16 * kb + 8 * h + (i & 7);
    out[p.off[l] + i] = w[p.off[l] + (FLIP ? ((int64_t)k * T + (T - 1 - t)) * Cin + row : ((int64_t)row * T + t) * Cin + k)];
}

PFN_cuTensorMapEncodeTiled_v12000 tc_encoder() {
    static std::atomic<PFN_cuTensorMapEncodeTiled_v12000> fn{nullptr};   // every thread finds the same
    if (!fn) {
        void *ptr = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &ptr, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (PFN_cuTensorMapEncodeTiled_v12000)ptr;
    }
    return fn;
}

// The epilogue warps bound these kernels, so shared memory is budgeted for the four blocks of 192 threads
// that an SM's registers hold.
constexpr uint32_t SMEM_PER_BLOCK = 55 * 1024;

// the weights of one output-channel block of N stay in shared memory
bool tc_resident(const TcConvArgs &a, int N) { return a.nblocks == 1 && a.Cin * a.T * 2 * N <= 48 * 1024; }

template <int N, int T, int CB>
cudaError_t tc_launch(const CUtensorMap &map, TcConvArgs a, cudaStream_t st) {
    using IN = InTile<T, CB>;
    struct Limits {
        int nsm, occ_threads;
    };
    static PerDevice<Limits> cache;
    const uint32_t wbytes = (uint32_t)T * 2 * CB * N;
    const uint32_t wall = (uint32_t)(a.Cin / CB) * wbytes;
    a.resident = tc_resident(a, N) ? 1 : 0;
    size_t smem;
    if (a.resident) {
        int S = ((int)SMEM_PER_BLOCK - (int)wall) / (int)IN::PITCH;
        a.stages = S < 2 ? 2 : (S > 8 ? 8 : S);
        smem = wall + (size_t)a.stages * IN::PITCH;
    } else {
        const uint32_t stage = IN::PITCH + wbytes;
        int S = (int)(SMEM_PER_BLOCK / stage);
        a.stages = S < 2 ? 2 : (S > 4 ? 4 : S);
        smem = (size_t)a.stages * stage;
    }
    smem += 8 * (2 * a.stages + 5) + 16;
    // blocks per SM: registers and threads (occupancy without shared memory), shared memory
    // (228 KB, 1 KB reserved per block) and tensor memory (512 columns, 2N per block); the
    // shared-memory request is raised so that the SM cannot host more blocks than its tensor
    // memory holds
    const int tmem_cap = 512 / (2 * N);
    const size_t smem_floor = (size_t)(227 * 1024) / (size_t)(tmem_cap + 1) + 1024;
    if (smem < smem_floor) smem = smem_floor;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    Limits lim{};
    e = cache.get(dev, lim, [&](Limits &v) {
        cudaError_t e = cudaFuncSetAttribute(k_tc_conv<N, T, CB>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
        if (e != cudaSuccess) return e;
        e = cudaDeviceGetAttribute(&v.nsm, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return e;
        // registers and threads per SM from the kernel's attributes
        cudaFuncAttributes fa;
        e = cudaFuncGetAttributes(&fa, k_tc_conv<N, T, CB>);
        if (e != cudaSuccess) return e;
        const int regs_warp = ((fa.numRegs * 32 + 255) / 256) * 256;
        v.occ_threads = 65536 / (regs_warp * (TC_THREADS / 32));
        if (v.occ_threads > 2048 / TC_THREADS) v.occ_threads = 2048 / TC_THREADS;
        return cudaSuccess;
    });
    if (e != cudaSuccess) return e;
    int per_sm = (int)((228 * 1024) / (smem + 1024));
    if (per_sm > lim.occ_threads) per_sm = lim.occ_threads;
    if (per_sm > tmem_cap) per_sm = tmem_cap;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    int64_t grid = (int64_t)lim.nsm * per_sm;
    if (grid > a.ntiles) grid = a.ntiles;
    k_tc_conv<N, T, CB><<<(unsigned)grid, TC_THREADS, smem, st>>>(map, a);
    return cudaGetLastError();
}

// [B][H][W][C] viewed as (channel in block, x, y, image, channel block) with blocks of cb = 32 or 16
// channels, swizzled over a block's bytes; blocks_box of them per copy
bool encode_nhwc_blocks(CUtensorMap &map, const __nv_bfloat16 *p, int B, int H, int W, int C, int cb, int bx, int by,
                        int blocks_box) {
    auto enc = tc_encoder();
    if (!enc) return false;
    cuuint64_t dims[5] = {(cuuint64_t)cb, (cuuint64_t)W, (cuuint64_t)H, (cuuint64_t)B, (cuuint64_t)(C / cb)};
    cuuint64_t strides[4] = {(cuuint64_t)C * 2, (cuuint64_t)W * C * 2, (cuuint64_t)H * W * C * 2, (cuuint64_t)cb * 2};
    cuuint32_t box[5] = {(cuuint32_t)cb, (cuuint32_t)bx, (cuuint32_t)by, 1, (cuuint32_t)blocks_box};
    cuuint32_t es[5] = {1, 1, 1, 1, 1};
    return enc(&map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, (void *)p, dims, strides, box, es,
               CU_TENSOR_MAP_INTERLEAVE_NONE, cb == 32 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B,
               CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

int tc_block_n(int Cout) { return Cout < 128 ? Cout : 128; }

cudaError_t tc_wgrad(TcWgradArgs a, float *dw, float *db, cudaStream_t st) {
    if ((a.Cin != 16 && a.Cin % 32) || a.Cout % 32 || a.Cin < 16 || a.Cout < 32 || (a.T != 1 && a.T != 9) || a.B < 1 || a.H < 1 || a.W < 1)
        return cudaErrorInvalidValue;
    // the narrow layers (64 x 64 would fill M = 128 with two taps, no fewer operand bytes per tap)
    const bool stack = a.T == 9 && a.Cin <= 32 && a.Cout <= 64;
    a.N = stack ? a.Cout : (a.Cin <= 256 ? a.Cin : 256);
    if (!stack && a.Cin % a.N) return cudaErrorInvalidValue;
    a.nbn = stack ? 1 : a.Cin / a.N;
    a.nbm = stack ? 1 : (a.Cout + 127) / 128;
    // M = 64 for at most 64 output channels: an MMA reads half as much of A (24 cycles against 40 at
    // N = 32; 222 -> 180 us for 32 x 32 x 9 over 2.1 M pixels)
    a.M = stack ? 4 * a.Cin : (a.Cout <= 64 ? 64 : 128);
    a.ga = stack ? a.Cout / 32 : (a.Cout < a.M ? a.Cout : a.M) / 32;
    a.cbx = a.Cin % 32 == 0 ? 32 : 16;
    // taps per block: as many N-column accumulators as the 512 TMEM columns hold, in groups of
    // balanced size
    const int maxt = stack ? 9 : 512 / a.N;
    a.ngroups = (a.T + maxt - 1) / maxt;
    a.tpc = (a.T + a.ngroups - 1) / a.ngroups;
    const int h = a.T == 9 ? 1 : 0;
    // tile height: 8 pixel rows when three stages of it fit in shared memory, else 4
    auto stage_bytes = [&](int ky) {
        return stack ? wg_stacked_x_bytes(a.Cin, ky) + (uint32_t)(a.ga * WG_KX * ky * 64) : wg_stage_bytes(a.M, a.ga, a.N, ky, h);
    };
    a.ky = stage_bytes(8) * 3 <= 196u * 1024u ? 8 : 4;
    const uint32_t stage = stage_bytes(a.ky);
    a.stage = (int)stage;
    a.xbytes = stack ? (int)wg_stacked_x_bytes(a.Cin, a.ky) : 0;
    // (32 input channels with taps stacked: one block per SM.  Two are 12 % faster on those layers, with
    // the FP32 sums grouped by twice as many chunks: not taken so far)
    const bool two = (stack ? a.Cin == 16 : a.tpc * a.N <= 256) && stage * 3 <= 100u * 1024u;   // room for two blocks per SM
    int S = (int)((two ? 100u * 1024u : 196u * 1024u) / stage);
    a.stages = S > 6 ? 6 : S;
    if (a.stages < 2) return cudaErrorInvalidConfiguration;
    a.tiles_x = (a.W + WG_KX - 1) / WG_KX;
    a.tiles_y = (a.H + a.ky - 1) / a.ky;
    a.ktiles = (int64_t)a.B * a.tiles_y * a.tiles_x;
    static PerDevice<int> sms;
    int dev = 0, nsm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    e = sms.get(dev, nsm, [&](int &v) {
        cudaError_t e = cudaFuncSetAttribute(k_tc_wgrad<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
        if (e != cudaSuccess) return e;
        e = cudaFuncSetAttribute(k_tc_wgrad<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
        if (e != cudaSuccess) return e;
        return cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
    });
    if (e != cudaSuccess) return e;
    // blocks: about one per SM per resident slot over (chunk, tap group, output block, input
    // block); every chunk's partial sums must fit the buffer
    const int64_t per_chunk_blocks = (int64_t)a.ngroups * a.nbm * a.nbn;
    const int64_t count = (int64_t)a.Cout * a.T * a.Cin;
    const int resident = two ? 2 : 1;
    // (rounded down: one block more than the SMs hold is a second round for all)
    int64_t chunks = (int64_t)resident * nsm / per_chunk_blocks;
    if (chunks < 1) chunks = 1;
    if (chunks > a.ktiles) chunks = a.ktiles;
    if (chunks * (count + a.Cout) > a.part_cap) chunks = a.part_cap / (count + a.Cout);
    if (chunks < 1) return cudaErrorInvalidValue;
    a.per_chunk = (a.ktiles + chunks - 1) / chunks;
    a.chunks = (int)((a.ktiles + a.per_chunk - 1) / a.per_chunk);
    const size_t smem = (size_t)a.stages * stage + 8 * (2 * a.stages + 1) + 16;
    CUtensorMap gmap, xmap;
    if (!encode_nhwc_blocks(gmap, a.g, a.B, a.H, a.W, a.Cout, 32, WG_KX, a.ky, a.ga) ||
        !encode_nhwc_blocks(xmap, a.in, a.B, a.H, a.W, a.Cin, a.cbx, WG_KX + 2 * h, a.ky + 2 * h, stack ? 1 : a.N / a.cbx))
        return cudaErrorInvalidValue;
    const int64_t grid = (int64_t)a.chunks * per_chunk_blocks;
    if (stack) k_tc_wgrad<true><<<(unsigned)grid, WG_THREADS, smem, st>>>(gmap, xmap, a);
    else k_tc_wgrad<false><<<(unsigned)grid, WG_THREADS, smem, st>>>(gmap, xmap, a);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return reduce_wgrad(a.part, a.chunks, count, a.Cout, dw, db, st);
}

cudaError_t tc_pack_weights(const __nv_bfloat16 *w, TcPackLayers p, bool flip, __nv_bfloat16 *out, cudaStream_t st) {
    int blocks = 0;
    for (int l = 0; l < p.n; ++l) {
        p.block0[l] = blocks;
        blocks += (p.cout[l] * p.taps[l] * p.cin[l] + 255) / 256;
    }
    if (flip) k_tc_pack<true><<<blocks, 256, 0, st>>>(w, p, out);
    else k_tc_pack<false><<<blocks, 256, 0, st>>>(w, p, out);
    return cudaGetLastError();
}

cudaError_t tc_conv(const __nv_bfloat16 *in, TcConvArgs a, cudaStream_t st) {
    const int N = tc_block_n(a.Cout);
    if ((a.T != 1 && a.T != 9) || a.Cin % 16 || a.Cout % N || (N != 32 && N != 64 && N != 128) || a.W < 1 ||
        a.H < 1 || a.B < 1)
        return cudaErrorInvalidValue;
    if (a.pool_out && (a.H % 2 || a.W % 2)) return cudaErrorInvalidValue;
    if (a.up_out && (!a.up_skip || a.T != 1)) return cudaErrorInvalidValue;
    if ((a.head_w && (a.Cout != 32 || a.T != 9)) || (a.pool_out && a.T != 9)) return cudaErrorInvalidValue;
    auto enc = tc_encoder();
    if (!enc) return cudaErrorNotSupported;
    a.nblocks = a.Cout / N;
    a.tiles_x = (a.W + TILE_X - 1) / TILE_X;
    a.tiles_y = (a.H + TILE_Y - 1) / TILE_Y;
    a.ntiles = (int64_t)a.B * a.tiles_y * a.tiles_x * a.nblocks;
    if (a.ntiles > INT32_MAX) return cudaErrorInvalidValue;
    // 32 channels per stage where the weights are resident or small; else 16, so that a stage with its
    // weight slab stays small enough for two or three blocks per SM
    const int cb = a.Cin % 32 == 0 && (tc_resident(a, N) || a.T == 1) ? 32 : 16;
    // activation tensor [B][H][W][Cin] BF16, box of cb channels x the staged pixels of 1 image
    CUtensorMap map;
    const int halo = a.T == 9 ? 2 : 0;
    cuuint64_t dims[4] = {(cuuint64_t)a.Cin, (cuuint64_t)a.W, (cuuint64_t)a.H, (cuuint64_t)a.B};
    cuuint64_t strides[3] = {(cuuint64_t)a.Cin * 2, (cuuint64_t)a.W * a.Cin * 2, (cuuint64_t)a.H * a.W * a.Cin * 2};
    cuuint32_t box[4] = {(cuuint32_t)cb, (cuuint32_t)(TILE_X + halo), (cuuint32_t)(TILE_Y + halo), 1};
    cuuint32_t es[4] = {1, 1, 1, 1};
    CUresult r = enc(&map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, (void *)in, dims, strides, box, es,
                     CU_TENSOR_MAP_INTERLEAVE_NONE, cb == 32 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B,
                     CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return cudaErrorInvalidValue;
#define GABP_CONV(NN) \
    if (N == NN && a.T == 9) return cb == 32 ? tc_launch<NN, 9, 32>(map, a, st) : tc_launch<NN, 9, 16>(map, a, st); \
    if (N == NN) return cb == 32 ? tc_launch<NN, 1, 32>(map, a, st) : tc_launch<NN, 1, 16>(map, a, st);
    GABP_CONV(32)
    GABP_CONV(64)
    GABP_CONV(128)
#undef GABP_CONV
    return cudaErrorInvalidValue;
}


}  // namespace nn
}  // namespace gabp
