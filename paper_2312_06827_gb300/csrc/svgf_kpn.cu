// Learned part: a kernel-predicting network (KPN) that stands in for a-trous iterations 2-5.
//
//   features  10 channels from the pass-0 output and the G-buffer (BF16, padded to 16)
//   conv x4   3x3, 10 -> 32 -> 32 -> 32 -> 25 (ReLU between), BF16 operands, FP32 accumulation,
//             as implicit GEMMs on the 5th-generation tensor cores (tcgen05.mma, accumulators in
//             tensor memory); the same kernel computes the data gradient (dgrad) with the
//             flipped, transposed weights; the weight gradient (wgrad) is a second tcgen05
//             GEMM, reduced over pixels
//   apply     softmax of the 25 logits = a 5x5 kernel per pixel (computed in the last layer's
//             epilogue, stored as 25 planes), applied to the pass-0 colour at dilation 1 and then
//             at dilation 4 (renormalised over in-image taps)
//   train     MSE in tone-mapped space against the plain pipeline's output, backward through
//             the applications, the softmax and the convolutions, Adam on FP32 master weights.
//
// Tensors: images [B][H][W][C] (pixel-major, channels contiguous); activations BF16 with 32
// channels (features 16); predicted kernels K and their gradients FP32 planar [25][B*H*W];
// colours float4.  Weights of the
// conv kernel: [9 taps][32 outputs][CI inputs] BF16 (inputs contiguous), tap = (dy+1)*3 + (dx+1).
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <math.h>
#include <stdint.h>

#include "svgf_device.cuh"
#include "svgf_kpn.h"

namespace svgf {
namespace kpn {
namespace {

__device__ __forceinline__ unsigned smem_addr(const void* p) {
    return (unsigned)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ float ex2_fast(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ unsigned pack_bf16(float lo, float hi) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const unsigned*>(&v);
}
__device__ __forceinline__ unsigned pack_f16(float lo, float hi) {
    const __half2 v = __floats2half2_rn(lo, hi);
    return *reinterpret_cast<const unsigned*>(&v);
}
__device__ __forceinline__ float2 unpack_f16(unsigned u) {
    return __half22float2(*reinterpret_cast<const __half2*>(&u));
}

// ---- the 3x3 convolution on the 5th-generation tensor cores (tcgen05) ------------------------
// An output row segment = 128 consecutive pixels of one image row (M = 128) x 32 output channels.
// Input rows of pixels x0-1 .. x0+128 are staged in shared memory so that the K-major operand A
// of horizontal tap dx and channel chunk kc (K = 16) is a descriptor start address dx pixels
// further on -- no im2col copy.  32 channels: each pixel a 64-byte row in the 64-byte swizzled
// layout (8-row groups every 512 B), A starting at dx * 64 + kc * 32 bytes.  16 channels (the
// first layer): channel groups outermost, [group of 8 channels][pixel][8 channels], 8 x 16 B
// core matrices stacked along M every 128 B (SBO) and along K every 130 x 16 B (LBO).  Input row r enters output
// rows r+1, r and r-1 through the kernel rows dy = 0, 1, 2, so one MMA per (dx, kc) with the
// three kernel rows side by side along N (N = 96) adds row r's share to all three outputs: the
// weights sit as [dx][group][dy = 2, 1, 0][co][8] (B operand: SBO 128 B, LBO 96 x 16 B), and
// the output rows' FP32 accumulators are consecutive 32-column slots of a ring in tensor memory
// (a triple that wraps around the ring is issued as two MMAs).  One thread issues the MMAs of
// each input row and commits them to an mbarrier; an output row is complete once the row below
// it has been issued, and the four epilogue warps then read their 32 accumulator lanes (one
// pixel per thread, 32 channels) and zero the slot for its next use.
namespace tc {
constexpr int M = 128;
constexpr int HP = M + 2;
// Shared memory left free beyond the staged rows (none: the operand extents end inside them).
constexpr int kSlack = 0;
// Instruction descriptor of tcgen05.mma kind::f16: FP32 accumulator (bits 4-5 = 1), BF16 A and
// B (bits 7-9, 10-12 = 1), both K-major (bits 15, 16 = 0), N >> 3 at bits 17-22, M >> 4 at bits
// 24-28.
constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((32u >> 3) << 17) | ((128u >> 4) << 24);

// Shared-memory matrix descriptor, no swizzle: start address >> 4 (bits 0-13), leading-
// dimension byte offset >> 4 (bits 16-29, the K stride of core matrices), stride-dimension byte
// offset >> 4 (bits 32-45, the M/N stride of 8-row groups), descriptor version 1 (bit 46).
__device__ __forceinline__ uint64_t sdesc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46);
}
__device__ __forceinline__ void mma(uint32_t dtmem, uint64_t a, uint64_t b, uint32_t accumulate,
                                    uint32_t idesc = kIdesc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %3, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %4, p;\n\t}"
        ::"r"(dtmem), "l"(a), "l"(b), "r"(accumulate), "r"(idesc) : "memory");
}
// The instruction descriptor of kIdesc with N = n (a multiple of 16, at most 256) columns.
__device__ __forceinline__ uint32_t idesc_n(uint32_t n) {
    return (kIdesc & ~(0x3Fu << 17)) | ((n >> 3) << 17);
}
__device__ __forceinline__ void commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
                 ::"r"(smem_addr(bar)) : "memory");
}
// The MMA (accumulating) and the commit issued by the lane elect.sync picks, for a whole warp
// walking the issue loop: its values are then warp-uniform, and the descriptors stay on the
// uniform datapath (one lane walking the loop inside a lane branch measured at about 240 cycles
// an MMA against 56 for N = 96).  In a converged warp elect.sync picks the same lane every
// time, so a commit tracks that lane's MMAs.
__device__ __forceinline__ void mma_elect(uint32_t dtmem, uint64_t a, uint64_t b, uint32_t idesc) {
    asm volatile(
        "{\n\t.reg .pred p, e;\n\tsetp.ne.u32 p, 1, 0;\n\telect.sync _|e, 0xffffffff;\n\t"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(dtmem), "l"(a), "l"(b), "r"(idesc) : "memory");
}
__device__ __forceinline__ void commit_elect(uint64_t* bar) {
    asm volatile(
        "{\n\t.reg .pred e;\n\telect.sync _|e, 0xffffffff;\n\t"
        "@e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}"
        ::"r"(smem_addr(bar)) : "memory");
}
__device__ __forceinline__ void tmem_alloc(uint32_t* slot, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 ::"r"(smem_addr(slot)), "r"(ncols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
// Zeros into 32 lanes x 32 columns of tensor memory (the warp's lanes), complete on return.
__device__ __forceinline__ void st32_zero(uint32_t taddr) {
    const uint32_t z = 0;
    asm volatile("tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1};"
                 ::"r"(taddr), "r"(z) : "memory");
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}
// 32 lanes x 32 columns of 32-bit accumulator: thread i of the warp gets lane (lane base + i).
__device__ __forceinline__ void ld32(uint32_t (&r)[32], uint32_t taddr) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
                 : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count = 1) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}
// One arrival that also expects `bytes` of asynchronous copies to complete on the barrier.
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes) : "memory");
}
// A TMA copy of one box of a 4-D tensor map (coordinates innermost first) into shared memory,
// completing its bytes on `bar`.
__device__ __forceinline__ void tma_load_4d(void* dst, const CUtensorMap* map, int c0, int c1, int c2, int c3,
                                            uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];"
        ::"r"(smem_addr(dst)), "l"((unsigned long long)map), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(smem_addr(bar))
        : "memory");
}
// Named barrier ID (an immediate) over 128 threads (a group of four warps), returning whether
// `ok` held for all of them.
template <int ID>
__device__ __forceinline__ bool all_of_128(bool ok) {
    uint32_t r;
    asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.u32 q, %1, 0;\n\tbar.red.and.pred p, %2, 128, q;\n\t"
                 "selp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(r) : "r"((uint32_t)ok), "n"(ID) : "memory");
    return r != 0;
}
// Bounded wait (about a second at most with the default number of tries) for the given phase of
// the barrier; false when it gave up.
constexpr int kWaitTries = 1 << 20;
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, int tries = kWaitTries) {
    for (int i = 0; i < tries; ++i) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred P;\n\tmbarrier.try_wait.parity.shared::cta.b64 P, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, P;\n\t}"
            : "=r"(done) : "r"(smem_addr(bar)), "r"(parity) : "memory");
        if (done) return true;
    }
    return false;
}
}  // namespace tc

// Bulk asynchronous shared -> global copy (16-byte aligned, size a multiple of 16), its group
// commit, and the waits for its source to be read / its writes to be done.
__device__ __forceinline__ void bulk_s2g(void* gdst, const void* ssrc, uint32_t bytes) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;"
                 ::"l"((unsigned long long)__cvta_generic_to_global(gdst)), "r"(smem_addr(ssrc)), "r"(bytes)
                 : "memory");
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}
// at most N of the bulk groups committed last still reading their source
template <int N = 0>
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(N) : "memory"); }
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

// 16-byte asynchronous global -> shared copy; src_bytes = 0 fills the 16 bytes with zeros.
__device__ __forceinline__ void cp_async16(void* dst, const void* src, uint32_t src_bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_addr(dst)), "l"(src),
                 "r"(src_bytes) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Staged input rows: a ring of kRing.
constexpr int kRing = 6;
// Accumulator slots (32 tensor-memory columns each) of the output-row ring.
constexpr unsigned kSlots = 8;
// Commit barriers of the input rows' MMAs.
constexpr unsigned kDone = 8;
// Output-row staging buffers of the epilogue (each M x 64 bytes): with two, an output row is
// written while the bulk store of the previous one still reads its buffer.  Two measured no
// faster at 1080p (nor a ring of 8 rows with 5 in flight), so one is kept.
constexpr int kOutBufs = 1;
// A staged 32-channel row in the 64-byte swizzled layout: 130 pixels x 64 bytes, padded to a
// multiple of the 512-byte swizzle pattern so that every ring slot starts on one.
constexpr int kRowSw64Bytes = 17 * 512;
// A 16-channel row in the 32-byte swizzled layout: 130 x 32 bytes padded to 17 x 256.
constexpr int kRowSw32Bytes = 17 * 256;
// Dynamic shared memory of a convolution block, at least: two blocks per SM, whose 2 x 8 slots
// fill the SM's 512 tensor-memory columns (a third block would wait in tcgen05.alloc).
constexpr size_t kMinConvSmem = 80 * 1024;

// One staged input row (image row gy of image n, pixels x0-1 .. x0+128, zeros outside the image,
// by a warp's 32 lanes with 16-byte cp.async) for CI = 32 in the 64-byte swizzled K-major
// layout: pixel px is a 64-byte row, its 16-byte chunk c (8 channels) stored at chunk
// c ^ ((px >> 1) & 3).  The tensor core applies the
// swizzle to the absolute shared-memory address bits (bits 4-5 ^= bits 7-8), so with the row
// slot 512-byte aligned, a tap shift of dx pixels is a start address dx * 64 bytes further on.
template <int NT>
__device__ __forceinline__ void tc_stage_row_sw64(unsigned char* dst, const __nv_bfloat16* __restrict__ in,
                                                  int n, int gy, int x0, int H, int W, int tid) {
    for (int i = tid; i < tc::HP * 4; i += NT) {
        const int kg = i % 4, px = i / 4, gx = x0 + px - 1;
        const bool ok = gx >= 0 && gx < W && gy >= 0 && gy < H;
        const __nv_bfloat16* src = ok ? in + (((long)n * H + gy) * W + gx) * 32 + kg * 8 : in;
        cp_async16(dst + px * 64 + ((kg ^ ((px >> 1) & 3)) << 4), src, ok ? 16u : 0u);
    }
    cp_async_commit();
}

// The same row for CI = 16 in the 32-byte swizzled K-major layout: pixel px is a 32-byte row,
// its chunk c stored at chunk c ^ ((px >> 2) & 1) (address bit 4 ^= bit 7), slots 256-byte
// aligned.
template <int NT>
__device__ __forceinline__ void tc_stage_row_sw32(unsigned char* dst, const __nv_bfloat16* __restrict__ in,
                                                  int n, int gy, int x0, int H, int W, int tid) {
    for (int i = tid; i < tc::HP * 2; i += NT) {
        const int kg = i & 1, px = i >> 1, gx = x0 + px - 1;
        const bool ok = gx >= 0 && gx < W && gy >= 0 && gy < H;
        const __nv_bfloat16* src = ok ? in + (((long)n * H + gy) * W + gx) * 16 + kg * 8 : in;
        cp_async16(dst + px * 32 + ((kg ^ ((px >> 2) & 1)) << 4), src, ok ? 16u : 0u);
    }
    cp_async_commit();
}

// Epilogue of one pixel: the 32 accumulated channels f (bias added) of pixel p.  EPI 1 writes
// the 25 kernel planes directly (a warp's 32 pixels are contiguous in each plane); EPI 0 / 2 write
// the pixel's 64 output bytes to `stage` (the tile's output row, stored in bulk afterwards).
template <int EPI>
__device__ __forceinline__ void tc_epilogue(float (&f)[32], long p, long npx,
                                            const __nv_bfloat16* __restrict__ mask, void* out,
                                            uint4* stage) {
    if (EPI == 1 || EPI == 3) {
        float mx = -INFINITY;
#pragma unroll
        for (int j = 0; j < 25; ++j) mx = fmaxf(mx, f[j]);
        float sum = 0.f;
#pragma unroll
        for (int j = 0; j < 25; ++j) {
            f[j] = ex2_fast((f[j] - mx) * 1.4426950408889634f);
            sum += f[j];
        }
        const float r = 1.0f / sum;
        if constexpr (EPI == 1) {
#pragma unroll
            for (int j = 0; j < 25; ++j) reinterpret_cast<float*>(out)[j * npx + p] = f[j] * r;
        } else {
#pragma unroll
            for (int j = 0; j < 32; ++j) f[j] = j < 25 ? f[j] * r : 0.f;
#pragma unroll
            for (int q = 0; q < 4; ++q)
                stage[q] = make_uint4(pack_f16(f[8 * q], f[8 * q + 1]), pack_f16(f[8 * q + 2], f[8 * q + 3]),
                                      pack_f16(f[8 * q + 4], f[8 * q + 5]), pack_f16(f[8 * q + 6], f[8 * q + 7]));
        }
        return;
    }
    if (EPI == 2) {
        const uint4* mk = reinterpret_cast<const uint4*>(mask + p * 32);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const uint4 m4 = mk[q];
            const unsigned mw[4] = {m4.x, m4.y, m4.z, m4.w};
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                const __nv_bfloat162 m2 = *reinterpret_cast<const __nv_bfloat162*>(&mw[h]);
                if (!(__low2float(m2) > 0.f)) f[8 * q + 2 * h] = 0.f;
                if (!(__high2float(m2) > 0.f)) f[8 * q + 2 * h + 1] = 0.f;
            }
        }
    } else {
#pragma unroll
        for (int j = 0; j < 32; ++j) f[j] = fmaxf(f[j], 0.f);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q)
        stage[q] = make_uint4(pack_bf16(f[8 * q], f[8 * q + 1]), pack_bf16(f[8 * q + 2], f[8 * q + 3]),
                              pack_bf16(f[8 * q + 4], f[8 * q + 5]), pack_bf16(f[8 * q + 6], f[8 * q + 7]));
}

// 3x3 convolution, 32 output channels: out[p][co] = epilogue(sum_{tap,ci} Wt[tap][co][ci] in[p+off][ci])
// EPI 0: + bias, ReLU, BF16 out.  EPI 1: + bias, then the softmax over the 25 logits of each
// pixel, written as 25 planes K[i][p] (FP32; npx = B*H*W).  EPI 2: x (mask[p][co] > 0), BF16 out
// (data gradient through the ReLU of the layer below).  EPI 3: the softmax of EPI 1 as FP16,
// pixel-major (25 weights and 7 zeros, 64 B per pixel, stored like a BF16 activation row; the
// inference form).  A block walks chunks of `chunk` output
// rows down one 128-pixel column of an image, reading input rows y0-1 .. y0+chunk.  Three roles,
// each walking the same chunks and rows (NG epilogue groups, 128 NG + 64 threads):
//   warp 4 NG + 1, the producer: copies each input row into a ring of kRing (one TMA copy a row,
//     completing on the slot's barrier) once the MMAs that read the slot's previous row have
//     completed;
//   warp 4 NG, the issuer (the whole warp walks the rows, one elected lane issues): per input
//     row, the MMAs into the output rows' accumulators;
//   warps 0 .. 4 NG - 1, the epilogue: group g takes the output rows of running index g modulo
//     NG; per output row, read its accumulator lanes, zero them, store.
// They meet at mbarriers, each waited for phase by phase (a parity wait must find its barrier at
// most one phase behind and not past the phase it waits for):
//   full[slot]     the producer's row has landed (TMA bytes)        -> the issuer;
//   rfree[slot]    the MMAs of the slot's row completed (commit)     -> the producer;
//   done[o % kDone] output row o complete: the MMAs of input row o + 1 (commit) -> the epilogue;
//   drained[acc]   the epilogue read and zeroed the accumulator slot -> the issuer.
// Rows take ring slots and output rows accumulator slots in the order the roles walk them (a
// running count), so a slot comes back kRing rows or kSlots output rows later.  The issuer can
// complete at most five output rows past the one the epilogue waits for (an accumulator slot
// is first written only after its previous output row was drained), below kDone = 8.
// Every wait is bounded: one that gives up sets kErrWaitGaveUp in *err and its side stops (the
// others' waits then run out too); the issuer commits once more to a barrier of its own and
// waits for it (all its MMAs done), and the block frees its tensor memory and returns.
template <int CI, int EPI, int NG>
__global__ void __launch_bounds__(128 * NG + 64, 2) k_conv3x3_tc(const __grid_constant__ CUtensorMap rows,
                                                       const __nv_bfloat16* __restrict__ in,
                                                       const __nv_bfloat16* __restrict__ wt,
                                                       const float* __restrict__ bias,
                                                       const __nv_bfloat16* __restrict__ mask,
                                                       void* out, int B, int H, int W, int chunk,
                                                       int* err) {
    using namespace tc;
    constexpr int KG = CI / 8;
    // rows and weights in the swizzled K-major layouts: CI = 32 rows of 64 bytes (slots of
    // 17 x 512 bytes), CI = 16 rows of 32 bytes (slots of 17 x 256 bytes)
    constexpr bool SW64 = CI == 32;     // else 32-byte swizzle
    constexpr bool SW64B = SW64;
    constexpr int RB = CI * 2;                       // bytes per pixel row (64 or 32)
    constexpr int ROW_BYTES = SW64 ? kRowSw64Bytes : kRowSw32Bytes;
    constexpr int W_BYTES = 9 * KG * 32 * 16, A_BYTES = kRing * ROW_BYTES, O_BYTES = NG * kOutBufs * M * 64;
    constexpr int NT = 128 * NG + 64;
    extern __shared__ __align__(1024) unsigned char tc_smem[];   // ring slots on 512-byte boundaries
    unsigned char* sw = tc_smem;
    unsigned char* sa = tc_smem + W_BYTES;
    uint4* so = reinterpret_cast<uint4*>(tc_smem + W_BYTES + A_BYTES);      // output rows [NG][kOutBufs][M][64 B]
    uint64_t* bar = reinterpret_cast<uint64_t*>(tc_smem + W_BYTES + A_BYTES + O_BYTES + kSlack);
    uint64_t* done = bar;                              // [kDone]
    uint64_t* full = done + kDone;                     // [kRing]
    uint64_t* rfree = full + kRing;                    // [kRing]
    uint64_t* drained = rfree + kRing;                 // [kSlots]
    uint64_t* fin = drained + kSlots;                  // the issuer's last commit
    uint32_t* tslot = reinterpret_cast<uint32_t*>(fin + 1);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // weights [tap][co][ci] -> per dx the 96 rows (2 - dy) * 32 + co of the B operand, swizzled
    // like the input rows (64-byte rows for 32 channels, 32-byte rows for 16).  Read ahead of pdl_wait,
    // beside the previous launch's end: earlier calls wrote them, and no launch of this one does.
    for (int i = tid; i < 9 * 32 * KG; i += NT) {
        const int kg = i % KG, co = (i / KG) % 32, tap = i / (KG * 32), dy = tap / 3, dx = tap % 3;
        const int r = (2 - dy) * 32 + co;
        const int off = SW64B ? dx * 96 * 64 + r * 64 + ((kg ^ ((r >> 1) & 3)) << 4)
                              : dx * 96 * 32 + r * 32 + ((kg ^ ((r >> 2) & 1)) << 4);
        *reinterpret_cast<uint4*>(sw + off) = *reinterpret_cast<const uint4*>(wt + ((long)tap * 32 + co) * CI + kg * 8);
    }
    if (tid == 0) {
        for (unsigned i = 0; i < kDone; ++i) mbar_init(&done[i]);
        for (int r = 0; r < kRing; ++r) {
            mbar_init(&full[r], 1);
            mbar_init(&rfree[r]);
        }
        for (unsigned i = 0; i < kSlots; ++i) mbar_init(&drained[i], 128);
        mbar_init(fin);
    }
    pdl_wait();   // before the tensor memory: the previous launch's blocks may still hold theirs
    if (warp == 0) tmem_alloc(tslot, 32 * kSlots);
    fence_proxy_async();
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = *tslot;
    if (warp < 4) {                    // every accumulator slot starts at zero
#pragma unroll 1
        for (unsigned sl = 0; sl < kSlots; ++sl) st32_zero(tmem + sl * 32u + ((uint32_t)(warp * 32) << 16));
    }
    fence_before();
    __syncthreads();
    fence_after();
    const long npx = (long)B * H * W;
    const int segs = (W + M - 1) / M, chunks_y = (H + chunk - 1) / chunk;
    const long total = (long)B * segs * chunks_y;

    if (warp == 4 * NG + 1) {
        // ---- the producer: each input row into the ring by one TMA copy (the tensor map's box
        // is the row's 130 pixels x CI channels, swizzled as the MMAs read it; pixels and rows
        // outside the image read as zeros) once the MMAs that read the slot's previous row have
        // completed; the copy completes on the slot's full barrier (one arrival, expected bytes)
        constexpr uint32_t kRowTx = (uint32_t)tc::HP * CI * 2;
        uint32_t used = 0, rpar = 0, ipar = 0;   // ipar: per slot, parity of the next copy's phase
        unsigned rs = 0;                // rows staged so far: the row's ring slot is rs % kRing
        bool fail = false;
        for (long c = blockIdx.x; c < total && !fail; c += gridDim.x) {
            const int n = (int)(c / ((long)segs * chunks_y));
            const int rc = (int)(c - (long)n * segs * chunks_y);
            const int seg = rc / chunks_y, y0 = (rc - seg * chunks_y) * chunk, x0 = seg * M;
            const int y1 = y0 + chunk < H ? y0 + chunk : H;
            for (int q = y0 - 1; q <= y1; ++q) {
                const int sl = (int)(rs++ % kRing);
                if ((used >> sl) & 1u) {        // the slot's previous row must have been read
                    const bool ok = __all_sync(0xffffffffu, mbar_wait(&rfree[sl], (rpar >> sl) & 1u));
                    rpar ^= 1u << sl;
                    if (!ok) {
                        fail = true;
                        break;
                    }
                }
                used |= 1u << sl;
                if (lane == 0) {
                    mbar_arrive_expect_tx(&full[sl], kRowTx);
                    tma_load_4d(sa + sl * ROW_BYTES, &rows, 0, x0 - 1, q, n, &full[sl]);
                }
                ipar ^= 1u << sl;
                __syncwarp();
            }
        }
        // the block's shared memory is released at its end: every copy issued must have landed
        for (int sl = 0; sl < kRing; ++sl)
            if ((used >> sl) & 1u) mbar_wait(&full[sl], ((ipar >> sl) & 1u) ^ 1u);
        if (fail && lane == 0) atomicOr(err, kErrWaitGaveUp);
    } else if (warp == 4 * NG) {
        // ---- the MMA issuer: the whole warp walks the rows, one elected lane issues
        {
            const uint32_t a0 = smem_addr(sa), b0 = smem_addr(sw);
            // descriptors of the ring's first slot and of the weights; an operand's descriptor
            // adds its byte offset / 16 to the start-address field (no carry: shared addresses
            // stay below 256 KB)
            // swizzled K-major operands: SBO = one 8-row group (512 or 256 bytes), swizzle mode at
            // bits 61-63 (64B = 4, 32B = 6); LBO is not used by these layouts
            const uint64_t A0 = SW64 ? (sdesc(a0, 16, 512) | (4ull << 61)) : (sdesc(a0, 16, 256) | (6ull << 61));
            const uint64_t B0 = SW64B ? (sdesc(b0, 16, 512) | (4ull << 61)) : (sdesc(b0, 16, 256) | (6ull << 61));
            unsigned nb = 0;           // input rows issued: ring slot nb % kRing
            unsigned obase = 0;        // output rows of earlier chunks (accumulator slot numbering)
            uint32_t fpar = 0;         // per ring slot: parity of the next row-ready phase
            uint32_t dused = 0, dpar = 0;   // per accumulator slot: used before, next drained parity
            bool fail = false;
            for (long c = blockIdx.x; c < total && !fail; c += gridDim.x) {
                const int rc = (int)(c % ((long)segs * chunks_y));
                const int y0 = (rc % chunks_y) * chunk;
                const int y1 = y0 + chunk < H ? y0 + chunk : H;
                for (int r = y0 - 1; r <= y1; ++r) {
                    const int sl = (int)(nb % kRing);
                    fail = !__all_sync(0xffffffffu, mbar_wait(&full[sl], (fpar >> sl) & 1u));
                    fpar ^= 1u << sl;
                    // output row r + 1 starts here: its slot's previous output must be drained
                    if (!fail && r + 1 <= y1 - 1) {
                        const unsigned ts = (obase + (unsigned)(r + 1 - y0)) % kSlots;
                        if ((dused >> ts) & 1u) {
                            fail = !__all_sync(0xffffffffu, mbar_wait(&drained[ts], (dpar >> ts) & 1u));
                            dpar ^= 1u << ts;
                        }
                        dused |= 1u << ts;
                    }
                    if (fail) break;
                    fence_after();
                    // output rows lo..hi of this chunk take input row r; output o uses kernel
                    // row dy = r - o + 1, stored as weight block 2 - dy = o - r + 1
                    const int lo = r - 1 > y0 ? r - 1 : y0, hi = r + 1 < y1 - 1 ? r + 1 : y1 - 1;
                    const int nblk = hi - lo + 1, blk0 = lo - r + 1;
                    const unsigned s0 = (obase + (unsigned)(lo - y0)) % kSlots;
                    const int first = nblk < (int)(kSlots - s0) ? nblk : (int)(kSlots - s0);
                    const uint32_t id1 = idesc_n(32u * first), id2 = idesc_n(32u * (nblk - first));
                    const uint64_t arow = A0 + (uint64_t)((sl * ROW_BYTES) >> 4);
#pragma unroll
                    for (int dx = 0; dx < 3; ++dx)
#pragma unroll
                        for (int kc = 0; kc < KG / 2; ++kc) {
                            const uint64_t a = arow + (uint64_t)((dx * RB + kc * 32) >> 4);
                            // B rows of block blk0 on: 32 rows per block (2048 B swizzled, 512 B plain)
                            const uint64_t bb = B0 + (uint64_t)((dx * 96 * RB + blk0 * 32 * RB + kc * 32) >> 4);
                            mma_elect(tmem + s0 * 32u, a, bb, id1);
                            if (first < nblk) mma_elect(tmem, a, bb + (uint64_t)((first * 32 * RB) >> 4), id2);
                        }
                    if (r - 1 >= y0) commit_elect(&done[(obase + (unsigned)(r - 1 - y0)) % kDone]);   // output r - 1 complete
                    commit_elect(&rfree[sl]);
                    ++nb;
                }
                obase += (unsigned)(y1 - y0);
            }
            if (fail && lane == 0) atomicOr(err, kErrWaitGaveUp);
            // the tensor memory is freed below: every MMA of the issuing lane must have completed
            if (nb > 0) {
                commit_elect(fin);
                mbar_wait(fin, 0u);
            }
        }
        __syncwarp();
    } else {
        // ---- warps 0 .. 4 NG - 1: the epilogue, NG groups of four warps, group g draining the
        // output rows whose running index is g modulo NG (with NG = 2 two rows drain at once;
        // kSlots and kDone are even, so each accumulator slot and done barrier has one group)
        const int g = warp >> 2, lx = (warp & 3) * 32 + lane;
        float bv[32];
#pragma unroll
        for (int j = 0; j < 32; ++j) bv[j] = EPI == 2 ? 0.f : bias[j];
        unsigned obase = 0;             // output rows of earlier chunks
        unsigned nst = 0;               // rows this group has stored (its staging buffer)
        bool fail = false;
        for (long c = blockIdx.x; c < total && !fail; c += gridDim.x) {
            const int n = (int)(c / ((long)segs * chunks_y));
            const int rc = (int)(c - (long)n * segs * chunks_y);
            const int seg = rc / chunks_y, y0 = (rc - seg * chunks_y) * chunk, x0 = seg * M;
            const int y1 = y0 + chunk < H ? y0 + chunk : H;
            for (int o = y0; o < y1; ++o) {
                // output row o is complete with input row o + 1, whose MMAs commit to done[oi % kDone]
                const unsigned oi = obase + (unsigned)(o - y0);
                if ((int)(oi % NG) != g) continue;
                const bool ok = mbar_wait(&done[oi % kDone], (oi / kDone) & 1u);
                if (EPI != 1 && lx == 0) bulk_wait_read<kOutBufs - 1>();   // the row's buffer is free
                if (!(g == 0 ? all_of_128<2>(ok) : all_of_128<3>(ok))) {
                    if (lx == 0) atomicOr(err, kErrWaitGaveUp);
                    fail = true;
                    break;
                }
                fence_after();
                const unsigned ts = oi % kSlots;
                const uint32_t ta = tmem + ts * 32u + ((uint32_t)((warp & 3) * 32) << 16);
                uint32_t v[32];
                ld32(v, ta);
                st32_zero(ta);
                fence_before();
                mbar_arrive(&drained[ts]);
                const long prow = ((long)n * H + o) * W;
                const int x = x0 + lx;
                uint4* buf = so + (g * kOutBufs + nst % kOutBufs) * M * 4;
                if (x < W) {
                    float f[32];
#pragma unroll
                    for (int j = 0; j < 32; ++j) f[j] = __uint_as_float(v[j]) + bv[j];
                    tc_epilogue<EPI>(f, prow + x, npx, mask, out, buf + lx * 4);
                }
                if (EPI != 1) {
                    // the output pixels x0 .. min(x0 + 128, W) - 1 are contiguous: one bulk store
                    fence_proxy_async();
                    if (g == 0) asm volatile("bar.sync 4, 128;" ::: "memory");
                    else asm volatile("bar.sync 5, 128;" ::: "memory");
                    if (lx == 0) {
                        const int nv = W - x0 < M ? W - x0 : M;
                        bulk_s2g(reinterpret_cast<__nv_bfloat16*>(out) + (prow + x0) * 32, buf, (uint32_t)(nv * 64));
                    }
                }
                ++nst;
            }
            obase += (unsigned)(y1 - y0);
        }
        if (lx == 0) bulk_wait_all();
    }
    fence_before();
    __syncthreads();
    fence_after();
    if (warp == 0) tmem_dealloc(tmem, 32 * kSlots);
}

// ---- the four layers in one kernel (inference) -------------------------------------------------
// The network's four convolutions in one pass, the activations never leaving the SM.  A block
// walks a chunk of output rows down one column segment; each layer's output row, once complete,
// goes from an epilogue (bias, ReLU, BF16) straight into the next layer's ring of input rows in
// shared memory, in the same 64-byte swizzled layout the per-layer kernel stages from global
// memory, and the last layer's softmax weights (FP16, pixel-major) are the only output.  Layer l
// has its own quarter of tensor memory: kNetSlots output-row accumulator slots of 32 columns.
// Columns: every layer computes the same 128 lanes, pixel x = s + lane.  Ring rows hold the
// pixels s - 1 .. s + 128 and the epilogues fill 1 .. 128 of them, so layer l is exact on lanes
// l .. 127 - l and a segment keeps lanes 3 .. 124 of the last layer: segments start kNetSeg = 122
// pixels apart (s = 122 seg - 3).  Outside the image the epilogue writes zeros, the zero padding
// each layer's input has in the per-layer form, so the result is that form's, bit for bit.
// Rows: for the chunk's output rows y0 .. y1 - 1, layer l reads rows y0 - 4 + l .. y1 + 3 - l
// (input k at y0 - 4 + l + k) and completes rows y0 - 3 + l .. y1 + 2 - l (output o at
// y0 - 3 + l + o, complete once input o + 2 is in); layer l's outputs are layer l + 1's inputs.
// Roles (20 warps): warp 16 + l issues layer l's MMAs (one elected lane), input row by input
// row, once the row is in its ring and the accumulator slot of the output row it starts was
// drained, and warp 16 also stages the feature rows into ring 0 (cp.async, kNetAhead rows ahead);
// epilogue warps 4l .. 4l + 3 drain layer l's output rows in order, each once its MMAs completed.
// One warp a layer issues and one group a layer drains, so the four layers' waits overlap: one
// thread issuing all four layers spent most of its time in its waits, and one group draining
// two layers set the pace at about 2,400 cycles a row each.  Barriers: per ring slot of layers
// 1-3 full (row written) and per ring slot rfree (its MMAs completed), per layer done (an output
// row's MMAs completed) and drained (an accumulator slot read), and a last commit per issuer;
// every wait is bounded as in the per-layer kernel.
constexpr int kNetSeg = 122;
constexpr int kNetRing0 = 4, kNetAhead = 2;       // feature rows (16 channels): ring, rows staged ahead
constexpr int kNetRing = 4;                       // input rows of layers 1-3
constexpr unsigned kNetSlots = 4;                 // 4 layers x 4 slots x 32 columns = 512
constexpr unsigned kNetDone = 4;
constexpr int kNetOutBufs = 2;
constexpr int kNetThreads = 20 * 32;
constexpr int kNetW0Bytes = 3 * 96 * 32, kNetW1Bytes = 3 * 96 * 64;
// shared memory: layers 1-3 weights, layer 0 weights, rings of layers 1-3, ring of layer 0,
// output staging, biases, barriers (every ring slot on a 512-byte boundary)
constexpr int kNetOffW0 = 3 * kNetW1Bytes;
constexpr int kNetOffRing = kNetOffW0 + kNetW0Bytes;
constexpr int kNetOffRing0 = kNetOffRing + 3 * kNetRing * kRowSw64Bytes;
constexpr int kNetOffOut = kNetOffRing0 + kNetRing0 * kRowSw32Bytes;
constexpr int kNetOffBias = kNetOffOut + kNetOutBufs * tc::M * 64;
constexpr int kNetOffBar = kNetOffBias + 4 * 32 * 4;
constexpr int kNetBars = kNetRing0 + 6 * kNetRing + 4 * (int)kNetDone + 4 * (int)kNetSlots + 4;
constexpr int kNetSmemBytes = kNetOffBar + kNetBars * 8 + 8;
static_assert(kNetOffRing % 512 == 0 && kNetOffRing0 % 512 == 0 && kNetOffOut % 16 == 0, "ring alignment");
static_assert(kNetRing >= 2 && kNetAhead < kNetRing0 && kNetAhead <= 2, "ring sizes");

struct NetWeights {
    const __nv_bfloat16* wt[4];
    const float* bias[4];
};

// Shared-memory state of the four-layer kernel.
struct NetSmem {
    unsigned char* ring0;      // [kNetRing0][kRowSw32Bytes]
    unsigned char* ring;       // [3][kNetRing][kRowSw64Bytes]: the input rows of layer l + 1
    unsigned char* sw0;        // layer 0 weights
    unsigned char* sw1;        // [3][kNetW1Bytes]
    uint4* so;                 // [kNetOutBufs][M][64 B]
    float* bias;               // [4][32]
    uint64_t *rfree0, *full, *rfree, *done, *drained, *fin;
};

// One chunk: image n, first kept row y0, rows output rows, first lane's pixel s.
struct NetChunk {
    int n, y0, rows, s;
};
__device__ __forceinline__ NetChunk net_chunk_of(long c, int H, int chunk, int segs, int chunks_y) {
    NetChunk ch;
    ch.n = (int)(c / ((long)segs * chunks_y));
    const int rc = (int)(c - (long)ch.n * segs * chunks_y);
    const int seg = rc / chunks_y;
    ch.y0 = (rc - seg * chunks_y) * chunk;
    ch.rows = (ch.y0 + chunk < H ? ch.y0 + chunk : H) - ch.y0;
    ch.s = seg * kNetSeg - 3;
    return ch;
}

// The MMAs of one input row of a layer (CI input channels): kernel-row blocks blk0.. of the
// weights into the accumulator slots s0.. of the layer's ring (two MMAs when the triple wraps).
template <int CI>
__device__ __forceinline__ void net_issue_row(uint32_t acc, uint64_t arow, uint64_t B0, int blk0, unsigned s0,
                                              int nblk) {
    using namespace tc;
    constexpr int RB = CI * 2;
    const int first = nblk < (int)(kNetSlots - s0) ? nblk : (int)(kNetSlots - s0);
    const uint32_t id1 = idesc_n(32u * first), id2 = idesc_n(32u * (nblk - first));
#pragma unroll
    for (int dx = 0; dx < 3; ++dx)
#pragma unroll
        for (int kc = 0; kc < CI / 16; ++kc) {
            const uint64_t a = arow + (uint64_t)((dx * RB + kc * 32) >> 4);
            const uint64_t bb = B0 + (uint64_t)((dx * 96 * RB + blk0 * 32 * RB + kc * 32) >> 4);
            mma_elect(acc + s0 * 32u, a, bb, id1);
            if (first < nblk) mma_elect(acc, a, bb + (uint64_t)((first * 32 * RB) >> 4), id2);
        }
}

// The issuer of layer L (a whole warp, one elected lane issuing): its input rows in order,
// across the block's chunks; layer 0's warp stages its rows too.
template <int L>
__device__ __forceinline__ void net_issuer(const NetSmem& sm, uint32_t tmem, const __nv_bfloat16* __restrict__ feats,
                                           int H, int W, int chunk, int segs, int chunks_y, long total, int* err) {
    using namespace tc;
    constexpr int CI = L == 0 ? 16 : 32;
    constexpr int NR = L == 0 ? kNetRing0 : kNetRing;
    constexpr int ROWB = L == 0 ? kRowSw32Bytes : kRowSw64Bytes;
    uint64_t* full = L == 0 ? nullptr : sm.full + (L - 1) * kNetRing;
    uint64_t* rfree = L == 0 ? sm.rfree0 : sm.rfree + (L - 1) * kNetRing;
    uint64_t* done = sm.done + L * kNetDone;
    uint64_t* drained = sm.drained + L * kNetSlots;
    // swizzled K-major operands: SBO = one 8-row group (256 or 512 bytes), swizzle mode at bits
    // 61-63 (32B = 6, 64B = 4)
    const uint64_t A0 = L == 0 ? (sdesc(smem_addr(sm.ring0), 16, 256) | (6ull << 61))
                               : (sdesc(smem_addr(sm.ring + (L - 1) * kNetRing * kRowSw64Bytes), 16, 512) | (4ull << 61));
    const uint64_t B0 = L == 0 ? (sdesc(smem_addr(sm.sw0), 16, 256) | (6ull << 61))
                               : (sdesc(smem_addr(sm.sw1 + (L - 1) * kNetW1Bytes), 16, 512) | (4ull << 61));
    const uint32_t acc = tmem + (uint32_t)(L * 32 * kNetSlots);
    unsigned nb = 0, ob = 0;
    uint32_t fpar = 0, dused = 0, dpar = 0;
    bool fail = false;
    // layer 0: this warp also stages the feature rows into ring 0, kNetAhead rows ahead of the
    // one it issues (rows y0 - 4 .. y1 + 3 of each chunk, in order across the block's chunks)
    long cs = blockIdx.x;
    int ks = 0;
    unsigned staged = 0;
    uint32_t used0 = 0, rpar0 = 0;
    const int lane = threadIdx.x & 31;
    auto stage_next = [&]() -> bool {
        if (cs >= total) return true;
        const NetChunk sc = net_chunk_of(cs, H, chunk, segs, chunks_y);
        const int sl = (int)(staged % kNetRing0);
        if ((used0 >> sl) & 1u) {           // the MMAs of the slot's previous row must be complete
            if (!__all_sync(0xffffffffu, mbar_wait(&sm.rfree0[sl], (rpar0 >> sl) & 1u))) return false;
            rpar0 ^= 1u << sl;
        }
        used0 |= 1u << sl;
        tc_stage_row_sw32<32>(sm.ring0 + sl * kRowSw32Bytes, feats, sc.n, sc.y0 - 4 + ks, sc.s, H, W, lane);
        ++staged;
        if (++ks == sc.rows + 8) {
            ks = 0;
            cs += gridDim.x;
        }
        return true;
    };
    for (long c = blockIdx.x; c < total && !fail; c += gridDim.x) {
        const NetChunk ch = net_chunk_of(c, H, chunk, segs, chunks_y);
        const int nin = ch.rows + 8 - 2 * L, nout = nin - 2;
        for (int k = 0; k < nin; ++k) {
            const int sl = (int)(nb % NR);
            if constexpr (L == 0) {
                while (!fail && staged < nb + 1 + kNetAhead && cs < total) fail = !stage_next();
                if (fail) break;
                // row nb's copies have landed once at most staged - nb - 1 later groups are pending
                const unsigned later = staged - nb - 1;
                if (later >= 2) cp_async_wait<2>();
                else if (later == 1) cp_async_wait<1>();
                else cp_async_wait<0>();
                fence_proxy_async();
                __syncwarp();
            } else {
                fail = !__all_sync(0xffffffffu, mbar_wait(&full[sl], (fpar >> sl) & 1u));
                fpar ^= 1u << sl;
            }
            // output row k starts here: its slot's previous row must be drained
            if (!fail && k < nout) {
                const unsigned ts = (ob + (unsigned)k) % kNetSlots;
                if ((dused >> ts) & 1u) {
                    fail = !__all_sync(0xffffffffu, mbar_wait(&drained[ts], (dpar >> ts) & 1u));
                    dpar ^= 1u << ts;
                }
                dused |= 1u << ts;
            }
            if (fail) break;
            fence_after();
            // outputs lo .. hi take input k; output o uses kernel row dy = k - o, stored as
            // weight block 2 - dy
            const int lo = k - 2 > 0 ? k - 2 : 0, hi = k < nout - 1 ? k : nout - 1;
            net_issue_row<CI>(acc, A0 + (uint64_t)((sl * ROWB) >> 4), B0, 2 - k + lo, (ob + (unsigned)lo) % kNetSlots,
                              hi - lo + 1);
            if (k >= 2) commit_elect(&done[(ob + (unsigned)(k - 2)) % kNetDone]);
            commit_elect(&rfree[sl]);
            ++nb;
        }
        ob += (unsigned)nout;
    }
    if (L == 0) cp_async_wait<0>();
    if (fail && (threadIdx.x & 31) == 0) atomicOr(err, kErrWaitGaveUp);
    // the tensor memory is freed at the end: every MMA of the issuing lane must have completed
    if (nb > 0) {
        commit_elect(&sm.fin[L]);
        mbar_wait(&sm.fin[L], 0u);
    }
}

// Named barrier over the 128 threads of epilogue group g (ids 2..5), returning whether `ok`
// held for all of them.
__device__ __forceinline__ bool net_all_of_group(bool ok, int g) {
    uint32_t r;
    asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.u32 q, %1, 0;\n\tbar.red.and.pred p, %2, 128, q;\n\t"
                 "selp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(r) : "r"((uint32_t)ok), "r"(2 + g) : "memory");
    return r != 0;
}

// Epilogue state of one layer: output rows of earlier chunks, last-layer rows stored, and the
// use / parity bits of the next layer's ring slots.
struct NetEpi {
    unsigned ob, nst;
    uint32_t rused, rpar;
};

// Output row o of layer L in the chunk, by epilogue group g (thread lx = lane of tensor memory):
// once its MMAs completed, read and zero the accumulator slot, then bias and ReLU into the next
// layer's ring (zeros outside the image), or for the last layer the softmax, staged and stored
// in bulk (lanes 3 .. 124 of the segment).  False when a wait gave up.
template <int L>
__device__ __forceinline__ bool net_epi_item(const NetSmem& sm, NetEpi& e, const NetChunk& ch, int o, int g,
                                             uint32_t tmem, void* out, int H, int W, int lx, int* err) {
    using namespace tc;
    const unsigned oi = e.ob + (unsigned)o;
    bool ok = mbar_wait(&sm.done[L * kNetDone + oi % kNetDone], (oi / kNetDone) & 1u);
    const int q = (int)(oi % kNetRing);
    if (L < 3) {
        // the next layer's ring slot: the MMAs of its previous row must have completed
        if ((e.rused >> q) & 1u) {
            ok = mbar_wait(&sm.rfree[L * kNetRing + q], (e.rpar >> q) & 1u) && ok;
            e.rpar ^= 1u << q;
        }
        e.rused |= 1u << q;
    } else if (lx == 0) {
        bulk_wait_read<kNetOutBufs - 1>();   // the staging buffer is free
    }
    if (!net_all_of_group(ok, g)) {
        if (lx == 0) atomicOr(err, kErrWaitGaveUp);
        return false;
    }
    fence_after();
    const unsigned ts = oi % kNetSlots;
    const uint32_t ta = tmem + (uint32_t)(L * 32 * kNetSlots) + ts * 32u + ((uint32_t)((lx >> 5) * 32) << 16);
    uint32_t v[32];
    ld32(v, ta);
    st32_zero(ta);
    fence_before();
    mbar_arrive(&sm.drained[L * kNetSlots + ts]);
    const int x = ch.s + lx, y = ch.y0 - 3 + L + o;
    const float* bias = sm.bias + L * 32;
    float f[32];
#pragma unroll
    for (int j = 0; j < 32; ++j) f[j] = __uint_as_float(v[j]) + bias[j];
    if constexpr (L < 3) {
        uint4 st[4] = {make_uint4(0u, 0u, 0u, 0u), make_uint4(0u, 0u, 0u, 0u), make_uint4(0u, 0u, 0u, 0u),
                       make_uint4(0u, 0u, 0u, 0u)};
        if ((unsigned)x < (unsigned)W && (unsigned)y < (unsigned)H) tc_epilogue<0>(f, 0, 0, nullptr, nullptr, st);
        unsigned char* row = sm.ring + (L * kNetRing + q) * kRowSw64Bytes;
        const int px = lx + 1;
#pragma unroll
        for (int kg = 0; kg < 4; ++kg)
            *reinterpret_cast<uint4*>(row + px * 64 + ((kg ^ ((px >> 1) & 3)) << 4)) = st[kg];
        fence_proxy_async();
        mbar_arrive(&sm.full[L * kNetRing + q]);
    } else {
        uint4* buf = sm.so + (e.nst % kNetOutBufs) * tc::M * 4;
        tc_epilogue<3>(f, 0, 0, nullptr, nullptr, buf + lx * 4);
        fence_proxy_async();
        asm volatile("bar.sync 6, 128;" ::: "memory");
        if (lx == 0) {
            const int xs = ch.s + 3;
            const int nv = W - xs < kNetSeg ? W - xs : kNetSeg;
            if (nv > 0)
                bulk_s2g(reinterpret_cast<__half*>(out) + (((long)ch.n * H + y) * W + xs) * 32, buf + 3 * 4,
                         (uint32_t)(nv * 64));
        }
        ++e.nst;
    }
    return true;
}

__global__ void __launch_bounds__(kNetThreads, 1) k_kpn_net(const __nv_bfloat16* __restrict__ feats, NetWeights w,
                                                            void* out, int B, int H, int W, int chunk, int* err) {
    using namespace tc;
    extern __shared__ __align__(1024) unsigned char tc_smem[];
    NetSmem sm;
    sm.sw1 = tc_smem;
    sm.sw0 = tc_smem + kNetOffW0;
    sm.ring = tc_smem + kNetOffRing;
    sm.ring0 = tc_smem + kNetOffRing0;
    sm.so = reinterpret_cast<uint4*>(tc_smem + kNetOffOut);
    sm.bias = reinterpret_cast<float*>(tc_smem + kNetOffBias);
    sm.rfree0 = reinterpret_cast<uint64_t*>(tc_smem + kNetOffBar);
    sm.full = sm.rfree0 + kNetRing0;
    sm.rfree = sm.full + 3 * kNetRing;
    sm.done = sm.rfree + 3 * kNetRing;
    sm.drained = sm.done + 4 * kNetDone;
    sm.fin = sm.drained + 4 * kNetSlots;
    uint32_t* tslot = reinterpret_cast<uint32_t*>(sm.fin + 4);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // weights [tap][co][ci] -> per dx the 96 rows (2 - dy) * 32 + co, swizzled like the rows
    for (int i = tid; i < 9 * 32 * 2; i += kNetThreads) {
        const int kg = i % 2, co = (i / 2) % 32, tap = i / 64, dy = tap / 3, dx = tap % 3;
        const int r = (2 - dy) * 32 + co;
        *reinterpret_cast<uint4*>(sm.sw0 + dx * 96 * 32 + r * 32 + ((kg ^ ((r >> 2) & 1)) << 4)) =
            *reinterpret_cast<const uint4*>(w.wt[0] + ((long)tap * 32 + co) * 16 + kg * 8);
    }
    for (int i = tid; i < 3 * 9 * 32 * 4; i += kNetThreads) {
        const int l = i / (9 * 32 * 4), j = i % (9 * 32 * 4);
        const int kg = j % 4, co = (j / 4) % 32, tap = j / 128, dy = tap / 3, dx = tap % 3;
        const int r = (2 - dy) * 32 + co;
        *reinterpret_cast<uint4*>(sm.sw1 + l * kNetW1Bytes + dx * 96 * 64 + r * 64 + ((kg ^ ((r >> 1) & 3)) << 4)) =
            *reinterpret_cast<const uint4*>(w.wt[l + 1] + ((long)tap * 32 + co) * 32 + kg * 8);
    }
    for (int i = tid; i < 128; i += kNetThreads) sm.bias[i] = w.bias[i >> 5][i & 31];
    // pixels 0 and 129 of the epilogue-filled rows are never written (they reach only the lanes
    // a segment does not keep): zeros
    for (int i = tid; i < 3 * kNetRing * 2 * 4; i += kNetThreads) {
        const int slot = i / 8, px = (i / 4) % 2 ? 129 : 0, kg = i % 4;
        *reinterpret_cast<uint4*>(sm.ring + slot * kRowSw64Bytes + px * 64 + (kg << 4)) = make_uint4(0u, 0u, 0u, 0u);
    }
    if (tid == 0) {
        for (int r = 0; r < kNetRing0; ++r) mbar_init(&sm.rfree0[r]);
        for (int r = 0; r < 3 * kNetRing; ++r) {
            mbar_init(&sm.full[r], 128);
            mbar_init(&sm.rfree[r]);
        }
        for (unsigned i = 0; i < 4 * kNetDone; ++i) mbar_init(&sm.done[i]);
        for (unsigned i = 0; i < 4 * kNetSlots; ++i) mbar_init(&sm.drained[i], 128);
        for (int i = 0; i < 4; ++i) mbar_init(&sm.fin[i]);
    }
    if (warp == 0) tmem_alloc(tslot, 4 * 32 * kNetSlots);
    fence_proxy_async();
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = *tslot;
    if (warp < 4) {                    // every accumulator slot starts at zero
#pragma unroll 1
        for (unsigned sl = 0; sl < 4 * kNetSlots; ++sl) st32_zero(tmem + sl * 32u + ((uint32_t)(warp * 32) << 16));
    }
    fence_before();
    __syncthreads();
    fence_after();
    const int segs = (W + kNetSeg - 1) / kNetSeg, chunks_y = (H + chunk - 1) / chunk;
    const long total = (long)B * segs * chunks_y;

    if (warp >= 16) {
        // ---- the issuers, one warp a layer (one elected lane issues); warp 16 stages the features
        if (warp == 16) net_issuer<0>(sm, tmem, feats, H, W, chunk, segs, chunks_y, total, err);
        else if (warp == 17) net_issuer<1>(sm, tmem, feats, H, W, chunk, segs, chunks_y, total, err);
        else if (warp == 18) net_issuer<2>(sm, tmem, feats, H, W, chunk, segs, chunks_y, total, err);
        else net_issuer<3>(sm, tmem, feats, H, W, chunk, segs, chunks_y, total, err);
        __syncwarp();
    } else {
        // ---- the epilogues, warps 4l .. 4l + 3 for layer l, each output row in order
        const int g = warp >> 2, lx = (warp & 3) * 32 + lane;
        NetEpi e = {0, 0, 0, 0};
        bool ok = true;
        for (long c = blockIdx.x; c < total && ok; c += gridDim.x) {
            const NetChunk ch = net_chunk_of(c, H, chunk, segs, chunks_y);
            const int nout = ch.rows + 6 - 2 * g;
            for (int o = 0; o < nout && ok; ++o) {
                if (g == 0) ok = net_epi_item<0>(sm, e, ch, o, 0, tmem, out, H, W, lx, err);
                else if (g == 1) ok = net_epi_item<1>(sm, e, ch, o, 1, tmem, out, H, W, lx, err);
                else if (g == 2) ok = net_epi_item<2>(sm, e, ch, o, 2, tmem, out, H, W, lx, err);
                else ok = net_epi_item<3>(sm, e, ch, o, 3, tmem, out, H, W, lx, err);
            }
            e.ob += (unsigned)nout;
        }
        if (g == 3 && lx == 0) bulk_wait_all();
    }
    fence_before();
    __syncthreads();
    fence_after();
    if (warp == 0) tmem_dealloc(tmem, 4 * 32 * kNetSlots);
}

// ---- two layers in one kernel ------------------------------------------------------------------
// The network as two kernels of two layers each (layers 0-1, then 2-3): the first layer's output
// rows go from their drain straight into the second layer's ring in shared memory, so of the three
// activations only the second layer's output crosses HBM.  With two layers a block, each layer
// has 8 accumulator slots (2 x 8 x 32 = the SM's 512 tensor-memory columns) as in the per-layer
// kernel, so an output row's slot comes back 8 rows later, and each layer's rows are drained by
// two groups of four warps, even rows and odd rows, so that two drains of a layer overlap.
// Columns: both layers compute the lanes x = s + lane; the second layer is exact on lanes 1 ..
// 126, and segments start kPairSeg = 126 pixels apart (s = 126 seg - 1).  Rows: for the chunk's
// output rows y0 .. y1 - 1, the first layer reads rows y0 - 2 .. y1 + 1 and completes y0 - 1 ..
// y1; the second reads those and completes y0 .. y1 - 1.  Roles (18 warps): warp 16 stages the
// input rows (cp.async, kPairAhead rows ahead) and issues the first layer's MMAs, warp 17 the
// second's (one elected lane each); drain warps 4g .. 4g + 3 take layer g >> 1, the rows whose
// running index has parity g & 1.  Zeros outside the image, accumulation order and epilogues as
// in the per-layer kernel, so the results are its results bit for bit.
constexpr int kPairSeg = 126;
constexpr int kPairRingIn = 4, kPairAhead = 2;
constexpr int kPairRing = 4;                      // even: all rows of a slot have the same parity
constexpr unsigned kPairSlots = 8;
constexpr unsigned kPairDone = 8;
constexpr int kPairOutBufs = 2;                   // output staging buffers a second-layer group
constexpr int kPairThreads = 18 * 32;
static_assert(kPairRing % 2 == 0 && kPairSlots % 2 == 0 && kPairDone % 2 == 0, "row parity owns slots");
static_assert(kPairAhead < kPairRingIn && kPairAhead <= 2, "ring sizes");

template <int LF>
struct PairCfg {
    static constexpr int CI0 = LF == 0 ? 16 : 32;                       // first layer's inputs
    static constexpr int ROW0 = LF == 0 ? kRowSw32Bytes : kRowSw64Bytes;
    static constexpr int W0B = 3 * 96 * CI0 * 2, W1B = 3 * 96 * 64;
    static constexpr int OFF_W0 = W1B;
    static constexpr int OFF_RIN = OFF_W0 + W0B;
    static constexpr int OFF_RMID = OFF_RIN + kPairRingIn * ROW0;
    static constexpr int OFF_OUT = OFF_RMID + kPairRing * kRowSw64Bytes;
    static constexpr int OFF_BIAS = OFF_OUT + 2 * kPairOutBufs * tc::M * 64;
    static constexpr int OFF_BAR = OFF_BIAS + 2 * 32 * 4;
    static constexpr int NBARS = kPairRingIn + 2 * kPairRing + 2 * (int)kPairDone + 2 * (int)kPairSlots + 2;
    static constexpr int SMEM_USED = OFF_BAR + NBARS * 8 + 8;
    // at least 120 KB, so that one block holds an SM (and its 512 tensor-memory columns)
    static constexpr int SMEM = SMEM_USED > 120 * 1024 ? SMEM_USED : 120 * 1024;
    static_assert(OFF_RIN % 512 == 0 && OFF_RMID % 512 == 0 && OFF_OUT % 16 == 0, "ring alignment");
};

struct PairSmem {
    unsigned char *rin, *rmid, *sw0, *sw1;
    uint4* so;                 // [2 groups][kPairOutBufs][M][64 B]
    float* bias;               // [2][32]
    uint64_t *rfree_in, *full, *rfree, *done, *drained, *fin;
};

__device__ __forceinline__ NetChunk pair_chunk_of(long c, int H, int chunk, int segs, int chunks_y) {
    NetChunk ch;
    ch.n = (int)(c / ((long)segs * chunks_y));
    const int rc = (int)(c - (long)ch.n * segs * chunks_y);
    const int seg = rc / chunks_y;
    ch.y0 = (rc - seg * chunks_y) * chunk;
    ch.rows = (ch.y0 + chunk < H ? ch.y0 + chunk : H) - ch.y0;
    ch.s = seg * kPairSeg - 1;
    return ch;
}

// The MMAs of one input row (CI input channels) into accumulator slots s0.. of a ring of
// kPairSlots (two MMAs when the triple wraps).
template <int CI>
__device__ __forceinline__ void pair_issue_row(uint32_t acc, uint64_t arow, uint64_t B0, int blk0, unsigned s0,
                                               int nblk) {
    using namespace tc;
    constexpr int RB = CI * 2;
    const int first = nblk < (int)(kPairSlots - s0) ? nblk : (int)(kPairSlots - s0);
    const uint32_t id1 = idesc_n(32u * first), id2 = idesc_n(32u * (nblk - first));
#pragma unroll
    for (int dx = 0; dx < 3; ++dx)
#pragma unroll
        for (int kc = 0; kc < CI / 16; ++kc) {
            const uint64_t a = arow + (uint64_t)((dx * RB + kc * 32) >> 4);
            const uint64_t bb = B0 + (uint64_t)((dx * 96 * RB + blk0 * 32 * RB + kc * 32) >> 4);
            mma_elect(acc + s0 * 32u, a, bb, id1);
            if (first < nblk) mma_elect(acc, a, bb + (uint64_t)((first * 32 * RB) >> 4), id2);
        }
}

// The issuer of layer J of the pair (a whole warp, one elected lane issuing); J = 0 also stages
// the input rows (rows y0 - 2 .. y1 + 1 of each chunk, kPairAhead rows ahead).
template <int LF, int J>
__device__ __forceinline__ void pair_issuer(const PairSmem& sm, uint32_t tmem, const __nv_bfloat16* __restrict__ in,
                                            int H, int W, int chunk, int segs, int chunks_y, long total, int* err) {
    using namespace tc;
    using C = PairCfg<LF>;
    constexpr int CI = J == 0 ? C::CI0 : 32;
    constexpr int NR = J == 0 ? kPairRingIn : kPairRing;
    constexpr int ROWB = J == 0 ? C::ROW0 : kRowSw64Bytes;
    constexpr uint64_t MODE = CI == 16 ? 6ull : 4ull;   // 32-byte / 64-byte swizzle
    constexpr uint32_t SBO = CI == 16 ? 256u : 512u;
    uint64_t* rfree = J == 0 ? sm.rfree_in : sm.rfree;
    uint64_t* done = sm.done + J * kPairDone;
    uint64_t* drained = sm.drained + J * kPairSlots;
    const uint64_t A0 = sdesc(smem_addr(J == 0 ? sm.rin : sm.rmid), 16, SBO) | (MODE << 61);
    const uint64_t B0 = sdesc(smem_addr(J == 0 ? sm.sw0 : sm.sw1), 16, SBO) | (MODE << 61);
    const uint32_t acc = tmem + (uint32_t)(J * 32 * kPairSlots);
    unsigned nb = 0, ob = 0;
    uint32_t fpar = 0, dused = 0, dpar = 0;
    bool fail = false;
    long cs = blockIdx.x;
    int ks = 0;
    unsigned staged = 0;
    uint32_t used0 = 0, rpar0 = 0;
    const int lane = threadIdx.x & 31;
    auto stage_next = [&]() -> bool {
        if (cs >= total) return true;
        const NetChunk sc = pair_chunk_of(cs, H, chunk, segs, chunks_y);
        const int sl = (int)(staged % kPairRingIn);
        if ((used0 >> sl) & 1u) {           // the MMAs of the slot's previous row must be complete
            if (!__all_sync(0xffffffffu, mbar_wait(&sm.rfree_in[sl], (rpar0 >> sl) & 1u))) return false;
            rpar0 ^= 1u << sl;
        }
        used0 |= 1u << sl;
        if constexpr (C::CI0 == 16) tc_stage_row_sw32<32>(sm.rin + sl * C::ROW0, in, sc.n, sc.y0 - 2 + ks, sc.s, H, W, lane);
        else tc_stage_row_sw64<32>(sm.rin + sl * C::ROW0, in, sc.n, sc.y0 - 2 + ks, sc.s, H, W, lane);
        ++staged;
        if (++ks == sc.rows + 4) {
            ks = 0;
            cs += gridDim.x;
        }
        return true;
    };
    for (long c = blockIdx.x; c < total && !fail; c += gridDim.x) {
        const NetChunk ch = pair_chunk_of(c, H, chunk, segs, chunks_y);
        const int nin = ch.rows + 4 - 2 * J, nout = nin - 2;
        for (int k = 0; k < nin; ++k) {
            const int sl = (int)(nb % NR);
            if constexpr (J == 0) {
                while (!fail && staged < nb + 1 + kPairAhead && cs < total) fail = !stage_next();
                if (fail) break;
                // row nb's copies have landed once at most staged - nb - 1 later groups are pending
                const unsigned later = staged - nb - 1;
                if (later >= 2) cp_async_wait<2>();
                else if (later == 1) cp_async_wait<1>();
                else cp_async_wait<0>();
                fence_proxy_async();
                __syncwarp();
            } else {
                fail = !__all_sync(0xffffffffu, mbar_wait(&sm.full[sl], (fpar >> sl) & 1u));
                fpar ^= 1u << sl;
            }
            // output row k starts here: its slot's previous row must be drained
            if (!fail && k < nout) {
                const unsigned ts = (ob + (unsigned)k) % kPairSlots;
                if ((dused >> ts) & 1u) {
                    fail = !__all_sync(0xffffffffu, mbar_wait(&drained[ts], (dpar >> ts) & 1u));
                    dpar ^= 1u << ts;
                }
                dused |= 1u << ts;
            }
            if (fail) break;
            fence_after();
            // outputs lo .. hi take input k; output o uses kernel row dy = k - o, stored as
            // weight block 2 - dy
            const int lo = k - 2 > 0 ? k - 2 : 0, hi = k < nout - 1 ? k : nout - 1;
            pair_issue_row<CI>(acc, A0 + (uint64_t)((sl * ROWB) >> 4), B0, 2 - k + lo, (ob + (unsigned)lo) % kPairSlots,
                               hi - lo + 1);
            if (k >= 2) commit_elect(&done[(ob + (unsigned)(k - 2)) % kPairDone]);
            commit_elect(&rfree[sl]);
            ++nb;
        }
        ob += (unsigned)nout;
    }
    if (J == 0) cp_async_wait<0>();
    if (fail && lane == 0) atomicOr(err, kErrWaitGaveUp);
    // the tensor memory is freed at the end: every MMA of the issuing lane must have completed
    if (nb > 0) {
        commit_elect(&sm.fin[J]);
        mbar_wait(&sm.fin[J], 0u);
    }
}

// Drain state of one group: output rows of earlier chunks, second-layer rows stored, and the use /
// parity bits of the second layer's ring slots it writes.
struct PairEpi {
    unsigned ob, nst;
    uint32_t rused, rpar;
};

// Output row o of pair layer J (running index oi, parity P) by drain group g: once its MMAs
// completed, read and zero the accumulator slot; the first layer's row goes (bias, ReLU, BF16,
// zeros outside the image) into the second layer's ring; the second layer's row is staged and
// stored in bulk (lanes 1 .. 126): bias, ReLU, BF16 for layer 1, the softmax as FP16 for layer
// 3.  False when a wait gave up.
template <int LF, int J>
__device__ __forceinline__ bool pair_epi_item(const PairSmem& sm, PairEpi& e, const NetChunk& ch, int o, int g,
                                              uint32_t tmem, void* out, int H, int W, int lx, int* err) {
    using namespace tc;
    const unsigned oi = e.ob + (unsigned)o;
    bool ok = mbar_wait(&sm.done[J * kPairDone + oi % kPairDone], (oi / kPairDone) & 1u);
    const int q = (int)(oi % kPairRing);
    if (J == 0) {
        if ((e.rused >> q) & 1u) {           // the MMAs of the slot's previous row must be complete
            ok = mbar_wait(&sm.rfree[q], (e.rpar >> q) & 1u) && ok;
            e.rpar ^= 1u << q;
        }
        e.rused |= 1u << q;
    } else if (lx == 0) {
        bulk_wait_read<kPairOutBufs - 1>();   // the staging buffer is free
    }
    if (!net_all_of_group(ok, g)) {
        if (lx == 0) atomicOr(err, kErrWaitGaveUp);
        return false;
    }
    fence_after();
    const unsigned ts = oi % kPairSlots;
    const uint32_t ta = tmem + (uint32_t)(J * 32 * kPairSlots) + ts * 32u + ((uint32_t)((lx >> 5) * 32) << 16);
    uint32_t v[32];
    ld32(v, ta);
    st32_zero(ta);
    fence_before();
    mbar_arrive(&sm.drained[J * kPairSlots + ts]);
    const int x = ch.s + lx, y = ch.y0 - 1 + J + o;
    const float* bias = sm.bias + J * 32;
    float f[32];
#pragma unroll
    for (int j = 0; j < 32; ++j) f[j] = __uint_as_float(v[j]) + bias[j];
    if constexpr (J == 0) {
        uint4 st[4] = {make_uint4(0u, 0u, 0u, 0u), make_uint4(0u, 0u, 0u, 0u), make_uint4(0u, 0u, 0u, 0u),
                       make_uint4(0u, 0u, 0u, 0u)};
        if ((unsigned)x < (unsigned)W && (unsigned)y < (unsigned)H) tc_epilogue<0>(f, 0, 0, nullptr, nullptr, st);
        unsigned char* row = sm.rmid + q * kRowSw64Bytes;
        const int px = lx + 1;
#pragma unroll
        for (int kg = 0; kg < 4; ++kg)
            *reinterpret_cast<uint4*>(row + px * 64 + ((kg ^ ((px >> 1) & 3)) << 4)) = st[kg];
        fence_proxy_async();
        mbar_arrive(&sm.full[q]);
    } else {
        const int p = g & 1;
        uint4* buf = sm.so + (p * kPairOutBufs + e.nst % kPairOutBufs) * tc::M * 4;
        if constexpr (LF == 0) tc_epilogue<0>(f, 0, 0, nullptr, nullptr, buf + lx * 4);
        else tc_epilogue<3>(f, 0, 0, nullptr, nullptr, buf + lx * 4);
        fence_proxy_async();
        if (p == 0) asm volatile("bar.sync 6, 128;" ::: "memory");
        else asm volatile("bar.sync 7, 128;" ::: "memory");
        if (lx == 0) {
            const int xs = ch.s + 1;
            const int nv = W - xs < kPairSeg ? W - xs : kPairSeg;
            if (nv > 0)
                bulk_s2g(reinterpret_cast<__nv_bfloat16*>(out) + (((long)ch.n * H + y) * W + xs) * 32, buf + 1 * 4,
                         (uint32_t)(nv * 64));
        }
        ++e.nst;
    }
    return true;
}

template <int LF>
__global__ void __launch_bounds__(kPairThreads, 1) k_kpn_pair(const __nv_bfloat16* __restrict__ in,
                                                              const __nv_bfloat16* __restrict__ w0,
                                                              const __nv_bfloat16* __restrict__ w1,
                                                              const float* __restrict__ b0, const float* __restrict__ b1,
                                                              void* out, int B, int H, int W, int chunk, int* err) {
    using namespace tc;
    using C = PairCfg<LF>;
    extern __shared__ __align__(1024) unsigned char tc_smem[];
    PairSmem sm;
    sm.sw1 = tc_smem;
    sm.sw0 = tc_smem + C::OFF_W0;
    sm.rin = tc_smem + C::OFF_RIN;
    sm.rmid = tc_smem + C::OFF_RMID;
    sm.so = reinterpret_cast<uint4*>(tc_smem + C::OFF_OUT);
    sm.bias = reinterpret_cast<float*>(tc_smem + C::OFF_BIAS);
    sm.rfree_in = reinterpret_cast<uint64_t*>(tc_smem + C::OFF_BAR);
    sm.full = sm.rfree_in + kPairRingIn;
    sm.rfree = sm.full + kPairRing;
    sm.done = sm.rfree + kPairRing;
    sm.drained = sm.done + 2 * kPairDone;
    sm.fin = sm.drained + 2 * kPairSlots;
    uint32_t* tslot = reinterpret_cast<uint32_t*>(sm.fin + 2);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // weights [tap][co][ci] -> per dx the 96 rows (2 - dy) * 32 + co, swizzled like the rows
    constexpr int KG0 = C::CI0 / 8;
    for (int i = tid; i < 9 * 32 * KG0; i += kPairThreads) {
        const int kg = i % KG0, co = (i / KG0) % 32, tap = i / (KG0 * 32), dy = tap / 3, dx = tap % 3;
        const int r = (2 - dy) * 32 + co;
        const int off = C::CI0 == 32 ? dx * 96 * 64 + r * 64 + ((kg ^ ((r >> 1) & 3)) << 4)
                                     : dx * 96 * 32 + r * 32 + ((kg ^ ((r >> 2) & 1)) << 4);
        *reinterpret_cast<uint4*>(sm.sw0 + off) = *reinterpret_cast<const uint4*>(w0 + ((long)tap * 32 + co) * C::CI0 + kg * 8);
    }
    for (int i = tid; i < 9 * 32 * 4; i += kPairThreads) {
        const int kg = i % 4, co = (i / 4) % 32, tap = i / 128, dy = tap / 3, dx = tap % 3;
        const int r = (2 - dy) * 32 + co;
        *reinterpret_cast<uint4*>(sm.sw1 + dx * 96 * 64 + r * 64 + ((kg ^ ((r >> 1) & 3)) << 4)) =
            *reinterpret_cast<const uint4*>(w1 + ((long)tap * 32 + co) * 32 + kg * 8);
    }
    for (int i = tid; i < 64; i += kPairThreads) sm.bias[i] = i < 32 ? b0[i] : b1[i - 32];
    // pixels 0 and 129 of the second layer's ring rows are never written (they reach only lanes
    // 0 and 127, which a segment does not keep): zeros
    for (int i = tid; i < kPairRing * 2 * 4; i += kPairThreads) {
        const int slot = i / 8, px = (i / 4) % 2 ? 129 : 0, kg = i % 4;
        *reinterpret_cast<uint4*>(sm.rmid + slot * kRowSw64Bytes + px * 64 + (kg << 4)) = make_uint4(0u, 0u, 0u, 0u);
    }
    if (tid == 0) {
        for (int r = 0; r < kPairRingIn; ++r) mbar_init(&sm.rfree_in[r]);
        for (int r = 0; r < kPairRing; ++r) {
            mbar_init(&sm.full[r], 128);
            mbar_init(&sm.rfree[r]);
        }
        for (unsigned i = 0; i < 2 * kPairDone; ++i) mbar_init(&sm.done[i]);
        for (unsigned i = 0; i < 2 * kPairSlots; ++i) mbar_init(&sm.drained[i], 128);
        for (int i = 0; i < 2; ++i) mbar_init(&sm.fin[i]);
    }
    if (warp == 0) tmem_alloc(tslot, 2 * 32 * kPairSlots);
    fence_proxy_async();
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = *tslot;
    if (warp < 4) {                    // every accumulator slot starts at zero
#pragma unroll 1
        for (unsigned sl = 0; sl < 2 * kPairSlots; ++sl) st32_zero(tmem + sl * 32u + ((uint32_t)(warp * 32) << 16));
    }
    fence_before();
    __syncthreads();
    fence_after();
    const int segs = (W + kPairSeg - 1) / kPairSeg, chunks_y = (H + chunk - 1) / chunk;
    const long total = (long)B * segs * chunks_y;
    if (warp >= 16) {
        if (warp == 16) pair_issuer<LF, 0>(sm, tmem, in, H, W, chunk, segs, chunks_y, total, err);
        else pair_issuer<LF, 1>(sm, tmem, in, H, W, chunk, segs, chunks_y, total, err);
        __syncwarp();
    } else {
        // drain groups: warps 4g .. 4g + 3 take layer g >> 1, rows of running parity g & 1
        const int g = warp >> 2, lx = (warp & 3) * 32 + lane, j = g >> 1, par = g & 1;
        PairEpi e = {0, 0, 0, 0};
        bool ok = true;
        for (long c = blockIdx.x; c < total && ok; c += gridDim.x) {
            const NetChunk ch = pair_chunk_of(c, H, chunk, segs, chunks_y);
            const int nout = ch.rows + 2 - 2 * j;
            for (int o = 0; o < nout && ok; ++o) {
                if (((e.ob + (unsigned)o) & 1u) != (unsigned)par) continue;
                if (j == 0) ok = pair_epi_item<LF, 0>(sm, e, ch, o, g, tmem, out, H, W, lx, err);
                else ok = pair_epi_item<LF, 1>(sm, e, ch, o, g, tmem, out, H, W, lx, err);
            }
            e.ob += (unsigned)nout;
        }
        if (j == 1 && lx == 0) bulk_wait_all();
    }
    fence_before();
    __syncthreads();
    fence_after();
    if (warp == 0) tmem_dealloc(tmem, 2 * 32 * kPairSlots);
}

// Weight and bias gradient of one layer: dW[co][tap][ci] += sum_p dZ[p][co] X[p + off(tap)][ci] and
// db[co] += sum_p dZ[p][co], over co < co_real, ci < ci_real (the padded channels carry no
// parameters), on the tensor cores (tcgen05).  The reduction runs over pixels, so both operands
// are read MN-major straight from the staged rows: 16 pixels of an X row are K, and M = 128 covers
// (dx, ci) because the descriptor's stride between channel groups is one pixel (the groups past
// dx = 2 are not used).  N = 96 covers (dy, co): the three dZ rows that X row r meets, r - 1, r and
// r + 1, which carry dy = 2, 1, 0.  One product of 16 pixels is thus 9 x 32 x CI of the gradient's
// sums, and they stay in tensor memory over all of a block's rows (in kWgSets interleaved sets,
// so that a sum's chain of additions stays short).
//
// A block walks chunks of X rows down one 128-pixel column of an image (two blocks a SM):
//   warp 5, the producer: X rows (130 pixels) and dZ rows (128) into two rings by TMA, zeros
//     outside the image from the tensor maps; dZ runs one row ahead and behind the chunk;
//   warp 4, the issuer (the whole warp walks the rows, one elected lane issues);
//   warps 0-3: the bias sums, from each staged dZ row of the chunk (a pixel a thread, its 32 sums
//     in registers), and at the end the accumulators, one atomic add an entry and block.
// They meet at mbarriers, waited for phase by phase as in k_conv3x3_tc: fullX / fullD (the row
// landed) -> issuer, bias warps; freeX (commit) and freeD (commit of the last X row that meets it,
// and one arrival a bias warp) -> the producer.  Slots follow running counts.
// 16 crops of 256 x 256, 32 -> 32 channels: 124 + 26 us (mma.sync and a
// separate bias sum) -> 40 us; layer 0, 10 -> 32 channels, 102 + 26 -> 39 us.  The products take 12
// us of that and the operands' bytes 20 us of HBM; the rest is the row hand-offs and the blocks'
// start and end.
constexpr int kWgXRing = 4, kWgDRing = 6;
constexpr unsigned kWgSets = 2;
constexpr int kWgThreads = 192;
constexpr int kWgDRow = tc::M * 64;                  // a staged dZ row: 128 pixels x 32 channels
template <int CI>
struct WgradCfg {
    static constexpr int XROW = CI == 32 ? kRowSw64Bytes : kRowSw32Bytes;
    static constexpr int OFF_D = kWgXRing * XROW;
    static constexpr int OFF_BIAS = OFF_D + kWgDRing * kWgDRow;      // [4][32] floats
    static constexpr int OFF_BAR = OFF_BIAS + 4 * 32 * 4;
    static constexpr int BARS = 2 * kWgXRing + 2 * kWgDRing + 1;
    static constexpr int SMEM = OFF_BAR + BARS * 8 + 8;
    static_assert(OFF_D % 512 == 0 && kWgDRow % 512 == 0, "row slots on swizzle boundaries");
};

template <int CI>
__global__ void __launch_bounds__(kWgThreads, 2) k_wgrad(const __grid_constant__ CUtensorMap xmap,
                                                         const __grid_constant__ CUtensorMap dmap, float* dW, float* db,
                                                         int B, int H, int W, int chunk, int ci_real, int co_real,
                                                         int* err) {
    using namespace tc;
    using Cfg = WgradCfg<CI>;
    constexpr int RB = CI * 2;
    extern __shared__ __align__(1024) unsigned char wg_smem[];
    unsigned char *sx = wg_smem, *sd = wg_smem + Cfg::OFF_D;
    float* sbias = reinterpret_cast<float*>(wg_smem + Cfg::OFF_BIAS);
    uint64_t* full_x = reinterpret_cast<uint64_t*>(wg_smem + Cfg::OFF_BAR);
    uint64_t *free_x = full_x + kWgXRing, *full_d = free_x + kWgXRing, *free_d = full_d + kWgDRing;
    uint64_t* fin = free_d + kWgDRing;
    uint32_t* tslot = reinterpret_cast<uint32_t*>(fin + 1);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) {
        for (int i = 0; i < kWgXRing; ++i) {
            mbar_init(&full_x[i]);
            mbar_init(&free_x[i]);
        }
        for (int i = 0; i < kWgDRing; ++i) {
            mbar_init(&full_d[i]);
            mbar_init(&free_d[i], 1 + 4);
        }
        mbar_init(fin);
    }
    pdl_wait();                                      // before the tensor memory, as in k_conv3x3_tc
    if (warp == 0) tmem_alloc(tslot, 128 * kWgSets);
    fence_proxy_async();
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = *tslot;
    if (warp < 4) {                                  // every sum starts at zero
#pragma unroll 1
        for (unsigned c = 0; c < 128 * kWgSets; c += 32) st32_zero(tmem + c + ((uint32_t)(warp * 32) << 16));
    }
    fence_before();
    __syncthreads();
    fence_after();
    const int segs = (W + M - 1) / M, chunks_y = (H + chunk - 1) / chunk;
    const long total = (long)B * segs * chunks_y;
    struct Chunk {
        int n, x0, y0, rows;
    };
    auto chunk_of = [&](long c) {
        Chunk k;
        k.n = (int)(c / ((long)segs * chunks_y));
        const int rc = (int)(c - (long)k.n * segs * chunks_y), seg = rc / chunks_y;
        k.x0 = seg * M;
        k.y0 = (rc - seg * chunks_y) * chunk;
        k.rows = (k.y0 + chunk < H ? k.y0 + chunk : H) - k.y0;
        return k;
    };

    if (warp == 5) {
        // ---- the producer
        constexpr uint32_t kXTx = (uint32_t)HP * RB, kDTx = (uint32_t)kWgDRow;
        unsigned nx = 0, nd = 0;                     // rows staged so far
        uint32_t usedx = 0, usedd = 0, px = 0, pd = 0;   // per slot: used before, parity of its next free phase
        uint32_t fx = 0, fd = 0;                     // per slot: parity of the next copy's phase
        bool ok = true;
        auto stage_x = [&](const Chunk& k, int row) {
            const int sl = (int)(nx++ % kWgXRing);
            if ((usedx >> sl) & 1u) {
                ok = __all_sync(0xffffffffu, mbar_wait(&free_x[sl], (px >> sl) & 1u));
                px ^= 1u << sl;
                if (!ok) return;
            }
            usedx |= 1u << sl;
            fx ^= 1u << sl;
            if (lane == 0) {
                mbar_arrive_expect_tx(&full_x[sl], kXTx);
                tma_load_4d(sx + sl * Cfg::XROW, &xmap, 0, k.x0 - 1, row, k.n, &full_x[sl]);
            }
            __syncwarp();
        };
        auto stage_d = [&](const Chunk& k, int row) {
            const int sl = (int)(nd++ % kWgDRing);
            if ((usedd >> sl) & 1u) {
                ok = __all_sync(0xffffffffu, mbar_wait(&free_d[sl], (pd >> sl) & 1u));
                pd ^= 1u << sl;
                if (!ok) return;
            }
            usedd |= 1u << sl;
            fd ^= 1u << sl;
            if (lane == 0) {
                mbar_arrive_expect_tx(&full_d[sl], kDTx);
                tma_load_4d(sd + sl * kWgDRow, &dmap, 0, k.x0, row, k.n, &full_d[sl]);
            }
            __syncwarp();
        };
        for (long c = blockIdx.x; c < total && ok; c += gridDim.x) {
            const Chunk k = chunk_of(c);
            stage_d(k, k.y0 - 1);
            if (ok) stage_d(k, k.y0);
            for (int i = 0; i < k.rows && ok; ++i) {
                stage_x(k, k.y0 + i);
                if (ok) stage_d(k, k.y0 + i + 1);
            }
        }
        // the block's shared memory is released at its end: every copy issued must have landed
        for (int sl = 0; sl < kWgXRing; ++sl)
            if ((usedx >> sl) & 1u) mbar_wait(&full_x[sl], ((fx >> sl) & 1u) ^ 1u);
        for (int sl = 0; sl < kWgDRing; ++sl)
            if ((usedd >> sl) & 1u) mbar_wait(&full_d[sl], ((fd >> sl) & 1u) ^ 1u);
        if (!ok && lane == 0) atomicOr(err, kErrWaitGaveUp);
    } else if (warp == 4) {
        // ---- the issuer: both operands MN-major (descriptor bits 15 and 16).  A: channel groups of
        // one pixel's CI channels, one pixel apart (LBO), 8-pixel groups along K (SBO).  B: one dZ
        // row's 32 channels a group, rows a slot apart.
        const uint32_t mn = (1u << 15) | (1u << 16);
        const uint64_t A0 = sdesc(smem_addr(sx), RB, 8 * RB) | ((CI == 32 ? 4ull : 6ull) << 61);
        const uint64_t B0 = sdesc(smem_addr(sd), kWgDRow, 512) | (4ull << 61);
        unsigned nx = 0, nd = 0;                     // X rows issued; dZ row i = 0 of the chunk
        uint32_t px = 0, pd = 0;                     // per slot: parity of the next full phase
        bool ok = true, any = false;
        for (long c = blockIdx.x; c < total && ok; c += gridDim.x) {
            const Chunk k = chunk_of(c);
            const int kcs = ((W - k.x0 < M ? W - k.x0 : M) + 15) / 16;   // 16-pixel products a row
            for (int i = 0; i < k.rows && ok; ++i) {
                // dZ rows i .. i + 2 of the chunk meet X row i; the first X row waits for three
                for (int j = i == 0 ? 0 : 2; j <= 2 && ok; ++j) {
                    const int sl = (int)((nd + i + j) % kWgDRing);
                    ok = __all_sync(0xffffffffu, mbar_wait(&full_d[sl], (pd >> sl) & 1u));
                    pd ^= 1u << sl;
                }
                const int sl = (int)(nx % kWgXRing);
                if (ok) ok = __all_sync(0xffffffffu, mbar_wait(&full_x[sl], (px >> sl) & 1u));
                px ^= 1u << sl;
                if (!ok) break;
                fence_after();
                const int s0 = (int)((nd + i) % kWgDRing), first = kWgDRing - s0 < 3 ? kWgDRing - s0 : 3;
                const uint32_t id1 = idesc_n(32u * first) | mn, id2 = idesc_n(32u * (3 - first)) | mn;
                const uint32_t acc = tmem + (nx % kWgSets) * 128u;
                for (int kc = 0; kc < kcs; ++kc) {
                    const uint64_t a = A0 + (uint64_t)((sl * Cfg::XROW + kc * 16 * RB) >> 4);
                    mma_elect(acc, a, B0 + (uint64_t)((s0 * kWgDRow + kc * 16 * 64) >> 4), id1);
                    if (first < 3) mma_elect(acc + 32u * first, a, B0 + (uint64_t)((kc * 16 * 64) >> 4), id2);
                }
                any = true;
                commit_elect(&free_x[sl]);
                commit_elect(&free_d[s0]);
                if (i == k.rows - 1) {               // the chunk's last two dZ rows are done too
                    commit_elect(&free_d[(nd + i + 1) % kWgDRing]);
                    commit_elect(&free_d[(nd + i + 2) % kWgDRing]);
                }
                ++nx;
            }
            nd += (unsigned)k.rows + 2;
        }
        if (!ok && lane == 0) atomicOr(err, kErrWaitGaveUp);
        // the sums are read and the tensor memory freed below: every MMA must have completed
        if (any) {
            commit_elect(fin);
            mbar_wait(fin, 0u);
        }
        __syncwarp();
    } else {
        // ---- the bias sums: thread t adds up pixel t of every dZ row of its chunks
        float bs[32];
#pragma unroll
        for (int j = 0; j < 32; ++j) bs[j] = 0.f;
        unsigned nd = 0;
        uint32_t pd = 0;
        bool ok = true;
        for (long c = blockIdx.x; c < total && ok; c += gridDim.x) {
            const Chunk k = chunk_of(c);
            for (int j = 0; j < k.rows + 2; ++j, ++nd) {
                const int sl = (int)(nd % kWgDRing);
                ok = __all_sync(0xffffffffu, mbar_wait(&full_d[sl], (pd >> sl) & 1u));
                pd ^= 1u << sl;
                if (!ok) break;
                if (j >= 1 && j <= k.rows) {         // the halo rows belong to the neighbouring chunks
                    const unsigned char* row = sd + sl * kWgDRow + tid * 64;
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const uint4 v = *reinterpret_cast<const uint4*>(row + ((q ^ ((tid >> 1) & 3)) << 4));
                        const unsigned u[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                        for (int h = 0; h < 4; ++h) {
                            bs[8 * q + 2 * h] += __uint_as_float(u[h] << 16);
                            bs[8 * q + 2 * h + 1] += __uint_as_float(u[h] & 0xffff0000u);
                        }
                    }
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(&free_d[sl]);
            }
        }
        if (!ok && lane == 0) atomicOr(err, kErrWaitGaveUp);
#pragma unroll
        for (int j = 0; j < 32; ++j) {
            float v = bs[j];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if (lane == 0) sbias[warp * 32 + j] = v;
        }
    }
    fence_before();
    __syncthreads();
    fence_after();
    if (warp < 4) {
        // accumulator lane = (dx, ci), column = (2 - dy, co)
        if (tid < co_real) atomicAdd(&db[tid], (sbias[tid] + sbias[32 + tid]) + (sbias[64 + tid] + sbias[96 + tid]));
        const int m = warp * 32 + lane, dx = m / CI, ci = m % CI;
        if (warp * 32 < 3 * CI) {
#pragma unroll 1
            for (int blk = 0; blk < 3; ++blk) {
                float sum[32];
#pragma unroll
                for (int j = 0; j < 32; ++j) sum[j] = 0.f;
#pragma unroll 1
                for (unsigned st = 0; st < kWgSets; ++st) {
                    uint32_t v[32];
                    ld32(v, tmem + st * 128u + blk * 32u + ((uint32_t)(warp * 32) << 16));
#pragma unroll
                    for (int j = 0; j < 32; ++j) sum[j] += __uint_as_float(v[j]);
                }
                if (dx < 3 && ci < ci_real) {
                    const int tap = (2 - blk) * 3 + dx;
#pragma unroll
                    for (int co = 0; co < 32; ++co)
                        if (co < co_real) atomicAdd(&dW[((long)co * 9 + tap) * ci_real + ci], sum[co]);
                }
            }
        }
    }
    fence_before();
    __syncthreads();
    fence_after();
    if (warp == 0) tmem_dealloc(tmem, 128 * kWgSets);
}

// ---------------------------------------------------------------- softmax + kernel application

// A kernel application: c_out(p) = sum_i K_i(p) c_in(p + D o_i) / sum_{i in image} K_i(p).  A block
// of 32 x 8 threads takes 32 x 16 pixels (two a thread) and first copies their colour taps' window
// (the tile with a margin of 2 D) into shared memory, so that each of the 25 taps is read from
// there rather than through L1: at dilation 4 the taps reach 8 pixels away and L1 serves few of
// them.  k_apply_h takes the kernels as FP16, pixel-major (Kh[p][32], the first 25 used; conv
// EPI 3), k_apply as FP32 planes (K[i][p]; conv EPI 1).

// The 25 FP16 kernel weights of pixel p (pixel-major, 64 bytes: 25 used) as floats.
__device__ __forceinline__ void load_kernel_h(const uint4* __restrict__ Kh, long p, float (&kv)[32]) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const uint4 u = __ldg(&Kh[p * 4 + q]);
        const unsigned w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            const float2 f = unpack_f16(w[h]);
            kv[8 * q + 2 * h] = f.x;
            kv[8 * q + 2 * h + 1] = f.y;
        }
    }
}

// One kernel application at pixel (x, y), dilation D: the K-weighted mean of the in-image taps
// (x + D kx, y + D ky), renormalised over them, and the sum of their weights (w); the colours come
// from a shared-memory window `win` (pitch `pitch` float4) whose element (wx, wy) is the pixel
// (x, y).
template <int D>
__device__ __forceinline__ float4 apply_taps(const float (&kv)[32], const float4* win, int pitch, int wx, int wy,
                                             int x, int y, int W, int H) {
    float s = 0.f, r = 0.f, g = 0.f, b = 0.f;
#pragma unroll
    for (int ky = -2; ky <= 2; ++ky)
#pragma unroll
        for (int kx = -2; kx <= 2; ++kx) {
            const int qx = x + D * kx, qy = y + D * ky;
            if (qx < 0 || qy < 0 || qx >= W || qy >= H) continue;
            const float k = kv[(ky + 2) * 5 + (kx + 2)];
            const float4 c = win[(wy + D * ky) * pitch + wx + D * kx];
            s += k;
            r = fmaf(k, c.x, r);
            g = fmaf(k, c.y, g);
            b = fmaf(k, c.z, b);
        }
    const float inv = 1.0f / s;
    return make_float4(r * inv, g * inv, b * inv, s);
}

// The window of a 32 x TYp tile at (x0, y0) with a margin of M pixels, zeros outside the image.
template <int M, int TYp>
__device__ __forceinline__ void load_window(float4 (*win)[32 + 2 * M], const float4* __restrict__ img, int x0, int y0,
                                            int H, int W) {
    constexpr int HX = 32 + 2 * M, HY = TYp + 2 * M;
    for (int i = threadIdx.y * 32 + threadIdx.x; i < HX * HY; i += 256) {
        const int ly = i / HX, lx = i - ly * HX;
        const int gx = x0 - M + lx, gy = y0 - M + ly;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (gx >= 0 && gx < W && gy >= 0 && gy < H) v = __ldg(&img[(long)gy * W + gx]);
        win[ly][lx] = v;
    }
}

// The inverse tone map of the library's Params (exact or the paper-literal form).
__device__ __forceinline__ float3 inverse_tm(const Params& P, float3 c) {
    if (P.tonemap) {
        const float l = 0.2126f * c.x + 0.7152f * c.y + 0.0722f * c.z;
        float f;
        if (P.inverse_mode == 1) {
            f = (1.0f + l) * P.inv_weight;
        } else {
            float dd = 1.0f - P.luma_k * l;
            dd = dd < 1e-6f ? 1e-6f : dd;
            f = 1.0f / dd;
        }
        c = make_float3(c.x * f, c.y * f, c.z * f);
    }
    return c;
}

template <int D>
__global__ void __launch_bounds__(256) k_apply_h(const uint4* __restrict__ Kh, const float4* __restrict__ c_in,
                                                 float4* c_out, int H, int W, Params P, float4* rgb_out,
                                                 const float4* __restrict__ var_src) {
    constexpr int TXp = 32, TYp = 16, HX = TXp + 4 * D, HY = TYp + 4 * D;
    __shared__ float4 tile[HY][HX];
    pdl_wait();
    const int x0 = blockIdx.x * TXp, y0 = blockIdx.y * TYp;
    const long base = (long)blockIdx.z * H * W;
    load_window<2 * D, TYp>(tile, c_in + base, x0, y0, H, W);
    __syncthreads();
#pragma unroll 1
    for (int half = 0; half < 2; ++half) {
        const int lx = threadIdx.x, ly = threadIdx.y + 8 * half;
        const int x = x0 + lx, y = y0 + ly;
        if (x >= W || y >= H) continue;
        const long p = base + (long)y * W + x;
        float kv[32];
        load_kernel_h(Kh, p, kv);
        const float4 o = apply_taps<D>(kv, &tile[0][0], HX, lx + 2 * D, ly + 2 * D, x, y, W, H);
        if (rgb_out) {
            const float3 c = inverse_tm(P, make_float3(o.x, o.y, o.z));
            rgb_out[p] = make_float4(c.x, c.y, c.z, var_src ? var_src[p].w : 0.f);
        } else {
            c_out[p] = make_float4(o.x, o.y, o.z, 0.f);
        }
    }
}

// An application of the training forward, kernels as FP32 planes K[i][np].  EPI 0: c_out = the
// colour, channel 3 zero.  EPI 1: channel 3 = the sum S of the in-image weights (the backward pass
// divides by it).  EPI 2, the second application of a gradient: c_out as EPI 0, and with the target
// T the squared error added to *loss_sum and u = g2 / S, g2 = scale (c_out - T) the loss's gradient.
// A thread's 25 weights are loaded before its taps, so their latency is paid once a pixel, and the
// taps come from the window: 51 -> 28 us at dilation 1 and 51 -> 38 at dilation 4 with the loss (16
// crops of 256 x 256; 18 us of that are the weights' bytes).
template <int D, int EPI>
__global__ void __launch_bounds__(256, 4) k_apply(const float* __restrict__ K, const float4* __restrict__ c_in,
                                                  float4* c_out, long np, int H, int W, const float4* __restrict__ T,
                                                  float4* u, float* loss_sum, float scale) {
    constexpr int TYp = 16, HX = 32 + 4 * D, HY = TYp + 4 * D;
    __shared__ float4 tile[HY][HX];
    pdl_wait();
    const int x0 = blockIdx.x * 32, y0 = blockIdx.y * TYp;
    const long base = (long)blockIdx.z * H * W;
    load_window<2 * D, TYp>(tile, c_in + base, x0, y0, H, W);
    __syncthreads();
    float sq = 0.f;
#pragma unroll 1
    for (int half = 0; half < 2; ++half) {
        const int lx = threadIdx.x, ly = threadIdx.y + 8 * half;
        const int x = x0 + lx, y = y0 + ly;
        if (x >= W || y >= H) continue;
        const long p = base + (long)y * W + x;
        float kv[32];
#pragma unroll
        for (int i = 0; i < 25; ++i) kv[i] = __ldg(&K[i * np + p]);
        const float4 o = apply_taps<D>(kv, &tile[0][0], HX, lx + 2 * D, ly + 2 * D, x, y, W, H);
        c_out[p] = make_float4(o.x, o.y, o.z, EPI == 1 ? o.w : 0.f);
        if constexpr (EPI == 2) {
            const float4 t = __ldg(&T[p]);
            const float e0 = o.x - t.x, e1 = o.y - t.y, e2 = o.z - t.z;
            sq += e0 * e0 + e1 * e1 + e2 * e2;
            const float rS = 1.0f / o.w;
            u[p] = make_float4(scale * e0 * rS, scale * e1 * rS, scale * e2 * rS, 0.f);
        }
    }
    if constexpr (EPI == 2) {
        // block sum of the squared error, one atomic add a block
        for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
        __shared__ float red[8];
        if (threadIdx.x == 0) red[threadIdx.y] = sq;
        __syncthreads();
        if (threadIdx.x == 0 && threadIdx.y == 0) {
            float s = 0.f;
            for (int w = 0; w < 8; ++w) s += red[w];
            atomicAdd(loss_sum, s);
        }
    }
}

// Backward through both applications and the softmax, per pixel q, from u = g2 / S2 and the
// applications' outputs c1 (channel 3: S1) and c2:
//   the gradient reaching c1: g1 = sum_i [p = q - 4 o_i in image] u(p) K_i(p);
//   the kernel's gradient:    gK_i = u (c1(q + 4 o_i) - c2) + g1 (c0(q + o_i) - c1) / S1, each term
//                             over its in-image taps;
//   the logits' gradient:     dz_j = K_j (gK_j - sum_i K_i gK_i), BF16 [p][32] (zeros past 25).
// The second application's term is formed here from shared-memory windows of u, c1 and c0 rather
// than by a kernel of its own that passes 25 FP32 planes (200 B a pixel written and read back)
// through memory.  Bound by the latency of its weight loads (12 of 16 waiting warps an issue): the
// weights K_j are read again for the last line instead of being kept, and the budget is five blocks a
// SM (48 registers): 566 us a training step of 16 crops of 256 x 256, against 579, 598 and 644 with
// four, three and two blocks.  The windows of five blocks leave L1 about 30 KB, so the second reads are
// mostly the L2's (hit rates 12 % in L1, 60 % in L2).  The two kernels before took 53 + 188 us of that
// step, this one 115.
__global__ void __launch_bounds__(256, 5) k_bwd_apply(const float* __restrict__ K, const float4* __restrict__ u,
                                                      const float4* __restrict__ c0, const float4* __restrict__ c1,
                                                      const float4* __restrict__ c2, __nv_bfloat16* dz, long np,
                                                      int H, int W) {
    __shared__ float4 wu[8 + 16][32 + 16], w1[8 + 16][32 + 16], w0[8 + 4][32 + 4];
    pdl_wait();
    const int x0 = blockIdx.x * 32, y0 = blockIdx.y * 8;
    const long base = (long)blockIdx.z * H * W;
    load_window<8, 8>(wu, u + base, x0, y0, H, W);
    load_window<8, 8>(w1, c1 + base, x0, y0, H, W);
    load_window<2, 8>(w0, c0 + base, x0, y0, H, W);
    __syncthreads();
    const int x = x0 + threadIdx.x, y = y0 + threadIdx.y;
    if (x >= W || y >= H) return;
    const int lx = threadIdx.x, ly = threadIdx.y;
    const long q = base + (long)y * W + x;
    float g0 = 0.f, g1 = 0.f, g2 = 0.f;
#pragma unroll
    for (int ky = -2; ky <= 2; ++ky)
#pragma unroll
        for (int kx = -2; kx <= 2; ++kx) {
            const int px = x - 4 * kx, py = y - 4 * ky;
            if (px < 0 || py < 0 || px >= W || py >= H) continue;
            const float k = __ldg(&K[((ky + 2) * 5 + (kx + 2)) * np + base + (long)py * W + px]);
            const float4 uu = wu[ly + 8 - 4 * ky][lx + 8 - 4 * kx];
            g0 = fmaf(k, uu.x, g0);
            g1 = fmaf(k, uu.y, g1);
            g2 = fmaf(k, uu.z, g2);
        }
    const float4 o1 = w1[ly + 8][lx + 8], o2 = __ldg(&c2[q]), uq = wu[ly + 8][lx + 8];
    const float rS = 1.0f / o1.w;
    float gq[25], dot = 0.f;
#pragma unroll
    for (int ky = -2; ky <= 2; ++ky)
#pragma unroll
        for (int kx = -2; kx <= 2; ++kx) {
            const int i = (ky + 2) * 5 + (kx + 2);
            float v = 0.f;
            if (x + 4 * kx >= 0 && y + 4 * ky >= 0 && x + 4 * kx < W && y + 4 * ky < H) {
                const float4 c = w1[ly + 8 + 4 * ky][lx + 8 + 4 * kx];
                v = uq.x * (c.x - o2.x) + uq.y * (c.y - o2.y) + uq.z * (c.z - o2.z);
            }
            if (x + kx >= 0 && y + ky >= 0 && x + kx < W && y + ky < H) {
                const float4 c = w0[ly + 2 + ky][lx + 2 + kx];
                v += (g0 * (c.x - o1.x) + g1 * (c.y - o1.y) + g2 * (c.z - o1.z)) * rS;
            }
            gq[i] = v;
            dot = fmaf(__ldg(&K[i * np + q]), v, dot);
        }
    uint4* out = reinterpret_cast<uint4*>(dz + q * 32);
#pragma unroll
    for (int h = 0; h < 4; ++h) {
        unsigned w[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int a = 8 * h + 2 * i, b = a + 1;
            const float va = a < 25 ? __ldg(&K[(a < 25 ? a : 0) * np + q]) * (gq[a < 25 ? a : 0] - dot) : 0.f;
            const float vb = b < 25 ? __ldg(&K[(b < 25 ? b : 0) * np + q]) * (gq[b < 25 ? b : 0] - dot) : 0.f;
            w[i] = pack_bf16(va, vb);
        }
        out[h] = make_uint4(w[0], w[1], w[2], w[3]);
    }
}

// ---------------------------------------------------------------- parameters

// From the flat FP32 parameters to the conv kernels' BF16 weights:
//  fwd[l]   [9][32][CIpad_l]: W_l[co][tap][ci] (zero for co >= 25 in layer 3, ci >= 10 in layer 0)
//  dgrad[l] [9][32][32]:      W_l[co][8 - tap][n = ci] transposed (l >= 1; zero for co >= 25)
//  bias[l]  [32]
__global__ void k_prep_weights(const float* __restrict__ prm, WeightPtrs w) {
    pdl_wait();
    const int l = blockIdx.y;
    const int cin = cin_of(l), cout = cout_of(l), cip = cin_pad_of(l);
    const float* Wl = prm + param_offset(l);
    const float* bl = Wl + cout * 9 * cin;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < 9 * 32 * cip; i += gridDim.x * blockDim.x) {
        const int ci = i % cip, co = (i / cip) % 32, tap = i / (cip * 32);
        const float v = (co < cout && ci < cin) ? Wl[((long)co * 9 + tap) * cin + ci] : 0.f;
        w.fwd[l][i] = __float2bfloat16_rn(v);
    }
    if (l >= 1)
        for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < 9 * 32 * 32; i += gridDim.x * blockDim.x) {
            const int co = i % 32, n = (i / 32) % 32, tap = i / (32 * 32);   // k = co, n = ci
            const float v = (co < cout && n < cin) ? Wl[((long)co * 9 + (8 - tap)) * cin + n] : 0.f;
            w.dgrad[l][i] = __float2bfloat16_rn(v);
        }
    if (blockIdx.x == 0 && threadIdx.x < 32) w.bias[l][threadIdx.x] = threadIdx.x < cout ? bl[threadIdx.x] : 0.f;
}

__global__ void k_adam(float* prm, const float* __restrict__ grad, float* m, float* v, int n,
                       float lr, float b1, float b2, float eps, float bc1, float bc2) {
    pdl_wait();
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const float g = grad[i];
        const float mi = b1 * m[i] + (1.0f - b1) * g;
        const float vi = b2 * v[i] + (1.0f - b2) * g * g;
        m[i] = mi;
        v[i] = vi;
        prm[i] -= lr * (mi / bc1) / (sqrtf(vi / bc2) + eps);
    }
}

// Features of the pass-0 output (tone-mapped colour, sqrt variance, log2 depth, octahedral
// normal, albedo), BF16 [H][W][16] (channels 10..15 zero).  cv in any storage precision.
template <class S>
__global__ void k_features_t(const typename S::Rec* __restrict__ cv, const float4* __restrict__ gbuf,
                             const float* __restrict__ albedo, __nv_bfloat16* feat, float4* c0,
                             int npx) {
    pdl_wait();
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < npx; p += gridDim.x * blockDim.x) {
        const float4 c = S::ld_cv(cv, p);
        const float4 g = gbuf[p];
        const float s = fabsf(g.x) + fabsf(g.y) + fabsf(g.z);
        float ox = g.x / s, oy = g.y / s;
        if (g.z < 0.f) {
            const float tx = (1.0f - fabsf(oy)) * (ox >= 0.f ? 1.f : -1.f);
            const float ty = (1.0f - fabsf(ox)) * (oy >= 0.f ? 1.f : -1.f);
            ox = tx;
            oy = ty;
        }
        float f[16] = {c.x, c.y, c.z, sqrtf(fmaxf(c.w, 0.f)), log2f(fmaxf(g.w, 1e-20f)), ox, oy,
                       albedo[3 * (long)p], albedo[3 * (long)p + 1], albedo[3 * (long)p + 2],
                       0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        uint4* o = reinterpret_cast<uint4*>(feat + (long)p * 16);
        o[0] = make_uint4(pack_bf16(f[0], f[1]), pack_bf16(f[2], f[3]), pack_bf16(f[4], f[5]), pack_bf16(f[6], f[7]));
        o[1] = make_uint4(pack_bf16(f[8], f[9]), 0u, 0u, 0u);
        if (c0) c0[p] = c;       // the pass-0 colour (and variance) the applications filter
    }
}

unsigned flat_grid(long n, int threads) {
    long b = (n + threads - 1) / threads;
    return (unsigned)(b > 152L * 32 ? 152L * 32 : (b < 1 ? 1 : b));
}

}  // namespace

cudaError_t prep_weights(const float* prm, const WeightPtrs& w, bool chained, cudaStream_t s) {
    return launch(chained, k_prep_weights, dim3(36, 4), 256, 0, s, prm, w);
}

namespace {
// One thread initialises a single-arrival barrier and waits for its first phase, which no thread
// ever arrives at: the wait runs out after `tries` polls and the error bit is raised.
__global__ void k_wait_expiry(int tries, int* err) {
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x != 0) return;
    tc::mbar_init(&bar);
    if (!tc::mbar_wait(&bar, 0u, tries)) atomicOr(err, kErrWaitGaveUp);
}
}  // namespace

cudaError_t wait_expiry_probe(int tries, int* err, cudaStream_t s) {
    if (tries < 1 || tries > tc::kWaitTries || err == nullptr) return cudaErrorInvalidValue;
    k_wait_expiry<<<1, 32, 0, s>>>(tries, err);
    return cudaGetLastError();
}

// Chunk length of a convolution launch: the B x segs columns of 128 pixels, each cut into
// chunks_y chunks, give at most one chunk to each of the grid's blocks (2 per SM), so that no
// block takes one more chunk than the others while they wait (with a fixed 16-row chunk a 1080p
// layer had 1020 chunks for 304 blocks: 108 blocks took four, the rest three); the chunk's two
// halo rows are then a small share of its rows.
static int conv_chunk(int B, int H, int W, int sm_count) {
    const long cols = (long)B * ((W + tc::M - 1) / tc::M);
    const long cap = (long)sm_count * 2;
    long per = cols >= cap ? 1 : cap / cols;            // chunks a column
    if (per > H) per = H;
    return (int)((H + per - 1) / per);
}

// The tensor map of a convolution's input [B][H][W][CI] BF16 for the producer's row copies: box
// CI channels x px pixels (130: a row with its halo) x 1 row x 1 image, in the swizzle the MMAs read (64-byte rows for 32
// channels, 32-byte rows for 16), zeros outside the tensor.  cuTensorMapEncodeTiled is reached
// through the runtime's driver entry point.
static cudaError_t encode_rows(CUtensorMap* map, const __nv_bfloat16* in, int CI, int B, int H, int W, int px = tc::HP) {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        const cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q);
        if (e != cudaSuccess) return e;
        if (q != cudaDriverEntryPointSuccess || !p) return cudaErrorNotSupported;
        fn = (PFN_cuTensorMapEncodeTiled_v12000)p;
    }
    const cuuint64_t dims[4] = {(cuuint64_t)CI, (cuuint64_t)W, (cuuint64_t)H, (cuuint64_t)B};
    const cuuint64_t strides[3] = {(cuuint64_t)CI * 2, (cuuint64_t)W * CI * 2, (cuuint64_t)H * W * CI * 2};
    const cuuint32_t box[4] = {(cuuint32_t)CI, (cuuint32_t)px, 1, 1};
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    const CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, (void*)in, dims, strides, box, estr,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CI == 32 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B,
                          CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

cudaError_t conv(int layer, bool dgrad, const __nv_bfloat16* in, const WeightPtrs& w,
                 const __nv_bfloat16* mask, void* out, int B, int H, int W, int sm_count, bool chained,
                 cudaStream_t s, int* err) {
    {
        const int chunk = conv_chunk(B, H, W, sm_count);
        const long tiles = (long)B * ((W + tc::M - 1) / tc::M) * ((H + chunk - 1) / chunk);
        const long cap = (long)sm_count * 2;
        const int grid = (int)(tiles < cap ? tiles : cap);
        // ng drain groups of four warps (two, except for the FP32-plane softmax, whose epilogue
        // needs more registers than 320 threads a block at two blocks a SM leave)
        auto launch = [&](auto kernel, int ci, int ng, const __nv_bfloat16* wt, const float* bias) {
            size_t smem = (size_t)9 * (ci / 8) * 32 * 16 + (size_t)kRing * (ci == 32 ? kRowSw64Bytes : kRowSw32Bytes) +
                          (size_t)ng * kOutBufs * tc::M * 64 + tc::kSlack + (kDone + 2 * kRing + kSlots + 1) * 8 + 8;
            if (smem < kMinConvSmem) smem = kMinConvSmem;
            cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (e != cudaSuccess) return e;
            CUtensorMap rows;
            e = encode_rows(&rows, in, ci, B, H, W);
            if (e != cudaSuccess) return e;
            return svgf::launch(chained, kernel, grid, 128 * ng + 64, smem, s, rows, in, wt, bias, mask, out, B, H, W,
                                chunk, err);
        };
        if (!dgrad) {
            if (layer == 0) return launch(k_conv3x3_tc<16, 0, 2>, 16, 2, w.fwd[0], w.bias[0]);
            if (layer < 3) return launch(k_conv3x3_tc<32, 0, 2>, 32, 2, w.fwd[layer], w.bias[layer]);
            if (layer == 3) return launch(k_conv3x3_tc<32, 1, 1>, 32, 1, w.fwd[3], w.bias[3]);
            return launch(k_conv3x3_tc<32, 3, 2>, 32, 2, w.fwd[3], w.bias[3]);   // layer 3, FP16 kernels
        }
        return launch(k_conv3x3_tc<32, 2, 2>, 32, 2, w.dgrad[layer], nullptr);
    }
}

// Chunk length of the four-layer kernel: one block a SM (its shared memory), the B x segs column
// segments cut into at most one chunk a block.
static int net_chunk(int B, int H, int W, int sm_count) {
    const long cols = (long)B * ((W + kNetSeg - 1) / kNetSeg);
    long per = cols >= sm_count ? 1 : sm_count / cols;
    if (per > H) per = H;
    return (int)((H + per - 1) / per);
}

cudaError_t net_forward(const __nv_bfloat16* feats, const WeightPtrs& w, void* Kh, int B, int H, int W,
                        int sm_count, cudaStream_t s, int* err) {
    if (B <= 0 || H <= 0 || W <= 0) return cudaSuccess;
    const int chunk = net_chunk(B, H, W, sm_count);
    const long tiles = (long)B * ((W + kNetSeg - 1) / kNetSeg) * ((H + chunk - 1) / chunk);
    const int grid = (int)(tiles < sm_count ? tiles : sm_count);
    cudaError_t e = cudaFuncSetAttribute(k_kpn_net, cudaFuncAttributeMaxDynamicSharedMemorySize, kNetSmemBytes);
    if (e != cudaSuccess) return e;
    NetWeights nw;
    for (int l = 0; l < 4; ++l) {
        nw.wt[l] = w.fwd[l];
        nw.bias[l] = w.bias[l];
    }
    k_kpn_net<<<grid, kNetThreads, kNetSmemBytes, s>>>(feats, nw, Kh, B, H, W, chunk, err);
    return cudaGetLastError();
}

// Chunk length of the two-layer kernels: one block a SM, at most one chunk a block.
static int pair_chunk(int B, int H, int W, int sm_count) {
    const long cols = (long)B * ((W + kPairSeg - 1) / kPairSeg);
    long per = cols >= sm_count ? 1 : sm_count / cols;
    if (per > H) per = H;
    return (int)((H + per - 1) / per);
}

cudaError_t net_pairs(const __nv_bfloat16* feats, const WeightPtrs& w, __nv_bfloat16* mid, void* Kh, int B, int H,
                      int W, int sm_count, cudaStream_t s, int* err) {
    if (B <= 0 || H <= 0 || W <= 0) return cudaSuccess;
    const int chunk = pair_chunk(B, H, W, sm_count);
    const long tiles = (long)B * ((W + kPairSeg - 1) / kPairSeg) * ((H + chunk - 1) / chunk);
    const int grid = (int)(tiles < sm_count ? tiles : sm_count);
    cudaError_t e = cudaFuncSetAttribute(k_kpn_pair<0>, cudaFuncAttributeMaxDynamicSharedMemorySize, PairCfg<0>::SMEM);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_kpn_pair<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, PairCfg<2>::SMEM);
    if (e != cudaSuccess) return e;
    k_kpn_pair<0><<<grid, kPairThreads, PairCfg<0>::SMEM, s>>>(feats, w.fwd[0], w.fwd[1], w.bias[0], w.bias[1], mid,
                                                               B, H, W, chunk, err);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_kpn_pair<2><<<grid, kPairThreads, PairCfg<2>::SMEM, s>>>(mid, w.fwd[2], w.fwd[3], w.bias[2], w.bias[3], Kh,
                                                               B, H, W, chunk, err);
    return cudaGetLastError();
}

cudaError_t wgrad(int layer, const __nv_bfloat16* X, const __nv_bfloat16* dZ, float* grad_flat,
                  int B, int H, int W, int sm_count, cudaStream_t s, int* err) {
    const int chunk = conv_chunk(B, H, W, sm_count);
    const long tiles = (long)B * ((W + tc::M - 1) / tc::M) * ((H + chunk - 1) / chunk), cap = (long)sm_count * 2;
    const int grid = (int)(tiles < cap ? tiles : cap);
    float* dW = grad_flat + param_offset(layer);
    float* db = dW + cout_of(layer) * 9 * cin_of(layer);
    auto launch = [&](auto kernel, int ci, int smem) {
        CUtensorMap xmap, dmap;
        cudaError_t e = encode_rows(&xmap, X, ci, B, H, W);
        if (e == cudaSuccess) e = encode_rows(&dmap, dZ, 32, B, H, W, tc::M);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
        return svgf::launch(true, kernel, grid, kWgThreads, smem, s, xmap, dmap, dW, db, B, H, W, chunk, cin_of(layer),
                            cout_of(layer), err);
    };
    return layer == 0 ? launch(k_wgrad<16>, 16, WgradCfg<16>::SMEM) : launch(k_wgrad<32>, 32, WgradCfg<32>::SMEM);
}

cudaError_t apply(const float* K, const float4* c_in, float4* c_out, int B, int H, int W, int dilation,
                  const float4* T, float4* u, float* loss_sum, cudaStream_t s) {
    const long np = (long)B * H * W;
    const float scale = 2.0f / (3.0f * (float)np);
    const dim3 grid((W + 31) / 32, (H + 15) / 16, B), block(32, 8);
    if (dilation != 1 && dilation != 4) return cudaErrorInvalidValue;
    return launch(true, dilation == 1 ? k_apply<1, 1> : T ? k_apply<4, 2> : k_apply<4, 0>, grid, block, 0, s, K, c_in,
                  c_out, np, H, W, T, u, loss_sum, scale);
}

cudaError_t apply_h(const void* Kh, const float4* c_in, float4* c_out, int B, int H, int W,
                    int dilation, const Params& P, float4* rgb_out, const float4* var_src, bool chained, cudaStream_t s) {
    const dim3 grid((W + 31) / 32, (H + 15) / 16, B), block(32, 8);
    if (dilation != 1 && dilation != 4) return cudaErrorInvalidValue;
    return launch(chained, dilation == 1 ? k_apply_h<1> : k_apply_h<4>, grid, block, 0, s, (const uint4*)Kh, c_in, c_out,
                  H, W, P, rgb_out, var_src);
}

cudaError_t backward_apply(const float* K, const float4* c0, const float4* c1, const float4* c2, const float4* u,
                           __nv_bfloat16* dz, int B, int H, int W, cudaStream_t s) {
    const dim3 grid((W + 31) / 32, (H + 7) / 8, B), block(32, 8);
    return launch(true, k_bwd_apply, grid, block, 0, s, K, u, c0, c1, c2, dz, (long)B * H * W, H, W);
}

cudaError_t adam(float* prm, const float* grad, float* m, float* v, float lr, float b1, float b2,
                 float eps, float bc1, float bc2, cudaStream_t s) {
    return launch(true, k_adam, flat_grid(kParamCount, 256), 256, 0, s, prm, grad, m, v, kParamCount, lr, b1, b2, eps,
                  bc1, bc2);
}

cudaError_t features(int prec, const void* cv, const float4* gbuf, const float* albedo,
                     __nv_bfloat16* feat, float4* c0, int npx, bool chained, cudaStream_t s) {
    const unsigned g = flat_grid(npx, 256);
    switch (prec) {
        case 0: return launch(chained, k_features_t<dev::StoreF32>, g, 256, 0, s, (const float4*)cv, gbuf, albedo, feat, c0, npx);
        case 1: return launch(chained, k_features_t<dev::Store16<false>>, g, 256, 0, s, (const uint2*)cv, gbuf, albedo, feat, c0, npx);
        default: return launch(chained, k_features_t<dev::Store16<true>>, g, 256, 0, s, (const uint2*)cv, gbuf, albedo, feat, c0, npx);
    }
}

namespace {
// Per 32x32 tile: the population standard deviation of the pass-0 luminance (tone-mapped, the
// colour the network filters), two-pass; above the threshold -> flag = 1, counted.  Tiles with
// detail (edges, texture, contact shadows) are where the network's two narrow kernels depart
// from the wide, edge-stopped plain passes.
__global__ void __launch_bounds__(256) k_tile_flags(const float4* __restrict__ c0, int H, int W, float thr,
                                                    unsigned char* flags, int* count) {
    const int tx = blockIdx.x, ty = blockIdx.y;
    __shared__ float rs[256];
    __shared__ int rn[256];
    float l[4];
    bool in[4];
    float s = 0.f;
    int n = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int i = threadIdx.x + k * 256;
        const int x = tx * 32 + (i & 31), y = ty * 32 + (i >> 5);
        in[k] = x < W && y < H;
        l[k] = 0.f;
        if (in[k]) {
            const float4 c = c0[(long)y * W + x];
            l[k] = fmaf(0.0722f, c.z, fmaf(0.7152f, c.y, 0.2126f * c.x));
            s += l[k];
            ++n;
        }
    }
    rs[threadIdx.x] = s;
    rn[threadIdx.x] = n;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) {
            rs[threadIdx.x] += rs[threadIdx.x + o];
            rn[threadIdx.x] += rn[threadIdx.x + o];
        }
        __syncthreads();
    }
    const float cnt = (float)rn[0];
    const float mean = rs[0] / cnt;
    __syncthreads();
    float ss = 0.f;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const float d = l[k] - mean;
        if (in[k]) ss = fmaf(d, d, ss);
    }
    rs[threadIdx.x] = ss;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) rs[threadIdx.x] += rs[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        const unsigned char f = sqrtf(rs[0] / cnt) > thr ? 1 : 0;
        flags[ty * gridDim.x + tx] = f;
        if (f) atomicAdd(count, 1);
    }
}

// out = in dilated by r tiles (Chebyshev distance) over a tiles_x x tiles_y grid.
__global__ void k_dilate(const unsigned char* __restrict__ in, unsigned char* __restrict__ out,
                         int tiles_x, int tiles_y, int r) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= tiles_x * tiles_y) return;
    const int y = t / tiles_x, x = t - y * tiles_x;
    const int y0 = max(0, y - r), y1 = min(tiles_y - 1, y + r);
    const int x0 = max(0, x - r), x1 = min(tiles_x - 1, x + r);
    unsigned char v = 0;
    for (int yy = y0; yy <= y1 && !v; ++yy)
        for (int xx = x0; xx <= x1; ++xx) v |= in[yy * tiles_x + xx];
    out[t] = v;
}

// rgb_out <- plain for the pixels of flagged tiles.
__global__ void k_tile_select(const float4* __restrict__ plain, const unsigned char* __restrict__ flags,
                              float4* rgb_out, int H, int W) {
    const long n = (long)H * W;
    const int tiles_x = (W + 31) / 32;
    for (long p = blockIdx.x * (long)blockDim.x + threadIdx.x; p < n; p += (long)gridDim.x * blockDim.x) {
        const int x = (int)(p % W), y = (int)(p / W);
        if (flags[(y / 32) * tiles_x + x / 32]) rgb_out[p] = plain[p];
    }
}

__global__ void k_loss_finish(const float* sum, float* loss_out, float inv_n) {
    pdl_wait();
    if (threadIdx.x == 0) *loss_out = *sum * inv_n;
}
}  // namespace

cudaError_t tile_flags(const float4* c0, int H, int W, float thr, unsigned char* flags, int* count,
                       cudaStream_t s) {
    k_tile_flags<<<dim3((W + 31) / 32, (H + 31) / 32), 256, 0, s>>>(c0, H, W, thr, flags, count);
    return cudaGetLastError();
}

cudaError_t tile_dilate(const unsigned char* in, unsigned char* out, int tiles_x, int tiles_y, int r,
                        cudaStream_t s) {
    const int n = tiles_x * tiles_y;
    k_dilate<<<(n + 255) / 256, 256, 0, s>>>(in, out, tiles_x, tiles_y, r);
    return cudaGetLastError();
}

cudaError_t tile_select(const float4* plain, const unsigned char* flags, float4* rgb_out, int H, int W,
                        cudaStream_t s) {
    k_tile_select<<<flat_grid((long)H * W, 256), 256, 0, s>>>(plain, flags, rgb_out, H, W);
    return cudaGetLastError();
}

cudaError_t loss_finish(const float* sum, float* loss_out, long n, cudaStream_t s) {
    return launch(true, k_loss_finish, 1, 32, 0, s, sum, loss_out, 1.0f / (3.0f * (float)n));
}

}  // namespace kpn
}  // namespace svgf
