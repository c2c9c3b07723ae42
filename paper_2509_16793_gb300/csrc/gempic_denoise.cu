// Learned current denoiser: a 3-layer 3x3x3 convolutional net (16 hidden channels, ReLU) on
// the current j of the half-slice grid, BF16 operands with FP32 accumulation on the 5th-
// generation tensor cores (tcgen05.mma, accumulators in tensor memory), plus its training
// step (loss, backward pass, Adam).  The paper has no such component: it lets a run with few
// particles per cell stand in for one with many (include/gempic.h, gempic_denoiser_*).
//
// Tensors are channel-last, X[z][y][x][16] in BF16 (z = half-slice, periodic across, zero
// outside the window along zeta); rows of 128 voxels lie in memory in the tensor core's operand
// layout and take conv_ws_kernel, described there.  Other widths (conv_kernel): a convolution
// is an implicit GEMM: a tile of 128 voxels (consecutive in z, y, x order) is the M dimension,
// the 16 output channels N, and each of the 27 taps adds a K = 16 slice (the 16 input channels
// of the tap's neighbour).  Per tap the
// CTA gathers its tile's 128 neighbour voxels into shared memory in the tensor core's K-major
// layout without swizzle (8-row x 16-byte core matrices: 128 B apart along K, 256 B apart
// along M), one thread issues the MMA, and the 27 MMAs of a tile accumulate in 16 columns of
// tensor memory.  Taps are staged nine at a time into one of two buffers, so the gather of the
// next nine overlaps the MMAs of the last; an mbarrier that tcgen05.commit arrives on tells
// when a buffer is free.  The epilogue reads the accumulators back (tcgen05.ld, one warp per
// 32 rows) and applies the layer's bias, activation or mask.
//
// The backward pass through a layer's input is the same convolution with the kernel mirrored
// and its channels transposed (host-packed operand), masked by the ReLU of the layer below.
// The weight gradients contract X_shift^T dY over the voxels (wgrad_kernel); Adam
// updates FP32 master weights, which are then repacked into the BF16 operands.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <new>
#include <vector>

#include "../../include/gempic.h"

namespace {

constexpr int kCh = 16;            // channels of every activation tensor (inputs padded)
constexpr int kTaps = 27;
constexpr int kTile = 128;         // voxels per MMA tile (M)
constexpr int kRound = 9;          // taps staged per buffer
constexpr int kThreads = 128;      // 4 warps: one per 32 accumulator rows, one thread per row
static_assert(kThreads == kTile, "the gather gives each thread one row of the tile");
constexpr uint32_t kTapBytesA = kTile * kCh * 2;     // 4096
constexpr uint32_t kTapBytesB = kCh * kCh * 2;       // 512
constexpr uint32_t kLBO = 128;     // byte offset of the core matrix next along K
constexpr uint32_t kSBO = 256;     // byte offset of the core matrix next along M (N)
constexpr int kSpinLimit = 1 << 22;   // polls of an mbarrier before giving up

// instruction descriptor of tcgen05.mma kind::f16: D in FP32, A and B in BF16, both K-major,
// N = 16, M = 128
constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kCh >> 3) << 17) |
                            ((uint32_t)(kTile >> 4) << 24);

// Activation layouts in global memory.  Plain (any width): [z][y][x][16], 32 bytes a voxel.
// Padded rows (rows of 128 voxels, the 128 x 128 grids): [z][y] rows of kRowBytes holding
// voxels x = -1 .. 128 (the periodic neighbour at each end), a voxel's two 16-byte halves
// exchanged in every other group of four voxels.  That is byte for byte the operand layout of
// the row convolution in shared memory (32-byte swizzle), so a row goes there in one bulk copy.
constexpr int kRowVox = 128;                         // nx of the row path
constexpr int kRowHalo = kRowVox + 2;                // staged voxels: x = -1 .. 128
constexpr uint32_t kRowBytes = 17u * 256u;           // 130 x 32 bytes, rounded to 256
constexpr uint32_t kRowCopy = (uint32_t)kRowHalo * 32u;

// byte offset of half h of position xi (voxel x = xi - 1) in a padded row
__device__ __forceinline__ uint32_t seg_off(int xi, int h) {
  return (uint32_t)xi * 32u + (uint32_t)((h ^ (xi >> 2)) & 1) * 16u;
}
// the 16 channels of voxel v (v = (z ny + y) nx + x): read, or write with the row's halo copies
__device__ __forceinline__ void act_load(const __nv_bfloat16* x, int nx, long long v, uint4& a, uint4& b) {
  if (nx == kRowVox) {
    const char* row = reinterpret_cast<const char*>(x) + (v / kRowVox) * (long long)kRowBytes;
    const int xi = (int)(v % kRowVox) + 1;
    a = *reinterpret_cast<const uint4*>(row + seg_off(xi, 0));
    b = *reinterpret_cast<const uint4*>(row + seg_off(xi, 1));
  } else {
    const uint4* d = reinterpret_cast<const uint4*>(x + v * 16);
    a = d[0];
    b = d[1];
  }
}
__device__ __forceinline__ void act_store(__nv_bfloat16* x, int nx, long long v, uint4 a, uint4 b) {
  if (nx == kRowVox) {
    char* row = reinterpret_cast<char*>(x) + (v / kRowVox) * (long long)kRowBytes;
    const int xi = (int)(v % kRowVox) + 1;
    *reinterpret_cast<uint4*>(row + seg_off(xi, 0)) = a;
    *reinterpret_cast<uint4*>(row + seg_off(xi, 1)) = b;
    if (xi == 1 || xi == kRowVox) {
      const int xh = xi == 1 ? kRowVox + 1 : 0;
      *reinterpret_cast<uint4*>(row + seg_off(xh, 0)) = a;
      *reinterpret_cast<uint4*>(row + seg_off(xh, 1)) = b;
    }
  } else {
    uint4* d = reinterpret_cast<uint4*>(x + v * 16);
    d[0] = a;
    d[1] = b;
  }
}

enum Mode { MODE_HIDDEN = 0, MODE_LAST = 1, MODE_BWD = 2 };

struct ConvArgs {
  const __nv_bfloat16* x;     // [V][16] input activations
  const __nv_bfloat16* w;     // [27][256] operand B per tap, K-major canonical layout
  const float* bias;          // [16] (MODE_HIDDEN, MODE_LAST)
  int nx, ny, nz;
  int mode;
  __nv_bfloat16* out;         // [V][16] (MODE_HIDDEN, MODE_BWD)
  const __nv_bfloat16* mask;  // [V][16] activations whose sign masks the output (MODE_BWD)
  float* r;                   // [V][4] net output r (MODE_LAST, may be null)
  const float* jres;          // [nz][3][ny][nx] current added to scale r (MODE_LAST, may be null)
  float* jout;                // [nz][3][ny][nx] denoised current (MODE_LAST, may be null)
  float scale;
  int* err;
  int zlo, zhi;               // output half-slices [zlo, zhi) (inputs are read where needed)
};

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

// shared-memory matrix descriptor: start address, LBO, SBO (all >> 4), descriptor version 1
// (bit 46), no swizzle
__device__ __forceinline__ uint64_t sdesc(uint32_t saddr) {
  return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)(kLBO >> 4) << 16) |
         ((uint64_t)(kSBO >> 4) << 32) | (1ull << 46);
}

__device__ __forceinline__ void umma(uint32_t tmem_d, uint64_t a, uint64_t b, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem_d),
      "l"(a), "l"(b), "r"(kIdesc), "r"(acc));
}

__device__ __forceinline__ void umma_commit(uint64_t* mbar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                   smem_u32(mbar))
               : "memory");
}

__device__ __forceinline__ void mbar_init(uint64_t* m, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(m)), "r"(count) : "memory");
}

__device__ __forceinline__ bool mbar_test(uint64_t* m, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}\n"
      : "=r"(ok)
      : "r"(smem_u32(m)), "r"(parity)
      : "memory");
  return ok != 0;
}

// bounded wait for the phase `parity` of an mbarrier: false if it did not complete
__device__ __forceinline__ bool mbar_wait(uint64_t* m, uint32_t parity) {
  for (int i = 0; i < kSpinLimit; ++i)
    if (mbar_test(m, parity)) return true;
  return false;
}

// 16-byte asynchronous copy global -> shared through L1 (neighbouring taps reuse it);
// src_bytes = 0 fills the destination with zeros
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, uint32_t src_bytes) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(src_bytes)
               : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
  asm volatile("cp.async.wait_all;" ::: "memory");
}

__device__ __forceinline__ void fence_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}

// 16 FP32 accumulator columns of this warp's 32 rows (lane = row)
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float* v) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,"
      "%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// the layer's output for voxel v from its 16 accumulators: bias + ReLU in BF16 (hidden layers),
// the input's ReLU mask (backward through a layer's input), or bias, the net output r and the
// residual into the FP32 current (last layer)
__device__ __forceinline__ void epilogue(const ConvArgs& a, long long v, const float* acc) {
  if (a.mode == MODE_HIDDEN) {
    __align__(16) __nv_bfloat16 o[16];
#pragma unroll
    for (int c = 0; c < 16; ++c)
      o[c] = __float2bfloat16_rn(fmaxf(acc[c] + a.bias[c], 0.0f));
    act_store(a.out, a.nx, v, reinterpret_cast<const uint4*>(o)[0], reinterpret_cast<const uint4*>(o)[1]);
  } else if (a.mode == MODE_BWD) {
    __align__(16) __nv_bfloat16 m[16];
    act_load(a.mask, a.nx, v, reinterpret_cast<uint4*>(m)[0], reinterpret_cast<uint4*>(m)[1]);
    __align__(16) __nv_bfloat16 o[16];
#pragma unroll
    for (int c = 0; c < 16; ++c)
      o[c] = __float2bfloat16_rn(__bfloat162float(m[c]) > 0.0f ? acc[c] : 0.0f);
    act_store(a.out, a.nx, v, reinterpret_cast<const uint4*>(o)[0], reinterpret_cast<const uint4*>(o)[1]);
  } else {
    const float r0 = acc[0] + a.bias[0], r1 = acc[1] + a.bias[1], r2 = acc[2] + a.bias[2];
    if (a.r) *reinterpret_cast<float4*>(a.r + v * 4) = make_float4(r0, r1, r2, 0.0f);
    if (a.jout) {
      const long long plane = (long long)a.nx * a.ny;
      const long long z = v / plane, rem = v - z * plane;
      const long long base = z * 3 * plane + rem;
      const float rr[3] = {r0, r1, r2};
#pragma unroll
      for (int c = 0; c < 3; ++c)
        a.jout[base + c * plane] = __ldcg(a.jres + base + c * plane) + a.scale * rr[c];
    }
  }
}

__global__ void __launch_bounds__(kThreads) conv_kernel(ConvArgs a) {
  extern __shared__ __align__(1024) unsigned char smem[];
  unsigned char* sB = smem;                                   // 27 x 512
  unsigned char* sA = smem + kTaps * kTapBytesB;              // 2 x 9 x 4096
  __shared__ __align__(8) uint64_t mbar[2];
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const long long plane0 = (long long)a.nx * a.ny;
  const long long vlo = (long long)a.zlo * plane0;
  const long long V = (long long)a.zhi * plane0;            // output voxels [vlo, V)
  const long long ntiles = (V - vlo + kTile - 1) / kTile;

  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 32;" ::"r"(
                     smem_u32(&tmem_slot))
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 0) {
    mbar_init(&mbar[0], 1);
    mbar_init(&mbar[1], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    abort_flag = 0;
  }
  // the B operands of the 27 taps
  {
    const uint4* src = reinterpret_cast<const uint4*>(a.w);
    uint4* dst = reinterpret_cast<uint4*>(sB);
    for (int i = tid; i < (int)(kTaps * kTapBytesB / 16); i += kThreads) dst[i] = src[i];
  }
  fence_async_smem();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  const uint32_t aBase = smem_u32(sA), bBase = smem_u32(sB);
  uint32_t phase[2] = {0u, 0u};
  int pending[2] = {0, 0};
  int gr = 0;                                                 // rounds staged so far

  const long long plane = (long long)a.nx * a.ny;
  for (long long tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const long long v0 = vlo + tile * kTile;
    // this thread gathers tile row `tid` (one voxel) for every tap
    const long long vr = v0 + tid;
    const bool valid = vr < V;
    int z = 0, y = 0, x = 0;
    if (valid) {
      z = (int)(vr / plane);
      const int rem = (int)(vr - (long long)z * plane);
      y = rem / a.nx;
      x = rem - y * a.nx;
    }
    for (int round = 0; round < kTaps / kRound; ++round, ++gr) {
      const int buf = gr & 1;
      if (pending[buf]) {                                     // MMAs still reading this buffer
        if (!mbar_wait(&mbar[buf], phase[buf])) atomicExch(&abort_flag, 1);
        phase[buf] ^= 1u;
        pending[buf] = 0;
      }
      // gather: for each tap of the round, this thread's row = the 16 channels (two 16-byte
      // core-matrix rows) of its voxel's neighbour
      // (asynchronous copies: all of a round's loads are in flight at once; a neighbour
      // outside the window copies zero bytes, which fills zeros)
      const uint32_t dstA = aBase + (uint32_t)(buf * kRound) * kTapBytesA + (tid >> 3) * kSBO +
                            (tid & 7) * 16;
#pragma unroll
      for (int s = 0; s < kRound; ++s) {
        const int t = round * kRound + s;
        const int dz = t / 9 - 1, dy = (t / 3) % 3 - 1, dx = t % 3 - 1;
        const int zz = z + dz;
        const bool in = valid && zz >= 0 && zz < a.nz;
        int yy = y + dy, xx = x + dx;
        yy += yy < 0 ? a.ny : 0;
        yy -= yy >= a.ny ? a.ny : 0;
        xx += xx < 0 ? a.nx : 0;
        xx -= xx >= a.nx ? a.nx : 0;
        const __nv_bfloat16* src =
            in ? a.x + ((long long)zz * plane + (long long)yy * a.nx + xx) * kCh : a.x;
        const uint32_t nb = in ? 16u : 0u;
        cp_async16(dstA + (uint32_t)s * kTapBytesA, src, nb);
        cp_async16(dstA + (uint32_t)s * kTapBytesA + kLBO, src + 8, nb);
      }
      cp_async_wait_all();
      fence_async_smem();
      tc_fence_before();
      __syncthreads();
      tc_fence_after();
      if (tid == 0 && !abort_flag) {
        for (int s = 0; s < kRound; ++s) {
          const int t = round * kRound + s;
          umma(tmem, sdesc(aBase + (uint32_t)(buf * kRound + s) * kTapBytesA),
               sdesc(bBase + (uint32_t)t * kTapBytesB), (round > 0 || s > 0) ? 1u : 0u);
        }
        umma_commit(&mbar[buf]);
      }
      pending[buf] = abort_flag ? 0 : 1;                      // uniform after the barrier
    }
    // epilogue: wait for this tile's last MMAs, then one warp per 32 rows
    const int last = (gr - 1) & 1;
    if (pending[last]) {
      if (!mbar_wait(&mbar[last], phase[last])) atomicExch(&abort_flag, 1);
      phase[last] ^= 1u;
      pending[last] = 0;
    }
    tc_fence_after();
    float acc[16];
    tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16), acc);
    const long long v = v0 + warp * 32 + lane;
    if (v < V && !abort_flag) epilogue(a, v, acc);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
  }
  // no MMA may still be running when the accumulator is released
  for (int b = 0; b < 2; ++b)
    if (pending[b]) {
      if (!mbar_wait(&mbar[b], phase[b])) atomicExch(&abort_flag, 1);
      phase[b] ^= 1u;
    }
  tc_fence_before();
  __syncthreads();
  if (abort_flag && tid == 0) atomicOr(a.err, 1);
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 32;" ::"r"(tmem) : "memory");
}

// ---- row-staged operands (rows of 128 voxels) ------------------------------------------------
// For nx = 128 an output tile is one row (z, y), and the A operand of tap (dz, dy, dx) is the
// input row (z + dz, y + dy) shifted by dx: with the padded rows above in shared memory (256-byte
// aligned, 32-byte swizzled K-major rows in groups of eight) it is a descriptor advanced by
// dx x 32 bytes, with no per-tap gather.
__device__ __forceinline__ uint64_t sdesc_row(uint32_t saddr) {
  return (uint64_t)((saddr & 0x3FFFFu) >> 4) | (1ull << 16) | ((uint64_t)(256u >> 4) << 32) |
         (1ull << 46) | (6ull << 61);
}

// ---- warp-specialised row convolution with the three dy taps in one MMA (rows of 128 voxels) -
// An input row (z + dz, r) feeds the output rows r - 1, r, r + 1 of plane z through the taps
// dy = +1, 0, -1.  With the operand B of a (dz, dx) pair holding those three taps' 16 x 16
// weights one under the other (N = 48) and the accumulators of consecutive output rows in
// consecutive 16-column sets of tensor memory, one MMA per (input row, dz, dx) adds all three
// contributions: 9 MMAs per output row instead of 27, each reading its 4 KB operand A once.
// A CTA takes strips of kStripW output rows of one z; the input rows y0 - 1 .. y1 are staged
// as units (three z-planes each) in a ring; set s of tensor memory holds output row
// y0 - 1 + s (sets 0 and kStripW + 1 only collect the contributions to the rows beyond the
// strip, the first and last input rows use N = 16 MMAs of the one tap that reaches into it).
// Roles: one thread stages the units, three bulk copies each (cp.async.bulk, completing on the
// unit's `full` mbarrier; the rows lie in global memory as the tensor core reads them); one
// thread issues the MMAs (after the epilogue warps zeroed the strip's accumulators), frees each
// unit through `empty` and marks each finished output row through its set's `rowd` mbarrier;
// four epilogue warps zero the accumulators, then read each finished row back and write it.
// Every wait is bounded: a wait that gives up sets the abort flag and its role stops; the MMA
// thread waits for its MMAs in flight before the tensor memory is freed, the staging thread for
// its copies before the CTA ends.
// Bound: the issuing thread and the tensor pipe, about half each.  An MMA of K = 16 takes 62-68
// cycles on its CTA whatever N <= 128 is; with two CTAs on the SM, as here, a CTA completes one in
// 88 and the SM's pipe one in 44.  MMAs are 596 of a unit's 1130 cycles; waits and commits take
// the rest.  128 x 128 x 512, 16 -> 16 channels: 346 us with
// asynchronous 16-byte copies by two warps, 325 us with bulk copies, 164 us with the two
// single-thread roles cut to a few instructions per unit (DRAM floor 75 us); last layer 500 ->
// 204 us.
constexpr int kUnits = 6;                            // ring of staged units
constexpr int kStripW = 14;                          // output rows per strip
constexpr int kSets = kStripW + 2;                   // accumulator sets (16 columns each)
constexpr int kWsThreads = 192;                      // warp 0 stages, 1 issues, 2-5 drain
constexpr uint32_t kUnitBytes = 3u * kRowBytes;      // three z-planes of one row
constexpr uint32_t kWsSmem = (uint32_t)kTaps * kTapBytesB + kUnits * kUnitBytes + 256u;
// instruction descriptors: M = 128, N = 48 (three taps) and N = 16 (one)
constexpr uint32_t kIdesc48 = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(48 >> 3) << 17) |
                              ((uint32_t)(kTile >> 4) << 24);

__device__ __forceinline__ void umma_n(uint32_t tmem_d, uint64_t a, uint64_t b, uint32_t idesc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, 1, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem_d),
      "l"(a), "l"(b), "r"(idesc));
}
__device__ __forceinline__ void mbar_arrive(uint64_t* m) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(m)) : "memory");
}
__device__ __forceinline__ void mbar_expect(uint64_t* m, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(m)), "r"(bytes)
               : "memory");
}
// bulk copy global -> shared, 16-byte aligned at both ends, completing on an mbarrier
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void* src, uint32_t bytes, uint64_t* m) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
      "l"(src), "r"(bytes), "r"(smem_u32(m))
      : "memory");
}
// zero 16 accumulator columns of this warp's 32 lanes
__device__ __forceinline__ void tmem_zero16(uint32_t taddr) {
  const uint32_t z = 0u;
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,"
      "%1,%1};" ::"r"(taddr), "r"(z)
      : "memory");
}

// What the epilogue of voxel x of row (z, y) reads: the current (last layer) or the mask
// (backward); loaded a row ahead, so that its latency passes meanwhile (the last layer took
// 0.49 ms at 128 x 128 x 512, 3.0 k cycles a row in these loads)
struct EpiIn {
  uint4 a, b;
};
__device__ __forceinline__ EpiIn epilogue_read(const ConvArgs& a, int z, int y, int x) {
  EpiIn in{};
  const long long rowi = (long long)z * a.ny + y;
  if (a.mode == MODE_LAST) {
    if (a.jout) {
      const long long plane = (long long)a.ny * kRowVox;
      const float* j = a.jres + (long long)z * 3 * plane + (long long)y * kRowVox + x;
      in.a.x = __float_as_uint(__ldcg(j));
      in.a.y = __float_as_uint(__ldcg(j + plane));
      in.a.z = __float_as_uint(__ldcg(j + 2 * plane));
    }
  } else if (a.mode == MODE_BWD) {
    const char* mr = reinterpret_cast<const char*>(a.mask) + rowi * kRowBytes;
    in.a = *reinterpret_cast<const uint4*>(mr + seg_off(x + 1, 0));
    in.b = *reinterpret_cast<const uint4*>(mr + seg_off(x + 1, 1));
  }
  return in;
}

// epilogue() for voxel x of row (z, y) of a grid of 128-voxel rows (bias already added)
__device__ __forceinline__ void epilogue_row(const ConvArgs& a, int z, int y, int x, const EpiIn& in,
                                             const float* acc) {
  const long long rowi = (long long)z * a.ny + y;
  const uint32_t o0 = seg_off(x + 1, 0), o1 = seg_off(x + 1, 1);
  if (a.mode == MODE_LAST) {
    if (a.r) *reinterpret_cast<float4*>(a.r + (rowi * kRowVox + x) * 4) = make_float4(acc[0], acc[1], acc[2], 0.0f);
    if (a.jout) {
      const long long plane = (long long)a.ny * kRowVox;
      float* j = a.jout + (long long)z * 3 * plane + (long long)y * kRowVox + x;
      j[0] = __uint_as_float(in.a.x) + a.scale * acc[0];
      j[plane] = __uint_as_float(in.a.y) + a.scale * acc[1];
      j[2 * plane] = __uint_as_float(in.a.z) + a.scale * acc[2];
    }
    return;
  }
  __align__(16) __nv_bfloat16 o[16];
  if (a.mode == MODE_HIDDEN) {
#pragma unroll
    for (int c = 0; c < 16; ++c) o[c] = __float2bfloat16_rn(fmaxf(acc[c], 0.0f));
  } else {
    __align__(16) __nv_bfloat16 m[16];
    reinterpret_cast<uint4*>(m)[0] = in.a;
    reinterpret_cast<uint4*>(m)[1] = in.b;
#pragma unroll
    for (int c = 0; c < 16; ++c) o[c] = __float2bfloat16_rn(__bfloat162float(m[c]) > 0.0f ? acc[c] : 0.0f);
  }
  char* row = reinterpret_cast<char*>(a.out) + rowi * kRowBytes;
  const uint4 h0 = reinterpret_cast<const uint4*>(o)[0], h1 = reinterpret_cast<const uint4*>(o)[1];
  *reinterpret_cast<uint4*>(row + o0) = h0;
  *reinterpret_cast<uint4*>(row + o1) = h1;
  if (x == 0 || x == kRowVox - 1) {                            // the row's periodic halo copies
    const int xh = x == 0 ? kRowVox + 1 : 0;
    *reinterpret_cast<uint4*>(row + seg_off(xh, 0)) = h0;
    *reinterpret_cast<uint4*>(row + seg_off(xh, 1)) = h1;
  }
}

__global__ void __launch_bounds__(kWsThreads) conv_ws_kernel(ConvArgs a) {
  extern __shared__ __align__(1024) unsigned char smem[];
  unsigned char* sB = smem;                                   // [9 (dz, dx)][3 (dy = +1, 0, -1)][512]
  unsigned char* sU = smem + kTaps * kTapBytesB;              // [kUnits][3 planes][kRowBytes]
  __shared__ __align__(8) uint64_t full[kUnits], empty[kUnits], rowd[kSets], zeroed, drain;
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 256;" ::"r"(
                     smem_u32(&tmem_slot))
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 0) {
    for (int u = 0; u < kUnits; ++u) {
      mbar_init(&full[u], 1);
      mbar_init(&empty[u], 1);
    }
    for (int c = 0; c < kSets; ++c) mbar_init(&rowd[c], 1);
    mbar_init(&zeroed, 4);
    mbar_init(&drain, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    abort_flag = 0;
  }
  {
    // operand B regrouped by (dz, dx): the taps dy = +1, 0, -1 one under the other
    const uint4* src = reinterpret_cast<const uint4*>(a.w);
    uint4* dst = reinterpret_cast<uint4*>(sB);
    constexpr int kBlk = (int)(kTapBytesB / 16);              // 32 uint4 per tap
    for (int i = tid; i < kTaps * kBlk; i += kWsThreads) {
      const int blk = i / kBlk, e = i - blk * kBlk;
      const int pair = blk / 3, b = blk - pair * 3;           // b = 0, 1, 2: dy = +1, 0, -1
      const int pz = pair / 3, px = pair - pz * 3;
      const int t = pz * 9 + (2 - b) * 3 + px;                // tap (dz, dy, dx) + 1
      dst[i] = src[t * kBlk + e];
    }
  }
  fence_async_smem();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  const uint32_t uBase = smem_u32(sU);
  const int nyb = (a.ny + kStripW - 1) / kStripW;
  const int nstrips = (a.zhi - a.zlo) * nyb;

  // The two single-thread roles run a few instructions per unit: ring slot and phase are
  // counters (a 64-bit modulo per unit and barrier cost the issuing thread more than its MMAs
  // take: 190 cycles per MMA where a CTA alone completes one in 62-68), descriptors advance by
  // constants.
  if (warp == 0) {
    // ---- staging: units (z, r) for r = y0-1 .. y1 of every strip, in order; one thread ----
    if (lane == 0) {
      int slot = 0;
      uint32_t phase = 0, staged = 0;               // staged: units so far, at most kUnits
      bool ok = true;
      for (int strip = blockIdx.x; strip < nstrips && ok && !abort_flag; strip += gridDim.x) {
        const int zq = strip / nyb;
        const int z = a.zlo + zq, y0 = (strip - zq * nyb) * kStripW, y1 = min(a.ny, y0 + kStripW);
        const int p0 = z == 0 ? 1 : 0, p1 = z == a.nz - 1 ? 1 : 2;   // planes inside the window
        const uint32_t bytes = (uint32_t)(p1 - p0 + 1) * kRowCopy;
        const long long plane = (long long)a.ny * kRowBytes;
        const char* base = reinterpret_cast<const char*>(a.x) + (z - 1) * plane;
        for (int r = y0 - 1; r <= y1; ++r) {
          if (!mbar_wait(&empty[slot], phase ^ 1u)) {
            atomicExch(&abort_flag, 1);
            ok = false;
            break;
          }
          const int yr = r < 0 ? r + a.ny : (r >= a.ny ? r - a.ny : r);
          const char* src = base + (long long)yr * kRowBytes;
          const uint32_t dst = uBase + (uint32_t)slot * kUnitBytes;
          mbar_expect(&full[slot], bytes);
          for (int pl = p0; pl <= p1; ++pl) bulk_g2s(dst + (uint32_t)pl * kRowBytes, src + pl * plane, kRowCopy, &full[slot]);
          staged = min(staged + 1u, (uint32_t)kUnits);
          if (++slot == kUnits) {
            slot = 0;
            phase ^= 1u;
          }
        }
      }
      // no copy may land after the CTA has ended: the last staged units' copies, newest first
      for (uint32_t k = 0; k < staged; ++k) {
        if (--slot < 0) {
          slot = kUnits - 1;
          phase ^= 1u;
        }
        if (!mbar_wait(&full[slot], phase)) atomicExch(&abort_flag, 1);
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    // ---- MMA issue: one thread ----
    if (lane == 0) {
      const uint64_t bdesc = sdesc(smem_u32(sB));
      const uint64_t adesc = sdesc_row(uBase);
      constexpr uint64_t kPair = (3u * kTapBytesB) >> 4;     // B of the next (dz, dx) pair
      constexpr uint64_t kTap = kTapBytesB >> 4;
      int slot = 0;
      uint32_t phase = 0, zphase = 0;
      bool issued = false, ok = true;
      for (int strip = blockIdx.x; strip < nstrips && ok && !abort_flag; strip += gridDim.x) {
        const int zq = strip / nyb;
        const int z = a.zlo + zq, y0 = (strip - zq * nyb) * kStripW, y1 = min(a.ny, y0 + kStripW);
        const int p0 = z == 0 ? 1 : 0, p1 = z == a.nz - 1 ? 1 : 2;
        // the epilogue warps have zeroed the accumulators of this strip
        if (!mbar_wait(&zeroed, zphase)) {
          atomicExch(&abort_flag, 1);
          break;
        }
        zphase ^= 1u;
        tc_fence_after();
        for (int r = y0 - 1; r <= y1; ++r) {
          if (!mbar_wait(&full[slot], phase)) {
            atomicExch(&abort_flag, 1);
            ok = false;
            break;
          }
          tc_fence_after();
          // rows r - 1, r, r + 1: sets r - y0 .. r - y0 + 2 (N = 48); at the strip's ends only the
          // tap that reaches into it: dy = -1 into row y0 (set 1), dy = +1 into row y1 - 1
          const bool first = r == y0 - 1, last = r == y1;
          const uint32_t d = tmem + (uint32_t)(first ? 16 : 16 * (r - y0));
          const uint32_t id = first || last ? kIdesc : kIdesc48;
          uint64_t ad = adesc + (uint64_t)((slot * kUnitBytes + (uint32_t)p0 * kRowBytes) >> 4);
          uint64_t bd = bdesc + (uint64_t)(3 * p0) * kPair + (first ? 2 * kTap : 0);
          for (int pz = p0; pz <= p1; ++pz, ad += kRowBytes >> 4, bd += 3 * kPair) {
            umma_n(d, ad, bd, id);                            // dx = -1, 0, 1: 32 bytes a voxel
            umma_n(d, ad + 2, bd + kPair, id);
            umma_n(d, ad + 4, bd + 2 * kPair, id);
          }
          issued = true;
          umma_commit(&empty[slot]);
          // output row r - 1 has all its contributions (input rows r - 2 .. r)
          if (r - 1 >= y0) umma_commit(&rowd[r - y0]);
          if (++slot == kUnits) {
            slot = 0;
            phase ^= 1u;
          }
        }
      }
      if (issued) {
        umma_commit(&drain);
        if (!mbar_wait(&drain, 0u)) atomicExch(&abort_flag, 1);
      }
    }
    __syncwarp();
  } else {
    // ---- epilogue: warps 2..5 own lanes 32 (warp % 4) .. +31 of the accumulators ----
    const int q = warp & 3;
    float bias[16];
#pragma unroll
    for (int c = 0; c < 16; ++c) bias[c] = (a.bias && a.mode != MODE_BWD) ? a.bias[c] : 0.0f;
    const uint32_t lanes = (uint32_t)(q * 32) << 16;
    // phase of each row barrier (a short strip at the end of y completes only some of them)
    uint32_t rpar = 0u;                                       // bit c: parity of rowd[c]
    for (int strip = blockIdx.x; strip < nstrips && !abort_flag; strip += gridDim.x) {
      const int zq = strip / nyb;
      const int z = a.zlo + zq, y0 = (strip - zq * nyb) * kStripW, y1 = min(a.ny, y0 + kStripW);
      // zero this strip's accumulators (the previous strip's rows have all been read)
      for (int c = 0; c < kSets; ++c) tmem_zero16(tmem + lanes + (uint32_t)(16 * c));
      asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&zeroed);
      bool ok = true;
      EpiIn next = epilogue_read(a, z, y0, q * 32 + lane);
      for (int y = y0; y < y1; ++y) {
        const int set = y - y0 + 1;
        const EpiIn in = next;
        if (y + 1 < y1) next = epilogue_read(a, z, y + 1, q * 32 + lane);
        if (!mbar_wait(&rowd[set], (rpar >> set) & 1u)) {
          atomicExch(&abort_flag, 1);
          ok = false;
          break;
        }
        rpar ^= 1u << set;
        tc_fence_after();
        float acc[16];
        tmem_ld16(tmem + lanes + (uint32_t)(16 * set), acc);
#pragma unroll
        for (int c = 0; c < 16; ++c) acc[c] += bias[c];
        epilogue_row(a, z, y, q * 32 + lane, in, acc);
      }
      tc_fence_before();
      if (!ok) break;
    }
  }
  tc_fence_before();
  __syncthreads();
  if (abort_flag && tid == 0) atomicOr(a.err, 1);
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 256;" ::"r"(tmem) : "memory");
}

// ---- element-wise kernels ------------------------------------------------------------------

// x0 = bf16(j / scale) channel-last, channels 3..15 zero, on the half-slices [zlo, zhi)
// (j is read through L2: it may have been written by a kernel still running)
__global__ void pack_input_kernel(const float* j, __nv_bfloat16* x0, int nx, int ny, int zlo,
                                  int zhi, float inv_scale) {
  const long long plane = (long long)nx * ny, v0 = plane * zlo, V = plane * zhi;
  const long long step = (long long)gridDim.x * blockDim.x;
  // four voxels in flight per thread: with one, the kernel moved 3.5 TB/s at 128 x 128 x 512
  for (long long w = v0 + blockIdx.x * (long long)blockDim.x + threadIdx.x; w < V; w += 4 * step) {
    float f[4][3];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const long long v = w + u * step;
      if (v >= V) break;
      const long long z = v / plane, rem = v - z * plane;
#pragma unroll
      for (int c = 0; c < 3; ++c) f[u][c] = __ldcg(j + (z * 3 + c) * plane + rem);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const long long v = w + u * step;
      if (v >= V) break;
      const __nv_bfloat162 lo = __floats2bfloat162_rn(f[u][0] * inv_scale, f[u][1] * inv_scale);
      const __nv_bfloat162 hi = __floats2bfloat162_rn(f[u][2] * inv_scale, 0.0f);
      uint4 a = make_uint4(0u, 0u, 0u, 0u);
      a.x = *reinterpret_cast<const uint32_t*>(&lo);
      a.y = *reinterpret_cast<const uint32_t*>(&hi);
      act_store(x0, nx, v, a, make_uint4(0u, 0u, 0u, 0u));
    }
  }
}

// e = j/scale + r - t/scale on the slices [zlo, zhi): loss += e^2 (FP64), dr = bf16(2 e / count)
// channel-last (zero elsewhere and in channels 3..15)
__global__ void loss_kernel(const float* j, const float* t, const float* r, __nv_bfloat16* dr,
                            int nx, int ny, int nz, int zlo, int zhi, float inv_scale,
                            float inv_count2, double* loss) {
  const long long plane = (long long)nx * ny, V = plane * nz;
  double acc = 0.0;
  for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < V;
       v += (long long)gridDim.x * blockDim.x) {
    const long long z = v / plane, rem = v - z * plane;
    __align__(16) __nv_bfloat16 o[16];
#pragma unroll
    for (int c = 0; c < 16; ++c) o[c] = __float2bfloat16_rn(0.0f);
    if (z >= zlo && z < zhi) {
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const long long e0 = (z * 3 + c) * plane + rem;
        const float e = (j[e0] - t[e0]) * inv_scale + r[v * 4 + c];
        acc += (double)e * e;
        o[c] = __float2bfloat16_rn(e * inv_count2);
      }
    }
    act_store(dr, nx, v, reinterpret_cast<const uint4*>(o)[0], reinterpret_cast<const uint4*>(o)[1]);
  }
  __shared__ double red[32];
  for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) acc += red[w];
    atomicAdd(loss, acc);
  }
}

// Weight gradients dW[t][ci][co] = sum over voxels v of X[v + off(t)][ci] dY[v][co] and bias
// gradients db[co] = sum dY[v][co] of the three layers in one launch (blockIdx.y = layer).  Per
// tap this is a 16 x 16 product contracted over all voxels: on the tensor cores with the voxels
// as K, straight from the channel-last rows (ldmatrix transposes both operands), FP32
// accumulators.  The warp-level mma carries it: the outputs are 16 x 16 tiles, so a tcgen05 tile
// (M >= 64) would have to gather several taps' shifted rows as one operand, and the tensor rate
// is not what binds (below).  A CTA takes a run of rows (z, x-segment, y) of up to 128 voxels:
// warp w owns the taps (dz, dy) = (w / 3 - 1, w % 3 - 1), dx = -1, 0, 1 and keeps their three
// accumulators; the nine staged input rows serve all 27 taps, and going to the next y stages
// only the three new rows (asynchronous copies, one row ahead of the products).  Each row's
// products are added to the running sums in FP32, so a chain inside the tensor core is at most
// 8 long.  Every CTA writes its partial sums; wgrad_reduce_kernel adds them in a fixed order
// (in FP64), so gradients are reproducible bit for bit.
// Bound: L2 and issue latency of the staging (16 KB per row and layer; the products are 1 % of
// the tensor rate).  A training step at 128 x 128 x 32 voxels took 3.10 ms with FP32 FMA reductions
// per tap and float atomics (2.7 ms of it here) and 0.43 ms with this kernel; 0.34 with the row
// convolution as it is now.
constexpr int kSeg = 128;                            // voxels of a row segment
constexpr int kGradWarps = 9;
constexpr int kGradThreads = 32 * kGradWarps;
constexpr uint32_t kSegBytes = (uint32_t)(kSeg + 2) * 32u;
constexpr uint32_t kGradSmem = 14u * kSegBytes;      // [4 y][3 z] input rows, 2 dY rows
constexpr int kPart = kTaps * kCh * kCh + kCh;       // partial sums per CTA and layer: dW, db

struct GradArgs {
  const __nv_bfloat16* x[3];    // layer inputs [V][16]
  const __nv_bfloat16* dy[3];   // gradients of the layer outputs [V][16]
  float* part;                  // [3][gridDim.x][kPart]
  int nx, ny, nz;
};

__device__ __forceinline__ void ldsm4t(uint32_t a, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(a)
               : "memory");
}
__device__ __forceinline__ void mma16816(float* d, const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

__global__ void __launch_bounds__(kGradThreads, 2) wgrad_kernel(GradArgs g) {
  extern __shared__ __align__(1024) unsigned char smem[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int layer = blockIdx.y;
  const __nv_bfloat16* const X = g.x[layer];
  const __nv_bfloat16* const dY = g.dy[layer];
  const uint32_t sx = smem_u32(smem), sy = sx + 12u * kSegBytes;
  const int nseg = (g.nx + kSeg - 1) / kSeg;
  const bool padded = g.nx == kRowVox;               // rows lie in memory as they are staged
  const long long rows = (long long)g.nz * nseg * g.ny;
  const long long r0 = rows * blockIdx.x / gridDim.x, r1 = rows * (blockIdx.x + 1) / gridDim.x;
  const int pz = warp / 3, py = warp - 3 * pz;       // this warp's (dz, dy) + 1
  // ldmatrix lane -> (voxel, half): matrices (v 0-7, c 0-7), (v 0-7, c 8-15), (v 8-15, c 0-7), ...
  const int lv = ((lane >> 4) & 1) * 8 + (lane & 7), lh = (lane >> 3) & 1;
  float sum[3][8], bsum[8];
#pragma unroll
  for (int i = 0; i < 24; ++i) sum[i >> 3][i & 7] = 0.0f;
#pragma unroll
  for (int i = 0; i < 8; ++i) bsum[i] = 0.0f;
  const uint32_t one2 = 0x3F803F80u;                 // two BF16 ones
  const uint32_t ones[4] = {one2, one2, one2, one2};

  // stage the input rows (z - 1 .. z + 1, y) of a segment with a halo voxel at each end; voxels
  // beyond the segment are zero (so are dY's: products beyond the row add nothing)
  auto stage_x = [&](int slot, int z, int y, int s0, int len, int kk) {
    for (int pl = 0; pl < 3; ++pl) {
      const int zz = z + pl - 1;
      if (zz < 0 || zz >= g.nz) continue;            // its warps skip their products
      const uint32_t dst = sx + (uint32_t)(slot * 3 + pl) * kSegBytes;
      if (padded) {                                  // as it lies in memory
        const char* row = reinterpret_cast<const char*>(X) + ((long long)zz * g.ny + y) * kRowBytes;
        for (int i = tid; i < (int)(kRowCopy / 16); i += kGradThreads) cp_async16(dst + i * 16, row + i * 16, 16u);
        continue;
      }
      const __nv_bfloat16* row = X + ((long long)zz * g.ny + y) * (long long)g.nx * kCh;
      for (int i = tid; i < 2 * (kk + 2); i += kGradThreads) {
        const int xi = i >> 1, h = i & 1;
        int x = s0 + xi - 1;
        x = x < 0 ? x + g.nx : x >= g.nx ? x - g.nx : x;
        const bool in = xi < len + 2;
        cp_async16(dst + seg_off(xi, h), in ? row + (long long)x * kCh + h * 8 : X, in ? 16u : 0u);
      }
    }
  };
  auto stage_y = [&](int buf, int z, int y, int s0, int len, int kk) {
    const uint32_t dst = sy + (uint32_t)buf * kSegBytes;
    if (padded) {
      const char* row = reinterpret_cast<const char*>(dY) + ((long long)z * g.ny + y) * kRowBytes;
      for (int i = tid; i < (int)(kRowCopy / 16); i += kGradThreads) cp_async16(dst + i * 16, row + i * 16, 16u);
      return;
    }
    const __nv_bfloat16* row = dY + (((long long)z * g.ny + y) * g.nx + s0) * kCh;
    for (int i = tid; i < 2 * kk; i += kGradThreads) {
      const int xi = i >> 1, h = i & 1;
      cp_async16(dst + seg_off(xi + 1, h), xi < len ? row + xi * kCh + h * 8 : dY, xi < len ? 16u : 0u);
    }
  };

  int base = 0, buf = 0;
  bool staged = false;                               // this row was staged during the last one
  for (long long r = r0; r < r1; ++r) {
    const int y = (int)(r % g.ny);
    const int zs = (int)(r / g.ny);
    const int z = zs / nseg, s0 = (zs - z * nseg) * kSeg;
    const int len = min(kSeg, g.nx - s0), kk = (len + 15) & ~15;
    if (!staged) {
      __syncthreads();                               // the last row's products are done
      for (int d = 0; d < 3; ++d) {
        int yy = y + d - 1;
        yy = yy < 0 ? yy + g.ny : yy >= g.ny ? yy - g.ny : yy;
        stage_x((base + d) & 3, z, yy, s0, len, kk);
      }
      stage_y(buf, z, y, s0, len, kk);
    }
    cp_async_wait_all();
    __syncthreads();
    staged = r + 1 < r1 && y + 1 < g.ny;
    if (staged) {
      const int yn = y + 2 >= g.ny ? y + 2 - g.ny : y + 2;
      stage_x((base + 3) & 3, z, yn, s0, len, kk);
      stage_y(buf ^ 1, z, y + 1, s0, len, kk);
    }
    if (z + pz - 1 >= 0 && z + pz - 1 < g.nz) {
      const uint32_t xrow = sx + (uint32_t)(((base + py) & 3) * 3 + pz) * kSegBytes;
      const uint32_t yrow = sy + (uint32_t)buf * kSegBytes;
      float acc[3][8], bacc[8];
#pragma unroll
      for (int i = 0; i < 24; ++i) acc[i >> 3][i & 7] = 0.0f;
#pragma unroll
      for (int i = 0; i < 8; ++i) bacc[i] = 0.0f;
      for (int k = 0; k < kk; k += 16) {
        uint32_t b[4];
        ldsm4t(yrow + seg_off(k + lv + 1, lh), b);
#pragma unroll
        for (int dx = 0; dx < 3; ++dx) {
          uint32_t a[4];
          ldsm4t(xrow + seg_off(k + lv + dx, lh), a);
          mma16816(acc[dx], a, b[0], b[2]);
          mma16816(acc[dx] + 4, a, b[1], b[3]);
        }
        if (warp == 4) {                             // column sums of dY: the bias gradient
          mma16816(bacc, ones, b[0], b[2]);
          mma16816(bacc + 4, ones, b[1], b[3]);
        }
      }
#pragma unroll
      for (int i = 0; i < 24; ++i) sum[i >> 3][i & 7] += acc[i >> 3][i & 7];
      if (warp == 4) {
#pragma unroll
        for (int i = 0; i < 8; ++i) bsum[i] += bacc[i];
      }
    }
    if (staged) {
      base = (base + 1) & 3;
      buf ^= 1;
    }
  }
  // accumulator (row, column): rows lane / 4 and + 8, columns 2 (lane % 4) + {0, 1} and + 8
  float* out = g.part + ((size_t)layer * gridDim.x + blockIdx.x) * kPart;
  const int row = lane >> 2, col = 2 * (lane & 3);
#pragma unroll
  for (int dx = 0; dx < 3; ++dx) {
    float* t = out + (pz * 9 + py * 3 + dx) * (kCh * kCh);
#pragma unroll
    for (int n = 0; n < 2; ++n)
#pragma unroll
      for (int m = 0; m < 2; ++m)
        *reinterpret_cast<float2*>(t + (row + 8 * m) * kCh + col + 8 * n) =
            make_float2(sum[dx][4 * n + 2 * m], sum[dx][4 * n + 2 * m + 1]);
  }
  if (warp == 4 && row == 0) {
#pragma unroll
    for (int n = 0; n < 2; ++n)
      *reinterpret_cast<float2*>(out + kTaps * kCh * kCh + col + 8 * n) =
          make_float2(bsum[4 * n], bsum[4 * n + 1]);
  }
}

// g[i] = the sum over the CTAs' partial sums, in FP64 and in a fixed order: 8 lanes of partial
// runs per parameter.  Parameter order: W1, b1, W2, b2, W3, b3 (W[tap][ci][co])
__global__ void __launch_bounds__(256) wgrad_reduce_kernel(const float* part, int ncta, float* g,
                                                           int n) {
  __shared__ double red[8][32];
  const int lane = threadIdx.x & 31, run = threadIdx.x >> 5;
  const int i = blockIdx.x * 32 + lane;
  double acc = 0.0;
  if (i < n) {
    constexpr int cin[3] = {3, 16, 16}, cout[3] = {16, 16, 3};
    int l = 0, o = i;
    while (l < 2 && o >= kTaps * cin[l] * cout[l] + cout[l]) {
      o -= kTaps * cin[l] * cout[l] + cout[l];
      ++l;
    }
    const int nw = kTaps * cin[l] * cout[l];
    int e;
    if (o < nw) {
      const int co = o % cout[l], tc = o / cout[l];
      e = (tc / cin[l]) * (kCh * kCh) + (tc % cin[l]) * kCh + co;
    } else {
      e = kTaps * kCh * kCh + (o - nw);
    }
    const float* p = part + (size_t)l * ncta * kPart + e;
#pragma unroll 4
    for (int c = run; c < ncta; c += 8) acc += (double)p[(size_t)c * kPart];
  }
  red[run][lane] = acc;
  __syncthreads();
  if (run == 0 && i < n) {
    double v = red[0][lane];
#pragma unroll
    for (int q = 1; q < 8; ++q) v += red[q][lane];
    g[i] = (float)v;
  }
}

// Adam (Kingma and Ba 2015) on the FP32 master parameters, bias-corrected
// (nothing is changed when a bounded wait of the gradient gave up: *err)
__global__ void adam_kernel(float* p, const float* g, float* m, float* v, int n, float lr,
                            float b1, float b2, float eps, float c1, float c2, const int* err) {
  if (*err) return;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.0f - b1) * gi;
    const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  }
}

// operands B from the FP32 parameters, one launch: blockIdx.y = layer, + 3 for the backward
// form.  K-major canonical layout, B_t[n][k] = W[t][k][n] (forward) or the mirrored tap with
// channels swapped, B_t[n][k] = W[26 - t][n][k] (backward through the input)
struct PackArgs {
  const float* W[3];
  __nv_bfloat16* B[6];
};
__global__ void pack_weights_kernel(PackArgs p) {
  constexpr int kci[3] = {3, 16, 16}, kco[3] = {16, 16, 3};
  const int t = blockIdx.x, l = blockIdx.y % 3;
  const bool bwd = blockIdx.y >= 3;
  const int cin = kci[l], cout = kco[l];
  const float* W = p.W[l];
  __nv_bfloat16* B = p.B[blockIdx.y];
  for (int e = threadIdx.x; e < 256; e += blockDim.x) {
    const int n = e >> 4, k = e & 15;
    float val = 0.0f;
    if (!bwd) {
      if (k < cin && n < cout) val = W[((size_t)t * cin + k) * cout + n];
    } else {
      if (n < cin && k < cout) val = W[((size_t)(26 - t) * cin + n) * cout + k];
    }
    const uint32_t off = (n >> 3) * kSBO + (k >> 3) * kLBO + (n & 7) * 16 + (k & 7) * 2;
    B[(size_t)t * 256 + off / 2] = __float2bfloat16_rn(val);
  }
}

}  // namespace

// ---- host side ------------------------------------------------------------------------------

struct gempic_denoiser {
  double scale = 1.0;
  int dev = 0, nsm = 0;
  float* p = nullptr;          // FP32 master parameters (layout of gempic_denoiser_params)
  float* g = nullptr;          // gradients
  float* m = nullptr;          // Adam moments
  float* v = nullptr;
  __nv_bfloat16* wf[3] = {};   // forward operands per layer
  __nv_bfloat16* wb[3] = {};   // backward operands (layers 2, 3)
  long long step = 0;
  // activations (grown on demand): x0, h1, h2, dr, dh2, dh1 channel-last; r FP32
  long long cap = 0;           // voxels of r
  size_t act_bytes = 0;        // bytes of each activation buffer
  __nv_bfloat16* act[6] = {};
  float* r = nullptr;
  float* part = nullptr;       // partial weight gradients [3][nsm][kPart] (first gradient)
  double* loss = nullptr;      // {loss sum, status word}: read back in one copy
  int* err = nullptr;          // the status word, in loss[1]
};

namespace {

constexpr int kCin[3] = {3, 16, 16}, kCout[3] = {16, 16, 3};
// offsets of W1, b1, W2, b2, W3, b3 in the parameter vector
size_t woff(int l) {
  size_t o = 0;
  for (int i = 0; i < l; ++i) o += (size_t)kTaps * kCin[i] * kCout[i] + kCout[i];
  return o;
}
size_t boff(int l) { return woff(l) + (size_t)kTaps * kCin[l] * kCout[l]; }
size_t nparams() { return woff(3); }

size_t conv_smem() { return (size_t)kTaps * kTapBytesB + 2u * kRound * kTapBytesA; }

// buffers for nx x ny x nz voxels (activations in their layout's size)
cudaError_t grow(gempic_denoiser* d, int nx, int ny, int nz) {
  long long V = (long long)nx * ny * nz;
  size_t bytes = nx == kRowVox ? (size_t)ny * nz * kRowBytes : (size_t)V * kCh * sizeof(__nv_bfloat16);
  if (bytes <= d->act_bytes && V <= d->cap) return cudaSuccess;
  bytes = std::max(bytes, d->act_bytes);           // neither shrinks: calls may alternate layouts
  V = std::max(V, d->cap);
  for (auto*& a : d->act) {
    if (a) cudaFree(a);
    a = nullptr;
  }
  if (d->r) cudaFree(d->r);
  d->r = nullptr;
  d->cap = 0;
  d->act_bytes = 0;
  cudaError_t e = cudaSuccess;
  for (auto*& a : d->act)
    if (e == cudaSuccess) e = cudaMalloc(&a, bytes);
  if (e == cudaSuccess) e = cudaMalloc(&d->r, (size_t)V * 4 * sizeof(float));
  if (e == cudaSuccess) {
    d->cap = V;
    d->act_bytes = bytes;
  }
  return e;
}

cudaError_t repack(gempic_denoiser* d, cudaStream_t s) {
  PackArgs a;
  for (int l = 0; l < 3; ++l) {
    a.W[l] = d->p + woff(l);
    a.B[l] = d->wf[l];
    a.B[3 + l] = d->wb[l];
  }
  pack_weights_kernel<<<dim3(kTaps, 6), 256, 0, s>>>(a);
  return cudaGetLastError();
}

cudaError_t conv(gempic_denoiser* d, ConvArgs a, cudaStream_t s) {
  a.err = d->err;
  if (a.zhi <= a.zlo) {                  // whole window unless a range was given
    a.zlo = 0;
    a.zhi = a.nz;
  }
  if (a.nx == kRowVox) {
    const long long strips = (long long)(a.zhi - a.zlo) * ((a.ny + kStripW - 1) / kStripW);
    const int grid = (int)std::min<long long>(strips, 2LL * d->nsm);
    conv_ws_kernel<<<grid, kWsThreads, kWsSmem, s>>>(a);
    return cudaGetLastError();
  }
  const long long V = (long long)a.nx * a.ny * (a.zhi - a.zlo);
  const long long tiles = (V + kTile - 1) / kTile;
  const int grid = (int)std::min<long long>(tiles, 2LL * d->nsm);
  conv_kernel<<<grid, kThreads, conv_smem(), s>>>(a);
  return cudaGetLastError();
}

bool grid_ok(int nx, int ny, int nz) { return nx >= 1 && ny >= 1 && nz >= 1; }

// forward pass of the three layers on x0 = act[0]; h1 -> act[1], h2 -> act[2]; last layer's
// epilogue as requested, for the output half-slices [z0, z1): each layer is computed where the
// next one reads it (one more half-slice on each side per layer below the last)
cudaError_t forward(gempic_denoiser* d, int nx, int ny, int nz, int z0, int z1, const float* jres,
                    float* jout, float* r, cudaStream_t s) {
  ConvArgs a{};
  a.nx = nx;
  a.ny = ny;
  a.nz = nz;
  a.zlo = std::max(0, z0 - 2);
  a.zhi = std::min(nz, z1 + 2);
  a.mode = MODE_HIDDEN;
  a.x = d->act[0];
  a.w = d->wf[0];
  a.bias = d->p + boff(0);
  a.out = d->act[1];
  cudaError_t e = conv(d, a, s);
  if (e != cudaSuccess) return e;
  a.x = d->act[1];
  a.w = d->wf[1];
  a.bias = d->p + boff(1);
  a.out = d->act[2];
  a.zlo = std::max(0, z0 - 1);
  a.zhi = std::min(nz, z1 + 1);
  e = conv(d, a, s);
  if (e != cudaSuccess) return e;
  ConvArgs l{};
  l.nx = nx;
  l.ny = ny;
  l.nz = nz;
  l.zlo = z0;
  l.zhi = z1;
  l.mode = MODE_LAST;
  l.x = d->act[2];
  l.w = d->wf[2];
  l.bias = d->p + boff(2);
  l.r = r;
  l.jres = jres;
  l.jout = jout;
  l.scale = (float)d->scale;
  return conv(d, l, s);
}

gempic_status check_err(gempic_denoiser* d, cudaStream_t s) {
  int err = 0;
  cudaError_t e = cudaMemcpyAsync(&err, d->err, sizeof(int), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return GEMPIC_ECUDA;
  return err ? GEMPIC_ETIMEOUT : GEMPIC_OK;
}

}  // namespace

namespace gempic {

// The net on the output half-slices [z0, z1) of j_in (read where needed: z0 - 3 .. z1 + 2),
// into the same half-slices of j_out, on stream s (no wait).  For the denoised chain of
// marches: j_in may still be written elsewhere outside the half-slices the net reads.
int denoise_range(gempic_denoiser* d, const float* j_in, float* j_out, int nx, int ny, int nz,
                  int z0, int z1, cudaStream_t s) {
  if (!d || !j_in || !j_out || !grid_ok(nx, ny, nz) || z0 < 0 || z1 > nz || z0 >= z1)
    return GEMPIC_EINVAL;
  cudaError_t e = grow(d, nx, ny, nz);
  if (e != cudaSuccess) return e == cudaErrorMemoryAllocation ? GEMPIC_ENOMEM : GEMPIC_ECUDA;
  const int p0 = std::max(0, z0 - 3), p1 = std::min(nz, z1 + 3);
  const long long V = (long long)nx * ny * (p1 - p0);
  const int blocks = (int)std::min<long long>((V + 255) / 256, 8LL * d->nsm);
  pack_input_kernel<<<blocks, 256, 0, s>>>(j_in, d->act[0], nx, ny, p0, p1, (float)(1.0 / d->scale));
  e = cudaGetLastError();
  if (e == cudaSuccess) e = forward(d, nx, ny, nz, z0, z1, j_in, j_out, nullptr, s);
  return e == cudaSuccess ? GEMPIC_OK : GEMPIC_ECUDA;
}

// the denoiser's device status word (a bounded wait that gave up): GEMPIC_ETIMEOUT
int denoise_status(gempic_denoiser* d, cudaStream_t s) { return check_err(d, s); }

// working buffers for nx x ny x nz currents, allocated now: growing them frees the old ones,
// and cudaFree waits for the whole device -- while the chain of marches runs, that would wait
// for marches that wait for the net
int denoise_reserve(gempic_denoiser* d, int nx, int ny, int nz) {
  if (!d || !grid_ok(nx, ny, nz)) return GEMPIC_EINVAL;
  cudaError_t e = grow(d, nx, ny, nz);
  // the net's kernels are loaded now: with lazy module loading a kernel's first launch loads
  // its module, which can wait for the device -- for marches that wait for that kernel
  cudaFuncAttributes fa;
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, pack_input_kernel);
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, conv_kernel);
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, conv_ws_kernel);
  return e == cudaSuccess ? GEMPIC_OK : e == cudaErrorMemoryAllocation ? GEMPIC_ENOMEM : GEMPIC_ECUDA;
}

}  // namespace gempic

extern "C" {

size_t gempic_denoiser_param_count(void) { return nparams(); }

gempic_status gempic_denoiser_create(const float* params, double scale, gempic_denoiser** out) {
  if (!out || !(scale > 0) || !std::isfinite(scale)) return GEMPIC_EINVAL;
  *out = nullptr;
  gempic_denoiser* d = new (std::nothrow) gempic_denoiser();
  if (!d) return GEMPIC_ENOMEM;
  d->scale = scale;
  cudaError_t e = cudaGetDevice(&d->dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&d->nsm, cudaDevAttrMultiProcessorCount, d->dev);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(conv_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)conv_smem());
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(conv_ws_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)kWsSmem);
  const size_t n = nparams();
  float** bufs[4] = {&d->p, &d->g, &d->m, &d->v};
  for (float** b : bufs)
    if (e == cudaSuccess) e = cudaMalloc(b, n * sizeof(float));
  for (int l = 0; l < 3 && e == cudaSuccess; ++l) {
    e = cudaMalloc(&d->wf[l], kTaps * 256 * sizeof(__nv_bfloat16));
    if (e == cudaSuccess) e = cudaMalloc(&d->wb[l], kTaps * 256 * sizeof(__nv_bfloat16));
  }
  if (e == cudaSuccess) e = cudaMalloc(&d->loss, 2 * sizeof(double));
  if (e == cudaSuccess) e = cudaMemset(d->loss, 0, 2 * sizeof(double));
  if (e == cudaSuccess) d->err = reinterpret_cast<int*>(d->loss + 1);
  if (e == cudaSuccess) e = cudaMemset(d->m, 0, n * sizeof(float));
  if (e == cudaSuccess) e = cudaMemset(d->v, 0, n * sizeof(float));
  if (e == cudaSuccess) {
    if (params) {
      e = cudaMemcpy(d->p, params, n * sizeof(float), cudaMemcpyHostToDevice);
    } else {
      e = cudaMemset(d->p, 0, n * sizeof(float));   // all zero: the identity on j
    }
  }
  if (e == cudaSuccess) e = repack(d, nullptr);
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  if (e != cudaSuccess) {
    gempic_denoiser_destroy(d);
    cudaGetLastError();
    return e == cudaErrorMemoryAllocation ? GEMPIC_ENOMEM : GEMPIC_ECUDA;
  }
  *out = d;
  return GEMPIC_OK;
}

gempic_status gempic_denoiser_set_params(gempic_denoiser* d, const float* params, size_t n) {
  if (!d || !params || n != nparams()) return GEMPIC_EINVAL;
  cudaError_t e = cudaMemcpy(d->p, params, n * sizeof(float), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemset(d->m, 0, n * sizeof(float));
  if (e == cudaSuccess) e = cudaMemset(d->v, 0, n * sizeof(float));
  if (e == cudaSuccess) e = repack(d, nullptr);
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  d->step = 0;
  return e == cudaSuccess ? GEMPIC_OK : GEMPIC_ECUDA;
}

gempic_status gempic_denoiser_get_params(gempic_denoiser* d, float* params, size_t n) {
  if (!d || !params || n != nparams()) return GEMPIC_EINVAL;
  cudaError_t e = cudaMemcpy(params, d->p, n * sizeof(float), cudaMemcpyDeviceToHost);
  return e == cudaSuccess ? GEMPIC_OK : GEMPIC_ECUDA;
}

gempic_status gempic_denoiser_apply(gempic_denoiser* d, const float* j_in, float* j_out,
                                    int32_t nx, int32_t ny, int32_t nz, void* cuda_stream) {
  if (!d || !j_in || !j_out || !grid_ok(nx, ny, nz)) return GEMPIC_EINVAL;
  cudaStream_t s = (cudaStream_t)cuda_stream;
  const long long V = (long long)nx * ny * nz;
  cudaError_t e = grow(d, nx, ny, nz);
  if (e != cudaSuccess) return e == cudaErrorMemoryAllocation ? GEMPIC_ENOMEM : GEMPIC_ECUDA;
  const int blocks = (int)std::min<long long>((V + 255) / 256, 8LL * d->nsm);
  pack_input_kernel<<<blocks, 256, 0, s>>>(j_in, d->act[0], nx, ny, 0, nz, (float)(1.0 / d->scale));
  e = cudaGetLastError();
  if (e == cudaSuccess) e = forward(d, nx, ny, nz, 0, nz, j_in, j_out, nullptr, s);
  if (e != cudaSuccess) return GEMPIC_ECUDA;
  return check_err(d, s);
}

}  // extern "C"

namespace {

// the loss sum and the gradient of the parameters into d->loss, d->g (device), no wait
gempic_status gradient(gempic_denoiser* d, const float* j_in, const float* j_target, int nx, int ny,
                       int nz, int z_margin, cudaStream_t s) {
  const long long V = (long long)nx * ny * nz;
  cudaError_t e = grow(d, nx, ny, nz);
  if (e == cudaSuccess && !d->part) {
    e = cudaFuncSetAttribute(wgrad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGradSmem);
    if (e == cudaSuccess) e = cudaMalloc(&d->part, (size_t)3 * d->nsm * kPart * sizeof(float));
    if (e != cudaSuccess) d->part = nullptr;
  }
  if (e != cudaSuccess) return e == cudaErrorMemoryAllocation ? GEMPIC_ENOMEM : GEMPIC_ECUDA;
  const int blocks = (int)std::min<long long>((V + 255) / 256, 8LL * d->nsm);
  if (cudaMemsetAsync(d->loss, 0, sizeof(double), s) != cudaSuccess) return GEMPIC_ECUDA;
  pack_input_kernel<<<blocks, 256, 0, s>>>(j_in, d->act[0], nx, ny, 0, nz, (float)(1.0 / d->scale));
  e = forward(d, nx, ny, nz, 0, nz, nullptr, nullptr, d->r, s);
  if (e != cudaSuccess) return GEMPIC_ECUDA;
  const double count = 3.0 * (double)nx * ny * (nz - 2 * z_margin);
  loss_kernel<<<blocks, 256, 0, s>>>(j_in, j_target, d->r, d->act[3], nx, ny, nz, z_margin,
                                     nz - z_margin, (float)(1.0 / d->scale), (float)(2.0 / count),
                                     d->loss);
  // backward: dr = act[3]; dh2 = mask(h2) conv(dr, W3'); dh1 = mask(h1) conv(dh2, W2')
  __nv_bfloat16* const dr = d->act[3];
  __nv_bfloat16* const dh2 = d->act[4];
  __nv_bfloat16* const dh1 = d->act[5];
  ConvArgs b{};
  b.nx = nx;
  b.ny = ny;
  b.nz = nz;
  b.mode = MODE_BWD;
  b.x = dr;
  b.w = d->wb[2];
  b.mask = d->act[2];
  b.out = dh2;
  e = conv(d, b, s);
  if (e == cudaSuccess) {
    b.x = dh2;
    b.w = d->wb[1];
    b.mask = d->act[1];
    b.out = dh1;
    e = conv(d, b, s);
  }
  if (e != cudaSuccess) return GEMPIC_ECUDA;
  // two CTAs per SM over the three layers, at least one row each
  const long long rows = (long long)nz * ny * ((nx + kSeg - 1) / kSeg);
  const int gx = (int)std::min<long long>(rows, std::max(1, 2 * d->nsm / 3));
  const GradArgs ga{{d->act[0], d->act[1], d->act[2]}, {dh1, dh2, dr}, d->part, nx, ny, nz};
  wgrad_kernel<<<dim3((unsigned)gx, 3), kGradThreads, kGradSmem, s>>>(ga);
  const int n = (int)nparams();
  wgrad_reduce_kernel<<<(n + 31) / 32, 256, 0, s>>>(d->part, gx, d->g, n);
  return cudaGetLastError() == cudaSuccess ? GEMPIC_OK : GEMPIC_ECUDA;
}

// wait for the stream; the loss and the status word
gempic_status finish(gempic_denoiser* d, double count, double* loss, cudaStream_t s) {
  double back[2] = {0.0, 0.0};
  cudaError_t e = cudaMemcpyAsync(back, d->loss, sizeof(back), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return GEMPIC_ECUDA;
  if (loss) *loss = back[0] / count;
  int err = 0;
  std::memcpy(&err, &back[1], sizeof(err));
  return err ? GEMPIC_ETIMEOUT : GEMPIC_OK;
}

bool grad_args_ok(gempic_denoiser* d, const float* j_in, const float* j_target, int nx, int ny, int nz,
                  int z_margin) {
  return d && j_in && j_target && grid_ok(nx, ny, nz) && z_margin >= 0 && 2 * z_margin < nz;
}

}  // namespace

extern "C" {

gempic_status gempic_denoiser_grad(gempic_denoiser* d, const float* j_in, const float* j_target,
                                   int32_t nx, int32_t ny, int32_t nz, int32_t z_margin,
                                   double* loss, float* grad_host, void* cuda_stream) {
  if (!grad_args_ok(d, j_in, j_target, nx, ny, nz, z_margin)) return GEMPIC_EINVAL;
  cudaStream_t s = (cudaStream_t)cuda_stream;
  const gempic_status st = gradient(d, j_in, j_target, nx, ny, nz, z_margin, s);
  if (st != GEMPIC_OK) return st;
  if (grad_host && cudaMemcpyAsync(grad_host, d->g, nparams() * sizeof(float), cudaMemcpyDeviceToHost,
                                   s) != cudaSuccess)
    return GEMPIC_ECUDA;
  return finish(d, 3.0 * (double)nx * ny * (nz - 2 * z_margin), loss, s);
}

// one wait per step: Adam and the repacking are queued behind the gradient and change nothing
// when a bounded wait in it gave up
gempic_status gempic_denoiser_train_step(gempic_denoiser* d, const float* j_in,
                                         const float* j_target, int32_t nx, int32_t ny,
                                         int32_t nz, int32_t z_margin, double lr, double* loss,
                                         void* cuda_stream) {
  if (!(lr > 0) || !std::isfinite(lr)) return GEMPIC_EINVAL;
  if (!grad_args_ok(d, j_in, j_target, nx, ny, nz, z_margin)) return GEMPIC_EINVAL;
  cudaStream_t s = (cudaStream_t)cuda_stream;
  gempic_status st = gradient(d, j_in, j_target, nx, ny, nz, z_margin, s);
  if (st != GEMPIC_OK) return st;
  const long long step = d->step + 1;
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = (float)(1.0 - std::pow(0.9, (double)step));
  const float c2 = (float)(1.0 - std::pow(0.999, (double)step));
  const int n = (int)nparams();
  adam_kernel<<<(n + 255) / 256, 256, 0, s>>>(d->p, d->g, d->m, d->v, n, (float)lr, b1, b2, 1e-8f,
                                               c1, c2, d->err);
  if (cudaGetLastError() != cudaSuccess || repack(d, s) != cudaSuccess) return GEMPIC_ECUDA;
  st = finish(d, 3.0 * (double)nx * ny * (nz - 2 * z_margin), loss, s);
  if (st == GEMPIC_OK) d->step = step;
  return st;
}

void gempic_denoiser_destroy(gempic_denoiser* d) {
  if (!d) return;
  cudaDeviceSynchronize();
  float* bufs[4] = {d->p, d->g, d->m, d->v};
  for (float* b : bufs)
    if (b) cudaFree(b);
  for (int l = 0; l < 3; ++l) {
    if (d->wf[l]) cudaFree(d->wf[l]);
    if (d->wb[l]) cudaFree(d->wb[l]);
  }
  for (auto* a : d->act)
    if (a) cudaFree(a);
  if (d->r) cudaFree(d->r);
  if (d->part) cudaFree(d->part);
  if (d->loss) cudaFree(d->loss);
  cudaGetLastError();
  delete d;
}

}  // extern "C"
