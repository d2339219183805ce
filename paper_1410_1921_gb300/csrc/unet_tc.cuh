// unet_tc.cuh -- the 3x3x3 convolutions of the learned warm start's U-Net (it
// predicts the steady velocity and concentration fields from the structure)
// on the 5th-generation tensor cores: tcgen05.mma with the accumulator in
// tensor memory, operands staged in shared memory by TMA.
//
// Activations are BF16 in NDHWC layout (channels last); weights are kept in
// FP32 (master copy for Adam) and converted to BF16 operand layouts before
// each pass.  With o_k = (k/9 - 1, k/3 % 3 - 1, k % 3 - 1) over (z, y, x) and
// zero padding at the box faces:
//   forward    Y[v][n] = sum_k sum_c X[v + o_k][c] WT[k][n][c]
//   data grad  the forward kernels on dY with WT[k][ci][co] = W[26-k][ci][co]
//   weight grad  dW[k][ci][co] = sum_v X[v + o_k][ci] dY[v][co]
// Kernels: conv3d_tc (below), conv3d_tc_zm (inputs of up to 96 channels:
// resident weights, one plane at a time), conv3d_wgrad_tc and
// conv3d_wgrad_tc32 (the weight gradient; the second for at most 32 output
// channels).
//
// conv3d_tc: implicit GEMM  Y[v][n] = sum_k sum_c X[v + o_k][c] WT[k][n][c]  with a CTA
// tile of M = 128 voxels (a box of 8 x 8 x 2 voxels in x, y, z) and all N
// output channels (16..256).  For each of the 27 offsets o_k and each
// 64-channel chunk of each input, TMA copies
//   A: the voxel box shifted by o_k, 64 channels -- a 5-D box {64, 8, 8, 2, 1}
//      of the NDHWC activation tensor (channels, x, y, z, batch); the box's
//      part outside the grid (and channels past the input's count) is
//      filled with zeros by the copy itself, which is the convolution's
//      zero padding at the box faces;
//   B: 64 columns of the N weight rows of offset k, a 2-D box {64, N} of
//      WT[27 N][K];
// both K-major with the 128-byte swizzle, into one of three stages.  One
// thread (warp 0) issues the copies, another (warp 1) per stage four MMAs of
// K = 16 (cta_group::1, kind::f16: BF16 x BF16 -> FP32, M = 128)
// accumulating in TMEM; tcgen05.commit frees a stage when its MMAs have
// read it.  The epilogue reads the accumulator with tcgen05.ld (warp w owns
// TMEM lanes = tile rows 32w..32w+31), adds the bias, applies ReLU and
// stores BF16 (and an FP32 copy) for the rows inside the grid.
//
// Every wait on an mbarrier is bounded; a wait that runs out stops both
// issuing threads, sets the error word, lets what was issued finish (again
// bounded), frees the CTA's TMEM and returns without writing.
#pragma once

#include <cuda.h>  // CUtensorMap (the type only; the encoder is fetched through the runtime)

#include <cuda_bf16.h>

#include "common.cuh"

namespace om {
namespace nn {

typedef __nv_bfloat16 bf16;

struct Grid {
  int B, D, H, W;
  __host__ __device__ int64_t voxels() const { return (int64_t)B * D * H * W; }
};

constexpr int kTcM = 128;            // voxels per CTA tile (8 x 8 x 2 box)
constexpr int kTcKc = 64;            // channels per stage (128 bytes of BF16: one swizzle span)
constexpr int kTcStages = 3;
constexpr int kTcThreads = 128;
constexpr uint32_t kTcATile = kTcM * kTcKc * 2;  // 16 KB
constexpr unsigned long long kTcSpin = 1ull << 26;  // try_wait rounds before giving up
// the plane-marching form's and the weight gradient's tile (8 x 16 voxels at one z) and its halo box
constexpr int kTcTx = 8, kTcTy = 16;
constexpr int kTcHx = kTcTx + 2, kTcHy = kTcTy + 2;

struct TcConvArgs {
  int c1, c2;         // channels of the two inputs (c2 = 0: one input)
  int N;              // output channels (multiple of 16, <= 256)
  const float* bias;  // [N] or null
  bf16* y;            // output rows of ldy elements, channels [oy, oy + N)
  int ldy, oy;
  int relu;
  Grid g;
  int tx, ty, tz;     // tiles along x, y, z (8, 8, 2 voxels each; the plane-marching form: 8, 16)
  // the plane-marching form: N is one part's output channels, of npart parts
  int nhalo, nacc;    // its halo buffers and the planes of its accumulator ring
  int nw, npart;      // weight rows per offset in WT (all parts), parts
  int* err;           // set when a wait ran out
};

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
// bounded wait for the phase with the given parity to complete; false if it
// ran out or (checked every 1024 rounds) another thread set *stop
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, const volatile int* stop = nullptr) {
  for (unsigned long long i = 0; i < kTcSpin; ++i) {
    uint32_t done;
    asm volatile(
        "{\n.reg .pred p;\n"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        "selp.u32 %0, 1, 0, p;\n}"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    if (done) return true;
    if (stop && (i & 1023) == 1023 && *stop) return false;
  }
  return false;
}

__device__ __forceinline__ void tma_load_5d(uint32_t dst, const CUtensorMap* map, int c0, int c1, int c2, int c3,
                                            int c4, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.5d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, "
      "%5, %6}], [%7];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, int c0, int c1, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], "
      "[%4];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(bar)
      : "memory");
}

// Shared-memory matrix descriptor of a K-major operand tile with the
// 128-byte swizzle: rows of 128 bytes (64 BF16), 8-row atoms 1024 bytes
// apart (stride byte offset), the leading byte offset unused for this
// layout (encoded 1), descriptor version 1, layout type 2 (128-byte
// swizzle).  The tile starts 1024-byte aligned; the k-th 16-element slice
// of the 64 starts 32 k bytes further.
__device__ __forceinline__ uint64_t sw128_desc(uint32_t addr) {
  return (uint64_t)((addr >> 4) & 0x3FFFu) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) |
         ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}

// Instruction descriptor, kind::f16: FP32 accumulator (bits 4-5 = 1), A and
// B BF16 (bits 7-9, 10-12 = 1), both K-major (bits 15, 16 = 0), N / 8 in
// bits 17-22, M / 16 in bits 24-28.
__host__ __device__ constexpr uint32_t tc_idesc(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// One MMA / one commit, issued by one lane of a converged warp (`lead`: elect_lane(), taken once).
// The whole warp runs the issuing loop, its warp index taken through a shuffle, and the
// instruction is predicated instead of branched around: then the compiler keeps descriptors in
// uniform registers, where the instruction wants them, and only their low words change.  Under a
// single thread's branch, with 64-bit descriptor arithmetic, issuing cost 70 to 110 clocks per MMA,
// more than most of these MMAs take.
__device__ __forceinline__ uint32_t elect_lane() {
  uint32_t lead;
  asm volatile("{\n.reg .pred q;\nelect.sync _|q, 0xffffffff;\nselp.u32 %0, 1, 0, q;\n}" : "=r"(lead));
  return lead;
}
// descriptors as (low word, high word): the start-address field lies in the low word
__device__ __forceinline__ void mma_f16(uint32_t lead, uint32_t d, uint32_t alo, uint32_t ahi, uint32_t blo, uint32_t bhi,
                                        uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n.reg .pred p, q;\n.reg .b64 a, b;\nsetp.ne.b32 q, %0, 0;\nsetp.ne.b32 p, %7, 0;\n"
      "mov.b64 a, {%2, %3};\nmov.b64 b, {%4, %5};\n"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%1], a, b, %6, p;\n}" ::"r"(lead),
      "r"(d), "r"(alo), "r"(ahi), "r"(blo), "r"(bhi), "r"(idesc), "r"(acc)
      : "memory");
}
__device__ __forceinline__ void mma_commit(uint32_t lead, uint32_t bar) {
  asm volatile(
      "{\n.reg .pred q;\nsetp.ne.b32 q, %0, 0;\n"
      "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%1];\n}" ::"r"(lead),
      "r"(bar)
      : "memory");
}
__device__ __forceinline__ uint32_t lo32(uint64_t v) { return (uint32_t)v; }
__device__ __forceinline__ uint32_t hi32(uint64_t v) { return (uint32_t)(v >> 32); }
// mbar_wait by a whole warp with one answer for all its lanes
__device__ __forceinline__ bool warp_wait(uint32_t bar, uint32_t parity, const volatile int* stop) {
  uint32_t now;
  asm volatile(
      "{\n.reg .pred p;\n"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      "selp.u32 %0, 1, 0, p;\n}"
      : "=r"(now)
      : "r"(bar), "r"(parity)
      : "memory");
  if (__all_sync(0xffffffffu, now)) return true;
  return __all_sync(0xffffffffu, mbar_wait(bar, parity, stop)) != 0;
}
__device__ __forceinline__ int warp_index() { return __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0); }

__global__ void __launch_bounds__(kTcThreads) conv3d_tc(const __grid_constant__ CUtensorMap map1,
                                                        const __grid_constant__ CUtensorMap map2,
                                                        const __grid_constant__ CUtensorMap mapw, TcConvArgs a) {
  extern __shared__ uint8_t tc_smem_raw[];
  // stages 1024-byte aligned: [A 16 KB][B N x 128 B] x kTcStages, then the barriers
  const uint32_t raw = smem_u32(tc_smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* gbase = tc_smem_raw + (base - raw);
  const uint32_t btile = (uint32_t)a.N * 128u;
  const uint32_t stage_bytes = kTcATile + btile;
  uint64_t* bars = reinterpret_cast<uint64_t*>(gbase + kTcStages * stage_bytes);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * kTcStages + 1);
  __shared__ volatile int stop;         // a wait ran out: issue nothing more
  __shared__ int n_issued, n_consumed;  // copies issued / waited for by the MMA thread
  const uint32_t full0 = smem_u32(bars), empty0 = full0 + 8u * kTcStages, done = full0 + 16u * kTcStages;
  const int tid = threadIdx.x, warp = warp_index(), lane = tid & 31;

  // tile coordinates
  int t = blockIdx.x;
  const int bx = t % a.tx;
  t /= a.tx;
  const int by = t % a.ty;
  t /= a.ty;
  const int bz = t % a.tz;
  const int bb = t / a.tz;
  const int x0 = bx * 8, y0 = by * 8, z0 = bz * 2;

  const uint32_t ncols = a.N <= 32 ? 32u : (a.N <= 64 ? 64u : (a.N <= 128 ? 128u : 256u));
  if (tid == 0) {
    stop = 0;
    n_issued = 0;
    n_consumed = 0;
    for (int s = 0; s < kTcStages; ++s) {
      mbar_init(full0 + 8u * s, 1);
      mbar_init(empty0 + 8u * s, 1);
    }
    mbar_init(done, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(ncols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;

  const int n1 = (a.c1 + kTcKc - 1) / kTcKc, n2 = (a.c2 + kTcKc - 1) / kTcKc;
  const int per_k = n1 + n2, nsteps = 27 * per_k;
  if (tid == 0) {
    // producer: step s = (offset k, chunk j) into stage s % kTcStages once
    // the MMAs of step s - kTcStages have read that stage
    int s = 0;
    for (; s < nsteps; ++s) {
      const int st = s % kTcStages;
      if (s >= kTcStages && !mbar_wait(empty0 + 8u * st, (uint32_t)(s / kTcStages - 1) & 1u, &stop)) break;
      if (stop) break;
      const int k = s / per_k, j = s % per_k;
      const int dz = k / 9 - 1, dy = (k / 3) % 3 - 1, dx = k % 3 - 1;
      const uint32_t sa = base + (uint32_t)st * stage_bytes, sb = sa + kTcATile;
      const uint32_t fb = full0 + 8u * st;
      mbar_expect_tx(fb, kTcATile + btile);
      int cw;  // column of WT's K dimension
      if (j < n1) {
        tma_load_5d(sa, &map1, j * kTcKc, x0 + dx, y0 + dy, z0 + dz, bb, fb);
        cw = j * kTcKc;
      } else {
        tma_load_5d(sa, &map2, (j - n1) * kTcKc, x0 + dx, y0 + dy, z0 + dz, bb, fb);
        cw = a.c1 + (j - n1) * kTcKc;
      }
      tma_load_2d(sb, &mapw, cw, k * a.N, fb);
    }
    n_issued = s;
    if (s < nsteps) stop = 1;
  } else if (warp == 1) {
    // MMA issue: four K = 16 slices per stage, accumulating in TMEM
    const uint32_t idesc = tc_idesc(kTcM, a.N), lead = elect_lane(), dhi = hi32(sw128_desc(0u));
    int s = 0;
    for (; s < nsteps; ++s) {
      const int st = s % kTcStages;
      if (!warp_wait(full0 + 8u * st, (uint32_t)(s / kTcStages) & 1u, &stop)) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t sa = base + (uint32_t)st * stage_bytes, sb = sa + kTcATile;
      const uint32_t alo = lo32(sw128_desc(sa)), blo = lo32(sw128_desc(sb));
#pragma unroll
      for (int kk = 0; kk < kTcKc / 16; ++kk)
        mma_f16(lead, tmem, alo + 2u * kk, dhi, blo + 2u * kk, dhi, idesc, (s > 0 || kk > 0) ? 1u : 0u);
      mma_commit(lead, empty0 + 8u * st);
    }
    n_consumed = s;
    if (s < nsteps) stop = 1;
    // `done` fires when every MMA issued above has completed
    mma_commit(lead, done);
  }
  const bool fin = mbar_wait(done, 0);
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  // one decision for the whole CTA (the epilogue's TMEM loads are warp-collective)
  const bool failed = __syncthreads_or(!fin || stop) != 0;
  if (failed && tid == 0) {
    atomicExch(a.err, 1);
    // copies still in flight land in their stages: wait for them (bounded)
    for (int s = n_consumed; s < n_issued; ++s)
      (void)mbar_wait(full0 + 8u * (s % kTcStages), (uint32_t)(s / kTcStages) & 1u);
  }

  // epilogue: warp w reads TMEM lanes 32w..32w+31 = tile rows
  if (!failed) {
    const int r = warp * 32 + lane;
    const int xx = x0 + (r & 7), yy = y0 + ((r >> 3) & 7), zz = z0 + (r >> 6);
    const bool inside = xx < a.g.W && yy < a.g.H && zz < a.g.D;
    const int64_t v = inside ? (((int64_t)bb * a.g.D + zz) * a.g.H + yy) * a.g.W + xx : 0;
    for (int c0 = 0; c0 < a.N; c0 += 16) {
      uint32_t q[16];
      const uint32_t taddr = tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c0;
      asm volatile(
          "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, "
          "%14, %15}, [%16];"
          : "=r"(q[0]), "=r"(q[1]), "=r"(q[2]), "=r"(q[3]), "=r"(q[4]), "=r"(q[5]), "=r"(q[6]), "=r"(q[7]),
            "=r"(q[8]), "=r"(q[9]), "=r"(q[10]), "=r"(q[11]), "=r"(q[12]), "=r"(q[13]), "=r"(q[14]), "=r"(q[15])
          : "r"(taddr));
      asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
      if (!inside) continue;
      float f[16];
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        f[i] = __uint_as_float(q[i]) + (a.bias ? a.bias[c0 + i] : 0.f);
        if (a.relu) f[i] = fmaxf(f[i], 0.f);
      }
      uint32_t p[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const __nv_bfloat162 h = __floats2bfloat162_rn(f[2 * i], f[2 * i + 1]);
        p[i] = *reinterpret_cast<const uint32_t*>(&h);
      }
      uint4* dst = reinterpret_cast<uint4*>(a.y + v * a.ldy + a.oy + c0);
      dst[0] = make_uint4(p[0], p[1], p[2], p[3]);
      dst[1] = make_uint4(p[4], p[5], p[6], p[7]);
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ncols) : "memory");
}

// ------------------------------------------------------------------ plane-marching form
// conv3d_tc_zm: inputs of up to 96 channels (three chunks of 32).  A CTA keeps the weights of `np`
// output channels resident and walks the z planes of an 8 x 16-voxel column.  One input plane
// contributes to three output planes, through the filter's dz = +1, 0, -1 parts, so the three
// output planes' accumulators sit side by side in TMEM and the weight rows of the three parts side
// by side in shared memory: one MMA of N = 3 np does what three of N = np did, on one read of its A
// operand, and a plane's halo (10 x 18 voxels, rows of 64 bytes, 64-byte swizzle) is copied once
// instead of three times.  With N = 32 the shared-memory reads of A (4 KB per 128 x 32 x 16 MMA)
// and the issue of 54 small MMAs a tile set the pace (the form before this one, three planes of halo
// per tile: 20 % tensor-pipe activity).  Measured (4 x 64^3; K in, N out channels): 16 -> 32 from
// 110 to 50 us, 32 -> 32 110 to 65, 96 -> 32 (then on conv3d_tc) 448 to 160, 64 -> 64 at 32^3 51 to 33.
// What is left above the MMAs' own ~56 clocks each is the issuing warp's work between planes
// (~1200 clocks: waits, commits, ring bookkeeping); where the weights are few enough, two or three
// CTAs on an SM, each with its part of the TMEM, overlap one's bookkeeping with another's MMAs (a
// forward pass at 128 x 120 x 136 with 16-32-64-128 channels from 881 to 731 us, with two CTAs 746;
// a training step of 4 x 64^3 with 32-64-128 channels from 2256 to 2177).
//
// The accumulators form a ring of R planes in TMEM: input plane z adds to planes z - 1, z, z + 1
// (two MMAs where the ring wraps), plane z - 1 is then complete and drained by warps 2-5 (bias,
// ReLU, BF16 store) while the next planes accumulate.  Planes outside the box are skipped: they
// are zeros.  Every output sums its products in the order of conv3d_tc: filter offsets k = 0..26,
// per offset the channels upwards.
//
// Warp 0 issues the copies (weights once, then 32-channel planes into a ring of nhalo buffers),
// warp 1 the MMAs.  CTA i of a part (blockIdx.x % npart) takes an equal share of the planes of all
// columns laid end to end; a share that starts inside a column reads up to two planes more than it
// puts out.  Waits are bounded as in conv3d_tc.
constexpr int kZmThreads = 192;
constexpr int kZmPerSm = 3;  // CTAs per SM where the weights leave room
constexpr int kZmMaxRing = 32, kZmMaxHalo = 12;
constexpr uint32_t kZmBox = (uint32_t)(kTcHx * kTcHy) * 64u;      // 11520 bytes
constexpr uint32_t kZmBuf = (kZmBox + 1023u) / 1024u * 1024u;     // 12288
constexpr uint32_t kZmBars = 8u * (2 * kZmMaxHalo + 2 * kZmMaxRing + 2) + 16u;

__device__ __forceinline__ uint64_t sw64_desc(uint32_t addr, uint32_t sbo) {
  return (uint64_t)((addr >> 4) & 0x3FFFu) | ((uint64_t)1 << 16) | ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) |
         ((uint64_t)1 << 46) | ((uint64_t)4 << 61);
}

// shared memory of a launch: alignment slack, halo buffers, weights, barriers
__host__ __device__ constexpr size_t zm_smem(int nhalo, int nch, int np) {
  return 1024 + (size_t)nhalo * kZmBuf + (size_t)27 * nch * np * 64 + kZmBars;
}

// NCH: 32-channel chunks of the input(s); KK: K = 16 slices of a chunk (1: one input of 16 channels)
template <int NCH, int KK>
__global__ void __launch_bounds__(kZmThreads) conv3d_tc_zm(const __grid_constant__ CUtensorMap map1,
                                                           const __grid_constant__ CUtensorMap map2,
                                                           const __grid_constant__ CUtensorMap mapw, TcConvArgs a) {
  extern __shared__ uint8_t tc_smem_raw[];
  const uint32_t raw = smem_u32(tc_smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* gbase = tc_smem_raw + (base - raw);
  const int NH = a.nhalo, R = a.nacc;
  const uint32_t np = (uint32_t)a.N;                                    // output channels of this CTA
  const uint32_t wres = base + (uint32_t)NH * kZmBuf, brow = np * 64u;  // weights; bytes of one part's rows
  uint64_t* bars = reinterpret_cast<uint64_t*>(gbase + (size_t)NH * kZmBuf + (size_t)27 * NCH * brow);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * kZmMaxHalo + 2 * kZmMaxRing + 2);
  const uint32_t wfull = smem_u32(bars), done = wfull + 8u, hfull0 = done + 8u, hempty0 = hfull0 + 8u * kZmMaxHalo,
                 afull0 = hempty0 + 8u * kZmMaxHalo, aempty0 = afull0 + 8u * kZmMaxRing;
  __shared__ volatile int stop;
  __shared__ int h_issued, h_used;
  __shared__ __align__(16) float sbias[256];
  const int tid = threadIdx.x, warp = warp_index(), lane = tid & 31;
  const int D = a.g.D, n1 = (a.c1 + 31) / 32;
  const int part = (int)blockIdx.x % a.npart, n0 = part * a.N;
  // this CTA's planes of all columns laid end to end
  const int64_t planes = (int64_t)a.g.B * a.ty * a.tx * D;
  const int64_t share = blockIdx.x / a.npart, shares = gridDim.x / a.npart;
  const int64_t lo = planes * share / shares, hi = planes * (share + 1) / shares;
  uint32_t ncols = 32u;
  while (ncols < (uint32_t)R * np) ncols <<= 1;

  for (int i = tid; i < (int)np; i += kZmThreads) sbias[i] = a.bias ? a.bias[n0 + i] : 0.f;
  if (tid == 0) {
    stop = 0;
    h_issued = h_used = 0;
    mbar_init(wfull, 1);
    mbar_init(done, 1);
    for (int i = 0; i < NH; ++i) {
      mbar_init(hfull0 + 8u * i, 1);
      mbar_init(hempty0 + 8u * i, 1);
    }
    for (int i = 0; i < R; ++i) {
      mbar_init(afull0 + 8u * i, 1);
      mbar_init(aempty0 + 8u * i, 4);  // one arrival per epilogue warp
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(ncols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;

  // a run of planes [zs, ze) of one column starting at plane p of the whole
  struct Run {
    int x0, y0, bb, zs, ze;
  };
  auto run_at = [&](int64_t p) {
    Run r;
    int64_t c = p / D;
    r.zs = (int)(p - c * D);
    r.ze = (int)min((int64_t)D, r.zs + (hi - p));
    r.x0 = (int)(c % a.tx) * kTcTx;
    c /= a.tx;
    r.y0 = (int)(c % a.ty) * kTcTy;
    r.bb = (int)(c / a.ty);
    return r;
  };

  if (tid == 0) {
    // producer: the weights, rows of the parts dz = +1, 0, -1 of each (dy, dx) and chunk together
    mbar_expect_tx(wfull, 27u * NCH * brow);
    for (int k9 = 0; k9 < 9; ++k9)
      for (int c = 0; c < NCH; ++c)
        for (int d = 0; d < 3; ++d)
          tma_load_2d(wres + (uint32_t)((k9 * NCH + c) * 3 + d) * brow, &mapw, c < n1 ? 32 * c : a.c1 + 32 * (c - n1),
                      ((2 - d) * 9 + k9) * a.nw + n0, wfull);
    int i = 0, hb = 0;
    uint32_t lap = 1u;  // parity of the release that frees buffer hb; the first lap waits for none
    bool ok = true;
    for (int64_t p = lo; ok && p < hi;) {
      const Run r = run_at(p);
      const int zl = min(r.ze, D - 1);
      for (int z = max(r.zs - 1, 0); ok && z <= zl; ++z)
        for (int c = 0; c < NCH; ++c) {
          if (i >= NH && !mbar_wait(hempty0 + 8u * hb, lap, &stop)) ok = false;
          if (stop) ok = false;
          if (!ok) break;
          mbar_expect_tx(hfull0 + 8u * hb, kZmBox);
          tma_load_5d(base + (uint32_t)hb * kZmBuf, c < n1 ? &map1 : &map2, c < n1 ? 32 * c : 32 * (c - n1), r.x0 - 1,
                      r.y0 - 1, z, r.bb, hfull0 + 8u * hb);
          h_issued = ++i;
          if (++hb == NH) {
            hb = 0;
            lap ^= 1u;
          }
        }
      p += r.ze - r.zs;
    }
    if (!ok) stop = 1;
  } else if (warp == 1) {
    // MMA issue.  Ring positions advance by counting, not by division: this warp's instructions between
    // two MMAs are time the tensor pipe may wait for.
    const uint32_t idesc1 = tc_idesc(kTcM, (int)np) - ((np >> 3) << 17);  // without N
    const uint32_t lead = elect_lane();
    bool ok = warp_wait(wfull, 0, &stop);
    int used = 0;                  // planes of 32 channels taken
    int hb = 0;                    // the next one's buffer
    uint32_t hlap = 0u;            // and the parity of its lap
    int nslot = 0, cslot = 0;      // ring slots of the next plane to start and the next to complete
    uint32_t nlap = 1u;            // parity of the drain that frees nslot; the first lap waits for none
    bool lap0 = true;
    for (int64_t p = lo; ok && p < hi;) {
      const Run r = run_at(p);
      const int zl = min(r.ze, D - 1);
      int olo = r.zs, slo = nslot;  // first output plane this input adds to, and its slot
      for (int z = max(r.zs - 1, 0); z <= zl; ++z) {
        if (z - 1 > olo) {
          ++olo;
          if (++slo == R) slo = 0;
        }
        const int ohi = min(z + 1, r.ze - 1), onew = max(olo, z == 0 ? 0 : z + 1);
        for (int o = onew; o <= ohi; ++o) {  // a slot is free again once drained
          if (!lap0) ok = ok && warp_wait(aempty0 + 8u * nslot, nlap, &stop);
          if (++nslot == R) {
            nslot = 0;
            nlap ^= 1u;
            lap0 = false;
          }
        }
        if (!ok) break;
        uint32_t alo[NCH], hbar[NCH], hpar[NCH];
#pragma unroll
        for (int c = 0; c < NCH; ++c) {
          alo[c] = lo32(sw64_desc(base + (uint32_t)hb * kZmBuf, 0u));
          hbar[c] = 8u * hb;
          hpar[c] = hlap;
          if (++hb == NH) {
            hb = 0;
            hlap ^= 1u;
          }
        }
        const uint32_t ahi = hi32(sw64_desc(0u, kTcHx * 64u)), bhi = hi32(sw64_desc(0u, 512u));
        const int cnt = ohi - olo + 1, first = min(cnt, R - slo);  // planes before the ring wraps
        for (int w = 0; w < 2; ++w) {
          const int plo = w ? olo + first : olo, pn = w ? cnt - first : first;
          if (pn <= 0) break;
          const uint32_t dcol = tmem + (uint32_t)(w ? 0 : slo) * np;
          const uint32_t idesc = idesc1 + (((uint32_t)pn * np >> 3) << 17);
          uint32_t blo = lo32(sw64_desc(wres + (uint32_t)(plo - (z - 1)) * brow, 0u));
          const uint32_t bstep = 3u * brow >> 4;
          const int old = min(max(onew - plo, 0), pn);  // planes that already hold sums
          constexpr uint32_t kRow = 64u / 16u;          // a halo row in units of 16 bytes
#pragma unroll
          for (int k9 = 0; k9 < 9; ++k9) {
            const uint32_t shift = (uint32_t)((k9 / 3) * kTcHx + k9 % 3) * kRow;
#pragma unroll
            for (int c = 0; c < NCH; ++c) {
              if (k9 == 0) {
                if (w == 0) {  // the chunk's first use
                  ok = ok && warp_wait(hfull0 + hbar[c], hpar[c], &stop);
                  if (!ok) break;
                  h_used = ++used;
                  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                }
                if (c == 0 && old < pn) {
                  // the first product of the planes that start here overwrites their slots
                  if (old > 0)
                    mma_f16(lead, dcol, alo[0], ahi, blo, bhi, idesc1 + (((uint32_t)old * np >> 3) << 17), 1u);
                  mma_f16(lead, dcol + (uint32_t)old * np, alo[0], ahi, blo + (uint32_t)old * (brow >> 4), bhi,
                          idesc1 + (((uint32_t)(pn - old) * np >> 3) << 17), 0u);
                } else {
                  mma_f16(lead, dcol, alo[c], ahi, blo, bhi, idesc, 1u);
                }
              } else {
                mma_f16(lead, dcol, alo[c] + shift, ahi, blo, bhi, idesc, 1u);
              }
              if (KK > 1) mma_f16(lead, dcol, alo[c] + shift + 2u, ahi, blo + 2u, bhi, idesc, 1u);
              blo += bstep;
            }
            if (k9 == 0 && !ok) break;
          }
          if (!ok) break;
        }
        if (!ok) break;
#pragma unroll
        for (int c = 0; c < NCH; ++c) mma_commit(lead, hempty0 + hbar[c]);
        // planes complete after this one: z - 1, and z itself at the far face
        if (z - 1 >= r.zs) {
          mma_commit(lead, afull0 + 8u * cslot);
          if (++cslot == R) cslot = 0;
        }
        if (z == D - 1 && z < r.ze) {
          mma_commit(lead, afull0 + 8u * cslot);
          if (++cslot == R) cslot = 0;
        }
      }
      p += r.ze - r.zs;
    }
    if (!ok) stop = 1;
    mma_commit(lead, done);
  } else if (warp >= 2) {
    // epilogue: warp w reads TMEM lanes 32 (w % 4) .. + 31 = tile rows
    const int qd = warp & 3, rr = qd * 32 + lane;
    int slot = 0;
    uint32_t lap = 0u;
    bool ok = true;
    for (int64_t p = lo; ok && p < hi;) {
      const Run r = run_at(p);
      const int xx = r.x0 + (rr & 7), yy = r.y0 + (rr >> 3);
      const bool inside = xx < a.g.W && yy < a.g.H;
      const int64_t plane = (int64_t)a.g.H * a.g.W * a.ldy;
      bf16* dst = inside ? a.y + ((((int64_t)r.bb * D + r.zs) * a.g.H + yy) * a.g.W + xx) * a.ldy + a.oy + n0 : a.y;
      for (int z = r.zs; z < r.ze; ++z, dst += plane) {
        if (!warp_wait(afull0 + 8u * slot, lap, &stop)) {
          if (lane == 0) stop = 1;
          ok = false;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        for (int c0 = 0; c0 < (int)np; c0 += 16) {
          uint32_t qv[16];
          const uint32_t taddr = tmem + ((uint32_t)(qd * 32) << 16) + (uint32_t)slot * np + (uint32_t)c0;
          asm volatile(
              "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, "
              "%14, %15}, [%16];"
              : "=r"(qv[0]), "=r"(qv[1]), "=r"(qv[2]), "=r"(qv[3]), "=r"(qv[4]), "=r"(qv[5]), "=r"(qv[6]),
                "=r"(qv[7]), "=r"(qv[8]), "=r"(qv[9]), "=r"(qv[10]), "=r"(qv[11]), "=r"(qv[12]), "=r"(qv[13]),
                "=r"(qv[14]), "=r"(qv[15])
              : "r"(taddr));
          float bias[16];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const float4 b = *reinterpret_cast<const float4*>(&sbias[c0 + 4 * j]);
            bias[4 * j] = b.x, bias[4 * j + 1] = b.y, bias[4 * j + 2] = b.z, bias[4 * j + 3] = b.w;
          }
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
          if (!inside) continue;
          uint32_t o[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            float f0 = __uint_as_float(qv[2 * j]) + bias[2 * j], f1 = __uint_as_float(qv[2 * j + 1]) + bias[2 * j + 1];
            if (a.relu) f0 = fmaxf(f0, 0.f), f1 = fmaxf(f1, 0.f);
            const __nv_bfloat162 h = __floats2bfloat162_rn(f0, f1);
            o[j] = *reinterpret_cast<const uint32_t*>(&h);
          }
          uint4* d4 = reinterpret_cast<uint4*>(dst + c0);
          d4[0] = make_uint4(o[0], o[1], o[2], o[3]);
          d4[1] = make_uint4(o[4], o[5], o[6], o[7]);
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(aempty0 + 8u * slot) : "memory");
        if (++slot == R) {
          slot = 0;
          lap ^= 1u;
        }
      }
      p += r.ze - r.zs;
    }
  }
  const bool fin = mbar_wait(done, 0);
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const bool failed = __syncthreads_or(!fin || stop) != 0;
  if (failed && tid == 0) {
    atomicExch(a.err, 1);
    (void)mbar_wait(wfull, 0);  // the weight copies, if they never landed
    for (int i = h_used; i < h_issued; ++i) (void)mbar_wait(hfull0 + 8u * (i % NH), (uint32_t)(i / NH) & 1u);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 1)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ncols) : "memory");
}

// ------------------------------------------------------------------ weight gradient
// dW[k][ci][co] = sum over voxels v of X[v + o_k][ci] dY[v][co], read in
// place: no transposed copies.  Both operands are "MN-major" (channels
// contiguous, voxels along K) views of TMA copies with the 64-byte swizzle:
// A of the input's halo (rows of 32 channels, as conv3d_tc_zm loads it), B
// of the 8 x 16-voxel tile of dY (one 32-channel atom per 8 KB).  An MN atom
// of A is 32 channels; its four atoms sit one halo row (64 bytes) apart, so
// one MMA's 128 rows of D are the channels of the offsets dx = -1, 0, +1 (and
// a fourth, discarded).  A K-group of 8 voxels is one x row of the tile (10
// halo rows apart in A, 8 in B); one K = 16 MMA covers two y rows.  A CTA
// takes one 32-channel chunk of the input, one dz with its three dy and up
// to 128 output channels, keeps one TMEM accumulator per dy over every
// gridDim.x-th tile and adds them to dW with FP32 atomics (four columns each)
// at the end.  It serves more than 32 output channels.
// Waits are bounded as in conv3d_tc.
struct TcWgradArgs {
  int c1, c2;     // input channels of the two concatenated parts
  int nch1;       // 32-channel chunks of the first part
  int N, Nm;      // output channels, and the MMA's N (min(N, 128) rounded up to 32)
  int npart;      // parts of Nm output channels (N / 128 rounded up)
  int nstage;     // pipeline stages
  float* dw;      // [27][c1 + c2][N], accumulated
  Grid g;
  int tx, ty;     // tiles along x (8) and y (16); one z plane per tile
  int vec4;       // dw 16-byte aligned: add four columns per atomic
  int* err;
};

constexpr uint32_t kWgPlane = (uint32_t)(kTcHx * kTcHy) * 64u;              // 11520: one z plane of the halo
constexpr uint32_t kWgHalo = (kWgPlane + 1023u) / 1024u * 1024u;            // 12288: its buffer
constexpr uint32_t kWgAtom = 128u * 64u;                                     // 8192: 32 channels of the dY tile

__host__ __device__ constexpr uint32_t wg_stage_bytes(int Nm) { return kWgHalo + (uint32_t)(Nm / 32) * kWgAtom; }

// MN-major shared-memory descriptor, 64-byte swizzle: MN atoms of 32
// elements `lbo` bytes apart, K-groups of 8 rows (64 bytes each) `sbo` apart
__device__ __forceinline__ uint64_t mn_sw64_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  return (uint64_t)((addr >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
         ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | ((uint64_t)1 << 46) | ((uint64_t)4 << 61);
}

__global__ void __launch_bounds__(kTcThreads) conv3d_wgrad_tc(const __grid_constant__ CUtensorMap xm1,
                                                              const __grid_constant__ CUtensorMap xm2,
                                                              const __grid_constant__ CUtensorMap dym, TcWgradArgs a) {
  extern __shared__ uint8_t tc_smem_raw[];
  // [halo + dY atoms] x nstage (1024-byte aligned), then the barriers and the TMEM address
  const uint32_t raw = smem_u32(tc_smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* gbase = tc_smem_raw + (base - raw);
  const int S = a.nstage;
  const uint32_t stage_bytes = wg_stage_bytes(a.Nm);
  uint64_t* bars = reinterpret_cast<uint64_t*>(gbase + (size_t)S * stage_bytes);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * S + 1);
  const uint32_t full0 = smem_u32(bars), empty0 = full0 + 8u * S, done = full0 + 16u * S;
  __shared__ volatile int stop;
  __shared__ int n_issued, n_used;
  const int tid = threadIdx.x, warp = warp_index(), lane = tid & 31;
  const int ntiles = a.g.B * a.g.D * a.ty * a.tx;
  // this CTA's output channels, input chunk and dz (0..2 for -1..+1)
  const int part = (int)blockIdx.y % a.npart, n0 = part * a.Nm;
  const int chunk = (int)blockIdx.y / a.npart / 3, dz = (int)blockIdx.y / a.npart % 3;
  const bool second = chunk >= a.nch1;
  const int ch0 = second ? (chunk - a.nch1) * 32 : chunk * 32;            // channel coordinate in its part
  const int cnt = min(32, (second ? a.c2 : a.c1) - ch0);                  // real channels of the chunk
  const int row0 = second ? a.c1 + ch0 : ch0;                             // its first row of dW
  const CUtensorMap* xm = second ? &xm2 : &xm1;
  const uint32_t tx_bytes = kWgPlane + (uint32_t)(a.Nm / 32) * kWgAtom;
  uint32_t ncols = 32u;
  while (ncols < (uint32_t)(3 * a.Nm)) ncols <<= 1;
  int mytiles = 0;
  for (int t = blockIdx.x; t < ntiles; t += gridDim.x) ++mytiles;

  if (tid == 0) {
    stop = 0;
    n_issued = n_used = 0;
    for (int i = 0; i < S; ++i) {
      mbar_init(full0 + 8u * i, 1);
      mbar_init(empty0 + 8u * i, 1);
    }
    mbar_init(done, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(ncols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;

  if (tid == 0) {
    // producer: per tile the input halo's plane at dz and the dY atoms
    int i = 0;
    for (; i < mytiles; ++i) {
      const int st = i % S;
      if (i >= S && !mbar_wait(empty0 + 8u * st, (uint32_t)(i / S - 1) & 1u, &stop)) break;
      if (stop) break;
      int t = blockIdx.x + i * gridDim.x;
      const int x0 = (t % a.tx) * kTcTx;
      t /= a.tx;
      const int y0 = (t % a.ty) * kTcTy;
      t /= a.ty;
      const int z0 = t % a.g.D, bb = t / a.g.D;
      const uint32_t sa = base + (uint32_t)st * stage_bytes, fb = full0 + 8u * st;
      mbar_expect_tx(fb, tx_bytes);
      tma_load_5d(sa, xm, ch0, x0 - 1, y0 - 1, z0 + dz - 1, bb, fb);
      for (int j = 0; j < a.Nm / 32; ++j)
        tma_load_5d(sa + kWgHalo + (uint32_t)j * kWgAtom, &dym, n0 + 32 * j, x0, y0, z0, bb, fb);
      n_issued = i + 1;
    }
    if (i < mytiles) stop = 1;
  } else if (warp == 1) {
    // MMA issue: per dy and two y rows, A = halo rows (y + dy, x + dx) for dx = 0..3
    const uint32_t idesc = tc_idesc(kTcM, a.Nm) | (1u << 15) | (1u << 16), lead = elect_lane();
    int i = 0;
    for (; i < mytiles; ++i) {
      const int st = i % S;
      if (!warp_wait(full0 + 8u * st, (uint32_t)(i / S) & 1u, &stop)) break;
      n_used = i + 1;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t sa = base + (uint32_t)st * stage_bytes;
      const uint64_t ad0 = mn_sw64_desc(sa, 64u, kTcHx * 64u), bd0 = mn_sw64_desc(sa + kWgHalo, kWgAtom, 512u);
      for (int dy = 0; dy < 3; ++dy) {
        const uint32_t acc_addr = tmem + (uint32_t)(dy * a.Nm);
        const uint32_t alo = lo32(ad0) + (uint32_t)(dy * kTcHx) * 4u;  // 64-byte rows in units of 16 bytes
        const uint32_t acc = i > 0 ? 1u : 0u;
#pragma unroll
        for (int kk = 0; kk < 8; ++kk)  // two y rows: 2 halo rows of A, 1024 bytes of B
          mma_f16(lead, acc_addr, alo + (uint32_t)kk * 8u * kTcHx, hi32(ad0), lo32(bd0) + (uint32_t)kk * 64u, hi32(bd0),
                  idesc, kk > 0 ? 1u : acc);
      }
      mma_commit(lead, empty0 + 8u * st);
    }
    if (i < mytiles) stop = 1;
    mma_commit(lead, done);
  }
  const bool fin = mbar_wait(done, 0);
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const bool failed = __syncthreads_or(!fin || stop) != 0;
  if (failed && tid == 0) {
    atomicExch(a.err, 1);
    for (int j = n_used; j < n_issued; ++j) (void)mbar_wait(full0 + 8u * (j % S), (uint32_t)(j / S) & 1u);
  }
  // epilogue: warp w < 3 holds TMEM lanes 32 w .. + 31 = offset dx = w - 1, channel ch0 + lane
  if (!failed && mytiles > 0 && warp < 3) {
    for (int dy = 0; dy < 3; ++dy) {
      const int k = (dz * 3 + dy) * 3 + warp;
      float* dst = a.dw + ((int64_t)k * (a.c1 + a.c2) + row0 + lane) * a.N + n0;
      for (int c0 = 0; c0 < a.Nm && n0 + c0 < a.N; c0 += 16) {
        uint32_t q[16];
        const uint32_t taddr = tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(dy * a.Nm + c0);
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, "
            "%14, %15}, [%16];"
            : "=r"(q[0]), "=r"(q[1]), "=r"(q[2]), "=r"(q[3]), "=r"(q[4]), "=r"(q[5]), "=r"(q[6]), "=r"(q[7]),
              "=r"(q[8]), "=r"(q[9]), "=r"(q[10]), "=r"(q[11]), "=r"(q[12]), "=r"(q[13]), "=r"(q[14]), "=r"(q[15])
            : "r"(taddr));
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        if (lane >= cnt) continue;
        if (a.vec4) {
#pragma unroll
          for (int j = 0; j < 16; j += 4)
            atomicAdd(reinterpret_cast<float4*>(dst + c0 + j),
                      make_float4(__uint_as_float(q[j]), __uint_as_float(q[j + 1]), __uint_as_float(q[j + 2]),
                                  __uint_as_float(q[j + 3])));
        } else {
#pragma unroll
          for (int j = 0; j < 16; ++j) atomicAdd(dst + c0 + j, __uint_as_float(q[j]));
        }
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 1)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ncols) : "memory");
}

// Weight gradient for at most 32 output channels: the roles swapped, so that
// one MMA is 128 x 96 x 16 instead of 128 x 32 x 16.  A = dY from a copy of
// the tile's rows y0 - 2 .. y0 + 15 (box {32, 8, 18, 1, 1}); its four 32-channel
// atoms are those rows shifted by a = 0..3 in y (one tile row, 512 bytes,
// apart).  B = the input's rows y0 - 1 .. y0 + 14 of planes z0 - 1 .. z0 + 1
// (box {32, 10, 16, 3, 1}); its three atoms are shifted by b = 0..2 in x (one
// halo row apart).  For the dY voxel u the product pairs dY[u] with
// X[u + (b - 1, 1 - a, dz)]: D row (a, co), column (b, ci) of the accumulator
// of plane dz is the gradient of offset (dz, dy = 1 - a, dx = b - 1), and
// a = 3 is discarded.  Tile row j sums u over y0 - 2 + a + [0, 16); one more
// tile row (j = ty) with only its first two rows closes the gap this leaves
// at the far face for a < 2.  A CTA takes one 32-channel input chunk and all
// 27 offsets (3 accumulators of 96 columns).
constexpr uint32_t kWnB = 3u * 160u * 64u;  // 30720: B, three planes of 16 x 10 rows
constexpr uint32_t kWnA = 10240u;           // A: 18 x 8 rows (9216 bytes) and the discarded atom's overrun
constexpr uint32_t kWnStage = kWnB + kWnA;
constexpr uint32_t kWnTx = kWnB + 144u * 64u;

__global__ void __launch_bounds__(kTcThreads) conv3d_wgrad_tc32(const __grid_constant__ CUtensorMap xm1,
                                                                const __grid_constant__ CUtensorMap xm2,
                                                                const __grid_constant__ CUtensorMap dym, TcWgradArgs a) {
  extern __shared__ uint8_t tc_smem_raw[];
  const uint32_t raw = smem_u32(tc_smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* gbase = tc_smem_raw + (base - raw);
  const int S = a.nstage;
  uint64_t* bars = reinterpret_cast<uint64_t*>(gbase + (size_t)S * kWnStage);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * S + 1);
  const uint32_t full0 = smem_u32(bars), empty0 = full0 + 8u * S, done = full0 + 16u * S;
  __shared__ volatile int stop;
  __shared__ int n_issued, n_used;
  const int tid = threadIdx.x, warp = warp_index(), lane = tid & 31;
  const int tyx = a.ty + 1;  // tile rows, the last one two rows high
  const int ntiles = a.g.B * a.g.D * tyx * a.tx;
  const int chunk = (int)blockIdx.y;
  const bool second = chunk >= a.nch1;
  const int ch0 = second ? (chunk - a.nch1) * 32 : chunk * 32;
  const int cnt = min(32, (second ? a.c2 : a.c1) - ch0);
  const int row0 = second ? a.c1 + ch0 : ch0;
  const CUtensorMap* xm = second ? &xm2 : &xm1;
  constexpr uint32_t ncols = 512u;  // 3 x 96
  int mytiles = 0;
  for (int t = blockIdx.x; t < ntiles; t += gridDim.x) ++mytiles;

  if (tid == 0) {
    stop = 0;
    n_issued = n_used = 0;
    for (int i = 0; i < S; ++i) {
      mbar_init(full0 + 8u * i, 1);
      mbar_init(empty0 + 8u * i, 1);
    }
    mbar_init(done, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(ncols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;

  if (tid == 0) {
    int i = 0;
    for (; i < mytiles; ++i) {
      const int st = i % S;
      if (i >= S && !mbar_wait(empty0 + 8u * st, (uint32_t)(i / S - 1) & 1u, &stop)) break;
      if (stop) break;
      int t = blockIdx.x + i * gridDim.x;
      const int x0 = (t % a.tx) * kTcTx;
      t /= a.tx;
      const int y0 = (t % tyx) * kTcTy;
      t /= tyx;
      const int z0 = t % a.g.D, bb = t / a.g.D;
      const uint32_t sa = base + (uint32_t)st * kWnStage, fb = full0 + 8u * st;
      mbar_expect_tx(fb, kWnTx);
      tma_load_5d(sa, xm, ch0, x0 - 1, y0 - 1, z0 - 1, bb, fb);
      tma_load_5d(sa + kWnB, &dym, 0, x0, y0 - 2, z0, bb, fb);
      n_issued = i + 1;
    }
    if (i < mytiles) stop = 1;
  } else if (warp == 1) {
    const uint32_t idesc = tc_idesc(kTcM, 96) | (1u << 15) | (1u << 16), lead = elect_lane();
    int i = 0;
    for (; i < mytiles; ++i) {
      const int st = i % S;
      if (!warp_wait(full0 + 8u * st, (uint32_t)(i / S) & 1u, &stop)) break;
      n_used = i + 1;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const int yt = (blockIdx.x + i * gridDim.x) / a.tx % tyx;
      const int nk = yt == a.ty ? 1 : 8;  // the last tile row: its first two rows only
      const uint32_t sa = base + (uint32_t)st * kWnStage;
      // A: dY, atoms one tile row (512 bytes) apart, K-groups one tile row apart;
      // B: the planes, atoms one halo row (64 bytes) apart, K-groups 10 rows apart
      const uint64_t ad0 = mn_sw64_desc(sa + kWnB, 512u, 512u), bd0 = mn_sw64_desc(sa, 64u, kTcHx * 64u);
      const uint32_t acc = i > 0 ? 1u : 0u;
#pragma unroll
      for (int dz = 0; dz < 3; ++dz) {
#pragma unroll
        for (int kk = 0; kk < 8; ++kk) {
          if (kk > 0 && kk >= nk) break;
          // A 1024 bytes a K = 16 step; B 64-byte rows, two halo rows a step
          mma_f16(lead, tmem + (uint32_t)(dz * 96), lo32(ad0) + (uint32_t)kk * 64u, hi32(ad0),
                  lo32(bd0) + ((uint32_t)dz * 160u + (uint32_t)kk * 2u * kTcHx) * 4u, hi32(bd0), idesc, kk > 0 ? 1u : acc);
        }
      }
      mma_commit(lead, empty0 + 8u * st);
    }
    if (i < mytiles) stop = 1;
    mma_commit(lead, done);
  }
  const bool fin = mbar_wait(done, 0);
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const bool failed = __syncthreads_or(!fin || stop) != 0;
  if (failed && tid == 0) {
    atomicExch(a.err, 1);
    for (int j = n_used; j < n_issued; ++j) (void)mbar_wait(full0 + 8u * (j % S), (uint32_t)(j / S) & 1u);
  }
  // epilogue: warp w < 3 holds TMEM lanes 32 w .. + 31 = dy = 1 - w, output channel lane;
  // columns dz * 96 + b * 32 + ci
  if (!failed && mytiles > 0 && warp < 3) {
    const bool live = lane < a.N;
    for (int dz = 0; dz < 3; ++dz)
      for (int b = 0; b < 3; ++b) {
        const int k = dz * 9 + (2 - warp) * 3 + b;
        float* dst = a.dw + ((int64_t)k * (a.c1 + a.c2) + row0) * a.N + lane;
        for (int c0 = 0; c0 < 32; c0 += 16) {
          uint32_t q[16];
          const uint32_t taddr = tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(dz * 96 + b * 32 + c0);
          asm volatile(
              "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, "
              "%14, %15}, [%16];"
              : "=r"(q[0]), "=r"(q[1]), "=r"(q[2]), "=r"(q[3]), "=r"(q[4]), "=r"(q[5]), "=r"(q[6]), "=r"(q[7]),
                "=r"(q[8]), "=r"(q[9]), "=r"(q[10]), "=r"(q[11]), "=r"(q[12]), "=r"(q[13]), "=r"(q[14]),
                "=r"(q[15])
              : "r"(taddr));
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
          if (!live) continue;
#pragma unroll
          for (int j = 0; j < 16; ++j)
            if (c0 + j < cnt) atomicAdd(dst + (int64_t)(c0 + j) * a.N, __uint_as_float(q[j]));
        }
      }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 1)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ncols) : "memory");
}

}  // namespace nn
}  // namespace om
