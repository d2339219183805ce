// label.cu -- connected-phase labelling (Sec. 4.1) on the GPU.
//
// Pore voxels are joined with their 18 neighbours (the D3Q19 links; y and z
// periodic, x not) by a lock-free union-find: a root is only ever linked
// below a smaller index, so every component ends as a tree rooted at its
// smallest voxel index, the canonical label.  Transport voxels belong to a
// component with voxels on both x faces.
//
// The nodes of the union-find are the runs of pore voxels along z, each
// named by its first voxel.  Rows are packed to bits first; contacts between
// neighbouring rows are then word operations, and only one union is issued
// per pair of overlapping runs, plus the diagonal contacts that no overlap
// implies.  256^3 at porosity 0.35: 280 us of kernels; with a tree
// node per voxel and 27 mask reads per voxel (the form that
// om_label_connectivity_noalloc still takes, for want of scratch for the
// packed rows) 1430 us.
#include <algorithm>

#include "common.cuh"

namespace om {
namespace {

__device__ __forceinline__ int uf_find(volatile int* par, int x) {
  int p = par[x];
  while (p != x) {
    const int gp = par[p];
    if (gp != p) par[x] = gp;  // path halving: only ever points further up
    x = p;
    p = gp;
  }
  return x;
}

__device__ __forceinline__ void uf_union(int* par, int a, int b) {
  for (;;) {
    a = uf_find(par, a);
    b = uf_find(par, b);
    if (a == b) return;
    if (a < b) {
      const int t = a;
      a = b;
      b = t;
    }
    const int old = atomicCAS(par + a, a, b);  // link the larger root below the smaller
    if (old == a) return;
    a = old;
  }
}

// Runs of pore voxels along z (not wrapping at z = 0) start as one tree
// each: every voxel points at the first voxel of its run, which is its own
// root and the run's smallest index.  One thread per (x, y) column.
__global__ void uf_init_runs(const uint8_t* mask, int64_t ncol, int nz, int* par) {
  for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < ncol; c += (int64_t)gridDim.x * blockDim.x) {
    const int64_t base = c * nz;
    int head = -1;
    for (int z = 0; z < nz; ++z) {
      const int64_t v = base + z;
      if (!mask[v]) {
        par[v] = -1;
        head = -1;
        continue;
      }
      if (head < 0) head = (int)v;
      par[v] = head;
    }
  }
}

// The forward half of the 18 neighbour offsets (the other half is the same
// pairs seen from the other voxel).  Voxel v is joined to its neighbour u =
// v + o unless the pair one step lower in z, (v - 1, u - 1), is a pore pair
// inside the same two runs: that pair already joins the two runs.  So each
// overlap of two runs issues one union, at its lowest voxel.  One block row
// of threads per (x, y) column, threads along z: no 64-bit index division.
__global__ void uf_link_runs(const uint8_t* mask, int nx, int ny, int nz, int* par) {
  constexpr int8_t H[9][3] = {{1, 0, 0}, {1, 1, 0}, {1, -1, 0}, {1, 0, 1}, {1, 0, -1},
                              {0, 1, 0}, {0, 1, 1}, {0, 1, -1}, {0, 0, 1}};
  const int64_t ncol = (int64_t)nx * ny;
  for (int64_t c = blockIdx.x; c < ncol; c += gridDim.x) {
    const int x = (int)(c / ny), y = (int)(c - (int64_t)x * ny);
    const int64_t base = c * nz;
    for (int z = threadIdx.x; z < nz; z += blockDim.x) {
      const int64_t v = base + z;
      if (!mask[v]) continue;
      const bool below = z > 0 && mask[v - 1];  // v - 1 in the same run
#pragma unroll
      for (int k = 0; k < 9; ++k) {
        const int xx = x + H[k][0];
        if (xx >= nx) continue;
        int yy = y + H[k][1], zz = z + H[k][2];
        yy = yy < 0 ? yy + ny : (yy >= ny ? yy - ny : yy);
        zz = zz < 0 ? zz + nz : (zz >= nz ? zz - nz : zz);
        const int64_t u = ((int64_t)xx * ny + yy) * nz + zz;
        if (!mask[u]) continue;
        if (k == 8 && zz > 0) continue;              // z + 1 without wrap: the same run
        if (below && zz > 0 && mask[u - 1]) continue;  // (v-1, u-1) joins these runs
        uf_union(par, (int)v, (int)u);
      }
    }
  }
}

// Root without path compression.  The flatten pass must not compress: a
// compressing walk could overwrite a root another thread has just stored
// with an intermediate ancestor it read earlier.
__device__ __forceinline__ int uf_root(const volatile int* par, int x) {
  int p = par[x];
  while (p != x) {
    x = p;
    p = par[x];
  }
  return x;
}

__global__ void uf_flatten(int* par, int64_t N) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < N; v += (int64_t)gridDim.x * blockDim.x)
    if (par[v] >= 0) par[v] = uf_root(par, (int)v);
}

}  // namespace

namespace {

// Rows: bits[r * W + w], r = x * ny + y; bits past nz are zero.  Words are
// numbered in 32 bits (at most 2^27 of them): 64-bit divisions cost more than the rest of
// the per-word work.
struct Rows {
  const uint32_t* bits;
  int nx, ny, nz, W;
};

__global__ void row_pack(const uint8_t* mask, int64_t rows, int nz, int W, uint32_t* bits) {
  const int lane = threadIdx.x & 31;
  const uint32_t words = (uint32_t)(rows * W);
  for (uint32_t i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < words; i += (gridDim.x * blockDim.x) >> 5) {
    const uint32_t r = i / (uint32_t)W;
    const int z = 32 * (int)(i - r * W) + lane;
    const uint32_t b = __ballot_sync(0xffffffffu, z < nz && mask[(int64_t)r * nz + z] != 0);
    if (lane == 0) bits[i] = b;
  }
}

__global__ void row_pack16(const uint8_t* mask, uint32_t words, int nz, int W, uint32_t* bits) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < words; i += gridDim.x * blockDim.x) {
    const int64_t r = i / (uint32_t)W;
    const int w = (int)(i - r * W);
    bits[i] = pack_word(mask + r * nz + 32 * w, min(32, nz - 32 * w));
  }
}

// first voxel of the run that holds voxel z of a row
__device__ __forceinline__ int run_head(const uint32_t* row, int z) {
  int w = z >> 5;
  uint32_t gap = ~__ldg(row + w) & ((1u << (z & 31)) - 1u);
  while (!gap && w > 0) gap = ~__ldg(row + --w);
  return gap ? 32 * w + 32 - __clz((int)gap) : 0;
}

// run heads of word w (a run does not wrap at z = 0)
__device__ __forceinline__ uint32_t word_heads(const uint32_t* row, int w) {
  const uint32_t b = __ldg(row + w);
  return b & ~((b << 1) | (w > 0 ? __ldg(row + w - 1) >> 31 : 0u));
}

__global__ void run_init(Rows q, uint32_t words, int* par) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < words; i += gridDim.x * blockDim.x) {
    const int64_t r = i / (uint32_t)q.W;
    const int w = (int)(i - r * q.W);
    uint32_t h = word_heads(q.bits + r * q.W, w);
    for (; h; h &= h - 1) {
      const int64_t v = r * q.nz + 32 * w + __ffs((int)h) - 1;
      par[v] = (int)v;
    }
  }
}

// bit z of the result: voxel z + 1 (UP) or z - 1 of the row, periodic
template <bool UP>
__device__ __forceinline__ uint32_t row_shift(const uint32_t* row, int w, int W, int nz) {
  const uint32_t b = __ldg(row + w);
  if (UP) {
    if (w + 1 < W) return (b >> 1) | (__ldg(row + w + 1) << 31);
    return (b >> 1) | ((__ldg(row) & 1u) << ((nz - 1) & 31));
  }
  if (w > 0) return (b << 1) | (__ldg(row + w - 1) >> 31);
  return (b << 1) | ((__ldg(row + W - 1) >> ((nz - 1) & 31)) & 1u);
}

// The forward half of the 18 neighbours, one word of a row per thread.
// Overlaps of two rows' runs (dz = 0) are joined at their first voxel;
// contacts one voxel up or down only where neither voxel faces a pore of the
// other row: otherwise an overlap (and a row's own join of its two ends,
// where the contact wraps) already connects the runs.
__global__ void run_link(Rows q, uint32_t words, int* par) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < words; i += gridDim.x * blockDim.x) {
    const int64_t r = i / (uint32_t)q.W;
    const int w = (int)(i - r * q.W);
    const uint32_t* row = q.bits + r * q.W;
    const uint32_t a = __ldg(row + w);
    if (!a) continue;
    const int x = (int)((uint32_t)r / (uint32_t)q.ny), y = (int)(r - (int64_t)x * q.ny);
    const int yp = y + 1 == q.ny ? 0 : y + 1, ym = y == 0 ? q.ny - 1 : y - 1;
    const uint32_t valid = w + 1 < q.W || (q.nz & 31) == 0 ? 0xffffffffu : (1u << (q.nz & 31)) - 1u;
    auto join = [&](int z, int64_t r2, int z2) {
      uf_union(par, (int)(r * q.nz) + run_head(row, z), (int)(r2 * q.nz) + run_head(q.bits + r2 * q.W, z2));
    };
    auto overlap = [&](int64_t r2) {
      const uint32_t* row2 = q.bits + r2 * q.W;
      const uint32_t c = a & __ldg(row2 + w);
      uint32_t first = c & ~((c << 1) | (w > 0 ? (__ldg(row + w - 1) & __ldg(row2 + w - 1)) >> 31 : 0u));
      for (; first; first &= first - 1) {
        const int z = 32 * w + __ffs((int)first) - 1;
        join(z, r2, z);
      }
    };
    auto corners = [&](int64_t r2) {
      const uint32_t* row2 = q.bits + r2 * q.W;
      const uint32_t alone = a & ~__ldg(row2 + w);
      uint32_t up = alone & row_shift<true>(row2, w, q.W, q.nz) & ~row_shift<true>(row, w, q.W, q.nz) & valid;
      for (; up; up &= up - 1) {
        const int z = 32 * w + __ffs((int)up) - 1;
        join(z, r2, z + 1 == q.nz ? 0 : z + 1);
      }
      uint32_t dn = alone & row_shift<false>(row2, w, q.W, q.nz) & ~row_shift<false>(row, w, q.W, q.nz) & valid;
      for (; dn; dn &= dn - 1) {
        const int z = 32 * w + __ffs((int)dn) - 1;
        join(z, r2, z == 0 ? q.nz - 1 : z - 1);
      }
    };
    if (x + 1 < q.nx) {
      const int64_t e = (int64_t)(x + 1) * q.ny;
      overlap(e + y);
      corners(e + y);
      overlap(e + yp);
      overlap(e + ym);
    }
    overlap((int64_t)x * q.ny + yp);
    corners((int64_t)x * q.ny + yp);
    if (w == q.W - 1 && ((a >> ((q.nz - 1) & 31)) & 1u) && (__ldg(row) & 1u)) join(q.nz - 1, r, 0);  // round the row
  }
}

// every head to its root (no compression on the way: see uf_root), and the
// roots of the two x faces' runs marked (bit 0 inlet, bit 1 outlet)
__global__ void run_flatten(Rows q, uint32_t words, int* par) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < words; i += gridDim.x * blockDim.x) {
    const int64_t r = i / (uint32_t)q.W;
    const int w = (int)(i - r * q.W);
    uint32_t h = word_heads(q.bits + r * q.W, w);
    for (; h; h &= h - 1) {
      const int v = (int)(r * q.nz) + 32 * w + __ffs((int)h) - 1;
      par[v] = uf_root(par, v);
    }
  }
}

__global__ void run_faces(Rows q, const int* par, uint8_t* touch) {
  const int64_t face = (int64_t)q.ny * q.W;  // words of one x face
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < 2 * face; i += (int64_t)gridDim.x * blockDim.x) {
    const bool out = i >= face;
    const int64_t k = (out ? i - face : i) / q.W, r = (out ? (int64_t)(q.nx - 1) * q.ny : 0) + k;
    const int w = (int)((out ? i - face : i) - k * q.W);
    uint32_t h = word_heads(q.bits + r * q.W, w);
    for (; h; h &= h - 1) {
      const int a = par[r * q.nz + 32 * w + __ffs((int)h) - 1];
      atomicOr((unsigned int*)(touch + (a & ~3)), (out ? 2u : 1u) << (8 * (a & 3)));
    }
  }
}

// labels (LAB: in place of par, whose head entries already hold the labels),
// transport flags and the counts, one warp per word
template <bool LAB>
__global__ void run_labels(Rows q, uint32_t words, int* par, const uint8_t* touch, uint8_t* tr, unsigned long long* counts) {
  const int lane = threadIdx.x & 31;
  unsigned long long np = 0, nt = 0;
  for (uint32_t i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < words; i += (gridDim.x * blockDim.x) >> 5) {
    const int64_t r = i / (uint32_t)q.W;
    const int w = (int)(i - r * q.W), z = 32 * w + lane;
    const uint32_t* row = q.bits + r * q.W;
    const uint32_t b = __ldg(row + w);
    const bool pore = (b >> lane) & 1u;
    int lab = -1;
    bool t = false;
    if (pore) {
      lab = par[r * q.nz + run_head(row, z)];
      t = touch[lab] == 3;
    }
    if (z < q.nz) {
      if (LAB) par[r * q.nz + z] = lab;
      if (tr) tr[r * q.nz + z] = t ? 1 : 0;
    }
    np += __popc(b);
    nt += __popc(__ballot_sync(0xffffffffu, t));
  }
  if (lane == 0 && np) {
    atomicAdd(counts, np);
    atomicAdd(counts + 1, nt);
  }
}

}  // namespace

void launch_union_find(const uint8_t* mask_dev, const om_domain& d, int* labels_dev, cudaStream_t s);

// labels (int32 N, nullable) and transport flags (nullable) on the device;
// counts of pore and transport voxels returned through the host pointers
// when non-null.
om_status label_impl(const uint8_t* mask_dev, const om_domain& d, int* labels_dev, uint8_t* transport_dev,
                     int64_t* npore, int64_t* ntrans, cudaStream_t s) {
  const int64_t N = voxels(d);
  if (N >= (int64_t)0x7fffffff) return fail(OM_EINVAL, "labelling needs fewer than 2^31 voxels");
  const int W = (d.nz + 31) / 32;
  const int64_t rows = (int64_t)d.nx * d.ny, words = rows * W;
  // scratch: flag bytes (set through 32-bit words: padded to a multiple of 4), counters, packed rows, run parents
  const size_t touch_bytes = (size_t)(N + 3) / 4 * 4;
  StreamBuf buf(s);
  size_t at = 0, need = 0;
  for (size_t b : {touch_bytes, 2 * sizeof(unsigned long long), words * sizeof(uint32_t), labels_dev ? (size_t)0 : N * sizeof(int)})
    need += (b + 255) / 256 * 256;
  OM_TRY(buf.alloc(need));
  uint8_t* touch = carve<uint8_t>(buf.p, &at, touch_bytes);
  unsigned long long* cnt = carve<unsigned long long>(buf.p, &at, 2);
  OM_CUDA(cudaMemsetAsync(buf.p, 0, at, s));
  uint32_t* bits = carve<uint32_t>(buf.p, &at, words);
  int* par = labels_dev ? labels_dev : carve<int>(buf.p, &at, N);
  const Rows q{bits, d.nx, d.ny, d.nz, W};
  const unsigned warps = (unsigned)std::min<int64_t>((words + 7) / 8, 16 * 1216);
  const unsigned threads = (unsigned)std::min<int64_t>((words + 127) / 128, 16 * 1216);
  if (pack_aligned(mask_dev, d.nz)) row_pack16<<<threads, 128, 0, s>>>(mask_dev, words, d.nz, W, bits);
  else row_pack<<<warps, 256, 0, s>>>(mask_dev, rows, d.nz, W, bits);
  run_init<<<threads, 128, 0, s>>>(q, words, par);
  run_link<<<threads, 128, 0, s>>>(q, words, par);
  run_flatten<<<threads, 128, 0, s>>>(q, words, par);
  run_faces<<<(unsigned)std::min<int64_t>((2 * (int64_t)d.ny * W + 127) / 128, 1216), 128, 0, s>>>(q, par, touch);
  const unsigned few = std::min(warps, 4864u);
  if (labels_dev) run_labels<true><<<few, 256, 0, s>>>(q, words, par, touch, transport_dev, cnt);
  else run_labels<false><<<few, 256, 0, s>>>(q, words, par, touch, transport_dev, cnt);
  OM_CUDA(cudaGetLastError());
  unsigned long long h[2];
  OM_CUDA(cudaMemcpyAsync(h, cnt, sizeof h, cudaMemcpyDeviceToHost, s));
  OM_CUDA(cudaStreamSynchronize(s));
  if (npore) *npore = (int64_t)h[0];
  if (ntrans) *ntrans = (int64_t)h[1];
  return OM_OK;
}

// Union-find labelling alone (labels_dev: int32 N, written), for callers
// that bring their own flag storage.
void launch_union_find(const uint8_t* mask_dev, const om_domain& d, int* labels_dev, cudaStream_t s) {
  const int64_t N = voxels(d), ncol = (int64_t)d.nx * d.ny;
  const int zt = d.nz >= 128 ? 128 : (d.nz >= 64 ? 64 : 32);  // threads along z per column
  uf_init_runs<<<(unsigned)std::min<int64_t>((ncol + 255) / 256, 4864), 256, 0, s>>>(mask_dev, ncol, d.nz,
                                                                                     labels_dev);
  uf_link_runs<<<(unsigned)std::min<int64_t>(ncol, 152 * 64), zt, 0, s>>>(mask_dev, d.nx, d.ny, d.nz, labels_dev);
  uf_flatten<<<1216, 256, 0, s>>>(labels_dev, N);
}

}  // namespace om

using namespace om;

extern "C" om_status om_label_connectivity_dev(const uint8_t* mask_dev, om_domain d, int32_t* labels_dev,
                                               uint8_t* transport_dev, double* connectivity_out,
                                               void* stream) {
  if (!mask_dev) return fail(OM_EINVAL, "om_label_connectivity_dev: null mask");
  OM_TRY(check_domain(d));
  cudaStream_t s = as_stream(stream);
  int64_t np = 0, nt = 0;
  OM_TRY(label_impl(mask_dev, d, labels_dev, transport_dev, &np, &nt, s));
  if (connectivity_out) *connectivity_out = np > 0 ? (double)nt / (double)np : 0.0;
  return OM_OK;
}

extern "C" om_status om_label_connectivity(const uint8_t* mask, om_domain d, int32_t* labels,
                                           uint8_t* transport, double* connectivity_out) {
  if (!mask) return fail(OM_EINVAL, "om_label_connectivity: null mask");
  OM_TRY(check_domain(d));
  const int64_t N = voxels(d);
  cudaStream_t s;
  OM_CUDA(cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking));
  DevBuf<uint8_t> m, tr;
  DevBuf<int> lab;
  om_status st = m.alloc(N);
  if (st == OM_OK) st = tr.alloc(N);
  if (st == OM_OK) st = lab.alloc(N);
  if (st == OM_OK) {
    cudaError_t e = cudaMemcpyAsync(m.p, mask, N, cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) st = cuda_fail(e, "copy-in", __FILE__, __LINE__);
  }
  int64_t np = 0, nt = 0;
  if (st == OM_OK) st = label_impl(m.p, d, lab.p, tr.p, &np, &nt, s);
  if (st == OM_OK) {
    cudaError_t e = cudaSuccess;
    if (labels) e = cudaMemcpyAsync(labels, lab.p, N * sizeof(int), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess && transport) e = cudaMemcpyAsync(transport, tr.p, N, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) st = cuda_fail(e, "copy-out", __FILE__, __LINE__);
    if (connectivity_out) *connectivity_out = np > 0 ? (double)nt / (double)np : 0.0;
  }
  cudaStreamDestroy(s);
  return st;
}
