// nodeset.cu -- the fluid-node layout of the LB sweeps.
//
// Lattice nodes (transport voxels) are numbered in lexicographic voxel order
// and their populations stored densely by that number, so no solid voxel
// occupies memory or bandwidth.  A neighbour's node number is not stored:
// each (x, y) column keeps, per 32 voxels in z, a bit map of nodes and the
// number of nodes that precede the word, and
//     node(x, y, z) = rank[w] + popc(bits[w] & ((1 << (z & 31)) - 1)),
//     w = column word of z,
// plus the node numbers of the voxel just below the word's first and just
// above its last (periodic in z), so that z - 1, z, z + 1 of any column come
// from one 16-byte word without branches.  16 bytes per 32 voxels (the whole
// map sits in L2) instead of an 18-entry neighbour table per node.
#include <algorithm>

#include "lattice.cuh"

namespace om {

// One warp per word: 32 voxels of a column.  Words are numbered in 32 bits (at
// most 2^27 of them), which keeps the divisions short (ns_fill, 256^3 at porosity
// 0.35: 81 -> 62 us).
__global__ void ns_bits(const uint8_t* nodes, int nz, int W, uint32_t words, uint32_t* bits, uint32_t* cnt) {
  const int lane = threadIdx.x & 31;
  for (uint32_t k = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; k < words; k += (gridDim.x * blockDim.x) >> 5) {
    const int64_t c = k / (uint32_t)W;
    const int z = 32 * (int)(k - c * W) + lane;
    const uint32_t b = __ballot_sync(0xffffffffu, z < nz && nodes[c * nz + z] != 0);
    if (lane == 0) {
      bits[k] = b;
      cnt[k] = __popc(b);
    }
  }
}

__global__ void ns_bits16(const uint8_t* nodes, int nz, int W, uint32_t words, uint32_t* bits, uint32_t* cnt) {
  for (uint32_t k = blockIdx.x * blockDim.x + threadIdx.x; k < words; k += gridDim.x * blockDim.x) {
    const int64_t c = k / (uint32_t)W;
    const int w = (int)(k - c * W);
    const uint32_t b = pack_word(nodes + c * nz + 32 * w, min(32, nz - 32 * w));
    bits[k] = b;
    cnt[k] = __popc(b);
  }
}

// node number of voxel z of the column whose first word is k0, or kNoNode
__device__ __forceinline__ uint32_t ns_node(const uint32_t* bits, const uint32_t* rank, int64_t k0, int z) {
  const int64_t k = k0 + (z >> 5);
  const uint32_t bit = 1u << (z & 31);
  return (bits[k] & bit) ? rank[k] + __popc(bits[k] & (bit - 1u)) : kNoNode;
}

// one warp per word, a lane per voxel: consecutive nodes are written together
__global__ void ns_fill(const uint32_t* bits, const uint32_t* rank, int ny, int nz, int W,
                        uint32_t nwords, uint4* col, uint32_t* coord, int64_t* vox) {
  const int lane = threadIdx.x & 31;
  for (uint32_t k = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; k < nwords; k += (gridDim.x * blockDim.x) >> 5) {
    const uint32_t b = bits[k], r0 = rank[k];
    const int64_t c = k / (uint32_t)W;
    const int w = (int)(k - c * W);
    if (lane == 0) {
      const int zprev = w == 0 ? nz - 1 : 32 * w - 1;         // below the word's first voxel
      const int znext = 32 * w + 32 >= nz ? 0 : 32 * w + 32;  // above its last (nz - 1 in the last word)
      col[k] = make_uint4(b, r0, ns_node(bits, rank, c * W, zprev), ns_node(bits, rank, c * W, znext));
    }
    if ((b >> lane) & 1u) {
      const int x = (int)((uint32_t)c / (uint32_t)ny), y = (int)(c - (int64_t)x * ny), z = 32 * w + lane;
      const uint32_t r = r0 + __popc(b & ((1u << lane) - 1u));
      coord[r] = pack_xyz(x, y, z);
      vox[r] = c * nz + z;
    }
  }
}

// Links of the flow lattice across the periodic x boundary: node voxels
// (nx-1, y, z) whose neighbour (0, y + dy, z + dz), |dy| + |dz| <= 1, along
// one of the five velocities with e_x = +1, is a node voxel (y, z periodic).
// Without any, the x wrap is a wall for the flow and its steady net flux is
// zero.
__global__ void ns_wrap_links(const uint8_t* nodes, int nx, int ny, int nz, unsigned long long* count) {
  const int64_t plane = (int64_t)ny * nz;
  const uint8_t* last = nodes + (int64_t)(nx - 1) * plane;
  unsigned long long c = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < plane; i += (int64_t)gridDim.x * blockDim.x) {
    if (!last[i]) continue;
    const int y = (int)(i / nz), z = (int)(i - (int64_t)y * nz);
    const int yp = y + 1 == ny ? 0 : y + 1, ym = y == 0 ? ny - 1 : y - 1;
    const int zp = z + 1 == nz ? 0 : z + 1, zm = z == 0 ? nz - 1 : z - 1;
    c += nodes[(int64_t)y * nz + z] != 0;
    c += nodes[(int64_t)yp * nz + z] != 0;
    c += nodes[(int64_t)ym * nz + z] != 0;
    c += nodes[(int64_t)y * nz + zp] != 0;
    c += nodes[(int64_t)y * nz + zm] != 0;
  }
  if (c) atomicAdd(count, c);
}

// R_c(z) (nodes before voxel (x, y, z)) and whether that voxel is a node
__device__ __forceinline__ void ns_rank_bit(const uint4* col, int ny, int W, int x, int y, int z, uint32_t& r,
                                            uint32_t& bit) {
  const uint4 w = col[((int64_t)x * ny + y) * W + (z >> 5)];
  r = w.y + __popc(w.x & ((1u << (z & 31)) - 1u));
  bit = (w.x >> (z & 31)) & 1u;
}

// The neighbour records of lattice.cuh for every node, and a 0/1 "slow" flag
// per node (a face of the box, or a box beyond the record fields: !fit).
__global__ void ns_records(const uint4* col, const uint32_t* coord, int64_t nf, int nx, int ny, int nz, int W,
                           int fit, uint2* rec7, uint2* rec19, uint32_t* slow) {
  const int64_t n = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= nf) return;
  int x, y, z;
  unpack_xyz(coord[n], x, y, z);
  if (!fit || x == 0 || x == nx - 1 || y == 0 || y == ny - 1 || z == 0 || z == nz - 1) {
    rec7[n] = make_uint2(kRecSlow, 0u);
    rec19[n] = make_uint2(0u, 0u);
    slow[n] = 1u;
    return;
  }
  const uint32_t nn = (uint32_t)n;
  uint32_t rxp, bxp, rxm, bxm, ryp, byp, rym, bym, r;
  ns_rank_bit(col, ny, W, x + 1, y, z, rxp, bxp);
  ns_rank_bit(col, ny, W, x - 1, y, z, rxm, bxm);
  ns_rank_bit(col, ny, W, x, y + 1, z, ryp, byp);
  ns_rank_bit(col, ny, W, x, y - 1, z, rym, bym);
  uint32_t szp, szm;
  ns_rank_bit(col, ny, W, x, y, z + 1, r, szp);
  ns_rank_bit(col, ny, W, x, y, z - 1, r, szm);
  uint2 a;
  a.x = (rxp - nn - 1u) | ((ryp - nn - 1u) << 19) | (bxp << 29) | (byp << 30) | (szp << 31);
  a.y = (nn - rxm) | ((nn - rym) << 19) | (bxm << 29) | (bym << 30) | (szm << 31);
  uint32_t r1, b1, r2, b2, r3, b3, r4, b4;
  ns_rank_bit(col, ny, W, x + 1, y + 1, z, r1, b1);
  ns_rank_bit(col, ny, W, x + 1, y - 1, z, r2, b2);
  ns_rank_bit(col, ny, W, x - 1, y + 1, z, r3, b3);
  ns_rank_bit(col, ny, W, x - 1, y - 1, z, r4, b4);
  uint32_t zb[8];
  ns_rank_bit(col, ny, W, x + 1, y, z - 1, r, zb[0]);
  ns_rank_bit(col, ny, W, x + 1, y, z + 1, r, zb[1]);
  ns_rank_bit(col, ny, W, x - 1, y, z - 1, r, zb[2]);
  ns_rank_bit(col, ny, W, x - 1, y, z + 1, r, zb[3]);
  ns_rank_bit(col, ny, W, x, y + 1, z - 1, r, zb[4]);
  ns_rank_bit(col, ny, W, x, y + 1, z + 1, r, zb[5]);
  ns_rank_bit(col, ny, W, x, y - 1, z - 1, r, zb[6]);
  ns_rank_bit(col, ny, W, x, y - 1, z + 1, r, zb[7]);
  uint2 q;
  q.x = (r1 - rxp) | ((rxp - r2) << 10) | ((r3 - rxm) << 20) | (b1 << 30) | (b2 << 31);
  q.y = (rxm - r4) | (b3 << 10) | (b4 << 11);
  for (int k = 0; k < 8; ++k) q.y |= zb[k] << (12 + k);
  rec7[n] = a;
  rec19[n] = q;
  slow[n] = 0u;
}

__global__ void ns_slow_list(const uint32_t* flag, const uint32_t* pos, int64_t nf, uint32_t* list) {
  const int64_t n = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (n < nf && flag[n]) list[pos[n]] = (uint32_t)n;
}

}  // namespace om

using namespace om;

extern "C" om_status om_nodeset_create(const uint8_t* nodes_dev, om_domain d, void* stream,
                                       om_nodeset** out) {
  if (!nodes_dev || !out) return fail(OM_EINVAL, "om_nodeset_create: null pointer");
  OM_TRY(check_domain(d));
  cudaStream_t s = as_stream(stream);
  const int W = (d.nz + 31) / 32;
  const int64_t ncol = (int64_t)d.nx * d.ny;
  const int64_t nw = ncol * W;
  // scratch of the column pass
  StreamBuf tmp(s);
  size_t at = 0;
  OM_TRY(tmp.alloc(3 * ((size_t)nw * 4 + 256) + 512));
  uint64_t* total = carve<uint64_t>(tmp.p, &at, 2);  // nodes, and links across x
  uint32_t* bits = carve<uint32_t>(tmp.p, &at, nw);
  uint32_t* cnt = carve<uint32_t>(tmp.p, &at, nw);
  uint32_t* rank = carve<uint32_t>(tmp.p, &at, nw);
  OM_CUDA(cudaMemsetAsync(total, 0, 2 * sizeof(uint64_t), s));
  const unsigned warps = (unsigned)std::min<int64_t>((nw + 7) / 8, 16 * 1216);
  const unsigned threads = (unsigned)std::min<int64_t>((nw + 127) / 128, 16 * 1216);
  if (pack_aligned(nodes_dev, d.nz)) ns_bits16<<<threads, 128, 0, s>>>(nodes_dev, d.nz, W, nw, bits, cnt);
  else ns_bits<<<warps, 256, 0, s>>>(nodes_dev, d.nz, W, nw, bits, cnt);
  ns_wrap_links<<<152, 256, 0, s>>>(nodes_dev, d.nx, d.ny, d.nz, (unsigned long long*)(total + 1));
  OM_CUDA(cudaGetLastError());
  OM_TRY(exclusive_scan_u32(cnt, rank, nw, total, s));
  uint64_t got[2] = {0, 0};
  OM_CUDA(cudaMemcpyAsync(got, total, sizeof got, cudaMemcpyDeviceToHost, s));
  OM_CUDA(cudaStreamSynchronize(s));
  const int64_t nf = (int64_t)got[0];

  om_nodeset* ns = new om_nodeset();
  ns->dom = d;
  ns->W = W;
  ns->N = voxels(d);
  ns->nf = nf;
  ns->pitch = (nf + 63) / 64 * 64;
  ns->wrap_links = (int64_t)got[1];
  // one allocation for everything the node set keeps; the slow nodes (lattice.cuh) lie on the
  // faces of the box, or are all nodes of a box beyond the record fields
  const int fit = d.nz <= kRecMaxNz && (int64_t)d.ny * d.nz <= kRecMaxPlane;
  const int64_t inner = std::max(0, d.nx - 2) * (int64_t)std::max(0, d.ny - 2) * std::max(0, d.nz - 2);
  const int64_t slow_cap = fit ? std::min(nf, ns->N - inner) : nf;
  DevBuf<uint8_t> mem;
  const int64_t nrec = fit ? nf : 0;
  om_status st = mem.alloc((size_t)nw * 16 + (size_t)nf * 12 + (size_t)nrec * 16 + (size_t)slow_cap * 4 + 6 * 256);
  StreamBuf flags(s);
  if (st == OM_OK && nf > 0) st = flags.alloc(2 * ((size_t)nf * 4 + 256) + 256 + (fit ? 0 : (size_t)nf * 16 + 512));
  if (st != OM_OK) {
    delete ns;
    return st;
  }
  at = 0;
  ns->mem = mem.take();
  ns->col = carve<uint4>(ns->mem, &at, nw);
  ns->vox = carve<int64_t>(ns->mem, &at, nf);
  uint2 *r7 = nullptr, *r19 = nullptr;
  if (fit) {
    r7 = carve<uint2>(ns->mem, &at, nf);
    r19 = carve<uint2>(ns->mem, &at, nf);
  }
  ns->coord = carve<uint32_t>(ns->mem, &at, nf);
  ns->slow = carve<uint32_t>(ns->mem, &at, slow_cap);
  auto build = [&]() -> om_status {
    ns_fill<<<warps, 256, 0, s>>>(bits, rank, d.ny, d.nz, W, nw, ns->col, ns->coord, ns->vox);
    OM_CUDA(cudaGetLastError());
    uint64_t nslow = 0;
    if (nf > 0) {
      size_t f = 0;
      uint64_t* tslow = carve<uint64_t>(flags.p, &f, 1);
      uint32_t* flag = carve<uint32_t>(flags.p, &f, nf);
      uint32_t* pos = carve<uint32_t>(flags.p, &f, nf);
      if (!fit) {  // written, not kept
        r7 = carve<uint2>(flags.p, &f, nf);
        r19 = carve<uint2>(flags.p, &f, nf);
      }
      const unsigned nb = (unsigned)((nf + 255) / 256);
      ns_records<<<nb, 256, 0, s>>>(ns->col, ns->coord, nf, d.nx, d.ny, d.nz, W, fit, r7, r19, flag);
      OM_CUDA(cudaGetLastError());
      OM_TRY(exclusive_scan_u32(flag, pos, nf, tslow, s));
      ns_slow_list<<<nb, 256, 0, s>>>(flag, pos, nf, ns->slow);
      OM_CUDA(cudaGetLastError());
      OM_CUDA(cudaMemcpyAsync(&nslow, tslow, sizeof nslow, cudaMemcpyDeviceToHost, s));
    }
    OM_CUDA(cudaStreamSynchronize(s));
    ns->n_slow = (int64_t)nslow;
    if (fit && nf > 0) {
      ns->rec7 = r7;
      ns->rec19 = r19;
    }
    return OM_OK;
  };
  st = build();
  if (st != OM_OK) {
    om_nodeset_destroy(ns);
    return st;
  }
  *out = ns;
  return OM_OK;
}

extern "C" om_status om_nodeset_count(const om_nodeset* ns, int64_t* n_nodes) {
  if (!ns || !n_nodes) return fail(OM_EINVAL, "om_nodeset_count: null pointer");
  *n_nodes = ns->nf;
  return OM_OK;
}

extern "C" om_status om_nodeset_voxels(const om_nodeset* ns, int64_t* voxel_dev, void* stream) {
  if (!ns || !voxel_dev) return fail(OM_EINVAL, "om_nodeset_voxels: null pointer");
  if (ns->nf > 0)
    OM_CUDA(cudaMemcpyAsync(voxel_dev, ns->vox, sizeof(int64_t) * ns->nf, cudaMemcpyDeviceToDevice,
                            as_stream(stream)));
  return OM_OK;
}

extern "C" om_status om_nodeset_destroy(om_nodeset* ns) {
  if (!ns) return OM_OK;
  cudaFree(ns->mem);
  delete ns;
  return OM_OK;
}
