// poresize.cu -- local pore size on the GPU.
//
// CHORD13 (Sec. 4.1): for each pore voxel and each of the 13 line
// directions (3 axes, 6 face diagonals, 4 body diagonals) count the cells of
// the all-pore line through it; lines wrap in y and z, stop at the x faces,
// and a closed all-pore loop counts each of its cells once.  The pore size
// is the mean of the 13 lengths, a count along a diagonal weighing sqrt(2)
// or sqrt(3) cells.
//
// MIS: r2(c), the squared distance from pore voxel c to the nearest solid
// voxel (periodic y, z; nothing solid beyond the x faces), by three separable
// 1-D minimisations; then every pore voxel v takes the largest r2(c) over
// centres c with |v - c|^2 < r2(c) and d = dx (2 sqrt(r2) - 1).
//
// Counts and distances are integers; the final diameters are fixed
// sequences of IEEE double operations (no fused multiply-add) rounded once
// to float.
#include <algorithm>
#include <cmath>

#include "common.cuh"

namespace om {
namespace {

__constant__ int8_t c_dir13[13][3] = {{1, 0, 0},  {0, 1, 0},  {0, 0, 1},   {1, 1, 0},  {1, -1, 0},
                                      {1, 0, 1},  {1, 0, -1}, {0, 1, 1},   {0, 1, -1}, {1, 1, 1},
                                      {1, 1, -1}, {1, -1, 1}, {1, -1, -1}};

// CHORD13 from bit lines.  Walking from every pore voxel along its 26 half
// lines reads ~325 bytes per pore voxel, one dependent step at a time (256^3
// at porosity 0.35: 11.4 ms).  Instead every line is packed once into 32-bit
// words (chord_lines), and a voxel's run length follows from one to three
// words per direction by counting ones on either side of its bit
// (chord13_kernel).  The packed lines take 13 N / 8 bytes (27 MB at 256^3: they
// stay in L2).  The same structure: lines 50 us + rows 6 us + lengths 343 us (535 with a
// thread per voxel of the box).
// What bounds it now is instructions: ~26 word reads and bit scans per pore
// voxel.
//
// Lines per direction k (e of c_dir13), position p along them:
//   e_x = 1:         line (y0, z0), its voxel at x = 0; p = x, nx voxels, no wrap;
//   (0, 1, e_z):     segment (x, z0), its voxel at y = 0; p = y, ny voxels; past
//                    the last one the segment z0 + e_z ny (mod nz) follows, so
//                    nz / gcd-many segments close to a loop of `loop` voxels;
//   (0, 0, 1):       segment (x, y); p = z, nz voxels, closing on itself.
// Word w of line l is bits[off + w * lines + l], so that lanes adjacent in z
// read adjacent words; for k = 2 lines are (x, y) rows and lanes share them.
struct ChordLines {
  int nx, ny, nz;
  uint32_t N;            // voxels (check_domain keeps them below 2^32 - 1)
  int wx, wy, wz;        // words per line along x, y, z
  uint32_t loop;         // voxels of a closed (0, 1, +-1) loop: lcm(ny, nz)
  uint32_t* bits;
  uint64_t off[13];      // first word of each direction
};

__device__ __forceinline__ int wrap_once(int v, int n) { return v < 0 ? v + n : (v >= n ? v - n : v); }

// The 32 voxels zs .. zs + 31 (periodic; nz >= 32) of row r as bits
__device__ __forceinline__ uint32_t row_window(const uint32_t* __restrict__ rowbits, uint32_t rows, uint32_t r, int zs, int nz) {
  const int w = zs >> 5, W = (nz + 31) >> 5;
  const uint32_t lo = __ldg(rowbits + (uint64_t)w * rows + r);
  const uint32_t hi = w + 1 < W ? __ldg(rowbits + (uint64_t)(w + 1) * rows + r) : 0u;
  uint32_t b = __funnelshift_r(lo, hi, zs & 31);  // bits past nz are zero
  if (zs + 32 > nz) b |= __ldg(rowbits + r) << (nz - zs);
  return b;
}

// One word of 32 adjacent lines (z0 = 32 zb ..) per warp, nz >= 32, from the
// packed rows: lane t takes the 32 voxels that step t of the 32 lines passes
// through, one window of a row, and the warp transposes the 32 x 32 bits.
// Byte by byte (chord_lines, left for shorter rows) the same words took
// 202 us at 256^3, 50 us so.  blockIdx.y = direction (k = 2 excluded).
__global__ void chord_lines_rows(ChordLines c) {
  const int lane = threadIdx.x & 31, j = blockIdx.y, k = j < 2 ? j : j + 1;
  const int ex = c_dir13[k][0], ey = c_dir13[k][1], ez = c_dir13[k][2];
  const int na = ex ? c.ny : c.nx, W = ex ? c.wx : c.wy, len = ex ? c.nx : c.ny;
  const uint32_t lines = (uint32_t)na * c.nz, rows = (uint32_t)c.nx * c.ny;
  const uint64_t total = (uint64_t)W * na * c.wz;
  for (uint64_t i = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < total;
       i += ((uint64_t)gridDim.x * blockDim.x) >> 5) {
    const int zb = (int)(i % c.wz), a = (int)(i / c.wz % na), w = (int)(i / c.wz / na);
    const int p = 32 * w + lane;  // position along the line
    uint32_t b = 0;
    if (p < len) {
      const int x = ex ? p : a;
      int y = ex ? a : p, z = 32 * zb;
      if (ex && ey) y = wrap_once(y + ey * (p % c.ny), c.ny);
      if (ez) z = wrap_once(z + ez * (p % c.nz), c.nz);
      b = row_window(c.bits + c.off[2], rows, (uint32_t)x * c.ny + y, z, c.nz);
    }
    // transpose: bit t of lane s becomes bit s of lane t
    uint32_t m = 0x0000ffffu;
#pragma unroll
    for (int s = 16; s > 0; s >>= 1, m ^= m << s) {
      const uint32_t o = __shfl_xor_sync(0xffffffffu, b, s);
      b = lane & s ? (b & ~m) | ((o >> s) & m) : (b & m) | ((o << s) & ~m);
    }
    const int z0 = 32 * zb + lane;
    if (z0 < c.nz) c.bits[c.off[k] + (uint64_t)w * lines + (uint32_t)a * c.nz + z0] = b;
  }
}

// One word of one line per thread: 32 mask bytes along the line (all 32 loads
// are independent).  blockIdx.y = direction (k = 2 excluded).
__global__ void chord_lines(const uint8_t* __restrict__ m, ChordLines c) {
  const int j = blockIdx.y, k = j < 2 ? j : j + 1;
  const int ex = c_dir13[k][0], ey = c_dir13[k][1], ez = c_dir13[k][2];
  const uint32_t lines = ex ? (uint32_t)c.ny * c.nz : (uint32_t)c.nx * c.nz;
  const int W = ex ? c.wx : c.wy, len = ex ? c.nx : c.ny;
  const uint64_t total = (uint64_t)W * lines;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (uint64_t)gridDim.x * blockDim.x) {
    const int w = (int)(i / lines);
    const uint32_t l = (uint32_t)(i - (uint64_t)w * lines);
    const int a = (int)(l / (uint32_t)c.nz), z0 = (int)(l - (uint32_t)a * c.nz);
    const int p0 = 32 * w, cnt = min(32, len - p0);
    int x = ex ? p0 : a, y = ex ? a : p0, z = z0;
    if (ex && ey) y = wrap_once(y + ey * (p0 % c.ny), c.ny);
    if (ez) z = wrap_once(z + ez * (p0 % c.nz), c.nz);
    uint32_t b = 0;
#pragma unroll 8
    for (int t = 0; t < cnt; ++t) {
      b |= (uint32_t)(m[((uint32_t)x * c.ny + y) * (uint32_t)c.nz + z] != 0) << t;
      x += ex;
      y += ey;
      if (ex) y = wrap_once(y, c.ny);
      z = wrap_once(z + ez, c.nz);
    }
    c.bits[c.off[k] + i] = b;
  }
}

// the z lines (k = 2): one warp packs 32 voxels of a row
__global__ void chord_rows(const uint8_t* __restrict__ m, ChordLines c) {
  const int lane = threadIdx.x & 31;
  const uint32_t rows = (uint32_t)c.nx * c.ny, total = rows * (uint32_t)c.wz;
  for (uint32_t i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < total; i += (gridDim.x * blockDim.x) >> 5) {
    const uint32_t r = i / (uint32_t)c.wz, w = i - r * (uint32_t)c.wz;
    const int z = 32 * (int)w + lane;
    const uint32_t b = __ballot_sync(0xffffffffu, z < c.nz && m[(uint64_t)r * c.nz + z] != 0);
    if (lane == 0) c.bits[c.off[2] + (uint64_t)w * rows + r] = b;
  }
}

__global__ void chord_rows16(const uint8_t* __restrict__ m, ChordLines c) {
  const uint32_t rows = (uint32_t)c.nx * c.ny, total = rows * (uint32_t)c.wz;
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x) {
    const uint32_t r = i / (uint32_t)c.wz, w = i - r * (uint32_t)c.wz;
    c.bits[c.off[2] + (uint64_t)w * rows + r] = pack_word(m + (uint64_t)r * c.nz + 32 * w, min(32, c.nz - 32 * (int)w));
  }
}

// Pore voxels that follow position p of line l, along the line (UP) or
// against it; `stride` words lie between consecutive words of the line.  A
// looping line goes on at its neighbour segment (next(l, UP)) and the count
// stops at `most`.
template <bool UP, class Next>
__device__ __forceinline__ uint32_t chord_run(const uint32_t* __restrict__ bits, uint32_t stride, uint32_t l, int p, int len,
                                              uint32_t most, Next next) {
  uint32_t n = 0;
  p += UP ? 1 : -1;
  for (;;) {
    if (UP ? p >= len : p < 0) {  // off the end of this line
      if (most == 0 || n >= most) break;
      l = next(l);
      p = UP ? 0 : len - 1;
    }
    const uint32_t w = __ldg(bits + (uint64_t)((uint32_t)p >> 5) * stride + l);
    const int b = p & 31;
    uint32_t ones;
    int room;
    if (UP) {
      room = min(32 - b, len - p);
      const uint32_t gap = ~(w >> b);  // first zero at or above p; bits shifted in read as zero
      ones = gap ? (uint32_t)__ffs((int)gap) - 1u : 32u;
    } else {
      room = b + 1;
      ones = (uint32_t)__clz((int)~(w << (31 - b)));
    }
    ones = min(ones, (uint32_t)room);
    n += ones;
    if ((int)ones < room) break;
    p += UP ? (int)ones : -(int)ones;
  }
  return most ? min(n, most) : n;
}

// the mean of the 13 lengths from the counts by kind of direction: the exact
// sequence of the definition, every operation rounded once
__device__ __forceinline__ float chord_mean(uint32_t s0, uint32_t s1, uint32_t s2, double dx, double sq2, double sq3) {
  const double acc = __dadd_rn(__dadd_rn((double)s0, __dmul_rn(sq2, (double)s1)), __dmul_rn(sq3, (double)s2));
  // acc / 13 correctly rounded by Markstein's method: a quotient from the
  // rounded reciprocal, and one correction by its exact remainder
  const double y = 1.0 / 13.0;
  const double q = __dmul_rn(acc, y);
  const double quo = __fma_rn(__fma_rn(-13.0, q, acc), y, q);
  return (float)__dmul_rn(quo, dx);
}

// One block lists the pores of 256 * per consecutive voxels and then gives each
// thread one of the list at a time: a warp of 32 voxels in a row is part solid
// nearly everywhere, and its solid lanes would wait for the others' counts.
constexpr int kChordPer = 8;

__global__ void __launch_bounds__(256) chord13_kernel(const uint8_t* __restrict__ m, ChordLines c, int per, double dx,
                                                      double sq2, double sq3, float* d_nm, int32_t* witness) {
  __shared__ uint16_t list[256 * kChordPer];
  __shared__ int count;
  const uint32_t nz = (uint32_t)c.nz, ny = (uint32_t)c.ny;
  const uint32_t plane = ny * nz, xz = (uint32_t)c.nx * nz, rows = (uint32_t)c.nx * ny;
  const uint64_t base = (uint64_t)blockIdx.x * (256 * per);
  const int lane = threadIdx.x & 31;
  if (threadIdx.x == 0) count = 0;
  __syncthreads();
  for (int i = 0; i < per; ++i) {
    const int o = 256 * i + (int)threadIdx.x;
    const uint64_t v = base + o;
    const bool pore = v < c.N && m[v];
    if (v < c.N && !pore) {
      d_nm[v] = 0.f;
      if (witness)
        for (int k = 0; k < 13; ++k) witness[(int64_t)k * c.N + v] = 0;
    }
    const unsigned who = __ballot_sync(0xffffffffu, pore);
    int at = 0;
    if (lane == 0 && who) at = atomicAdd(&count, __popc(who));
    at = __shfl_sync(0xffffffffu, at, 0);
    if (pore) list[at + __popc(who & ((1u << lane) - 1u))] = (uint16_t)o;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < count; i += 256) {
    const uint32_t v = (uint32_t)(base + list[i]);
    const uint32_t row = v / nz;
    const int z = (int)(v - row * nz), x = (int)(row / ny), y = (int)(row - (uint32_t)x * ny);
    const int xy = (int)((uint32_t)x % ny), xzm = (int)((uint32_t)x % nz), yz = (int)((uint32_t)y % nz);
    uint32_t s[3] = {0, 0, 0};
#pragma unroll
    for (int k = 0; k < 13; ++k) {
      constexpr int8_t D[13][3] = {{1, 0, 0},  {0, 1, 0},  {0, 0, 1},  {1, 1, 0},  {1, -1, 0}, {1, 0, 1},  {1, 0, -1},
                                   {0, 1, 1},  {0, 1, -1}, {1, 1, 1},  {1, 1, -1}, {1, -1, 1}, {1, -1, -1}};
      const int ex = D[k][0], ey = D[k][1], ez = D[k][2];
      const uint32_t* b = c.bits + c.off[k];
      uint32_t n;
      if (ex) {
        const int y0 = ey == 0 ? y : wrap_once(y - ey * xy, c.ny), z0 = ez == 0 ? z : wrap_once(z - ez * xzm, c.nz);
        const uint32_t l = (uint32_t)y0 * nz + (uint32_t)z0;
        auto none = [](uint32_t q) { return q; };
        n = 1u + chord_run<true>(b, plane, l, x, c.nx, 0u, none) + chord_run<false>(b, plane, l, x, c.nx, 0u, none);
      } else if (ey) {
        const uint32_t most = ez ? c.loop - 1u : ny - 1u;
        const uint32_t z0 = ez == 0 ? (uint32_t)z : (uint32_t)wrap_once(z - ez * yz, c.nz);
        const uint32_t first = (uint32_t)x * nz;
        const int step = (int)(ny % nz);  // z0 moves by e_z ny from one segment to the next
        auto fwd = [&](uint32_t q) { return first + (uint32_t)wrap_once((int)(q - first) + ez * step, c.nz); };
        auto bwd = [&](uint32_t q) { return first + (uint32_t)wrap_once((int)(q - first) - ez * step, c.nz); };
        n = chord_run<true>(b, xz, first + z0, y, c.ny, most, fwd);
        if (n < most) n += chord_run<false>(b, xz, first + z0, y, c.ny, most, bwd);
        ++n;
      } else {
        auto same = [](uint32_t q) { return q; };
        n = chord_run<true>(b, rows, row, z, c.nz, nz - 1u, same);
        if (n < nz - 1u) n += chord_run<false>(b, rows, row, z, c.nz, nz - 1u, same);
        ++n;
      }
      if (witness) witness[(int64_t)k * c.N + v] = (int)n;
      s[k < 3 ? 0 : (k < 9 ? 1 : 2)] += n;
    }
    d_nm[v] = chord_mean(s[0], s[1], s[2], dx, sq2, sq3);
  }
}

// The walking form, without scratch memory: what is left when the packed
// lines cannot be allocated.
// Cells along +-e from (x,y,z), stopping at solid or the x faces; *closed is
// set when the walk comes back to its start (an all-pore loop).
__device__ int walk(const uint8_t* __restrict__ m, int nx, int ny, int nz, int x, int y, int z, int ex,
                    int ey, int ez, bool* closed) {
  int n = 0, cx = x, cy = y, cz = z;
  *closed = false;
  for (;;) {
    cx += ex;
    if (cx < 0 || cx >= nx) return n;
    cy += ey;
    cy = cy < 0 ? cy + ny : (cy >= ny ? cy - ny : cy);
    cz += ez;
    cz = cz < 0 ? cz + nz : (cz >= nz ? cz - nz : cz);
    if (cx == x && cy == y && cz == z) {
      *closed = true;
      return n;
    }
    if (!m[((int64_t)cx * ny + cy) * nz + cz]) return n;
    ++n;
  }
}

__global__ void chord13_walk(const uint8_t* __restrict__ m, int nx, int ny, int nz, double dx,
                               double sq2, double sq3, float* d_nm, int32_t* witness) {
  const int64_t N = (int64_t)nx * ny * nz;
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < N; v += (int64_t)gridDim.x * blockDim.x) {
    if (!m[v]) {
      d_nm[v] = 0.f;
      if (witness)
        for (int k = 0; k < 13; ++k) witness[k * N + v] = 0;
      continue;
    }
    const int x = (int)(v / ((int64_t)ny * nz));
    const int y = (int)((v / nz) % ny), z = (int)(v % nz);
    long long s[3] = {0, 0, 0};
    for (int k = 0; k < 13; ++k) {
      const int ex = c_dir13[k][0], ey = c_dir13[k][1], ez = c_dir13[k][2];
      bool closed;
      int n = 1 + walk(m, nx, ny, nz, x, y, z, ex, ey, ez, &closed);
      if (!closed) n += walk(m, nx, ny, nz, x, y, z, -ex, -ey, -ez, &closed);
      if (witness) witness[k * N + v] = n;
      s[k < 3 ? 0 : (k < 9 ? 1 : 2)] += n;
    }
    double acc = __dadd_rn(__dadd_rn((double)s[0], __dmul_rn(sq2, (double)s[1])), __dmul_rn(sq3, (double)s[2]));
    acc = __ddiv_rn(acc, 13.0);
    d_nm[v] = (float)__dmul_rn(acc, dx);
  }
}

constexpr int kFar = 0x3fffffff;  // "no solid on this line": larger than any squared distance

// The three passes look outward from the voxel and stop at the first step
// whose own square is no smaller than the best so far: farther voxels of the
// line cannot lower it.  A pore's radius, not the edge of the box, sets the
// number of steps (96^3 of the 2 nm workload, the three passes: 179 us over full lines, 39 us so).
// pass 1 (z, periodic): squared distance to the nearest solid in the z line;
// info[1] = 1 when the mask has a solid voxel
__global__ void edt_z(const uint8_t* __restrict__ m, int nx, int ny, int nz, int* g, int* info) {
  const int64_t N = (int64_t)nx * ny * nz;
  bool any = false;
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < N; v += (int64_t)gridDim.x * blockDim.x) {
    const int z = (int)((uint32_t)v % (uint32_t)nz);
    const uint8_t* line = m + (v - z);
    int best = kFar;
    if (!line[z]) {
      best = 0;
      any = true;
    } else {
      for (int k = 1; 2 * k <= nz; ++k) {
        const int a = z + k < nz ? z + k : z + k - nz, b = z - k >= 0 ? z - k : z - k + nz;
        if (!line[a] || !line[b]) {
          best = k * k;
          break;
        }
      }
    }
    g[v] = best;
  }
  if (any) info[1] = 1;
}

// pass 2 (y, periodic): min over y' of g(y') + dy^2
__global__ void edt_y(const int* __restrict__ g, int nx, int ny, int nz, int* h) {
  const int64_t N = (int64_t)nx * ny * nz;
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < N; v += (int64_t)gridDim.x * blockDim.x) {
    const int y = (int)((uint32_t)v / (uint32_t)nz % (uint32_t)ny);
    const int* line = g + (v - (int64_t)y * nz);
    int best = g[v];
    for (int k = 1; 2 * k <= ny && k * k < best; ++k) {
      const int a = y + k < ny ? y + k : y + k - ny, b = y - k >= 0 ? y - k : y - k + ny;
      best = min(best, min(line[(int64_t)a * nz], line[(int64_t)b * nz]) + k * k);
    }
    h[v] = min(best, kFar);
  }
}

// pass 3 (x, bounded): min over x' of h(x') + dx^2; pore voxels only
__global__ void edt_x(const uint8_t* __restrict__ m, const int* __restrict__ h, int nx, int ny, int nz,
                      int* r2, int* info) {
  const int64_t N = (int64_t)nx * ny * nz;
  const int64_t plane = (int64_t)ny * nz;
  int local = 0;
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < N; v += (int64_t)gridDim.x * blockDim.x) {
    if (!m[v]) {
      r2[v] = 0;
      continue;
    }
    const int x = (int)((uint32_t)v / (uint32_t)plane);
    int best = h[v];
    for (int k = 1; k * k < best && (k <= x || x + k < nx); ++k) {
      if (x + k < nx) best = min(best, h[v + k * plane] + k * k);
      if (k <= x) best = min(best, h[v - k * plane] + k * k);
    }
    best = min(best, kFar);
    r2[v] = best;
    local = max(local, best);
  }
  for (int o = 16; o > 0; o >>= 1) local = max(local, __shfl_down_sync(0xffffffffu, local, o));
  if ((threadIdx.x & 31) == 0) atomicMax(info, local);
}

// Largest inscribed ball holding each pore voxel.  Testing every centre of
// the (2R + 1)^3 box around a voxel is thousands of r2 reads per voxel
// (96^3 of the 2 nm workload: 4.8 ms).  Centres are taken in bricks of 4^3
// voxels instead, each with its largest r2 (brick_max).  One warp serves a
// target brick, two voxels a lane: it lists the bricks around it whose
// largest ball reaches the target brick and exceeds the smallest radius its
// voxels already have, and scans them from the largest on, until the next
// one's largest ball is no larger than what every voxel has or will get from a
// brick that lies within its own largest ball.  The ball that holds a voxel is
// usually among the first few: 4.79 ms -> 0.28 ms, bound by the instructions of
// the lists and scans (r2 and the brick maxima sit in L1/L2).
constexpr int kBrick = 4;

__global__ void brick_max(const int* __restrict__ r2, int nx, int ny, int nz, int nbx, int nby, int nbz, int* top) {
  const int lane = threadIdx.x & 31;
  const uint32_t nb = (uint32_t)nbx * nby * nbz;
  for (uint32_t b = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; b < nb; b += (gridDim.x * blockDim.x) >> 5) {
    const int bz = (int)(b % nbz), by = (int)(b / nbz % nby), bx = (int)(b / nbz / nby);
    const int y = by * kBrick + ((lane >> 2) & 3), z = bz * kBrick + (lane & 3);
    int t = 0;
    for (int h = 0; h < 2; ++h) {
      const int x = bx * kBrick + (lane >> 4) + 2 * h;
      if (x < nx && y < ny && z < nz) t = max(t, r2[((int64_t)x * ny + y) * nz + z]);
    }
    t = (int)__reduce_max_sync(0xffffffffu, (unsigned)t);
    if (lane == 0) top[b] = t;
  }
}

// voxels between the intervals [a, a + 3] and [b, b + 3] of a line of n voxels
// (0 when they meet), each cut at the line's end; periodic: either way round
__device__ __forceinline__ int brick_gap(int a, int b, int n, bool periodic) {
  const int a1 = min(a + kBrick, n) - 1, b1 = min(b + kBrick, n) - 1;
  if (a <= b1 && b <= a1) return 0;
  const int up = b - a1, down = a - b1;  // one of them positive
  const int direct = max(up, down);
  return periodic ? min(direct, n - (max(a1, b1) - min(a, b))) : direct;
}

// an upper bound of the largest distance along the line between voxels of the two intervals
__device__ __forceinline__ int brick_far(int a, int b, int n, bool periodic) {
  const int a1 = min(a + kBrick, n) - 1, b1 = min(b + kBrick, n) - 1;
  const int direct = max(a1 - b, b1 - a);
  return periodic ? min(direct, n - max(max(b - a1, a - b1), 0)) : direct;
}

constexpr int kMisWarps = 4;   // warps per block
constexpr int kMisList = 512;  // bricks listed at a time per warp

__global__ void __launch_bounds__(32 * kMisWarps) mis_gather(const uint8_t* __restrict__ m, const int* __restrict__ r2,
                                                             const int* __restrict__ top, int nx, int ny, int nz, int nbx,
                                                             int nby, int nbz, const int* info, double dx, float* d_nm) {
  __shared__ int list_top[kMisWarps][kMisList];
  __shared__ uint32_t list_at[kMisWarps][kMisList];
  if (!info[1]) return;  // no solid voxel: refused by the host
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int* lt = list_top[wid];
  uint32_t* la = list_at[wid];
  int R = (int)ceilf(sqrtf((float)info[0])) + 1;  // ball radius bound: |v - c| < sqrt(r2)
  const int K = (R + kBrick - 1) / kBrick;
  const uint32_t nb = (uint32_t)nbx * nby * nbz;
  for (uint32_t tb = blockIdx.x * kMisWarps + wid; tb < nb; tb += gridDim.x * kMisWarps) {
    const int bz = (int)(tb % nbz), by = (int)(tb / nbz % nby), bx = (int)(tb / nbz / nby);
    const int y = by * kBrick + ((lane >> 2) & 3), z = bz * kBrick + (lane & 3);
    const bool row = y < ny && z < nz;
    int x[2], best[2];
    int64_t v[2];
    bool in[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      x[h] = bx * kBrick + (lane >> 4) + 2 * h;
      in[h] = row && x[h] < nx;
      v[h] = in[h] ? ((int64_t)x[h] * ny + y) * nz + z : 0;
      best[h] = in[h] && m[v[h]] ? r2[v[h]] : 0;  // a pore's own ball holds it
    }
    // the smallest radius among the brick's pores
    auto least = [&]() {
      const unsigned a = best[0] ? (unsigned)best[0] : 0xffffffffu, b = best[1] ? (unsigned)best[1] : 0xffffffffu;
      return __reduce_min_sync(0xffffffffu, min(a, b));
    };
    unsigned low = least();
    if (low != 0xffffffffu) {
      // radii that every voxel of the target has for certain: the largest ball of a brick when even
      // the farthest pair of voxels lies within it.  First from the bricks next to the target.
      unsigned sure = 0;
      auto certain = [&](int qx, int qy, int qz, int t) {
        const int fx = brick_far(bx * kBrick, qx * kBrick, nx, false);
        const int fy = brick_far(by * kBrick, qy * kBrick, ny, true);
        const int fz = brick_far(bz * kBrick, qz * kBrick, nz, true);
        return fx * fx + fy * fy + fz * fz < t ? (unsigned)t : 0u;
      };
      if (lane < 27) {
        const int qx = min(max(bx + lane / 9 - 1, 0), nbx - 1);
        int qy = by + lane / 3 % 3 - 1, qz = bz + lane % 3 - 1;
        qy = qy < 0 ? nby - 1 : (qy == nby ? 0 : qy);
        qz = qz < 0 ? nbz - 1 : (qz == nbz ? 0 : qz);
        sure = certain(qx, qy, qz, top[((uint32_t)qx * nby + qy) * nbz + qz]);
      }
      sure = __reduce_max_sync(0xffffffffu, sure);
      if (sure > low) low = sure - 1;
      // candidate bricks: K either side in x; in y and z one more, since the
      // last brick of a line may be narrower, or all of the line once
      const int x0 = max(0, bx - K), cx = min(nbx - 1, bx + K) - x0 + 1;
      const int cy = min(nby, 2 * K + 3), cz = min(nbz, 2 * K + 3);
      const int y0 = ((by - K - 1) % nby + nby) % nby, z0 = ((bz - K - 1) % nbz + nbz) % nbz;
      const uint32_t total = (uint32_t)cx * cy * cz;
      // a lane's candidate (jx, jy, jz), moved on by 32 with carries instead of divisions
      int jz = lane % cz, jy = lane / cz % cy, jx = lane / cz / cy;
      const int sz = 32 % cz, sy = 32 / cz % cy, sx = 32 / cz / cy;
      uint32_t next = 0;
      while (next < total) {
        int cnt = 0;
        for (; next < total && cnt <= kMisList - 32; next += 32) {  // list bricks that can matter
          int t = 0;
          const int qx = x0 + jx;
          int qy = y0 + jy, qz = z0 + jz;
          qy -= qy >= nby ? nby : 0;
          qz -= qz >= nbz ? nbz : 0;
          const uint32_t at = ((uint32_t)qx * nby + qy) * nbz + qz;
          if (next + lane < total) t = top[at];
          jz += sz;
          const bool c0 = jz >= cz;
          jz -= c0 ? cz : 0;
          jy += sy + c0;
          const bool c1 = jy >= cy;
          jy -= c1 ? cy : 0;
          jx += sx + c1;
          if (!__any_sync(0xffffffffu, t > (int)low)) continue;
          const int gx = brick_gap(bx * kBrick, qx * kBrick, nx, false);
          const int gy = brick_gap(by * kBrick, qy * kBrick, ny, true);
          const int gz = brick_gap(bz * kBrick, qz * kBrick, nz, true);
          if (gx * gx + gy * gy + gz * gz >= t) t = 0;
          if (__any_sync(0xffffffffu, t > (int)low)) {
            sure = __reduce_max_sync(0xffffffffu, t > (int)low ? max(sure, certain(qx, qy, qz, t)) : sure);
            if (sure > low) low = sure - 1;
          }
          const bool keep = t > (int)low;
          const unsigned who = __ballot_sync(0xffffffffu, keep);
          if (keep) {
            const int p = cnt + __popc(who & ((1u << lane) - 1u));
            lt[p] = t;
            la[p] = at;
          }
          cnt += __popc(who);
        }
        __syncwarp();
        for (;;) {  // largest first
          unsigned t = 0;
          int where = 0;
          for (int p = lane; p < cnt; p += 32)
            if ((unsigned)lt[p] > t) {
              t = (unsigned)lt[p];
              where = p;
            }
          const unsigned big = __reduce_max_sync(0xffffffffu, t);
          if (big <= low) break;  // nothing larger than what every voxel has
          const int src = __ffs(__ballot_sync(0xffffffffu, t == big)) - 1;
          where = __shfl_sync(0xffffffffu, where, src);
          const uint32_t at = la[where];
          __syncwarp();
          if (lane == src) lt[where] = 0;
          const int qz = (int)(at % nbz) * kBrick, qy = (int)(at / nbz % nby) * kBrick, qx = (int)(at / nbz / nby) * kBrick;
          int rc[2];
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int ax = qx + (lane >> 4) + 2 * h, ay = qy + ((lane >> 2) & 3), az = qz + (lane & 3);
            rc[h] = ax < nx && ay < ny && az < nz ? r2[((int64_t)ax * ny + ay) * nz + az] : 0;
          }
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            unsigned who = __ballot_sync(0xffffffffu, rc[h] > (int)low);
            while (who) {
              const int i = __ffs(who) - 1;
              who &= who - 1;
              const int r = __shfl_sync(0xffffffffu, rc[h], i);
              const int ax = qx + (i >> 4) + 2 * h, ay = qy + ((i >> 2) & 3), az = qz + (i & 3);
              int dy = abs(ay - y), dz = abs(az - z);
              dy = min(dy, ny - dy);
              dz = min(dz, nz - dz);
              const int dyz = dy * dy + dz * dz;
#pragma unroll
              for (int g = 0; g < 2; ++g) {
                const int ddx = ax - x[g];
                if (best[g] && r > best[g] && ddx * ddx + dyz < r) best[g] = r;
              }
            }
          }
          low = max(least(), low);
          __syncwarp();
        }
        __syncwarp();
      }
    }
#pragma unroll
    for (int h = 0; h < 2; ++h)
      if (in[h]) {
        const double val = __dsub_rn(__dmul_rn(2.0, sqrt((double)best[h])), 1.0);
        d_nm[v[h]] = best[h] ? (float)__dmul_rn(val, dx) : 0.f;
      }
  }
}

om_status chord13(const uint8_t* m, const om_domain& d, float* d_nm, int32_t* witness, cudaStream_t s) {
  const double sq2 = std::sqrt(2.0), sq3 = std::sqrt(3.0);
  ChordLines c{};
  c.nx = d.nx, c.ny = d.ny, c.nz = d.nz, c.N = (uint32_t)voxels(d);
  c.wx = (d.nx + 31) / 32, c.wy = (d.ny + 31) / 32, c.wz = (d.nz + 31) / 32;
  int a = d.ny, b = d.nz;
  while (b) {
    const int r = a % b;
    a = b;
    b = r;
  }
  c.loop = (uint32_t)(d.ny / a) * (uint32_t)d.nz;
  const uint64_t wx = (uint64_t)c.wx * d.ny * d.nz, wy = (uint64_t)c.wy * d.nx * d.nz, wz = (uint64_t)c.wz * d.nx * d.ny;
  uint64_t words = 0;
  for (int k = 0; k < 13; ++k) {
    c.off[k] = words;
    words += k == 2 ? wz : (k == 1 || k == 7 || k == 8 ? wy : wx);
  }
  StreamBuf buf(s);
  if (!buf.try_alloc(words * sizeof(uint32_t))) {  // (allowed under stream capture, as the form without scratch)
    chord13_walk<<<4 * 1216, 128, 0, s>>>(m, d.nx, d.ny, d.nz, d.dx_nm, sq2, sq3, d_nm, witness);
    OM_CUDA(cudaGetLastError());
    return OM_OK;
  }
  c.bits = (uint32_t*)buf.p;
  if (pack_aligned(m, d.nz)) chord_rows16<<<(unsigned)std::min<uint64_t>((wz + 127) / 128, 16 * 1216), 128, 0, s>>>(m, c);
  else chord_rows<<<(unsigned)std::min<uint64_t>((wz + 7) / 8, 16 * 1216), 256, 0, s>>>(m, c);
  if (d.nz >= 32) {
    const uint64_t warps = (uint64_t)std::max((uint64_t)c.wx * d.ny, (uint64_t)c.wy * d.nx) * c.wz;
    chord_lines_rows<<<dim3((unsigned)std::min<uint64_t>((warps + 7) / 8, 65535), 12), 256, 0, s>>>(c);
  } else {
    const unsigned nb = (unsigned)std::min<uint64_t>((std::max(wx, wy) + 255) / 256, 65535);
    chord_lines<<<dim3(nb, 12), 256, 0, s>>>(m, c);
  }
  // voxels per thread: up to kChordPer while the blocks still fill the chip (152 SMs x 8 blocks)
  const int per = (int)std::min<uint64_t>(kChordPer, std::max<uint64_t>(1, c.N / (256u * 152 * 8)));
  const uint64_t span = 256u * (uint64_t)per;
  chord13_kernel<<<(unsigned)((c.N + span - 1) / span), 256, 0, s>>>(m, c, per, d.dx_nm, sq2, sq3, d_nm, witness);
  OM_CUDA(cudaGetLastError());
  return OM_OK;
}

om_status pore_impl(const uint8_t* m, const om_domain& d, int mode, float* d_nm, int32_t* witness,
                    cudaStream_t s) {
  OM_TRY(check_domain(d));
  if (!m || !d_nm) return fail(OM_EINVAL, "local_pore_diameter: null pointer");
  const int64_t N = voxels(d);
  if (mode == OM_PORE_CHORD13) {
    return chord13(m, d, d_nm, witness, s);
  }
  if (mode != OM_PORE_MIS) return fail(OM_EINVAL, "local_pore_diameter: unknown mode");
  const int nbx = (d.nx + kBrick - 1) / kBrick, nby = (d.ny + kBrick - 1) / kBrick, nbz = (d.nz + kBrick - 1) / kBrick;
  const int64_t nb = (int64_t)nbx * nby * nbz;
  StreamBuf buf(s);
  OM_TRY(buf.alloc(sizeof(int) * (2 + (size_t)(witness ? 2 : 3) * N + nb)));
  int* info = (int*)buf.p;  // largest r2, and whether there is a solid voxel
  int *g = info + 2, *h = g + N, *top = h + N, *r2 = witness ? witness : top + nb;
  OM_CUDA(cudaMemsetAsync(info, 0, 2 * sizeof(int), s));
  edt_z<<<1216, 256, 0, s>>>(m, d.nx, d.ny, d.nz, g, info);
  edt_y<<<1216, 256, 0, s>>>(g, d.nx, d.ny, d.nz, h);
  edt_x<<<1216, 256, 0, s>>>(m, h, d.nx, d.ny, d.nz, r2, info);
  const unsigned blocks = (unsigned)std::min<int64_t>((nb + kMisWarps - 1) / kMisWarps, 1 << 20);
  brick_max<<<blocks, 32 * kMisWarps, 0, s>>>(r2, d.nx, d.ny, d.nz, nbx, nby, nbz, top);
  mis_gather<<<blocks, 32 * kMisWarps, 0, s>>>(m, r2, top, d.nx, d.ny, d.nz, nbx, nby, nbz, info, d.dx_nm, d_nm);
  OM_CUDA(cudaGetLastError());
  int hm[2];
  OM_CUDA(cudaMemcpyAsync(hm, info, sizeof hm, cudaMemcpyDeviceToHost, s));
  OM_CUDA(cudaStreamSynchronize(s));
  if (!hm[1]) return fail(OM_EINVAL, "local_pore_diameter (MIS): the mask has no solid voxel");
  return OM_OK;
}

}  // namespace
}  // namespace om

using namespace om;

extern "C" om_status om_local_pore_diameter_dev(const uint8_t* mask_dev, om_domain d, int32_t mode,
                                                float* d_nm_dev, int32_t* witness_dev, void* stream) {
  return pore_impl(mask_dev, d, mode, d_nm_dev, witness_dev, as_stream(stream));
}

extern "C" om_status om_local_pore_diameter(const uint8_t* mask, om_domain d, int32_t mode, float* d_nm,
                                            int32_t* witness) {
  if (!mask || !d_nm) return fail(OM_EINVAL, "om_local_pore_diameter: null pointer");
  OM_TRY(check_domain(d));
  const int64_t N = voxels(d);
  const int64_t nw = mode == OM_PORE_CHORD13 ? 13 * N : N;
  cudaStream_t s;
  OM_CUDA(cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking));
  DevBuf<uint8_t> m;
  DevBuf<float> dd;
  DevBuf<int32_t> w;
  om_status st = m.alloc(N);
  if (st == OM_OK) st = dd.alloc(N);
  if (st == OM_OK && witness) st = w.alloc(nw);
  if (st == OM_OK) {
    cudaError_t e = cudaMemcpyAsync(m.p, mask, N, cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) st = cuda_fail(e, "copy-in", __FILE__, __LINE__);
  }
  if (st == OM_OK) st = pore_impl(m.p, d, mode, dd.p, witness ? w.p : nullptr, s);
  if (st == OM_OK) {
    cudaError_t e = cudaMemcpyAsync(d_nm, dd.p, N * sizeof(float), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess && witness) e = cudaMemcpyAsync(witness, w.p, nw * sizeof(int32_t), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) st = cuda_fail(e, "copy-out", __FILE__, __LINE__);
  }
  cudaStreamDestroy(s);
  return st;
}
