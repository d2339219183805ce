// recon.cu -- random pore-sphere reconstruction (Sec. 2).
//
// Host: the sequential acceptance loop.  Candidate spheres come from one
// SplitMix64 stream (Steele, Lea & Flood 2014) in a fixed draw order: for
// every sphere after the first an "overlap required" flag (u < p0), then per
// trial the centre x, y, z (uniform over the box, voxel units) and the
// diameter.  A trial is accepted when, against every placed sphere, the
// overlapped volume is at most xi times each sphere's own volume, and, if
// overlap is required, it overlaps at least one of them (steps 1-2).  The
// test visits only spheres in neighbouring cells of a uniform grid whose cell
// edge is the largest possible diameter, so it costs O(1) per trial.
//
// Device: accepted spheres are rasterised in batches.  Every voxel records
// the smallest index of the spheres covering it (atomicMin); the number of
// voxels a sphere k covers first is then the count of voxels owned by k, and
// the porosity after each acceptance is a prefix sum of those counts.  The
// reconstruction stops at the first acceptance that reaches the target
// porosity (step 3) and the mask is "owner <= that sphere".
//
// The decisions are floating-point comparisons, so their arithmetic is
// fixed: every distance, volume and voxel test below is a sequence of
// individually rounded IEEE double operations (no fused multiply-add: host
// code is compiled with -ffp-contract=off, device code uses the _rn
// intrinsics) and libm's log, cos and sqrt for the normal draws.
#include <algorithm>
#include <cmath>
#include <vector>

#include "common.cuh"

namespace om {
namespace {

constexpr double kPi = 3.14159265358979323846;

struct SplitMix64 {
  uint64_t s;
  uint64_t next() {
    s += 0x9E3779B97F4A7C15ULL;
    uint64_t z = s;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
    return z ^ (z >> 31);
  }
  double uniform() { return (double)(next() >> 11) * 0x1.0p-53; }
};

struct Ball {
  double c[3];
  double r;
  double v;  // ball_volume(r)
};

double ball_volume(double r) { return (4.0 * kPi / 3.0) * (r * r * r); }

// volume shared by balls of radii r1, r2 whose centres are `dist` apart
double overlap_volume(double r1, double r2, double dist) {
  const double rs = r1 + r2;
  if (dist >= rs) return 0.0;
  if (dist <= std::fabs(r1 - r2)) return ball_volume(std::min(r1, r2));
  const double h = rs - dist;
  const double dr = r1 - r2;
  const double q = dist * dist + 2.0 * dist * rs - 3.0 * (dr * dr);
  return kPi * (h * h) * q / (12.0 * dist);
}

double periodic_gap(double d, int n) {
  if (d > 0.5 * n) return d - n;
  if (d < -0.5 * n) return d + n;
  return d;
}

struct Placer {
  om_domain dom;
  om_recon_params p;
  SplitMix64 rng;
  std::vector<Ball> balls;
  // uniform grid of cells, each at least one maximal diameter wide
  int gx = 1, gy = 1, gz = 1;
  double hx = 1, hy = 1, hz = 1;
  std::vector<std::vector<Ball>> cells;  // copies, so that a cell's balls lie together
  int64_t trials = 0;

  void init(uint64_t seed) {
    rng.s = seed;
    const double dmax = (p.dist == 1 ? p.mean_d_nm + p.sd_d_nm : p.dmax_nm) / dom.dx_nm;
    const double h = std::max(1.0, dmax);
    gx = std::max(1, (int)(dom.nx / h));
    gy = std::max(1, (int)(dom.ny / h));
    gz = std::max(1, (int)(dom.nz / h));
    hx = (double)dom.nx / gx;
    hy = (double)dom.ny / gy;
    hz = (double)dom.nz / gz;
    cells.assign((size_t)gx * gy * gz, {});
  }
  int cell_of(double v, double h, int g) const { return std::min(g - 1, std::max(0, (int)(v / h))); }

  double draw_diameter() {
    if (p.dist == 1) {
      const double u = rng.uniform();
      return (p.mean_d_nm - p.sd_d_nm) + (2.0 * p.sd_d_nm) * u;
    }
    const double u1 = rng.uniform();
    const double u2 = rng.uniform();
    const double z = std::sqrt(-2.0 * std::log(1.0 - u1)) * std::cos(2.0 * kPi * u2);
    double d = p.mean_d_nm + p.sd_d_nm * z;
    if (d < p.dmin_nm) d = p.dmin_nm;
    if (d > p.dmax_nm) d = p.dmax_nm;
    return d;
  }

  // tolerance and overlap-requirement test of a trial against placed balls
  bool acceptable(const Ball& t, bool must_touch) const {
    const double vt = t.v;
    bool touched = false;
    const int ix = cell_of(t.c[0], hx, gx), iy = cell_of(t.c[1], hy, gy), iz = cell_of(t.c[2], hz, gz);
    int ys[3], zs[3], ny = 0, nz = 0;
    for (int d = -1; d <= 1; ++d) {
      int y = ((iy + d) % gy + gy) % gy, z = ((iz + d) % gz + gz) % gz;
      if (std::find(ys, ys + ny, y) == ys + ny) ys[ny++] = y;
      if (std::find(zs, zs + nz, z) == zs + nz) zs[nz++] = z;
    }
    for (int x = std::max(0, ix - 1); x <= std::min(gx - 1, ix + 1); ++x)
      for (int a = 0; a < ny; ++a)
        for (int b = 0; b < nz; ++b)
          for (const Ball& s : cells[((size_t)x * gy + ys[a]) * gz + zs[b]]) {
            // most balls of the cells are out of reach: then the overlap is 0 and changes nothing.
            // Clear by more than any rounding of the distance, without its square root
            const double reach = (t.r + s.r) * (1.0 + 1e-9);
            const double dx = t.c[0] - s.c[0];
            if (dx > reach || -dx > reach) continue;
            const double dy = periodic_gap(t.c[1] - s.c[1], dom.ny);
            const double dz = periodic_gap(t.c[2] - s.c[2], dom.nz);
            const double d2 = dx * dx + dy * dy + dz * dz;
            if (d2 > reach * reach) continue;
            const double v = overlap_volume(t.r, s.r, std::sqrt(d2));
            if (v > 0.0) touched = true;
            if (v / vt > p.overlap_tol || v / s.v > p.overlap_tol) return false;
          }
    return touched || !must_touch;
  }

  void add(const Ball& b) {
    const int ix = cell_of(b.c[0], hx, gx), iy = cell_of(b.c[1], hy, gy), iz = cell_of(b.c[2], hz, gz);
    cells[((size_t)ix * gy + iy) * gz + iz].push_back(b);
    balls.push_back(b);
  }

  // place the next sphere (steps 1-2); false when the trial cap is hit
  bool place_next() {
    const bool first = balls.empty();
    const bool must_touch = first ? false : rng.uniform() < p.p_overlap;
    for (;;) {
      if (trials >= p.max_trials) return false;
      ++trials;
      Ball t;
      t.c[0] = rng.uniform() * dom.nx;
      t.c[1] = rng.uniform() * dom.ny;
      t.c[2] = rng.uniform() * dom.nz;
      t.r = 0.5 * (draw_diameter() / dom.dx_nm);
      t.v = ball_volume(t.r);
      if (first || acceptable(t, must_touch)) {
        add(t);
        return true;
      }
    }
  }
};

// ------------------------------------------------------------------ device
struct DevBall {
  double cx, cy, cz, r;
  int x0, x1, y0, y1, z0, z1;  // bounding box (y, z may wrap)
};

__device__ __forceinline__ bool voxel_in_ball(int vx, int vy, int vz, const DevBall& b, int ny, int nz) {
  const double ddx = __dsub_rn(__dadd_rn((double)vx, 0.5), b.cx);
  const double r2 = __dmul_rn(b.r, b.r);
  const double xx = __dmul_rn(ddx, ddx);
  for (int ky = -1; ky <= 1; ++ky) {
    const double ddy = __dsub_rn(__dadd_rn((double)vy, 0.5), __dadd_rn(b.cy, (double)(ky * ny)));
    const double xy = __dadd_rn(xx, __dmul_rn(ddy, ddy));
    for (int kz = -1; kz <= 1; ++kz) {
      const double ddz = __dsub_rn(__dadd_rn((double)vz, 0.5), __dadd_rn(b.cz, (double)(kz * nz)));
      if (__dadd_rn(xy, __dmul_rn(ddz, ddz)) <= r2) return true;
    }
  }
  return false;
}

// One voxel of a ball's box.  The exact test is nine images of double
// arithmetic, and this chip does two double operations per clock and SM; nearly every
// voxel is decided by a single-precision distance from the ball's centre in the
// unwrapped box instead.  Its error is below slack: offsets of less than
// 2 r + 4 voxels carry 2^-23 relative error, their squares' sum 2^-21 of
// itself at most, and centre and radius, rounded to single precision relative
// to the box's first voxel, 2^-23 of the box's edge; 2^-17 (d2 + r2) + 1e-3
// covers these several times over.  Voxels nearer to the surface than that
// take the exact test, as do balls so large that a voxel may lie in two
// images (`alone` false).
struct BallBox {
  DevBall b;
  float fx, fy, fz, r2;  // centre relative to the centre of the box's first voxel, radius squared
  bool alone;            // the box is the unwrapped one (to_dev) and no voxel lies in two images
};

__device__ __forceinline__ BallBox ball_box(const DevBall& b, int ny, int nz) {
  BallBox q;
  q.b = b;
  q.fx = (float)(b.cx - ((double)b.x0 + 0.5));
  q.fy = (float)(b.cy - ((double)b.y0 + 0.5));
  q.fz = (float)(b.cz - ((double)b.z0 + 0.5));
  q.r2 = (float)(b.r * b.r);
  q.alone = 2.0 * b.r + 8.0 < (double)ny && 2.0 * b.r + 8.0 < (double)nz;
  return q;
}

// offset (i, j, k) in the box, voxel (x, y, z) of the grid
__device__ __forceinline__ bool box_voxel_in_ball(const BallBox& q, int i, int j, int k, int x, int y, int z, int ny, int nz) {
  if (q.alone) {
    const float ex = (float)i - q.fx, ey = (float)j - q.fy, ez = (float)k - q.fz;
    const float d2 = ex * ex + ey * ey + ez * ez;
    const float slack = 0x1p-17f * (d2 + q.r2) + 1e-3f;
    if (d2 > q.r2 + slack) return false;
    if (d2 < q.r2 - slack) return true;
  }
  return voxel_in_ball(x, y, z, q.b, ny, nz);
}

// owner[v] = smallest index of the balls covering v.  blockIdx.y takes every
// gridDim.y-th x plane of the ball's box, its threads the plane's voxels
// (lanes along z).  Diameters vary ninefold and boxes by their cube, so a
// ball is spread over many blocks.  256^3 at porosity 0.35: 4.51 ms with one
// block a ball and the exact test everywhere, 1.00 ms with the single-precision
// test and two blocks a ball, 0.29 ms so.
__global__ void __launch_bounds__(256) raster_balls(const DevBall* balls, int k0, int nx, int ny, int nz, int* owner) {
  const BallBox q = ball_box(balls[blockIdx.x], ny, nz);
  const int k = k0 + (int)blockIdx.x;
  const int bx = q.b.x1 - q.b.x0 + 1, by = q.b.y1 - q.b.y0 + 1, bz = q.b.z1 - q.b.z0 + 1;
  const uint32_t cells = (uint32_t)by * (uint32_t)bz;
  for (int i = blockIdx.y; i < bx; i += gridDim.y) {
    const int x = q.b.x0 + i;
    int* plane = owner + (int64_t)x * ny * nz;
    for (uint32_t t = threadIdx.x; t < cells; t += blockDim.x) {
      const int j = (int)(t / (uint32_t)bz), l = (int)(t - (uint32_t)j * bz);
      int y = q.b.y0 + j, z = q.b.z0 + l;  // the box is at most one period wide and overlaps the grid
      y = y < 0 ? y + ny : (y >= ny ? y - ny : y);
      z = z < 0 ? z + nz : (z >= nz ? z - nz : z);
      int* o = plane + (uint32_t)y * (uint32_t)nz + z;
      if (box_voxel_in_ball(q, i, j, l, x, y, z, ny, nz) && *o > k) atomicMin(o, k);
    }
  }
}

// cnt[o - k0] += voxels owned by ball o in [k0, k1).  Neighbouring voxels
// mostly share an owner: a thread counts the runs of 16 consecutive voxels
// and adds one run at a time, in shared memory while the counters fit (16 K
// of them), else in global memory.  One global atomic a voxel took 0.81 ms (now 17 us) on
// 256^3 at porosity 0.35.
constexpr int kCountSlots = 16384;
__global__ void __launch_bounds__(512) count_first_cover(const int* owner, int64_t N, int k0, int k1, unsigned long long* cnt) {
  extern __shared__ unsigned int slot[];
  const int n = k1 - k0;
  const bool local = n <= kCountSlots;
  if (local) {
    for (int i = threadIdx.x; i < n; i += blockDim.x) slot[i] = 0u;
    __syncthreads();
  }
  auto add = [&](int o, unsigned c) {
    if (o < k0 || o >= k1) return;
    if (local) atomicAdd(slot + (o - k0), c);
    else atomicAdd(cnt + (o - k0), (unsigned long long)c);
  };
  const int64_t quads = N / 16;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < quads; t += (int64_t)gridDim.x * blockDim.x) {
    int4 a[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) a[i] = reinterpret_cast<const int4*>(owner)[t * 4 + i];
    const int* o = reinterpret_cast<const int*>(a);
    unsigned run = 1;
#pragma unroll
    for (int i = 1; i < 16; ++i) {
      if (o[i] == o[i - 1]) {
        ++run;
      } else {
        add(o[i - 1], run);
        run = 1;
      }
    }
    add(o[15], run);
  }
  for (int64_t v = quads * 16 + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < N; v += (int64_t)gridDim.x * blockDim.x)
    add(owner[v], 1u);
  if (local) {
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += blockDim.x)
      if (slot[i]) atomicAdd(cnt + i, (unsigned long long)slot[i]);
  }
}

__global__ void owner_to_mask(const int* owner, int64_t N, int kstop, uint8_t* mask) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < N; v += (int64_t)gridDim.x * blockDim.x)
    mask[v] = owner[v] <= kstop ? 1 : 0;
}

__global__ void fill_int(int* p, int64_t n, int val) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    p[i] = val;
}

DevBall to_dev(const Ball& b, const om_domain& d) {
  DevBall o;
  o.cx = b.c[0];
  o.cy = b.c[1];
  o.cz = b.c[2];
  o.r = b.r;
  o.x0 = std::max(0, (int)std::floor(b.c[0] - b.r) - 1);
  o.x1 = std::min(d.nx - 1, (int)std::ceil(b.c[0] + b.r) + 1);
  o.y0 = (int)std::floor(b.c[1] - b.r) - 1;
  o.y1 = (int)std::ceil(b.c[1] + b.r) + 1;
  if (o.y1 - o.y0 + 1 > d.ny) { o.y0 = 0; o.y1 = d.ny - 1; }
  o.z0 = (int)std::floor(b.c[2] - b.r) - 1;
  o.z1 = (int)std::ceil(b.c[2] + b.r) + 1;
  if (o.z1 - o.z0 + 1 > d.nz) { o.z0 = 0; o.z1 = d.nz - 1; }
  if (o.x1 < o.x0) o.x1 = o.x0 - 1;  // empty in x (cannot happen for centres in the box)
  return o;
}

om_status reconstruct_impl(uint64_t seed, const om_domain& d, const om_recon_params& p, uint8_t* mask_dev,
                           double* eps_out, int64_t* nsph_out, cudaStream_t s) {
  OM_TRY(check_domain(d));
  if (!(p.porosity > 0.0 && p.porosity <= 1.0)) return fail(OM_EINVAL, "porosity must be in (0, 1]");
  if (!(p.overlap_tol >= 0.0) || !(p.p_overlap >= 0.0 && p.p_overlap <= 1.0) || p.max_trials <= 0)
    return fail(OM_EINVAL, "bad overlap tolerance, p_overlap or max_trials");
  if (p.dist != 0 && p.dist != 1) return fail(OM_EINVAL, "dist must be 0 (normal) or 1 (uniform)");
  if (p.dist == 0 && !(p.dmin_nm > 0.0 && p.dmax_nm >= p.dmin_nm))
    return fail(OM_EINVAL, "need 0 < dmin_nm <= dmax_nm");
  if (p.dist == 1 && !(p.mean_d_nm - p.sd_d_nm > 0.0)) return fail(OM_EINVAL, "uniform diameters must be positive");
  const int64_t N = voxels(d);
  Placer pl;
  pl.dom = d;
  pl.p = p;
  pl.init(seed);

  StreamBuf own(s);
  OM_TRY(own.alloc(sizeof(int) * (size_t)N));
  int* owner = (int*)own.p;
  fill_int<<<1216, 256, 0, s>>>(owner, N, 0x7fffffff);
  OM_CUDA(cudaGetLastError());

  const double rmean = 0.5 * p.mean_d_nm / d.dx_nm;
  const double vmean = std::max(1.0, ball_volume(rmean));
  int64_t covered = 0;
  int kstop = -1;
  bool infeasible = false;
  std::vector<DevBall> host_balls;
  std::vector<unsigned long long> cnt;
  while (kstop < 0 && !infeasible) {
    const double need = p.porosity * (double)N - (double)covered;
    // about what is needed: every sphere placed beyond the last one is wasted (serial) work, and a
    // second, small batch costs one round trip
    int64_t chunk = (int64_t)std::ceil(1.15 * std::max(0.0, need) / vmean) + 16;
    chunk = std::min<int64_t>(chunk, 1 << 18);
    const int k0 = (int)pl.balls.size();
    StreamBuf batch(s);
    size_t at = 0;
    OM_TRY(batch.alloc((size_t)chunk * (sizeof(DevBall) + sizeof(unsigned long long)) + 512));
    DevBall* dballs = carve<DevBall>(batch.p, &at, chunk);
    unsigned long long* dcnt = carve<unsigned long long>(batch.p, &at, chunk);
    host_balls.resize(chunk);
    // placed in a few parts, each rasterised while the host places the next
    const int64_t part = std::max<int64_t>(64, (chunk + 3) / 4);
    int done = k0;  // balls handed to the device
    for (int64_t i = 0; i < chunk && !infeasible; ++i) {
      infeasible = !pl.place_next();
      const int k = (int)pl.balls.size(), n = k - done;
      if (n == 0 || (n < part && i + 1 < chunk && !infeasible)) continue;
      for (int j = done; j < k; ++j) host_balls[j - k0] = to_dev(pl.balls[j], d);
      OM_CUDA(cudaMemcpyAsync(dballs + (done - k0), host_balls.data() + (done - k0), sizeof(DevBall) * n,
                              cudaMemcpyHostToDevice, s));
      // about 16 blocks for each of the 1216 that are resident, so that large balls do not trail
      const int split = std::max(1, std::min(64, 16 * 1216 / n));
      raster_balls<<<dim3((unsigned)n, (unsigned)split), 256, 0, s>>>(dballs + (done - k0), done, d.nx, d.ny, d.nz, owner);
      done = k;
    }
    const int k1 = (int)pl.balls.size(), nb = k1 - k0;
    if (nb == 0) break;
    OM_CUDA(cudaMemsetAsync(dcnt, 0, sizeof(unsigned long long) * nb, s));
    const size_t smem = nb <= kCountSlots ? sizeof(unsigned int) * (size_t)nb : 0;
    OM_CUDA(cudaFuncSetAttribute(count_first_cover, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)sizeof(unsigned int) * kCountSlots));
    count_first_cover<<<304, 512, smem, s>>>(owner, N, k0, k1, dcnt);
    OM_CUDA(cudaGetLastError());
    cnt.resize(k1 - k0);
    OM_CUDA(cudaMemcpyAsync(cnt.data(), dcnt, sizeof(unsigned long long) * (k1 - k0), cudaMemcpyDeviceToHost, s));
    OM_CUDA(cudaStreamSynchronize(s));
    for (int k = k0; k < k1; ++k) {
      covered += (int64_t)cnt[k - k0];
      if ((double)covered / (double)N >= p.porosity) {
        kstop = k;
        break;
      }
    }
  }
  const int klast = kstop >= 0 ? kstop : (int)pl.balls.size() - 1;
  owner_to_mask<<<1216, 256, 0, s>>>(owner, N, klast, mask_dev);
  OM_CUDA(cudaGetLastError());
  OM_CUDA(cudaStreamSynchronize(s));
  if (eps_out) *eps_out = (double)covered / (double)N;
  if (nsph_out) *nsph_out = klast + 1;
  if (kstop < 0)
    return fail(OM_EINFEASIBLE, "reconstruction: trial cap reached before the target porosity");
  return OM_OK;
}

}  // namespace
}  // namespace om

using namespace om;

extern "C" om_status om_reconstruct_dev(uint64_t seed, om_domain d, const om_recon_params* params,
                                        uint8_t* mask_dev, double* porosity_out, int64_t* n_spheres_out,
                                        void* stream) {
  if (!params || !mask_dev) return fail(OM_EINVAL, "om_reconstruct_dev: null pointer");
  return reconstruct_impl(seed, d, *params, mask_dev, porosity_out, n_spheres_out, as_stream(stream));
}

extern "C" om_status om_reconstruct(uint64_t seed, om_domain d, const om_recon_params* params,
                                    uint8_t* mask, double* porosity_out, int64_t* n_spheres_out) {
  if (!params || !mask) return fail(OM_EINVAL, "om_reconstruct: null pointer");
  OM_TRY(check_domain(d));
  cudaStream_t s;
  OM_CUDA(cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking));
  DevBuf<uint8_t> m;
  om_status st = m.alloc(voxels(d));
  if (st == OM_OK) st = reconstruct_impl(seed, d, *params, m.p, porosity_out, n_spheres_out, s);
  if (st == OM_OK || st == OM_EINFEASIBLE) {
    cudaError_t e = cudaMemcpyAsync(mask, m.p, voxels(d), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) st = cuda_fail(e, "om_reconstruct copy-out", __FILE__, __LINE__);
  }
  cudaStreamDestroy(s);
  return st;
}
