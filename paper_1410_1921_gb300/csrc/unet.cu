// unet.cu -- the learned warm start: a 3-D U-Net that maps the structure
// (pore mask, local pore size) to the steady fields the LB solves produce
// (velocity u_x, concentration C), trained on the GPU by this file's own
// forward and backward passes; the LB then iterates from the prediction to
// the same convergence test, so the plain solve stays the judge of the
// result.
//
// Network (levels L, channels c_0..c_{L-1}): per encoder level two 3x3x3
// convolutions with ReLU, 2x average pooling between levels; per decoder
// level nearest 2x upsampling, the skip tensor concatenated (read as a second
// conv input, never materialised) and two 3x3x3 convolutions with ReLU; a
// 1x1 head without activation.  Masked mean-squared error; Adam.
#include <algorithm>
#include <cmath>
#include <mutex>
#include <vector>

#include "unet_tc.cuh"

namespace om {
namespace nn {
namespace {

constexpr int kT = 256;
inline unsigned blocks(int64_t n, int t = kT) { return (unsigned)std::min<int64_t>((n + t - 1) / t, 1 << 20); }

// input [V][cin] FP32 -> [V][16] BF16, zero-padded: a thread per voxel, two 16-byte stores
__global__ void pack_input(const float* x, int cin, uint32_t V, bf16* out) {
  for (uint32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < V; v += gridDim.x * blockDim.x) {
    const float* p = x + (int64_t)v * cin;
    union {
      uint4 u[2];
      __nv_bfloat16 h[16];
    } o;
#pragma unroll
    for (int c = 0; c < 16; ++c) o.h[c] = __float2bfloat16_rn(c < cin ? p[c] : 0.f);
    uint4* q = reinterpret_cast<uint4*>(out + (int64_t)v * 16);
    q[0] = o.u[0];
    q[1] = o.u[1];
  }
}

// The element-wise kernels below move 8 channels (one 16-byte vector of
// BF16) per thread: every channel count and row offset of the network is a
// multiple of 16.  The resampling ones take a row of x per block, so that z,
// y and the batch are divided out once per row and not per element (element
// by element, with 64-bit divisions, a prediction of 128 x 120 x 136 spent 373 us
// in these kernels and the operand conversions, 93 us so).
union V8 {
  uint4 u;
  __nv_bfloat16 h[8];
};

// row r of grid g: its z, y and batch
__device__ __forceinline__ void row_zyb(int64_t r, const Grid& g, int& z, int& y, int& b) {
  const int64_t p = r / g.H;
  y = (int)(r - p * g.H);
  b = (int)(p / g.D);
  z = (int)(p - (int64_t)b * g.D);
}

// fine grid gf -> coarse grid (gf / 2)
__global__ void avgpool2(const bf16* in, Grid gf, int C, bf16* out) {
  const Grid gc{gf.B, gf.D / 2, gf.H / 2, gf.W / 2};
  const int C8 = C / 8;
  const int64_t rows = (int64_t)gc.B * gc.D * gc.H;
  for (int64_t r = blockIdx.x; r < rows; r += gridDim.x) {
    int z, y, b;
    row_zyb(r, gc, z, y, b);
    const int64_t f0 = (((int64_t)b * gf.D + 2 * z) * gf.H + 2 * y) * gf.W;
    for (int i = threadIdx.x; i < gc.W * C8; i += blockDim.x) {
      const int x = i / C8, c8 = i - x * C8;
      float s[8] = {0, 0, 0, 0, 0, 0, 0, 0};
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int64_t vf = f0 + ((int64_t)(q >> 2) * gf.H + ((q >> 1) & 1)) * gf.W + 2 * x + (q & 1);
        V8 a;
        a.u = *reinterpret_cast<const uint4*>(in + vf * C + 8 * c8);
#pragma unroll
        for (int j = 0; j < 8; ++j) s[j] += __bfloat162float(a.h[j]);
      }
      V8 o;
#pragma unroll
      for (int j = 0; j < 8; ++j) o.h[j] = __float2bfloat16_rn(0.125f * s[j]);
      *reinterpret_cast<uint4*>(out + (r * gc.W + x) * C + 8 * c8) = o.u;
    }
  }
}

// nearest 2x: coarse [V_c x C] -> fine rows of C
__global__ void upsample2(const bf16* in, Grid gf, int C, bf16* out) {
  const int C8 = C / 8;
  const int64_t rows = (int64_t)gf.B * gf.D * gf.H;
  for (int64_t r = blockIdx.x; r < rows; r += gridDim.x) {
    int z, y, b;
    row_zyb(r, gf, z, y, b);
    const uint4* src = reinterpret_cast<const uint4*>(
        in + (((int64_t)b * (gf.D / 2) + z / 2) * (gf.H / 2) + y / 2) * (gf.W / 2) * C);
    uint4* dst = reinterpret_cast<uint4*>(out + r * gf.W * C);
    for (int i = threadIdx.x; i < gf.W * C8; i += blockDim.x) {
      const int x = i / C8, c8 = i - x * C8;
      dst[i] = src[(x / 2) * C8 + c8];
    }
  }
}

// d(coarse) = sum of the 8 fine children, read from rows of ldi at offset oi
__global__ void upsample2_bwd(const bf16* dfine, int ldi, int oi, Grid gf, int C, bf16* dcoarse) {
  const Grid gc{gf.B, gf.D / 2, gf.H / 2, gf.W / 2};
  const int C8 = C / 8;
  const int64_t rows = (int64_t)gc.B * gc.D * gc.H;
  for (int64_t r = blockIdx.x; r < rows; r += gridDim.x) {
    int z, y, b;
    row_zyb(r, gc, z, y, b);
    const int64_t f0 = (((int64_t)b * gf.D + 2 * z) * gf.H + 2 * y) * gf.W;
    for (int i = threadIdx.x; i < gc.W * C8; i += blockDim.x) {
      const int x = i / C8, c8 = i - x * C8;
      float acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int64_t vf = f0 + ((int64_t)(q >> 2) * gf.H + ((q >> 1) & 1)) * gf.W + 2 * x + (q & 1);
        V8 a;
        a.u = *reinterpret_cast<const uint4*>(dfine + vf * ldi + oi + 8 * c8);
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[j] += __bfloat162float(a.h[j]);
      }
      V8 o;
#pragma unroll
      for (int j = 0; j < 8; ++j) o.h[j] = __float2bfloat16_rn(acc[j]);
      *reinterpret_cast<uint4*>(dcoarse + (r * gc.W + x) * C + 8 * c8) = o.u;
    }
  }
}

// The gradient at a pre-activation, out = g [y > 0], and the bias gradient
// db[c] += sum_v out[v][c], in one pass.  g is formed on the way:
//   kGradRows  read from rows of ldg at og;
//   kGradSkip  what the pooling below and the decoder's skip send to an
//              encoder level: BF16(BF16(coarse / 8) + skip), coarse rows of N
//              of the level below, skip from rows of ldg at og;
//   kGradHead  the head's: sum_o dy[v][o] w[c][o]; with y the head's input,
//              the head's own gradients dw[c][o] += y dy, dhb[o] += dy are
//              summed in the same pass (up to kHeadOut outputs).
// A thread keeps its 8 channels over every voxel it visits; the block's
// threads of a channel group are summed in shared memory, then added with
// one atomic per channel.  As separate passes (ReLU, bias sums, pooling
// gradient, skip addition, head) these took 510 us of a training step on
// 4 x 64^3 (channels 32-64-128), 238 us so; bound by their reads and writes.
enum { kGradRows = 0, kGradSkip = 1, kGradHead = 2 };
constexpr int kHeadOut = 4;
struct GradArgs {
  const bf16* g;
  int ldg, og;
  const bf16* coarse;
  Grid gf;           // the fine grid (kGradSkip)
  const float *dy, *w;
  int O;             // head outputs
  float *dw, *dhb;   // head gradients (null: not summed here)
  const bf16* y;
  int N;
  uint32_t V;
  bf16* out;
  float* db;
};

template <int SRC>
__global__ void __launch_bounds__(256) relu_grad(GradArgs a) {
  extern __shared__ float sh[];  // [8][256]
  const int N8 = a.N / 8, lanes = 256 / N8, c8 = threadIdx.x % N8, lane = threadIdx.x / N8;
  const bool live = lane < lanes;
  constexpr int kSums = SRC == kGradHead ? 1 + kHeadOut : 1;
  float acc[kSums][8], accb[kHeadOut] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int k = 0; k < kSums; ++k)
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[k][j] = 0.f;
  if (live)
    for (uint32_t v = blockIdx.x * lanes + lane; v < a.V; v += gridDim.x * lanes) {
      V8 yy, gg, o;
      yy.u = *reinterpret_cast<const uint4*>(a.y + (int64_t)v * a.N + 8 * c8);
      if (SRC == kGradHead) {
        float d[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        for (int k = 0; k < a.O; ++k) {
          const float t = a.dy[(int64_t)v * a.O + k];
#pragma unroll
          for (int j = 0; j < 8; ++j) d[j] += t * a.w[(8 * c8 + j) * a.O + k];
        }
        if (a.dw) {
#pragma unroll
          for (int k = 0; k < kHeadOut; ++k)
            if (k < a.O) {
              const float t = a.dy[(int64_t)v * a.O + k];
              accb[k] += t;
#pragma unroll
              for (int j = 0; j < 8; ++j) acc[SRC == kGradHead ? 1 + k : 0][j] += __bfloat162float(yy.h[j]) * t;
            }
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) gg.h[j] = __float2bfloat16_rn(d[j]);
      } else {
        gg.u = *reinterpret_cast<const uint4*>(a.g + (int64_t)v * a.ldg + a.og + 8 * c8);
        if (SRC == kGradSkip) {
          const uint32_t W = a.gf.W, H = a.gf.H, D = a.gf.D;
          const uint32_t r = v / W, x = v - r * W, p = r / H, yv = r - p * H, bb = p / D, z = p - bb * D;
          const int64_t vc = (((int64_t)bb * (D / 2) + z / 2) * (H / 2) + yv / 2) * (W / 2) + x / 2;
          V8 cc;
          cc.u = *reinterpret_cast<const uint4*>(a.coarse + vc * a.N + 8 * c8);
#pragma unroll
          for (int j = 0; j < 8; ++j)
            gg.h[j] = __float2bfloat16_rn(__bfloat162float(__float2bfloat16_rn(0.125f * __bfloat162float(cc.h[j]))) +
                                          __bfloat162float(gg.h[j]));
        }
      }
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        o.h[j] = __bfloat162float(yy.h[j]) > 0.f ? gg.h[j] : __float2bfloat16_rn(0.f);
        acc[0][j] += __bfloat162float(o.h[j]);
      }
      *reinterpret_cast<uint4*>(a.out + (int64_t)v * a.N + 8 * c8) = o.u;
    }
  auto reduce = [&](const float (&t)[8], auto put) {
    __syncthreads();
#pragma unroll
    for (int j = 0; j < 8; ++j) sh[j * 256 + threadIdx.x] = live ? t[j] : 0.f;
    __syncthreads();
    for (int c = threadIdx.x; c < a.N; c += 256) {
      float sum = 0.f;
      for (int l = 0; l < lanes; ++l) sum += sh[(c & 7) * 256 + l * N8 + (c >> 3)];
      put(c, sum);
    }
  };
  reduce(acc[0], [&](int c, float t) { atomicAdd(&a.db[c], t); });
  if (SRC == kGradHead && a.dw) {
#pragma unroll
    for (int k = 0; k < kHeadOut; ++k)
      if (k < a.O) {
        reduce(acc[SRC == kGradHead ? 1 + k : 0], [&](int c, float t) { atomicAdd(&a.dw[c * a.O + k], t); });
        __syncthreads();
        sh[threadIdx.x] = live && c8 == 0 ? accb[k] : 0.f;
        __syncthreads();
        if (threadIdx.x == 0) {
          float t = 0.f;
          for (int l = 0; l < lanes; ++l) t += sh[l * N8];
          atomicAdd(&a.dhb[k], t);
        }
      }
  }
}

// 1x1 head: y[v][o] = b[o] + sum_c x[v][c] w[c][o]  (FP32 out); a thread per voxel reads its row
// of C channels as 16-byte vectors
__global__ void head_fwd(const bf16* x, int C, const float* w, const float* b, int O, int64_t V, float* y) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < V; v += (int64_t)gridDim.x * blockDim.x) {
    const uint4* row = reinterpret_cast<const uint4*>(x + v * C);
    for (int o = 0; o < O; ++o) {
      float acc = b[o];
      for (int c8 = 0; c8 < C / 8; ++c8) {
        V8 q;
        q.u = row[c8];
#pragma unroll
        for (int j = 0; j < 8; ++j) acc += __bfloat162float(q.h[j]) * w[(8 * c8 + j) * O + o];
      }
      y[v * O + o] = acc;
    }
  }
}

// the mask's nonzero count, added to *cnt (a double: exact below 2^53)
__global__ void mask_count(const uint8_t* m, int64_t V, double* cnt) {
  unsigned long long k = 0;
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < V; v += (int64_t)gridDim.x * blockDim.x)
    k += m[v] != 0;
  for (int o = 16; o > 0; o >>= 1) k += __shfl_down_sync(0xffffffffu, k, o);
  if ((threadIdx.x & 31) == 0 && k) atomicAdd(cnt, (double)k);
}

// masked MSE: loss = sum m (y - t)^2 * scale, dy = 2 m (y - t) * scale, scale = 1 / (count O)
// with the mask's count read from *cnt
__global__ void mse_grad(const float* y, const float* t, const uint8_t* m, int O, int64_t V, const double* cnt,
                         float* dy, double* loss) {
  const int64_t nk = (int64_t)*cnt;
  const float scale = nk > 0 ? 1.f / (float)(nk * O) : 0.f;
  double acc = 0.0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < V * O; i += (int64_t)gridDim.x * blockDim.x) {
    const float keep = m[i / O] ? 1.f : 0.f;
    const float d = (y[i] - t[i]) * keep;
    dy[i] = 2.f * d * scale;
    acc += (double)d * d * scale;
  }
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) atomicAdd(loss, acc);
}

// The head's gradients where it has more than kHeadOut outputs:
// dw[c][o] and db[o] for o in [o0, o0 + 4): thread t of a block takes channel t % C of the
// voxels t / C, t / C + lanes, ... (coalesced rows); the lanes are reduced in shared memory
__global__ void head_bwd_dw(const bf16* x, const float* dy, int C, int O, int o0, int64_t V, float* dw, float* db) {
  extern __shared__ float sh[];  // [8][blockDim.x]
  const int lanes = blockDim.x / C, c = threadIdx.x % C, lane = threadIdx.x / C;
  const int no = min(4, O - o0);
  float aw[4] = {0, 0, 0, 0}, ab[4] = {0, 0, 0, 0};
  if (lane < lanes)
    for (int64_t v = (int64_t)blockIdx.x * lanes + lane; v < V; v += (int64_t)gridDim.x * lanes) {
      const float xv = __bfloat162float(x[v * C + c]);
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (j < no) {
          const float d = dy[v * O + o0 + j];
          aw[j] += xv * d;
          ab[j] += d;
        }
    }
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    sh[j * blockDim.x + threadIdx.x] = lane < lanes ? aw[j] : 0.f;
    sh[(4 + j) * blockDim.x + threadIdx.x] = lane < lanes ? ab[j] : 0.f;
  }
  __syncthreads();
  if ((int)threadIdx.x < C) {
    for (int j = 0; j < no; ++j) {
      float tw = 0.f, tb = 0.f;
      for (int l = 0; l < lanes; ++l) {
        tw += sh[j * blockDim.x + l * C + threadIdx.x];
        tb += sh[(4 + j) * blockDim.x + l * C + threadIdx.x];
      }
      atomicAdd(&dw[threadIdx.x * O + o0 + j], tw);
      if (threadIdx.x == 0) atomicAdd(&db[o0 + j], tb);
    }
  }
}

// Every convolution's operands from the FP32 master weights in one launch
// (a launch per convolution and operand was 20 to 28 of them): FWD the
// forward operand WT[27][N][K] of W[27][K][N], else the data gradient's
// WD[27][K][N] = W[26 - k][K][N], the forward kernel with inputs dY (N
// channels) and output channels K.  blockIdx.y = convolution.
constexpr int kMaxConvs = 24;
struct OperandTable {
  const float* W[kMaxConvs];
  bf16* out[kMaxConvs];
  int K[kMaxConvs], N[kMaxConvs];
};
template <bool FWD>
__global__ void convert_weights(const __grid_constant__ OperandTable t) {
  const int K = t.K[blockIdx.y], N = t.N[blockIdx.y];
  const uint32_t per = (uint32_t)K * N, n = 27u * per;
  const float* W = t.W[blockIdx.y];
  bf16* out = t.out[blockIdx.y];
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const uint32_t k = i / per, r = i - k * per;
    if (FWD) {
      const uint32_t ci = r / N, co = r - ci * N;
      out[((uint64_t)k * N + co) * K + ci] = __float2bfloat16_rn(W[i]);
    } else {
      out[i] = __float2bfloat16_rn(W[(26u - k) * per + r]);
    }
  }
}

__global__ void adam_step(float* w, const float* g, float* m, float* v, int64_t n, float lr, float b1, float b2,
                          float eps, float bc1, float bc2) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    w[i] -= lr * (mi / bc1) / (sqrtf(vi / bc2) + eps);
  }
}

// ------------------------------------------------------------------ host side
struct Conv {
  int cin1, cin2, cout;
  int64_t w_off, b_off;  // into the flat parameter vector
  bf16* wt = nullptr;    // forward operand
  bf16* wd = nullptr;    // data-gradient operand
};

template <class T>
struct Buf {
  T* p = nullptr;
  size_t n = 0;
  om_status ensure(size_t count) {
    if (count <= n) return OM_OK;
    if (p) cudaFree(p);
    p = nullptr;
    n = 0;
    if (cudaMalloc((void**)&p, sizeof(T) * std::max<size_t>(count, 1)) != cudaSuccess) {
      (void)cudaGetLastError();
      return fail(OM_ENOMEM, "U-Net: device allocation failed");
    }
    n = count;
    return OM_OK;
  }
  void release() {
    if (p) cudaFree(p);
    p = nullptr;
    n = 0;
  }
};

}  // namespace
}  // namespace nn
}  // namespace om

using namespace om;
using namespace om::nn;

struct om_unet {
  int in_ch = 0, out_ch = 0, L = 0;
  std::vector<int> ch;
  std::vector<Conv> enc1, enc2, dec1, dec2;  // per level (dec: levels 0..L-2)
  int64_t head_w = 0, head_b = 0, nparam = 0;
  float *w = nullptr, *g = nullptr, *m = nullptr, *v = nullptr;  // FP32 master, grad, Adam moments
  int64_t step = 0;
  Grid grid{0, 0, 0, 0};
  // activations per level
  Buf<bf16> x0;
  std::vector<Buf<bf16>> in, a, s, u, b, h;
  Buf<float> out, dout;
  // gradients (scratch)
  std::vector<Buf<bf16>> d1, d2, dcat, ds;
  Buf<double> loss;
  // the BF16 operands are those of the present weights (cleared where the weights change)
  bool wt_ready = false, wd_ready = false;
  Buf<int> tc_err;  // set by a tensor-core convolution whose wait ran out
};

namespace {

// ------------------------------------------------------------------ tensor-core convolutions (unet_tc.cuh)
using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                   const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// the driver's tensor-map encoder, fetched through the runtime (nothing links libcuda)
om_status tensor_map_encoder(EncodeTiledFn* out) {
  static std::mutex mu;
  static EncodeTiledFn fn = nullptr;
  std::lock_guard<std::mutex> lock(mu);
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q{};
    OM_CUDA(cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q));
    if (q != cudaDriverEntryPointSuccess || !p) return fail(OM_ECUDA, "U-Net: cuTensorMapEncodeTiled unavailable");
    fn = (EncodeTiledFn)p;
  }
  *out = fn;
  return OM_OK;
}

// 5-D map of an NDHWC activation tensor: rows of ld BF16, c channels from o,
// zero fill; box by mode: 0 = {64 channels, 8 x, 8 y, 2 z, 1 batch} with the
// 128-byte swizzle, and with the 64-byte swizzle 1 = one plane of the halo
// {32, 10, 18, 1, 1}, 2 = the 8 x 16 tile {32, 8, 16, 1, 1}, 3 = {32, 10, 16,
// 3, 1}, 4 = {32, 8, 18, 1, 1}
om_status activation_map(CUtensorMap* m, const bf16* x, int c, int ld, int o, const Grid& g, int mode = 0) {
  const bool halo = mode != 0;
  EncodeTiledFn enc;
  OM_TRY(tensor_map_encoder(&enc));
  const cuuint64_t row = (cuuint64_t)ld * 2;
  cuuint64_t dims[5] = {(cuuint64_t)c, (cuuint64_t)g.W, (cuuint64_t)g.H, (cuuint64_t)g.D, (cuuint64_t)g.B};
  cuuint64_t strides[4] = {row, row * g.W, row * g.W * g.H, row * g.W * g.H * g.D};
  cuuint32_t box[5] = {(cuuint32_t)kTcKc, 8, 8, 2, 1};
  if (mode == 1) box[0] = 32, box[1] = kTcHx, box[2] = kTcHy, box[3] = 1;
  if (mode == 2) box[0] = 32, box[1] = kTcTx, box[2] = kTcTy, box[3] = 1;
  if (mode == 3) box[0] = 32, box[1] = kTcHx, box[2] = kTcTy, box[3] = 3;
  if (mode == 4) box[0] = 32, box[1] = kTcTx, box[2] = kTcTy + 2, box[3] = 1;
  cuuint32_t es[5] = {1, 1, 1, 1, 1};
  const CUresult r = enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, (void*)(x + o), dims, strides, box, es,
                         CU_TENSOR_MAP_INTERLEAVE_NONE, halo ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B,
                         CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return fail(OM_ECUDA, "U-Net: activation tensor map rejected (" + std::to_string((int)r) + ")");
  return OM_OK;
}

// 2-D map of the operand WT[27 N][K]: box {64 columns, N rows}, 128-byte
// swizzle (narrow = true: {32 columns, rows (default N) rows}, 64-byte swizzle)
om_status weight_map(CUtensorMap* m, const bf16* wt, int K, int N, bool narrow = false, int rows = 0) {
  EncodeTiledFn enc;
  OM_TRY(tensor_map_encoder(&enc));
  cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)27 * N};
  cuuint64_t strides[1] = {(cuuint64_t)K * 2};
  cuuint32_t box[2] = {narrow ? 32u : (cuuint32_t)kTcKc, (cuuint32_t)(rows > 0 ? rows : N)};
  cuuint32_t es[2] = {1, 1};
  const CUresult r = enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, (void*)wt, dims, strides, box, es,
                         CU_TENSOR_MAP_INTERLEAVE_NONE, narrow ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B,
                         CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return fail(OM_ECUDA, "U-Net: weight tensor map rejected (" + std::to_string((int)r) + ")");
  return OM_OK;
}

// stages + 1 KB alignment slack + barriers and the TMEM address slot
size_t tc_smem_bytes(int N) { return 1024 + (size_t)kTcStages * (kTcATile + (size_t)N * 128) + 8 * (2 * kTcStages + 1) + 16; }

// Y (rows of ldy, channels [oy, oy + N)) = conv of concat(x1, x2) with WT[27][N][c1 + c2]
om_status conv_tc(const om_unet* U, const bf16* x1, int c1, int ld1, int o1, const bf16* x2, int c2, int ld2, int o2,
                  const bf16* wt, int N, const float* bias, bf16* y, int ldy, int oy, int relu, const Grid& g,
                  cudaStream_t s) {
  if (N % 16 || N < 16 || N > 256 || c1 < 8 || (c1 % 8) || (c2 % 8) || (ld1 % 8) || (o1 % 8) || (ldy % 8) || (oy % 8))
    return fail(OM_EINVAL, "U-Net: convolution shape outside the tensor-core kernel's layout");
  CUtensorMap m1, m2, mw;
  const int nch = (c1 + 31) / 32 + (c2 + 31) / 32;
  if (nch <= 3) {
    // planes marched with the weights of np output channels resident (conv3d_tc_zm): equal parts of
    // N, multiples of 16, as wide as 3 np <= 256 columns and the shared memory beside nch + 1 halo
    // buffers allow
    constexpr size_t kSmem = 227 * 1024 - 1280;  // static shared memory set aside
    int np = 0;
    for (int d = 5; d >= 1 && !np; --d)
      if ((N / 16) % d == 0 && zm_smem(nch + 1, nch, 16 * d) <= kSmem) np = 16 * d;
    if ((c2 > 0 && ((ld2 % 8) || (o2 % 8)))) return fail(OM_EINVAL, "U-Net: second input not 16-byte aligned");
    OM_TRY(activation_map(&m1, x1, c1, ld1, o1, g, 1));
    if (c2 > 0) OM_TRY(activation_map(&m2, x2, c2, ld2, o2, g, 1));
    else m2 = m1;
    OM_TRY(weight_map(&mw, wt, c1 + c2, N, true, np));
    int dev = 0, sms = 0;
    OM_CUDA(cudaGetDevice(&dev));
    OM_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    TcConvArgs a{};
    a.c1 = c1, a.c2 = c2, a.N = np, a.bias = bias, a.y = y, a.ldy = ldy, a.oy = oy, a.relu = relu, a.g = g;
    a.nw = N, a.npart = N / np;
    a.tx = (g.W + kTcTx - 1) / kTcTx, a.ty = (g.H + kTcTy - 1) / kTcTy;
    a.err = U->tc_err.p;
    // CTAs per SM: as many, up to kZmPerSm, as leave each its weights, two planes more than it works
    // on, a ring of at least 5 accumulators in an equal power of two of TMEM columns, and a run of 8
    // planes or more.  Each part's CTAs share the planes of all columns.
    const int64_t planes = (int64_t)g.B * a.ty * a.tx * g.D;
    int per = kZmPerSm;
    size_t room = 0;
    int cols = 0;
    for (;; --per) {
      room = per == 1 ? kSmem : 228 * 1024 / per - 1024 - 1280;
      cols = per == 1 ? 512 : (per == 2 ? 256 : 128);
      if (per == 1 || (zm_smem(nch + 2, nch, np) <= room && cols / np >= 5 && planes * a.npart >= 8ll * per * sms)) break;
    }
    a.nhalo = nch + 1;
    while (a.nhalo < kZmMaxHalo && zm_smem(a.nhalo + 1, nch, np) <= room) ++a.nhalo;
    a.nacc = std::min(kZmMaxRing, cols / np);
    const size_t smem = zm_smem(a.nhalo, nch, np);
    const unsigned grid = (unsigned)(a.npart * std::min<int64_t>(planes, std::max(1, per * sms / a.npart)));
    auto k = nch == 1 ? (c1 <= 16 ? conv3d_tc_zm<1, 1> : conv3d_tc_zm<1, 2>) : (nch == 2 ? conv3d_tc_zm<2, 2> : conv3d_tc_zm<3, 2>);
    OM_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    k<<<grid, kZmThreads, smem, s>>>(m1, m2, mw, a);
    OM_CUDA(cudaGetLastError());
    return OM_OK;
  }
  OM_TRY(activation_map(&m1, x1, c1, ld1, o1, g));
  if (c2 > 0) {
    if ((ld2 % 8) || (o2 % 8)) return fail(OM_EINVAL, "U-Net: second input not 16-byte aligned");
    OM_TRY(activation_map(&m2, x2, c2, ld2, o2, g));
  } else {
    m2 = m1;
  }
  OM_TRY(weight_map(&mw, wt, c1 + c2, N));
  TcConvArgs a{};
  a.c1 = c1, a.c2 = c2, a.N = N, a.bias = bias, a.y = y, a.ldy = ldy, a.oy = oy, a.relu = relu, a.g = g;
  a.tx = (g.W + 7) / 8, a.ty = (g.H + 7) / 8, a.tz = (g.D + 1) / 2;
  a.err = U->tc_err.p;
  OM_CUDA(cudaFuncSetAttribute(conv3d_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tc_smem_bytes(N)));
  const unsigned grid = (unsigned)((int64_t)g.B * a.tz * a.ty * a.tx);
  conv3d_tc<<<grid, kTcThreads, tc_smem_bytes(N), s>>>(m1, m2, mw, a);
  OM_CUDA(cudaGetLastError());
  return OM_OK;
}

// a tensor-core convolution gave up a wait: report (synchronises)
om_status check_tc(const om_unet* U, cudaStream_t s) {
  int h = 0;
  OM_CUDA(cudaMemcpyAsync(&h, U->tc_err.p, sizeof(int), cudaMemcpyDeviceToHost, s));
  OM_CUDA(cudaStreamSynchronize(s));
  if (h) return fail(OM_ETIMEOUT, "U-Net: a tensor-core convolution's wait ran out");
  return OM_OK;
}

om_status conv_forward(const om_unet* U, const Conv& c, const bf16* x1, int ld1, int o1, const bf16* x2, int ld2, int o2,
                       bf16* y, const Grid& g, cudaStream_t s) {
  return conv_tc(U, x1, c.cin1, ld1, o1, x2, c.cin2, ld2, o2, c.wt, c.cout, U->w + c.b_off, y, c.cout, 0, 1, g, s);
}

// dX (rows of cin1 + cin2) = data gradient of conv c for the pre-activation gradient dyp: the
// forward convolution of dyp with the flipped, transposed weights WD[27][cin][cout]
om_status conv_dgrad(const om_unet* U, const Conv& c, const bf16* dyp, bf16* dx, const Grid& g, cudaStream_t s) {
  const int N = c.cin1 + c.cin2;
  return conv_tc(U, dyp, c.cout, c.cout, 0, nullptr, 0, 0, 0, c.wd, N, nullptr, dx, N, 0, 0, g, s);
}

// dW += the weight gradient on tcgen05: conv3d_wgrad_tc32 for at most 32 output channels
// (one CTA per input chunk of 32 channels), else conv3d_wgrad_tc (one CTA per chunk, dz and
// part of 128 output channels); gridDim.x of them over the tiles
om_status wgrad_tc(om_unet* U, const Conv& c, const bf16* x1, int ld1, int o1, const bf16* x2, int ld2, int o2,
                   const bf16* dyp, const Grid& g, cudaStream_t s) {
  TcWgradArgs a{};
  a.c1 = c.cin1, a.c2 = c.cin2, a.nch1 = (c.cin1 + 31) / 32;
  const int nch2 = (c.cin2 + 31) / 32;
  a.N = c.cout, a.Nm = (std::min(c.cout, 128) + 31) / 32 * 32;
  a.npart = (c.cout + 127) / 128;
  a.dw = U->g + c.w_off;
  a.g = g;
  a.tx = (g.W + kTcTx - 1) / kTcTx, a.ty = (g.H + kTcTy - 1) / kTcTy;
  a.vec4 = reinterpret_cast<uintptr_t>(a.dw) % 16 == 0;
  a.err = U->tc_err.p;
  int dev = 0, sms = 0;
  OM_CUDA(cudaGetDevice(&dev));
  OM_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  if (a.Nm == 32) {
    // at most 32 output channels: the swapped form (conv3d_wgrad_tc32), all 27 offsets per CTA
    CUtensorMap m1, m2, md;
    OM_TRY(activation_map(&m1, x1, c.cin1, ld1, o1, g, 3));
    if (c.cin2 > 0) OM_TRY(activation_map(&m2, x2, c.cin2, ld2, o2, g, 3));
    else m2 = m1;
    OM_TRY(activation_map(&md, dyp, c.cout, c.cout, 0, g, 4));
    a.nstage = (int)std::min<size_t>(4, (227 * 1024 - 2048) / kWnStage);
    const size_t smem = 1024 + (size_t)a.nstage * kWnStage + 8 * (2 * a.nstage + 1) + 16;
    const int gy = a.nch1 + nch2;
    const int64_t ntiles = (int64_t)g.B * g.D * (a.ty + 1) * a.tx;
    const unsigned gx = (unsigned)std::max<int64_t>(1, std::min<int64_t>(ntiles, sms / gy));
    OM_CUDA(cudaFuncSetAttribute(conv3d_wgrad_tc32, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    conv3d_wgrad_tc32<<<dim3(gx, (unsigned)gy), kTcThreads, smem, s>>>(m1, m2, md, a);
    OM_CUDA(cudaGetLastError());
    return OM_OK;
  }
  // wider outputs: conv3d_wgrad_tc, one dz per CTA
  CUtensorMap m1, m2, md;
  OM_TRY(activation_map(&m1, x1, c.cin1, ld1, o1, g, 1));
  if (c.cin2 > 0) OM_TRY(activation_map(&m2, x2, c.cin2, ld2, o2, g, 1));
  else m2 = m1;
  OM_TRY(activation_map(&md, dyp, c.cout, c.cout, 0, g, 2));
  const size_t stage = wg_stage_bytes(a.Nm);
  a.nstage = (int)std::min<size_t>(4, (227 * 1024 - 2048) / stage);
  const size_t smem = 1024 + (size_t)a.nstage * stage + 8 * (2 * a.nstage + 1) + 16;
  const int gy = (a.nch1 + nch2) * 3 * a.npart;
  const int64_t ntiles = (int64_t)g.B * g.D * a.ty * a.tx;
  // one CTA per SM fits (shared memory); at most one wave, or the last CTAs run as a second
  const unsigned gx = (unsigned)std::max<int64_t>(1, std::min<int64_t>(ntiles, sms / gy));
  OM_CUDA(cudaFuncSetAttribute(conv3d_wgrad_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  conv3d_wgrad_tc<<<dim3(gx, (unsigned)gy), kTcThreads, smem, s>>>(m1, m2, md, a);
  OM_CUDA(cudaGetLastError());
  return OM_OK;
}

// dW += the weight gradient of conv c for the pre-activation gradient dyp (its bias gradient: relu_grad)
om_status conv_wgrad(om_unet* U, const Conv& c, const bf16* x1, int ld1, int o1, const bf16* x2, int ld2, int o2,
                     const bf16* dyp, const Grid& g, cudaStream_t s) {
  if (c.cout % 16 || c.cout > 256 || c.cin1 % 8 || c.cin2 % 8 || ld1 % 8 || o1 % 8 ||
      (c.cin2 > 0 && (ld2 % 8 || o2 % 8)))
    return fail(OM_EINVAL, "U-Net: weight-gradient shape outside the tensor-core kernel's layout");
  return wgrad_tc(U, c, x1, ld1, o1, x2, ld2, o2, dyp, g, s);
}

Grid level_grid(const Grid& g, int l) { return Grid{g.B, g.D >> l, g.H >> l, g.W >> l}; }

om_status prepare(om_unet* U, const Grid& g) {
  if (g.B == U->grid.B && g.D == U->grid.D && g.H == U->grid.H && g.W == U->grid.W) return OM_OK;
  U->grid = Grid{0, 0, 0, 0};  // until every buffer holds g: a failed allocation has freed its predecessor
  const int L = U->L;
  for (int l = 0; l < L; ++l) {
    const int64_t V = level_grid(g, l).voxels();
    const int cprev = l == 0 ? 16 : U->ch[l - 1];
    const int cnext = l + 1 < L ? U->ch[l + 1] : 0;
    const int c = U->ch[l];
    if (l > 0) OM_TRY(U->in[l].ensure(V * cprev));
    OM_TRY(U->a[l].ensure(V * c));
    OM_TRY(U->s[l].ensure(V * c));
    if (l + 1 < L) {
      OM_TRY(U->u[l].ensure(V * cnext));
      OM_TRY(U->b[l].ensure(V * c));
      OM_TRY(U->h[l].ensure(V * c));
      OM_TRY(U->dcat[l].ensure(V * (cnext + c)));
    }
    const int64_t wmax = std::max((int64_t)c, std::max((int64_t)cprev, (int64_t)(cnext + c)));
    OM_TRY(U->d1[l].ensure(V * wmax));
    OM_TRY(U->d2[l].ensure(V * wmax));
    OM_TRY(U->ds[l].ensure(V * c));
  }
  OM_TRY(U->x0.ensure(g.voxels() * 16));
  OM_TRY(U->out.ensure(g.voxels() * U->out_ch));
  OM_TRY(U->dout.ensure(g.voxels() * U->out_ch));
  U->grid = g;
  return OM_OK;
}

// the forward (or data-gradient) operands of the present weights
om_status refresh_operands(om_unet* U, bool fwd, cudaStream_t s) {
  bool& ready = fwd ? U->wt_ready : U->wd_ready;
  if (ready) return OM_OK;
  OperandTable t{};
  int n = 0, most = 0;
  auto conv = [&](Conv& c) {
    t.W[n] = U->w + c.w_off;
    t.out[n] = fwd ? c.wt : c.wd;
    t.K[n] = c.cin1 + c.cin2;
    t.N[n] = c.cout;
    most = std::max(most, 27 * t.K[n] * t.N[n]);
    ++n;
  };
  for (int l = 0; l < U->L; ++l) {
    conv(U->enc1[l]);
    conv(U->enc2[l]);
    if (l + 1 < U->L) {
      conv(U->dec1[l]);
      conv(U->dec2[l]);
    }
  }
  const dim3 grid(std::min<unsigned>(blocks(most), 608), (unsigned)n);
  if (fwd) convert_weights<true><<<grid, kT, 0, s>>>(t);
  else convert_weights<false><<<grid, kT, 0, s>>>(t);
  OM_CUDA(cudaGetLastError());
  ready = true;
  return OM_OK;
}

unsigned row_blocks(const Grid& g) { return (unsigned)std::min<int64_t>((int64_t)g.B * g.D * g.H, 8 * 1216); }

om_status launch_relu_grad(int src, const GradArgs& a, cudaStream_t s) {
  const int lanes = 256 / (a.N / 8);
  const unsigned nb = (unsigned)std::min<int64_t>(((int64_t)a.V + lanes - 1) / lanes, 1216);
  const size_t smem = 8 * 256 * sizeof(float);
  if (src == kGradRows) relu_grad<kGradRows><<<nb, 256, smem, s>>>(a);
  else if (src == kGradSkip) relu_grad<kGradSkip><<<nb, 256, smem, s>>>(a);
  else relu_grad<kGradHead><<<nb, 256, smem, s>>>(a);
  OM_CUDA(cudaGetLastError());
  return OM_OK;
}

om_status forward(om_unet* U, const float* x, const Grid& g, cudaStream_t s) {
  OM_TRY(prepare(U, g));
  OM_TRY(refresh_operands(U, true, s));
  const int L = U->L;
  pack_input<<<std::min<unsigned>(blocks(g.voxels()), 16 * 1216), kT, 0, s>>>(x, U->in_ch, (uint32_t)g.voxels(), U->x0.p);
  for (int l = 0; l < L; ++l) {
    const Grid gl = level_grid(g, l);
    const bf16* in = l == 0 ? U->x0.p : U->in[l].p;
    const int cin = l == 0 ? 16 : U->ch[l - 1];
    if (l > 0) avgpool2<<<row_blocks(gl), kT, 0, s>>>(U->s[l - 1].p, level_grid(g, l - 1), cin, U->in[l].p);
    OM_TRY(conv_forward(U, U->enc1[l], in, cin, 0, nullptr, 0, 0, U->a[l].p, gl, s));
    OM_TRY(conv_forward(U, U->enc2[l], U->a[l].p, U->ch[l], 0, nullptr, 0, 0, U->s[l].p, gl, s));
  }
  for (int l = L - 2; l >= 0; --l) {
    const Grid gl = level_grid(g, l);
    const bf16* below = l + 1 == L - 1 ? U->s[L - 1].p : U->h[l + 1].p;
    const int cb = U->ch[l + 1];
    upsample2<<<row_blocks(gl), kT, 0, s>>>(below, gl, cb, U->u[l].p);
    OM_TRY(conv_forward(U, U->dec1[l], U->u[l].p, cb, 0, U->s[l].p, U->ch[l], 0, U->b[l].p, gl, s));
    OM_TRY(conv_forward(U, U->dec2[l], U->b[l].p, U->ch[l], 0, nullptr, 0, 0, U->h[l].p, gl, s));
  }
  const bf16* top = L > 1 ? U->h[0].p : U->s[0].p;
  head_fwd<<<blocks(g.voxels()), kT, 0, s>>>(top, U->ch[0], U->w + U->head_w, U->w + U->head_b, U->out_ch,
                                                         g.voxels(), U->out.p);
  OM_CUDA(cudaGetLastError());
  return OM_OK;
}

// gradients of the masked MSE w.r.t. every parameter, into U->g
om_status backward(om_unet* U, const float* t, const uint8_t* mk, const Grid& g, double* loss_out, cudaStream_t s) {
  const int L = U->L;
  const int64_t V = g.voxels();
  OM_CUDA(cudaMemsetAsync(U->g, 0, sizeof(float) * U->nparam, s));
  OM_TRY(U->loss.ensure(2));
  OM_CUDA(cudaMemsetAsync(U->loss.p, 0, 2 * sizeof(double), s));
  // masked mean over pore voxels and output channels: the count in loss[1]
  mask_count<<<std::min<unsigned>(blocks(V), 1216), kT, 0, s>>>(mk, V, U->loss.p + 1);
  mse_grad<<<std::min<unsigned>(blocks(V * U->out_ch), 1216), kT, 0, s>>>(U->out.p, t, mk, U->out_ch, V, U->loss.p + 1,
                                                                           U->dout.p, U->loss.p);
  OM_TRY(refresh_operands(U, false, s));
  const int c0 = U->ch[0];
  const bf16* top = L > 1 ? U->h[0].p : U->s[0].p;
  const bool head_fused = U->out_ch <= kHeadOut;
  if (!head_fused)
    for (int o0 = 0; o0 < U->out_ch; o0 += 4)
      head_bwd_dw<<<1216, kT, 8 * kT * sizeof(float), s>>>(top, U->dout.p, c0, U->out_ch, o0, V, U->g + U->head_w,
                                                           U->g + U->head_b);
  // pre-activation gradient of the activation y (N channels) of conv c, and c's bias gradient
  auto grad_args = [&](const Conv& c, const bf16* y, const Grid& gl, bf16* out) {
    GradArgs a{};
    a.y = y, a.N = c.cout, a.V = (uint32_t)gl.voxels(), a.out = out, a.db = U->g + c.b_off;
    return a;
  };
  auto rows_grad = [&](const Conv& c, const bf16* g, const bf16* y, const Grid& gl, bf16* out) {
    GradArgs a = grad_args(c, y, gl, out);
    a.g = g, a.ldg = c.cout, a.og = 0;
    return launch_relu_grad(kGradRows, a, s);
  };
  auto head_grad = [&](const Conv& c, bf16* out) {
    GradArgs a = grad_args(c, top, g, out);
    a.dy = U->dout.p, a.w = U->w + U->head_w, a.O = U->out_ch;
    if (head_fused) a.dw = U->g + U->head_w, a.dhb = U->g + U->head_b;
    return launch_relu_grad(kGradHead, a, s);
  };
  // decoder, top level down: d1[l] holds the gradient of the level's output h_l
  for (int l = 0; l + 1 < L; ++l) {
    const Grid gl = level_grid(g, l);
    const int c = U->ch[l], cb = U->ch[l + 1];
    // h_l = relu(conv(b_l))
    if (l == 0) OM_TRY(head_grad(U->dec2[l], U->d2[l].p));
    else OM_TRY(rows_grad(U->dec2[l], U->d1[l].p, U->h[l].p, gl, U->d2[l].p));
    OM_TRY(conv_wgrad(U, U->dec2[l], U->b[l].p, c, 0, nullptr, 0, 0, U->d2[l].p, gl, s));
    OM_TRY(conv_dgrad(U, U->dec2[l], U->d2[l].p, U->d1[l].p, gl, s));
    // b_l = relu(conv(concat(u_l, s_l)))
    OM_TRY(rows_grad(U->dec1[l], U->d1[l].p, U->b[l].p, gl, U->d2[l].p));
    OM_TRY(conv_wgrad(U, U->dec1[l], U->u[l].p, cb, 0, U->s[l].p, c, 0, U->d2[l].p, gl, s));
    OM_TRY(conv_dgrad(U, U->dec1[l], U->d2[l].p, U->dcat[l].p, gl, s));
    // u_l = up(h_{l+1}) (or s_{L-1} at the bottom): gradient of the level below
    upsample2_bwd<<<row_blocks(level_grid(g, l + 1)), kT, 0, s>>>(U->dcat[l].p, cb + c, 0, gl, cb, U->d1[l + 1].p);
  }
  // encoder, bottom level up
  for (int l = L - 1; l >= 0; --l) {
    const Grid gl = level_grid(g, l);
    const int c = U->ch[l];
    const int cin = l == 0 ? 16 : U->ch[l - 1];
    // s_l = relu(conv(a_l)) receives: from the level below (pooling) and from the decoder's skip
    if (L == 1) {
      OM_TRY(head_grad(U->enc2[l], U->d1[l].p));
    } else if (l == L - 1) {
      OM_TRY(rows_grad(U->enc2[l], U->d1[l].p, U->s[l].p, gl, U->ds[l].p));
    } else {
      GradArgs a = grad_args(U->enc2[l], U->s[l].p, gl, U->ds[l].p);
      a.g = U->dcat[l].p, a.ldg = U->ch[l + 1] + c, a.og = U->ch[l + 1];
      a.coarse = U->d2[l + 1].p, a.gf = gl;
      OM_TRY(launch_relu_grad(kGradSkip, a, s));
    }
    const bf16* dp = L == 1 ? U->d1[l].p : U->ds[l].p;
    OM_TRY(conv_wgrad(U, U->enc2[l], U->a[l].p, c, 0, nullptr, 0, 0, dp, gl, s));
    OM_TRY(conv_dgrad(U, U->enc2[l], dp, U->d2[l].p, gl, s));
    // a_l = relu(conv(in_l))
    OM_TRY(rows_grad(U->enc1[l], U->d2[l].p, U->a[l].p, gl, U->d1[l].p));
    const bf16* in = l == 0 ? U->x0.p : U->in[l].p;
    OM_TRY(conv_wgrad(U, U->enc1[l], in, cin, 0, nullptr, 0, 0, U->d1[l].p, gl, s));
    // d2[l] = gradient of in_l (pooled s_{l-1}); not needed at the input
    if (l > 0) OM_TRY(conv_dgrad(U, U->enc1[l], U->d1[l].p, U->d2[l].p, gl, s));
  }
  double h = 0.0;
  OM_CUDA(cudaMemcpyAsync(&h, U->loss.p, sizeof(double), cudaMemcpyDeviceToHost, s));
  OM_TRY(check_tc(U, s));
  if (loss_out) *loss_out = h;
  return OM_OK;
}

uint64_t splitmix(uint64_t& st) {
  st += 0x9E3779B97F4A7C15ULL;
  uint64_t z = st;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
  return z ^ (z >> 31);
}

om_status check_grid(const om_unet* U, const Grid& g) {
  const int q = 1 << (U->L - 1);
  if (g.B <= 0 || g.D <= 0 || g.H <= 0 || g.W <= 0 || g.D % q || g.H % q || g.W % q)
    return fail(OM_EINVAL, "U-Net: box edges must be positive multiples of 2^(levels-1)");
  return OM_OK;
}

}  // namespace

extern "C" om_status om_unet_destroy(om_unet* U) {
  if (!U) return OM_OK;
  auto drop = [](std::vector<Buf<bf16>>& v) {
    for (auto& b : v) b.release();
  };
  drop(U->in), drop(U->a), drop(U->s), drop(U->u), drop(U->b), drop(U->h);
  drop(U->d1), drop(U->d2), drop(U->dcat), drop(U->ds);
  U->x0.release(), U->out.release(), U->dout.release(), U->loss.release(), U->tc_err.release();
  for (auto* v : {&U->enc1, &U->enc2, &U->dec1, &U->dec2})
    for (auto& c : *v) {
      cudaFree(c.wt);
      cudaFree(c.wd);
    }
  cudaFree(U->w), cudaFree(U->g), cudaFree(U->m), cudaFree(U->v);
  delete U;
  return OM_OK;
}

extern "C" om_status om_unet_create(int32_t in_ch, int32_t out_ch, int32_t levels, const int32_t* ch, uint64_t seed,
                                    om_unet** out) {
  if (!out || !ch || in_ch < 1 || in_ch > 16 || out_ch < 1 || levels < 1 || levels > 6)
    return fail(OM_EINVAL, "om_unet_create: 1..16 inputs, >= 1 output, 1..6 levels");
  for (int l = 0; l < levels; ++l)
    if (ch[l] < 16 || ch[l] % 16 || ch[l] > 256) return fail(OM_EINVAL, "om_unet_create: channels must be multiples of 16 up to 256");
  om_unet* U = new om_unet();
  U->in_ch = in_ch, U->out_ch = out_ch, U->L = levels;
  U->ch.assign(ch, ch + levels);
  int64_t off = 0;
  auto add = [&](int c1, int c2, int co) {
    Conv c;
    c.cin1 = c1, c.cin2 = c2, c.cout = co;
    c.w_off = off;
    off += 27LL * (c1 + c2) * co;
    c.b_off = off;
    off += co;
    return c;
  };
  for (int l = 0; l < levels; ++l) {
    U->enc1.push_back(add(l == 0 ? 16 : ch[l - 1], 0, ch[l]));
    U->enc2.push_back(add(ch[l], 0, ch[l]));
  }
  U->dec1.resize(std::max(0, levels - 1));
  U->dec2.resize(std::max(0, levels - 1));
  for (int l = levels - 2; l >= 0; --l) {
    U->dec1[l] = add(ch[l + 1], ch[l], ch[l]);
    U->dec2[l] = add(ch[l], 0, ch[l]);
  }
  U->head_w = off;
  off += (int64_t)ch[0] * out_ch;
  U->head_b = off;
  off += out_ch;
  U->nparam = off;
  const int L = levels;
  U->in.resize(L), U->a.resize(L), U->s.resize(L), U->u.resize(L), U->b.resize(L), U->h.resize(L);
  U->d1.resize(L), U->d2.resize(L), U->dcat.resize(L), U->ds.resize(L);
  // He-uniform initial weights from a SplitMix64 stream, zero biases
  std::vector<float> w((size_t)off, 0.f);
  uint64_t st = seed;
  auto init = [&](const Conv& c, int fan_in) {
    const double bound = std::sqrt(6.0 / fan_in);
    for (int64_t i = 0; i < 27LL * (c.cin1 + c.cin2) * c.cout; ++i)
      w[(size_t)(c.w_off + i)] = (float)(bound * (2.0 * ((double)(splitmix(st) >> 11) * 0x1.0p-53) - 1.0));
  };
  for (int l = 0; l < L; ++l) {
    init(U->enc1[l], 27 * (l == 0 ? in_ch : ch[l - 1]));
    init(U->enc2[l], 27 * ch[l]);
  }
  for (int l = L - 2; l >= 0; --l) {
    init(U->dec1[l], 27 * (ch[l + 1] + ch[l]));
    init(U->dec2[l], 27 * ch[l]);
  }
  // the 1x1 head starts at zero: the network's first output is 0 (the cold
  // start) and the first Adam steps cannot blow the decoder's ReLUs up (with
  // a He-initialised head the first outputs are O(10) and training stalls
  // in a state that predicts a constant)
  auto dal = [&](void** p, size_t bytes) -> bool {
    if (cudaMalloc(p, std::max<size_t>(bytes, 16)) != cudaSuccess) {
      (void)cudaGetLastError();
      *p = nullptr;
      return false;
    }
    return true;
  };
  bool ok = dal((void**)&U->w, sizeof(float) * off) && dal((void**)&U->g, sizeof(float) * off) &&
            dal((void**)&U->m, sizeof(float) * off) && dal((void**)&U->v, sizeof(float) * off);
  for (auto* v : {&U->enc1, &U->enc2, &U->dec1, &U->dec2})
    for (auto& c : *v) {
      const size_t n = 27ull * (c.cin1 + c.cin2) * c.cout;
      ok = ok && dal((void**)&c.wt, n * sizeof(bf16)) && dal((void**)&c.wd, n * sizeof(bf16));
    }
  ok = ok && U->tc_err.ensure(1) == OM_OK;
  if (!ok) {
    om_unet_destroy(U);
    return fail(OM_ENOMEM, "om_unet_create: device allocation failed");
  }
  if (cudaMemcpy(U->w, w.data(), sizeof(float) * off, cudaMemcpyHostToDevice) != cudaSuccess ||
      cudaMemset(U->tc_err.p, 0, sizeof(int)) != cudaSuccess ||
      cudaMemset(U->m, 0, sizeof(float) * off) != cudaSuccess || cudaMemset(U->v, 0, sizeof(float) * off) != cudaSuccess) {
    om_unet_destroy(U);
    return fail(OM_ECUDA, "om_unet_create: initialisation failed");
  }
  *out = U;
  return OM_OK;
}

extern "C" om_status om_unet_param_count(const om_unet* U, int64_t* n) {
  if (!U || !n) return fail(OM_EINVAL, "om_unet_param_count: null pointer");
  *n = U->nparam;
  return OM_OK;
}

extern "C" om_status om_unet_get_params(const om_unet* U, float* dst_dev, void* stream) {
  if (!U || !dst_dev) return fail(OM_EINVAL, "om_unet_get_params: null pointer");
  OM_CUDA(cudaMemcpyAsync(dst_dev, U->w, sizeof(float) * U->nparam, cudaMemcpyDeviceToDevice, as_stream(stream)));
  return OM_OK;
}

extern "C" om_status om_unet_set_params(om_unet* U, const float* src_dev, void* stream) {
  if (!U || !src_dev) return fail(OM_EINVAL, "om_unet_set_params: null pointer");
  U->wt_ready = U->wd_ready = false;
  OM_CUDA(cudaMemcpyAsync(U->w, src_dev, sizeof(float) * U->nparam, cudaMemcpyDeviceToDevice, as_stream(stream)));
  return OM_OK;
}

extern "C" om_status om_unet_get_grads(const om_unet* U, float* dst_dev, void* stream) {
  if (!U || !dst_dev) return fail(OM_EINVAL, "om_unet_get_grads: null pointer");
  OM_CUDA(cudaMemcpyAsync(dst_dev, U->g, sizeof(float) * U->nparam, cudaMemcpyDeviceToDevice, as_stream(stream)));
  return OM_OK;
}

extern "C" om_status om_unet_forward(om_unet* U, const float* x, int32_t B, int32_t D, int32_t H, int32_t W, float* y,
                                     void* stream) {
  if (!U || !x || !y) return fail(OM_EINVAL, "om_unet_forward: null pointer");
  const Grid g{B, D, H, W};
  OM_TRY(check_grid(U, g));
  cudaStream_t s = as_stream(stream);
  auto go = [&]() -> om_status {
    OM_TRY(forward(U, x, g, s));
    OM_CUDA(cudaMemcpyAsync(y, U->out.p, sizeof(float) * g.voxels() * U->out_ch, cudaMemcpyDeviceToDevice, s));
    return check_tc(U, s);
  };
  const om_status st = go();
  if (st != OM_OK) U->wt_ready = U->wd_ready = false;  // whatever was enqueued is not waited for
  return st;
}

extern "C" om_status om_unet_backward(om_unet* U, const float* x, const float* t, const uint8_t* m, int32_t B,
                                      int32_t D, int32_t H, int32_t W, double* loss_out, void* stream) {
  if (!U || !x || !t || !m) return fail(OM_EINVAL, "om_unet_backward: null pointer");
  const Grid g{B, D, H, W};
  OM_TRY(check_grid(U, g));
  cudaStream_t s = as_stream(stream);
  om_status st = forward(U, x, g, s);
  if (st == OM_OK) st = backward(U, t, m, g, loss_out, s);
  if (st != OM_OK) U->wt_ready = U->wd_ready = false;  // whatever was enqueued is not waited for
  return st;
}

namespace om {
namespace nn {
__global__ void pack_structure(const uint8_t* mask, const float* d, int64_t n, float ds, float* x) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
    x[2 * v] = mask[v] ? 1.f : 0.f;
    x[2 * v + 1] = d[v] * ds;
  }
}

__global__ void pack_structure3(const uint8_t* mask, const float* d, const float* e, int64_t n, float ds, float* x) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
    x[3 * v] = mask[v] ? 1.f : 0.f;
    x[3 * v + 1] = d[v] * ds;
    x[3 * v + 2] = e[v];
  }
}
}  // namespace nn
}  // namespace om

extern "C" om_status om_unet_pack_structure(const uint8_t* mask_dev, const float* d_nm_dev, int64_t n, double d_scale,
                                           float* x_dev, void* stream) {
  if (!mask_dev || !d_nm_dev || !x_dev || n < 0) return fail(OM_EINVAL, "om_unet_pack_structure: bad argument");
  if (n == 0) return OM_OK;
  om::nn::pack_structure<<<(unsigned)std::min<int64_t>((n + 255) / 256, 1 << 20), 256, 0, as_stream(stream)>>>(
      mask_dev, d_nm_dev, n, (float)d_scale, x_dev);
  OM_CUDA(cudaGetLastError());
  return OM_OK;
}

extern "C" om_status om_unet_pack_structure3(const uint8_t* mask_dev, const float* d_nm_dev, double d_scale,
                                            const float* extra_dev, int64_t n, float* x_dev, void* stream) {
  if (!mask_dev || !d_nm_dev || !extra_dev || !x_dev || n < 0)
    return fail(OM_EINVAL, "om_unet_pack_structure3: bad argument");
  if (n == 0) return OM_OK;
  om::nn::pack_structure3<<<(unsigned)std::min<int64_t>((n + 255) / 256, 1 << 20), 256, 0, as_stream(stream)>>>(
      mask_dev, d_nm_dev, extra_dev, n, (float)d_scale, x_dev);
  OM_CUDA(cudaGetLastError());
  return OM_OK;
}

extern "C" om_status om_unet_train_step(om_unet* U, const float* x, const float* t, const uint8_t* m, int32_t B,
                                        int32_t D, int32_t H, int32_t W, float lr, double* loss_out, void* stream) {
  OM_TRY(om_unet_backward(U, x, t, m, B, D, H, W, loss_out, stream));
  cudaStream_t s = as_stream(stream);
  ++U->step;
  const float b1 = 0.9f, b2 = 0.999f;
  const float bc1 = 1.f - std::pow(b1, (float)U->step), bc2 = 1.f - std::pow(b2, (float)U->step);
  U->wt_ready = U->wd_ready = false;
  adam_step<<<blocks(U->nparam), kT, 0, s>>>(U->w, U->g, U->m, U->v, U->nparam, lr, b1, b2, 1e-8f, bc1, bc2);
  OM_CUDA(cudaGetLastError());
  return OM_OK;
}
