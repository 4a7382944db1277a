// fh_nn.cu -- the learned warm start's 3-D convolutional network: forward,
// backward and Adam, all in hand-written kernels.
//
// Activations are float32 [channels][N0][N1][N2]; weights are kept as float32
// masters for Adam and rounded to bfloat16 (round to nearest even) for every
// product; products accumulate in float32.  Architecture (levels N, N/3,
// N/9, N/27; channels c0..c3; layers 0..10 in parameter order):
//   a0 = leaky(conv0(x))            a1 = leaky(conv1(pool(a0)))
//   a2 = leaky(conv2(pool(a1)))     a3 = leaky(conv3(pool(a2)))
//   v2 = up(leaky(conv4(a3))) + a2  u2 = leaky(conv5(v2))
//   v1 = up(leaky(conv6(u2))) + a1  u1 = leaky(conv7(v1))
//   v0 = up(leaky(conv8(u1))) + a0  u0 = leaky(conv9(v0))
//   y  = conv10(u0)
// conv = 3x3x3 with periodic padding (the unit cell is periodic), pool = mean
// over 3x3x3 blocks, up = nearest-neighbour upsampling by 3.
// All convolutions -- forward, data gradient and weight gradient -- run on the
// tensor cores (fh_conv_planes.cuh: tcgen05, bfloat16 weights, float32
// activations and gradients split into two bfloat16 halves).  The split, the
// pooling, upsampling and skip sums and the leaky ReLU's derivative are one
// pass that writes the operand planes of the next convolution; the forward
// ReLU is the convolution's epilogue.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <string>
#include <vector>

#include "../../include/fh_nn.h"
#include "fh_conv_planes.cuh"

namespace {

constexpr float kSlope = 0.1f;
constexpr int kThreads = 256;

struct Dims {
  int n0, n1, n2;
  __host__ __device__ long long v() const { return (long long)n0 * n1 * n2; }
};

// coarse[c][Z][Y][X] = sum of the fine block (adjoint of nearest upsampling)
__global__ void k_up_bwd(const float* __restrict__ fine, float* __restrict__ coarse, int C, Dims cd) {
  const long long Vc = cd.v();
  const long long n = Vc * C;
  const int f1 = 3 * cd.n1, f2 = 3 * cd.n2;
  const long long Vf = 27 * Vc;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const int c = (int)(i / Vc);
    const long long v = i - (long long)c * Vc;
    const int Z = (int)(v / ((long long)cd.n1 * cd.n2));
    const int rem = (int)(v - (long long)Z * cd.n1 * cd.n2);
    const int Y = rem / cd.n2, X = rem - Y * cd.n2;
    const float* fc = fine + (long long)c * Vf;
    float s = 0.0f;
    for (int a = 0; a < 3; ++a)
      for (int bb = 0; bb < 3; ++bb)
        for (int e = 0; e < 3; ++e) s += fc[((long long)(3 * Z + a) * f1 + 3 * Y + bb) * f2 + 3 * X + e];
    coarse[i] = s;
  }
}

// g = 2 (y - t) / n; per-block partial sums of (y - t)^2 in float64
__global__ void k_mse(const float* __restrict__ y, const float* __restrict__ t, float* __restrict__ g,
                      long long n, double* part) {
  double acc = 0.0;
  const float sc = 2.0f / (float)n;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const float dlt = y[i] - t[i];
    g[i] = sc * dlt;
    acc += (double)dlt * (double)dlt;
  }
  __shared__ double red[kThreads];
  red[threadIdx.x] = acc;
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = red[0];
}

__global__ void k_adam(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                       float* __restrict__ v, long long n, float lr, float b1, float b2, float eps,
                       float c1, float c2) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.0f - b1) * gi;
    const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  }
}

// x[0] = tab0[phase], x[1] = tab1[phase]  (input features from the phase image)
__global__ void k_features(const uint8_t* __restrict__ phase, const float* __restrict__ t0,
                           const float* __restrict__ t1, float* __restrict__ x, long long V) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < V; i += (long long)gridDim.x * blockDim.x) {
    const int p = phase[i];
    x[i] = t0[p];
    x[V + i] = t1[p];
  }
}

// target[b * d + a] = e^(b)_a - delta_ab (+ base[b * d + a] if base)
// (fields: d loads, each [d][V] float64)
__global__ void k_targets(const double* __restrict__ f0, const double* __restrict__ f1,
                          const double* __restrict__ f2, int d, const float* __restrict__ base,
                          float* __restrict__ t, long long V) {
  const double* f[3] = {f0, f1, f2};
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < V; i += (long long)gridDim.x * blockDim.x)
    for (int b = 0; b < d; ++b)
      for (int a = 0; a < d; ++a) {
        const long long k = (long long)(b * d + a) * V + i;
        float v = (float)(f[b][(long long)a * V + i] - (a == b ? 1.0 : 0.0));
        if (base) v += base[k];
        t[k] = v;
      }
}

// g[a] = sum_b E_b (pred[b * d + a] - base[b * d + a])  (fluctuation of load E
// predicted by the network; base = the residual base the network was trained
// against, or null)
__global__ void k_combine(const float* __restrict__ pred, const float* __restrict__ base, int d, double E0,
                          double E1, double E2, double* __restrict__ g, long long V) {
  const double E[3] = {E0, E1, E2};
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < V; i += (long long)gridDim.x * blockDim.x)
    for (int a = 0; a < d; ++a) {
      double s = 0.0;
      for (int b = 0; b < d; ++b) {
        const long long k = (long long)(b * d + a) * V + i;
        s += E[b] * ((double)pred[k] - (base ? (double)base[k] : 0.0));
      }
      g[(long long)a * V + i] = s;
    }
}

// x = E + g  (g already projected)
__global__ void k_add_E(double* __restrict__ x, int d, double E0, double E1, double E2, long long V) {
  const double E[3] = {E0, E1, E2};
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < (long long)d * V; i += (long long)gridDim.x * blockDim.x)
    x[i] += E[i / V];
}

// e[a][i] = delta_ab: the constant unit load b
template <typename T>
__global__ void k_unit_load(T* __restrict__ e, int b, int d, long long V) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < (long long)d * V; i += (long long)gridDim.x * blockDim.x)
    e[i] = (i / V == b) ? T(1) : T(0);
}

// x[a][i] = y[a][i] - delta_ab  (B e_b from y = (I + B) e_b), as float32
template <typename T>
__global__ void k_response(const T* __restrict__ y, int b, int d, float* __restrict__ x, long long V) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < (long long)d * V; i += (long long)gridDim.x * blockDim.x)
    x[i] = (float)(y[i] - ((i / V == b) ? T(1) : T(0)));
}

int grid1(long long n) {
  const long long g = (n + kThreads - 1) / kThreads;
  return (int)(g < 4096 ? (g < 1 ? 1 : g) : 4096);
}

}  // namespace

constexpr int kLayers = 11;
constexpr int kStaticSmem = 10 * 1024;  // at least the convolution kernels' static shared memory

using fh::tc::PlaneGeom;

struct fh_nn {
  Dims lv[4];
  PlaneGeom pg[4];                             // padded grids of the levels
  int cin = 0, cout = 0;
  int ch[4] = {16, 32, 48, 64};
  int lo[kLayers], li[kLayers], ll[kLayers];  // layer out / in channels, level
  long long woff[kLayers], boff[kLayers];      // offsets in the flat parameter vector
  long long nparam = 0;
  cudaStream_t st = nullptr;
  int sms = 0;
  size_t smem_cap = 0;
  float *P = nullptr, *G = nullptr, *Mo = nullptr, *Ve = nullptr;
  __nv_bfloat16* W[2][kLayers] = {};            // operand layouts: forward, data gradient
  int* dev_err = nullptr;                        // bounded waits that expired
  float* wpart[kLayers] = {};                    // weight-gradient partials
  // the weight gradients run beside the chain of data gradients on their own stream
  cudaStream_t side = nullptr;
  cudaEvent_t fork[kLayers] = {}, join = nullptr;
  // act[k]: output of layer k after the leaky ReLU; in[k]: operand planes of
  // its input (kept for the weight gradient); y: output
  float* act[kLayers - 1] = {};
  uint4* in[kLayers] = {};
  float* y = nullptr;
  // backward: gradients, planes with periodic padding (one layer at a time)
  // and with zero padding (per layer: the padding stays zero)
  float *gy = nullptr, *gu[3] = {}, *gv[3] = {}, *ga3 = nullptr, *gp[3] = {}, *gt = nullptr;
  uint4 *GA = nullptr, *GB[kLayers] = {};
  double* part = nullptr;
  double* h_part = nullptr;                      // pinned: loss partials, error word
  int npart = 0;
  void* slab = nullptr;                          // the one allocation behind all of it
  long long launches = 0;
};

namespace {

struct ConvShape {
  int T, sy, rows, tiles_z, grid, resident, cps, nstage;
  size_t smem;
};

// Compiled (T, NT): two accumulators of T NT columns per CTA.
#define FH_FOR_EACH_CONV(X) \
  X(4, 16) X(2, 16) X(1, 16) X(4, 32) X(2, 32) X(1, 32) X(4, 48) X(2, 48) X(1, 48) X(4, 64) X(2, 64) X(1, 64)

// Tile of a convolution: as many 128-voxel MMA tiles per CTA tile (4, 2, 1) as
// still give every SM a tile -- longer tiles copy their neighbouring rows less
// often -- with all chunks of channels in one stage where they fit and the
// weights beside them, and two stages where those fit.
ConvShape conv_shape(const fh_nn* n, const PlaneGeom& g, int chunks, int NT) {
  for (int cps : {chunks, 1})
    for (int nstage : {2, 1})
      for (int T : {4, 2, 1})
        for (int resident : {1, 0}) {
          if (!resident && cps > 1) continue;
          ConvShape c{};
          c.T = T;
          c.cps = cps;
          c.nstage = nstage;
          c.resident = resident;
          c.rows = std::min(128 * T, g.n1 * g.px);
          c.sy = std::min(g.px, c.rows + 2);
          c.tiles_z = (g.n1 * g.px + 128 * T - 1) / (128 * T);
          const long long tiles = (long long)c.tiles_z * g.n0;
          c.grid = (int)std::min<long long>(tiles, n->sms);
          c.smem = fh::tc::conv_smem(T, c.sy, c.rows, NT, chunks, resident != 0, cps, nstage);
          if (c.smem <= n->smem_cap && (tiles >= n->sms || T == 1)) return c;
        }
  return ConvShape{};
}

// y = leaky(conv(x; W) + b), or the data gradient gx = conv(gy; W^T, taps
// reversed) of layer k; slope 1: no ReLU
cudaError_t conv(fh_nn* n, int k, const uint4* planes, float* out, bool trans, float slope) {
  const PlaneGeom& g = n->pg[n->ll[k]];
  fh::tc::ConvPlanesArgs a;
  a.g = g;
  a.x = planes;
  a.nblk = fh::tc::chan_blocks(trans ? n->lo[k] : n->li[k]);
  a.w = n->W[trans][k];
  a.O = trans ? n->li[k] : n->lo[k];
  const int NT = (a.O + 15) / 16 * 16;
  a.y = out;
  a.b = trans ? nullptr : n->P + n->boff[k];
  a.slope = slope;
  const ConvShape c = conv_shape(n, g, a.nblk / 2, NT);
  a.sy = c.sy;
  a.rows = c.rows;
  a.tiles_z = c.tiles_z;
  a.resident = c.resident;
  a.cps = c.cps;
  a.nstage = c.nstage;
  a.err = n->dev_err;
  a.wait_ns = fh::tma::wait_limit_ns();
  ++n->launches;
#define FH_CONV(TT, NN) \
  if (c.T == TT && NT == NN) fh::tc::k_conv_planes<TT, NN><<<c.grid, fh::tc::kConvThreads, c.smem, n->st>>>(a);
  FH_FOR_EACH_CONV(FH_CONV)
#undef FH_CONV
  return cudaGetLastError();
}

template <int MODE>
cudaError_t split(fh_nn* n, int level, int C, const float* src, uint4* out, const float* coarse = nullptr,
                  const float* act = nullptr, uint4* out0 = nullptr) {
  fh::tc::SplitArgs a;
  a.g = n->pg[level];
  a.C = C;
  a.src = src;
  a.coarse = coarse;
  a.act = act;
  a.out = out;
  a.out0 = out0;
  a.slope = kSlope;
  const long long pv = (long long)(a.g.n0 + 2) * a.g.py * a.g.px;
  const dim3 grid((unsigned)std::min<long long>((pv + 255) / 256, 65535), fh::tc::chan_blocks(C));
  ++n->launches;
  fh::tc::k_split<MODE><<<grid, 256, 0, n->st>>>(a);
  return cudaGetLastError();
}

// CTAs of a layer's weight gradient along the voxels: one per SM and
// (16-channel chunk, 16 outputs), at most one per voxel tile
int wgrad_slices(const fh_nn* n, int k) {
  const PlaneGeom& g = n->pg[n->ll[k]];
  const int per = fh::tc::chan_blocks(n->li[k]) / 2 * (fh::tc::chan_blocks(n->lo[k]) / 2);
  return (int)std::max<long long>(1, std::min<long long>(n->sms / per, g.v() / fh::tc::kWgK + 1));
}

cudaError_t wgrad(fh_nn* n, int k) {
  const PlaneGeom& g = n->pg[n->ll[k]];
  fh::tc::WgradArgs a;
  a.g = g;
  a.x = n->in[k];
  a.nblk = fh::tc::chan_blocks(n->li[k]);
  a.gy = n->GB[k];
  a.oblk = fh::tc::chan_blocks(n->lo[k]);
  a.O = n->lo[k];
  a.C = n->li[k];
  a.slices = wgrad_slices(n, k);
  a.sy = std::min(g.px, fh::tc::kWgK);
  a.vox = (long long)(g.n0 - 1) * g.py * g.px + (long long)(g.n1 - 1) * g.px + g.n2 + 2;
  a.part = n->wpart[k];
  a.err = n->dev_err;
  a.wait_ns = fh::tma::wait_limit_ns();
  const int chunks = a.nblk / 2;
  ++n->launches;
  cudaError_t e = cudaEventRecord(n->fork[k], n->st);  // GB[k] is written
  if (e == cudaSuccess) e = cudaStreamWaitEvent(n->side, n->fork[k], 0);
  if (e != cudaSuccess) return e;
  fh::tc::k_wgrad_planes<16><<<dim3(a.slices, chunks, a.oblk / 2), fh::tc::kWgThreads, fh::tc::wg_smem(a.sy, 16), n->side>>>(a);
  return cudaGetLastError();
}

// Every layer's weight gradient from its partials; n->st waits for them.
cudaError_t wgrad_finish(fh_nn* n) {
  fh::tc::WgradSumArgs a;
  for (int k = 0; k < kLayers; ++k) {
    a.part[k] = n->wpart[k];
    a.gW[k] = n->G + n->woff[k];
    a.gb[k] = n->G + n->boff[k];
    a.O[k] = n->lo[k];
    a.C[k] = n->li[k];
    a.slices[k] = wgrad_slices(n, k);
  }
  ++n->launches;
  fh::tc::k_wgrad_sum<<<dim3(64, kLayers), 128, 0, n->side>>>(a);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaEventRecord(n->join, n->side);
  return e == cudaSuccess ? cudaStreamWaitEvent(n->st, n->join, 0) : e;
}

void up_bwd(fh_nn* n, const float* f, float* c, int C, Dims cd) {
  ++n->launches;
  k_up_bwd<<<grid1(cd.v() * C), kThreads, 0, n->st>>>(f, c, C, cd);
}

// decoder level l: (up convolution, post convolution) layer indices
constexpr int kUp[3] = {8, 6, 4};
constexpr int kPost[3] = {9, 7, 5};

#define FH_NN(call)                                  \
  do {                                               \
    const cudaError_t e_ = (call);                   \
    if (e_ != cudaSuccess) return e_;                \
  } while (0)

// y = net(x), both [channels][V] on the device
cudaError_t forward(fh_nn* n, const float* x, float* y) {
  using namespace fh::tc;
  WeightArgs wa;
  for (int k = 0; k < kLayers; ++k) {
    wa.w[k] = n->P + n->woff[k];
    wa.out[0][k] = n->W[0][k];
    wa.out[1][k] = n->W[1][k];
    wa.O[k] = n->lo[k];
    wa.C[k] = n->li[k];
  }
  ++n->launches;
  k_weight_planes<<<dim3(32, 2 * kLayers), kThreads, 0, n->st>>>(wa);
  FH_NN(cudaGetLastError());
  FH_NN(split<kSplitPlain>(n, 0, n->cin, x, n->in[0]));
  FH_NN(conv(n, 0, n->in[0], n->act[0], false, kSlope));
  for (int l = 1; l < 4; ++l) {
    FH_NN(split<kSplitPool>(n, l, n->ch[l - 1], n->act[l - 1], n->in[l]));
    FH_NN(conv(n, l, n->in[l], n->act[l], false, kSlope));
  }
  const float* cur = n->act[3];
  for (int l = 2; l >= 0; --l) {
    const int ku = kUp[l], kp = kPost[l];
    // v_l = up(leaky(conv_ku(cur))) + a_l ; u_l = leaky(conv_kp(v_l))
    FH_NN(split<kSplitPlain>(n, l + 1, n->li[ku], cur, n->in[ku]));
    FH_NN(conv(n, ku, n->in[ku], n->act[ku], false, kSlope));
    FH_NN(split<kSplitUp>(n, l, n->ch[l], n->act[l], n->in[kp], n->act[ku]));
    FH_NN(conv(n, kp, n->in[kp], n->act[kp], false, kSlope));
    cur = n->act[kp];
  }
  FH_NN(split<kSplitPlain>(n, 0, n->ch[0], cur, n->in[10]));
  return conv(n, 10, n->in[10], y, false, 1.0f);
}

// gradients of sum(gy * y) (gy already in n->gy)
cudaError_t backward(fh_nn* n) {
  using namespace fh::tc;
  FH_NN(split<kSplitPlain>(n, 0, n->cout, n->gy, n->GA, nullptr, nullptr, n->GB[10]));
  FH_NN(wgrad(n, 10));
  FH_NN(conv(n, 10, n->GA, n->gu[0], true, 1.0f));               // g_u0
  for (int l = 0; l < 3; ++l) {
    const int ku = kUp[l], kp = kPost[l];
    FH_NN(split<kSplitGrad>(n, l, n->ch[l], n->gu[l], n->GA, nullptr, n->act[kp], n->GB[kp]));  // g_z(post)
    FH_NN(wgrad(n, kp));
    FH_NN(conv(n, kp, n->GA, n->gv[l], true, 1.0f));              // g_v_l (= skip part of g_a_l)
    up_bwd(n, n->gv[l], n->gt, n->ch[l], n->lv[l + 1]);           // c_l at level l+1
    FH_NN(split<kSplitGrad>(n, l + 1, n->ch[l], n->gt, n->GA, nullptr, n->act[ku], n->GB[ku]));  // g_z(up)
    FH_NN(wgrad(n, ku));
    FH_NN(conv(n, ku, n->GA, l < 2 ? n->gu[l + 1] : n->ga3, true, 1.0f));  // g_u_{l+1} (or g_a3)
  }
  // encoder: g_a3 in ga3; g_a_l = g_v_l + poolT(g_p_l)
  for (int l = 3; l >= 1; --l) {
    if (l == 3)
      FH_NN(split<kSplitGrad>(n, 3, n->ch[3], n->ga3, n->GA, nullptr, n->act[3], n->GB[3]));
    else
      FH_NN(split<kSplitGradUp>(n, l, n->ch[l], n->gv[l], n->GA, n->gp[l], n->act[l], n->GB[l]));
    FH_NN(wgrad(n, l));
    FH_NN(conv(n, l, n->GA, n->gp[l - 1], true, 1.0f));           // g_p_{l-1}
  }
  FH_NN(split<kSplitGradUp>(n, 0, n->ch[0], n->gv[0], nullptr, n->gp[0], n->act[0], n->GB[0]));
  FH_NN(wgrad(n, 0));
  return wgrad_finish(n);
}
#undef FH_NN

// gy = gradient of the mean squared error of y, partial sums of the loss in part
cudaError_t loss_gradient(fh_nn* n, const float* target) {
  const long long cnt = n->lv[0].v() * n->cout;
  ++n->launches;
  k_mse<<<std::min(n->npart, grid1(cnt)), kThreads, 0, n->st>>>(n->y, target, n->gy, cnt, n->part);
  return cudaGetLastError();
}

// Waits for what is queued, reads the loss, the gradient (into grad_host, if
// any) and the device error word (bounded waits that expired, in this call or an
// earlier forward); a word that was set is reported once and cleared.
int finish(fh_nn* n, double* loss, float* grad_host) {
  const long long cnt = n->lv[0].v() * n->cout;
  const int g = std::min(n->npart, grid1(cnt));
  int* const h_err = reinterpret_cast<int*>(n->h_part + n->npart);
  if (cudaMemcpyAsync(n->h_part, n->part, g * sizeof(double), cudaMemcpyDeviceToHost, n->st) != cudaSuccess ||
      cudaMemcpyAsync(h_err, n->dev_err, sizeof(int), cudaMemcpyDeviceToHost, n->st) != cudaSuccess ||
      (grad_host && cudaMemcpyAsync(grad_host, n->G, n->nparam * sizeof(float), cudaMemcpyDeviceToHost, n->st) != cudaSuccess) ||
      cudaStreamSynchronize(n->st) != cudaSuccess)
    return FH_ERR_CUDA;
  if (*h_err != 0)
    return cudaMemsetAsync(n->dev_err, 0, sizeof(int), n->st) == cudaSuccess ? FH_ERR_TIMEOUT : FH_ERR_CUDA;
  double s = 0.0;
  for (int i = 0; i < g; ++i) s += n->h_part[i];
  if (loss) *loss = s / (double)cnt;
  return 0;
}

}  // namespace

extern "C" {

void fh_nn_destroy(fh_nn* n) {
  if (!n) return;
  if (n->st) cudaStreamSynchronize(n->st);
  if (n->side) cudaStreamSynchronize(n->side);
  if (n->slab) cudaFree(n->slab);
  for (cudaEvent_t e : n->fork)
    if (e) cudaEventDestroy(e);
  if (n->join) cudaEventDestroy(n->join);
  if (n->side) cudaStreamDestroy(n->side);
  if (n->h_part) cudaFreeHost(n->h_part);
  delete n;
}

fh_status fh_nn_create(fh_nn** out, const int* N, int cin, int cout, const int* channels, void* stream) {
  if (!out || !N || cin < 1 || cout < 1) return FH_ERR_ARG;
  *out = nullptr;
  for (int a = 0; a < 3; ++a)
    if (N[a] < 27 || N[a] % 27) return FH_ERR_ARG;
  fh_nn* n = new (std::nothrow) fh_nn();
  if (!n) return FH_ERR_OOM;
  n->cin = cin;
  n->cout = cout;
  if (channels)
    for (int k = 0; k < 4; ++k) {
      if (channels[k] < 1) {
        delete n;
        return FH_ERR_ARG;
      }
      n->ch[k] = channels[k];
    }
  for (int l = 0; l < 4; ++l) {
    int f = 1;
    for (int k = 0; k < l; ++k) f *= 3;
    n->lv[l] = Dims{N[0] / f, N[1] / f, N[2] / f};
  }
  const int c0 = n->ch[0], c1 = n->ch[1], c2 = n->ch[2], c3 = n->ch[3];
  const int io[kLayers][3] = {{cin, c0, 0}, {c0, c1, 1}, {c1, c2, 2}, {c2, c3, 3},
                              {c3, c2, 3},  {c2, c2, 2}, {c2, c1, 2}, {c1, c1, 1},
                              {c1, c0, 1},  {c0, c0, 0}, {c0, cout, 0}};
  long long off = 0;
  for (int k = 0; k < kLayers; ++k) {
    n->li[k] = io[k][0];
    n->lo[k] = io[k][1];
    n->ll[k] = io[k][2];
    n->woff[k] = off;
    off += (long long)n->lo[k] * n->li[k] * 27;
    n->boff[k] = off;
    off += n->lo[k];
  }
  n->nparam = off;
  for (int k = 0; k < kLayers; ++k)
    if (n->lo[k] > fh::tc::kNmax || n->li[k] > fh::tc::kNmax) {
      delete n;
      return FH_ERR_ARG;  // more than 64 channels on one side of a layer
    }
  for (int l = 0; l < 4; ++l) n->pg[l] = fh::tc::plane_geom(n->lv[l].n0, n->lv[l].n1, n->lv[l].n2);
  n->st = (cudaStream_t)stream;
  int dev = 0, optin = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&n->sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess ||
#define FH_CONV(TT, NN)                                                                          \
  cudaFuncSetAttribute(fh::tc::k_conv_planes<TT, NN>, cudaFuncAttributeMaxDynamicSharedMemorySize, \
                       optin - kStaticSmem) != cudaSuccess ||
      FH_FOR_EACH_CONV(FH_CONV)
#undef FH_CONV
      cudaFuncSetAttribute(fh::tc::k_wgrad_planes<16>, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - kStaticSmem) !=
          cudaSuccess) {
    delete n;
    return FH_ERR_CUDA;
  }
  n->smem_cap = (size_t)optin - kStaticSmem;
  const long long V[4] = {n->lv[0].v(), n->lv[1].v(), n->lv[2].v(), n->lv[3].v()};
  long long coarse_max = 0;  // largest c_l * |level l+1|
  for (int l = 0; l < 3; ++l) coarse_max = std::max(coarse_max, (long long)n->ch[l] * V[l + 1]);
  // one allocation; the operand planes come first (their padding and slack
  // start as zeros, and the zero-padded planes' padding stays zero)
  struct Want {
    void** p;
    size_t bytes;
  };
  std::vector<Want> want;
  size_t total = 0, planes = 0;
  auto need = [&](auto** p, long long count) {
    const size_t bytes = ((size_t)count * sizeof(**p) + 255) / 256 * 256;
    want.push_back({reinterpret_cast<void**>(p), bytes});
    total += bytes;
  };
  long long ga = 0;
  for (int k = 0; k < kLayers; ++k) {
    const PlaneGeom& g = n->pg[n->ll[k]];
    need(&n->in[k], fh::tc::plane_elems(g, n->li[k]));
    need(&n->GB[k], fh::tc::plane_elems(g, n->lo[k]));
    ga = std::max(ga, fh::tc::plane_elems(g, n->lo[k]));
  }
  need(&n->GA, ga);
  planes = total;
  for (int k = 0; k < kLayers; ++k) {
    need(&n->wpart[k], (long long)wgrad_slices(n, k) * (fh::tc::chan_blocks(n->li[k]) / 2) * 9 * 128 *
                           (fh::tc::chan_blocks(n->lo[k]) * 8));
    const int o16 = (n->lo[k] + 15) / 16 * 16, i16 = (n->li[k] + 15) / 16 * 16;
    need(&n->W[0][k], (long long)27 * o16 * i16);
    need(&n->W[1][k], (long long)27 * o16 * i16);
  }
  need(&n->P, off);
  need(&n->G, off);
  need(&n->Mo, off);
  need(&n->Ve, off);
  need(&n->dev_err, 1);
  for (int k = 0; k < kLayers - 1; ++k) need(&n->act[k], V[n->ll[k]] * (long long)n->lo[k]);
  need(&n->y, V[0] * cout);
  need(&n->gy, V[0] * cout);
  for (int k = 0; k < 3; ++k) need(&n->gu[k], V[k] * n->ch[k]);
  for (int k = 0; k < 3; ++k) need(&n->gv[k], V[k] * n->ch[k]);
  need(&n->ga3, V[3] * n->ch[3]);
  for (int k = 0; k < 3; ++k) need(&n->gp[k], V[k + 1] * n->ch[k]);
  need(&n->gt, coarse_max);
  n->npart = 4096;
  need(&n->part, n->npart);
  int rc = cudaMalloc(&n->slab, total) == cudaSuccess ? 0 : FH_ERR_OOM;
  if (!rc) {
    char* q = static_cast<char*>(n->slab);
    for (const Want& w : want) {
      *w.p = q;
      q += w.bytes;
    }
  }
  for (int k = 0; k <= kLayers && !rc; ++k)
    if (cudaEventCreateWithFlags(k < kLayers ? &n->fork[k] : &n->join, cudaEventDisableTiming) != cudaSuccess) rc = FH_ERR_CUDA;
  if (!rc && cudaStreamCreateWithFlags(&n->side, cudaStreamNonBlocking) != cudaSuccess) rc = FH_ERR_CUDA;
  if (!rc && cudaMallocHost(&n->h_part, (n->npart + 1) * sizeof(double)) != cudaSuccess) rc = FH_ERR_OOM;
  if (!rc && (cudaMemsetAsync(n->slab, 0, planes, n->st) != cudaSuccess ||
              cudaMemsetAsync(n->dev_err, 0, sizeof(int), n->st) != cudaSuccess ||
              cudaMemsetAsync(n->Mo, 0, off * sizeof(float), n->st) != cudaSuccess ||
              cudaMemsetAsync(n->Ve, 0, off * sizeof(float), n->st) != cudaSuccess ||
              cudaMemsetAsync(n->P, 0, off * sizeof(float), n->st) != cudaSuccess))
    rc = FH_ERR_CUDA;
  if (rc) {
    fh_nn_destroy(n);
    return FH_ERR_OOM;
  }
  *out = n;
  return FH_OK;
}

long long fh_nn_param_count(const fh_nn* n) { return n ? n->nparam : 0; }

long long fh_nn_launches(const fh_nn* n) { return n ? n->launches : 0; }

fh_status fh_nn_set_params(fh_nn* n, const float* host, long long count) {
  if (!n || !host || count != n->nparam) return FH_ERR_ARG;
  if (cudaMemcpyAsync(n->P, host, count * sizeof(float), cudaMemcpyHostToDevice, n->st) != cudaSuccess ||
      cudaMemsetAsync(n->Mo, 0, count * sizeof(float), n->st) != cudaSuccess ||
      cudaMemsetAsync(n->Ve, 0, count * sizeof(float), n->st) != cudaSuccess ||
      cudaStreamSynchronize(n->st) != cudaSuccess)
    return FH_ERR_CUDA;
  return FH_OK;
}

fh_status fh_nn_get_params(fh_nn* n, float* host, long long count) {
  if (!n || !host || count != n->nparam) return FH_ERR_ARG;
  if (cudaMemcpyAsync(host, n->P, count * sizeof(float), cudaMemcpyDeviceToHost, n->st) != cudaSuccess ||
      cudaStreamSynchronize(n->st) != cudaSuccess)
    return FH_ERR_CUDA;
  return FH_OK;
}

fh_status fh_nn_forward(fh_nn* n, const float* x, float* y) {
  if (!n || !x || !y) return FH_ERR_ARG;
  return forward(n, x, y) == cudaSuccess ? FH_OK : FH_ERR_CUDA;
}

fh_status fh_nn_gradients(fh_nn* n, const float* x, const float* target, double* loss, float* grad_host) {
  if (!n || !x || !target) return FH_ERR_ARG;
  // the error word is read behind the backward pass: its waits are bounded too
  if (forward(n, x, n->y) != cudaSuccess || loss_gradient(n, target) != cudaSuccess || backward(n) != cudaSuccess) {
    cudaStreamSynchronize(n->side);  // weight gradients that were launched read this call's planes
    return FH_ERR_CUDA;
  }
  return (fh_status)finish(n, loss, grad_host);
}

fh_status fh_nn_train_step(fh_nn* n, const float* x, const float* target, float lr, int step, double* loss) {
  if (!n || step < 1 || !(lr > 0.0f)) return FH_ERR_ARG;
  fh_status s = fh_nn_gradients(n, x, target, loss, nullptr);
  if (s != FH_OK) return s;
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = 1.0f - (float)std::pow(0.9, step), c2 = 1.0f - (float)std::pow(0.999, step);
  ++n->launches;
  k_adam<<<grid1(n->nparam), kThreads, 0, n->st>>>(n->P, n->G, n->Mo, n->Ve, n->nparam, lr, b1, b2, 1e-8f, c1, c2);
  return cudaGetLastError() == cudaSuccess ? FH_OK : FH_ERR_CUDA;
}

fh_status fh_nn_features(const uint8_t* phase, int nphase, const double* L, int d, long long nodes,
                         float* x, void* stream) {
  if (!phase || !L || !x || nphase < 1 || nphase > 256 || (d != 2 && d != 3)) return FH_ERR_ARG;
  // channel 0: log10(L_p / L_0) / 4 (isotropic phases, first diagonal entry), channel 1: indicator
  std::vector<float> h(512, 0.0f);
  const double l0 = L[0];
  if (!(l0 > 0.0)) return FH_ERR_NOT_SPD;
  for (int p = 0; p < nphase; ++p) {
    const double lp = L[(size_t)p * d * d];
    if (!(lp > 0.0)) return FH_ERR_NOT_SPD;
    h[p] = (float)(std::log10(lp / l0) / 4.0);
    h[256 + p] = p > 0 ? 1.0f : 0.0f;
  }
  float* dt = nullptr;
  cudaStream_t st = (cudaStream_t)stream;
  if (cudaMallocAsync((void**)&dt, 512 * sizeof(float), st) != cudaSuccess) return FH_ERR_OOM;
  cudaMemcpyAsync(dt, h.data(), 512 * sizeof(float), cudaMemcpyHostToDevice, st);
  k_features<<<grid1(nodes), kThreads, 0, st>>>(phase, dt, dt + 256, x, nodes);
  cudaError_t e = cudaGetLastError();
  cudaFreeAsync(dt, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  return e == cudaSuccess ? FH_OK : FH_ERR_CUDA;
}

fh_status fh_nn_targets(const double* const* fields, int d, long long nodes, const float* base, float* target,
                        void* stream) {
  if (!fields || !target || (d != 2 && d != 3)) return FH_ERR_ARG;
  for (int b = 0; b < d; ++b)
    if (!fields[b]) return FH_ERR_ARG;
  k_targets<<<grid1(nodes), kThreads, 0, (cudaStream_t)stream>>>(fields[0], fields[1], d > 2 ? fields[2] : fields[0], d,
                                                                  base, target, nodes);
  return cudaGetLastError() == cudaSuccess ? FH_OK : FH_ERR_CUDA;
}

}  // extern "C"

namespace {

template <typename T>
fh_status response_features(fh_ctx* ctx, int dtype, int d, long long nodes, float* x) {
  const long long len = (long long)d * nodes;
  T* buf = nullptr;
  if (cudaMalloc((void**)&buf, 2 * len * sizeof(T)) != cudaSuccess) return FH_ERR_OOM;
  fh_status s = FH_OK;
  for (int b = 0; b < d && s == FH_OK; ++b) {
    k_unit_load<T><<<grid1(len), kThreads>>>(buf, b, d, len / d);
    if (cudaGetLastError() != cudaSuccess || cudaDeviceSynchronize() != cudaSuccess) {
      s = FH_ERR_CUDA;
      break;
    }
    s = fh_apply(ctx, buf, buf + len, 0, dtype);
    if (s != FH_OK) break;
    if (cudaDeviceSynchronize() != cudaSuccess) {
      s = FH_ERR_CUDA;
      break;
    }
    k_response<T><<<grid1(len), kThreads>>>(buf + len, b, d, x + (long long)b * len, len / d);
    if (cudaGetLastError() != cudaSuccess) s = FH_ERR_CUDA;
  }
  if (cudaDeviceSynchronize() != cudaSuccess && s == FH_OK) s = FH_ERR_CUDA;
  cudaFree(buf);
  return s;
}

}  // namespace

extern "C" {

fh_status fh_nn_response_features(fh_ctx* ctx, int d, long long nodes, float* x) {
  if (!ctx || !x || (d != 2 && d != 3) || nodes < 1) return FH_ERR_ARG;
  // float32 products where the context has them (the features are float32),
  // else the float64 pipeline
  fh_status s = response_features<float>(ctx, FH_FP32, d, nodes, x);
  if (s == FH_ERR_ARG) s = response_features<double>(ctx, FH_FP64, d, nodes, x);
  return s;
}

fh_status fh_nn_warm_start(fh_ctx* ctx, const float* pred, const float* base, const double* E, int d,
                           long long nodes, double* x0, void* stream) {
  if (!ctx || !pred || !E || !x0 || (d != 2 && d != 3)) return FH_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  k_combine<<<grid1(nodes), kThreads, 0, st>>>(pred, base, d, E[0], E[1], d > 2 ? E[2] : 0.0, x0, nodes);
  if (cudaGetLastError() != cudaSuccess || cudaDeviceSynchronize() != cudaSuccess) return FH_ERR_CUDA;
  fh_status s = fh_project_compatible(ctx, x0, x0);
  if (s != FH_OK) return s;
  if (cudaDeviceSynchronize() != cudaSuccess) return FH_ERR_CUDA;
  k_add_E<<<grid1((long long)d * nodes), kThreads, 0, st>>>(x0, d, E[0], E[1], d > 2 ? E[2] : 0.0, nodes);
  if (cudaGetLastError() != cudaSuccess || cudaStreamSynchronize(st) != cudaSuccess) return FH_ERR_CUDA;
  return FH_OK;
}

}  // extern "C"
