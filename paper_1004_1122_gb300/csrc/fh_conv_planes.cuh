// fh_conv_planes.cuh -- the 3x3x3 periodic convolutions of the warm-start
// network on the fifth-generation tensor cores: forward and data gradient
// (k_conv_planes) and weight gradient (k_wgrad_planes).
//
// Operands.  The weights are bfloat16 (the network's definition); a float32
// activation or gradient is split as x = hi + lo with hi = bf16(x),
// lo = bf16(x - hi), and both halves are multiplied into the same float32
// accumulator, which keeps ~16 mantissa bits of x.
//
// Layout.  A tensor of C channels is stored as planes [half][C / 8][voxel][8]
// of bfloat16 (16 bytes per voxel) over the grid padded by one voxel on every
// side, the padding holding the periodic neighbours.  In the padded, flattened
// voxel index a tap (dz, dy, dx) is the constant shift (dz py + dy) px + dx,
// and 8 consecutive voxels of a plane are one 8-row x 16-byte core matrix of
// the unswizzled operand layout at any 16-byte address.  A tile of consecutive
// flattened voxels therefore needs only the rows around it copied to shared
// memory once (bulk copies, contiguous), and each of the 27 taps is a shared-
// memory descriptor with a shifted start address: nothing is gathered or
// converted per tap.  Flattening costs the padding columns, 2 / (n2 + 2) of
// the rows.
//
// What bounds them: an MMA of 128 voxels x 16 channels takes ~60 cycles here
// for N = 16 as for N = 32 (its 4 KB operand is read from shared memory); a
// 16 -> 16 channel layer at 135^3 is 1.07 M of them, 0.21 ms.  Stacking the
// three taps of a row along N (9 MMAs instead of 27, the epilogue adding
// neighbouring voxels) took 0.19 ms, but three shorter sums round differently
// from one long one (the tensor core's additions do not round to nearest), and
// a gradient then differs by 3e-5 from the one long sum's.  The weight
// gradient does stack three copies of the gradient, shifted by dx, along N.
#pragma once

#include "fh_conv_tc.cuh"

namespace fh {
namespace tc {

// Padded grid of one level.
struct PlaneGeom {
  int n0, n1, n2;
  int py, px;          // n1 + 2, n2 + 2
  long long stride;    // voxels between planes (slack for tiles that run over included)
  __host__ __device__ long long v() const { return (long long)n0 * n1 * n2; }
};
constexpr int kPlaneFront = 8;     // voxels before a plane's first (a tile may start one early)
constexpr int kTileMax = 512;      // most voxels of one tile
inline PlaneGeom plane_geom(int n0, int n1, int n2) {
  PlaneGeom g;
  g.n0 = n0;
  g.n1 = n1;
  g.n2 = n2;
  g.py = n1 + 2;
  g.px = n2 + 2;
  g.stride = (long long)(n0 + 2) * g.py * g.px + kTileMax + 2 * g.px + 64;
  return g;
}
inline int chan_blocks(int c) { return (c + 15) / 16 * 2; }  // blocks of 8 channels, pairs
// uint4 elements of a tensor's planes (both halves)
inline long long plane_elems(const PlaneGeom& g, int c) { return 2 * chan_blocks(c) * g.stride + kPlaneFront; }

// ----------------------------------------------------------------------------
// float32 [C][V] (or a function of it) -> planes
// ----------------------------------------------------------------------------
enum : int {
  kSplitPlain = 0,   // src
  kSplitUp = 1,      // src + up(coarse)
  kSplitPool = 2,    // mean of src's 3 x 3 x 3 blocks (src on the next finer level)
  kSplitGrad = 3,    // src leaky'(act)
  kSplitGradUp = 4   // (src + up(coarse) / 27) leaky'(act)
};
struct SplitArgs {
  PlaneGeom g;         // level of the planes
  int C;
  const float* src;
  const float* coarse;
  const float* act;    // activated values (their sign is the pre-activation's)
  uint4* out;          // planes with periodic padding
  uint4* out0;         // planes with zero padding (interior written only), or nullptr
  float slope;
};

template <int MODE> __global__ void __launch_bounds__(256) k_split(SplitArgs a) {
  const PlaneGeom& g = a.g;
  const int cb = blockIdx.y;
  const long long PV = (long long)(g.n0 + 2) * g.py * g.px, V = g.v();
  const int nblk = gridDim.y;
  for (long long f = blockIdx.x * (long long)blockDim.x + threadIdx.x; f < PV; f += (long long)gridDim.x * blockDim.x) {
    const int row = (int)(f / g.px), xp = (int)(f - (long long)row * g.px);
    const int zp = row / g.py, yp = row - zp * g.py;
    const int z = zp == 0 ? g.n0 - 1 : zp == g.n0 + 1 ? 0 : zp - 1;
    const int y = yp == 0 ? g.n1 - 1 : yp == g.n1 + 1 ? 0 : yp - 1;
    const int x = xp == 0 ? g.n2 - 1 : xp == g.n2 + 1 ? 0 : xp - 1;
    const bool inside = zp > 0 && zp <= g.n0 && yp > 0 && yp <= g.n1 && xp > 0 && xp <= g.n2;
    const long long v = ((long long)z * g.n1 + y) * g.n2 + x;
    const long long vc = (MODE == kSplitUp || MODE == kSplitGradUp)
                             ? ((long long)(z / 3) * (g.n1 / 3) + y / 3) * (g.n2 / 3) + x / 3
                             : 0;
    uint32_t h[4], l[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      float s[2];
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int c = cb * 8 + 2 * k + q;
        float t = 0.0f;
        if (c < a.C) {
          if (MODE == kSplitPool) {
            const float* fc = a.src + (long long)c * 27 * V;
            const int f1 = 3 * g.n1, f2 = 3 * g.n2;
#pragma unroll
            for (int i = 0; i < 3; ++i)
#pragma unroll
              for (int j = 0; j < 3; ++j)
#pragma unroll
                for (int m = 0; m < 3; ++m) t += __ldg(fc + ((long long)(3 * z + i) * f1 + 3 * y + j) * f2 + 3 * x + m);
            t *= 1.0f / 27.0f;
          } else {
            t = __ldg(a.src + c * V + v);
            if (MODE == kSplitUp) t = __ldg(a.coarse + c * (V / 27) + vc) + t;
            if (MODE == kSplitGradUp) t += (1.0f / 27.0f) * __ldg(a.coarse + c * (V / 27) + vc);
            if ((MODE == kSplitGrad || MODE == kSplitGradUp) && a.act && !(__ldg(a.act + c * V + v) > 0.0f)) t *= a.slope;
          }
        }
        s[q] = t;
      }
      const __nv_bfloat16 h0 = __float2bfloat16_rn(s[0]), h1 = __float2bfloat16_rn(s[1]);
      h[k] = pack2(h0, h1);
      l[k] = pack2(__float2bfloat16_rn(s[0] - __bfloat162float(h0)), __float2bfloat16_rn(s[1] - __bfloat162float(h1)));
    }
    const uint4 H = make_uint4(h[0], h[1], h[2], h[3]), Lo = make_uint4(l[0], l[1], l[2], l[3]);
    if (a.out) {
      a.out[kPlaneFront + cb * g.stride + f] = H;
      a.out[kPlaneFront + (nblk + cb) * g.stride + f] = Lo;
    }
    if (a.out0 && inside) {
      a.out0[kPlaneFront + cb * g.stride + f] = H;
      a.out0[kPlaneFront + (nblk + cb) * g.stride + f] = Lo;
    }
  }
}

// Weights of k_conv_planes, every layer in one launch (block row 2 k: forward
// of layer k, 2 k + 1: its data gradient, with the taps reversed and the
// channel roles swapped): [16-channel chunk][tap][k group 2][NT rows][8]
// bfloat16, zero beyond O x C.
constexpr int kMaxConvLayers = 11;
struct WeightArgs {
  const float* w[kMaxConvLayers];        // [O][C][27]
  __nv_bfloat16* out[2][kMaxConvLayers];
  int O[kMaxConvLayers], C[kMaxConvLayers];
};
__global__ void k_weight_planes(WeightArgs a) {
  const int k = blockIdx.y >> 1;
  const bool trans = blockIdx.y & 1;
  const int O = a.O[k], C = a.C[k];
  const int rows = trans ? C : O, cols = trans ? O : C;
  const int NT = (rows + 15) / 16 * 16;
  const float* const w = a.w[k];
  const int n = (cols + 15) / 16 * 27 * 2 * NT * 8;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const int e = i & 7;
    int r = i >> 3;
    const int row = r % NT;
    r /= NT;
    const int kg = r & 1;
    r >>= 1;
    const int t = r % 27, ck = r / 27;
    const int col = ck * 16 + kg * 8 + e;
    float v = 0.0f;
    if (row < rows && col < cols)
      v = trans ? w[((long long)col * C + row) * 27 + 26 - t] : w[((long long)row * C + col) * 27 + t];
    a.out[trans][k][i] = __float2bfloat16_rn(v);
  }
}

// Shared-memory descriptor of an unswizzled operand: lbo / sbo in bytes.
__device__ __forceinline__ uint64_t plane_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFF);
  d |= (uint64_t)((lbo >> 4) & 0x3FFF) << 16;
  d |= (uint64_t)((sbo >> 4) & 0x3FFF) << 32;
  d |= (uint64_t)1 << 46;
  return d;
}

// The same descriptor with the start address moved by `bytes` (the address
// field counts 16-byte words and shared memory is far from its end): one
// thread issues every MMA, so what it computes per MMA is what bounds the
// issue rate.
__device__ __forceinline__ uint64_t desc_at(uint64_t d, uint32_t bytes) { return d + (bytes >> 4); }

// ----------------------------------------------------------------------------
// forward convolution / data gradient
// ----------------------------------------------------------------------------
struct ConvPlanesArgs {
  PlaneGeom g;
  const uint4* x;              // planes of the input
  int nblk;                    // its 8-channel blocks per half (even)
  const __nv_bfloat16* w;      // k_weight_planes layout
  int O;                       // output channels
  float* y;                    // [O][V]
  const float* b;              // bias or nullptr
  float slope;                 // leaky slope applied to the result; 1: none
  int sy;                      // rows' distance in the shared tile: min(px, 128 T + 2) voxels
  int rows;                    // voxels of a tile that exist: min(128 T, n1 px)
  int tiles_z;                 // tiles per z plane
  int resident;                // every chunk's weights stay in shared memory
  int cps;                     // 16-channel chunks per stage: all of them, or 1
  int nstage;                  // stages in shared memory, 1 or 2
  int* err;
  unsigned long long wait_ns;
};
constexpr int kConvThreads = 192;  // warps 0-3: epilogue; 4: copies; 5: MMA

// Shared memory: [resident weights][stage 0][stage 1]; a stage holds cps
// 16-channel chunks, planes [chunk][half 2][dz 3][block 2][2 sy + rows + 2
// voxels], then (cps 1 only) the chunk's weights unless resident.  A tile of
// fewer than 128 T rows reads into the next plane (a tile's 128 T rows are
// allocated behind the last); those rows of the accumulator are not used.
__host__ __device__ inline uint32_t conv_plane_bytes(int sy, int rows) { return (uint32_t)(2 * sy + rows + 2) * 16; }
__host__ __device__ inline uint32_t conv_weight_bytes(int NT) { return 27u * 2 * NT * 16; }
inline size_t conv_smem(int T, int sy, int rows, int NT, int chunks, bool resident, int cps, int nstage) {
  return (resident ? (size_t)chunks : nstage) * conv_weight_bytes(NT) +
         (size_t)nstage * cps * 12 * conv_plane_bytes(sy, rows) + (rows < 128 * T ? (size_t)T * 2048 : 0);
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tma::saddr(bar)) : "memory");
}

// T: 128-voxel MMA tiles per CTA tile; NT: output channels padded to 16.
// Products of one output are summed tap by tap, chunk by chunk, hi then lo (cps
// 1, the few layers whose chunks do not fit together: chunk by chunk first).
template <int T, int NT> __global__ void __launch_bounds__(kConvThreads) k_conv_planes(ConvPlanesArgs a) {
  extern __shared__ __align__(1024) unsigned char smem[];
  __shared__ uint64_t full[2], empty[2], tfull[2], tempty[2], wfull;
  __shared__ uint32_t tmem_slot;
  __shared__ __align__(16) float bias[NT];
  __shared__ volatile int s_fail;
  const int tid = threadIdx.x, warp = tid >> 5;
  const PlaneGeom& g = a.g;
  const int chunks = a.nblk / 2, nstage = a.nstage, ssh = a.nstage - 1;  // it % nstage = it & ssh, it / nstage = it >> ssh
  const uint32_t P = conv_plane_bytes(a.sy, a.rows), wb = conv_weight_bytes(NT);
  unsigned char* const wres = smem;
  const int cps = a.cps, nst = chunks / cps;  // stages per tile
  const uint32_t stage_bytes = cps * 12 * P + (a.resident ? 0 : wb);
  unsigned char* const stage0 = smem + (a.resident ? (size_t)chunks * wb : 0);
  constexpr uint32_t cols = (uint32_t)(2 * T * NT);
  uint32_t ncols = 32;
  while (ncols < cols) ncols <<= 1;
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tma::saddr(&tmem_slot)),
                 "r"(ncols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 0) {
    for (int i = 0; i < 2; ++i) {
      tma::mbar_init(&full[i], 1);
      tma::mbar_init(&empty[i], 1);
      tma::mbar_init(&tfull[i], 1);
      tma::mbar_init(&tempty[i], 4);
    }
    tma::mbar_init(&wfull, 1);
    tma::fence_barrier_init();
    s_fail = 0;
  }
  if (tid < NT) bias[tid] = a.b && tid < a.O ? a.b[tid] : 0.0f;
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = tmem_slot;
  const int ntile = a.tiles_z * g.n0;
  int commits = 0;  // the issuing thread: accumulators committed
  const long long plane0 = (long long)g.py * g.px;

  if (warp == 4) {
    if ((tid & 31) == 0) {
      int it = 0;  // stages issued
      if (a.resident) {
        tma::mbar_arrive_expect_tx(&wfull, chunks * wb);
        tma::bulk_load(wres, a.w, chunks * wb, &wfull);
      }
      for (int tile = blockIdx.x; tile < ntile && !s_fail; tile += gridDim.x) {
        const int z = tile / a.tiles_z, k = tile - z * a.tiles_z;
        // first voxel of the rows the tile needs (row dy = -1, column -1), in plane dz = -1
        const long long f0 = z * plane0 + (long long)k * T * 128 - 1;
        for (int s = 0; s < nst; ++s, ++it) {
          const int st = it & ssh;
          if (it >= nstage && !tma::mbar_wait(&empty[st], ((it >> ssh) - 1) & 1, a.wait_ns)) {
            s_fail = 1;
            break;
          }
          unsigned char* const dst = stage0 + st * stage_bytes;
          tma::mbar_arrive_expect_tx(&full[st], stage_bytes);
          for (int h = 0; h < 2 * cps; ++h)  // (chunk, half)
            for (int dz = 0; dz < 3; ++dz)
              for (int cb = 0; cb < 2; ++cb) {
                const int ck = s * cps + (h >> 1), half = h & 1;
                const uint4* const src =
                    a.x + kPlaneFront + ((long long)half * a.nblk + 2 * ck + cb) * g.stride + f0 + dz * plane0;
                unsigned char* const d = dst + ((h * 3 + dz) * 2 + cb) * P;
                if (a.sy == g.px) {
                  tma::bulk_load(d, src, P, &full[st]);
                } else {
                  for (int dy = 0; dy < 3; ++dy)
                    tma::bulk_load(d + (uint32_t)dy * a.sy * 16, src + (long long)dy * g.px, (uint32_t)a.sy * 16, &full[st]);
                }
              }
          if (!a.resident)
            tma::bulk_load(dst + 12 * P, reinterpret_cast<const unsigned char*>(a.w) + (size_t)s * wb, wb, &full[st]);
        }
      }
      // no copy may land after the CTA has left
      for (int st = 0; st < nstage; ++st) {
        const int cnt = (it + nstage - 1 - st) >> ssh;  // loads issued into this stage
        if (cnt > 0) tma::mbar_wait(&full[st], (cnt - 1) & 1);
      }
      if (a.resident) tma::mbar_wait(&wfull, 0);
    }
  } else if (warp == 5) {
    if ((tid & 31) == 0) {
      const uint32_t idesc = instr_desc(NT);
      int it = 0, nt = 0;
      if (a.resident && !tma::mbar_wait(&wfull, 0, a.wait_ns)) s_fail = 1;
      for (int tile = blockIdx.x; tile < ntile && !s_fail; tile += gridDim.x, ++nt) {
        const int buf = nt & 1;
        if (nt >= 2 && !tma::mbar_wait(&tempty[buf], ((nt - 2) >> 1) & 1, a.wait_ns)) {
          s_fail = 1;
          break;
        }
        fence_after();
        for (int s = 0; s < nst; ++s, ++it) {
          const int st = it & ssh;
          if (!tma::mbar_wait(&full[st], (it >> ssh) & 1, a.wait_ns)) {
            s_fail = 1;
            break;
          }
          fence_after();
          const uint32_t base = tma::saddr(stage0 + st * stage_bytes);
          const uint32_t wbase = a.resident ? tma::saddr(wres) + s * wb : base + 12 * P;
          uint64_t bd0 = plane_desc(wbase, NT * 16, 128);
          const uint64_t ad0 = plane_desc(base, P, 128);
          const uint32_t td = tmem + (uint32_t)(buf * T * NT);
          uint32_t acc = s > 0 ? 1u : 0u;
          auto tap_chunk = [&](uint64_t ah, uint64_t bd) {
            const uint64_t al = desc_at(ah, 6 * P);
#pragma unroll
            for (int j = 0; j < T; ++j) mma(td + j * NT, desc_at(ah, 2048 * j), bd, idesc, acc);
#pragma unroll
            for (int j = 0; j < T; ++j) mma(td + j * NT, desc_at(al, 2048 * j), bd, idesc, 1u);
            acc = 1u;
          };
          if (cps == 1) {
            for (int dz = 0; dz < 3; ++dz) {
#pragma unroll
              for (int dy = 0; dy < 3; ++dy) {
                const uint64_t ay = desc_at(ad0, dz * 2 * P + (uint32_t)(dy * a.sy) * 16);
#pragma unroll
                for (int dx = 0; dx < 3; ++dx) {
                  tap_chunk(desc_at(ay, dx * 16), bd0);
                  bd0 = desc_at(bd0, 2 * NT * 16);
                }
              }
            }
          } else {
            for (int dz = 0; dz < 3; ++dz)
              for (int dy = 0; dy < 3; ++dy) {
                const uint64_t ay = desc_at(ad0, dz * 2 * P + (uint32_t)(dy * a.sy) * 16);
#pragma unroll
                for (int dx = 0; dx < 3; ++dx) {
                  uint64_t ah = desc_at(ay, dx * 16), bd = bd0;
                  for (int c = 0; c < cps; ++c) {
                    tap_chunk(ah, bd);
                    ah = desc_at(ah, 12 * P);
                    bd = desc_at(bd, wb);
                  }
                  bd0 = desc_at(bd0, 2 * NT * 16);
                }
              }
          }
          commit(&empty[st]);
        }
        commit(&tfull[buf]);
      }
      // every issued MMA has finished before tensor memory is released
      for (int st = 0; st < nstage; ++st) {
        const int cnt = (it + nstage - 1 - st) >> ssh;
        if (cnt > 0) tma::mbar_wait(&empty[st], (cnt - 1) & 1);
      }
      commits = nt;
    }
  } else {
    const long long V = g.v();
    int nt = 0;
    // a warp goes on or gives up as a whole (its tensor-memory loads need all lanes)
    for (int tile = blockIdx.x; tile < ntile && !__any_sync(0xffffffffu, s_fail); tile += gridDim.x, ++nt) {
      const int buf = nt & 1;
      if (!__all_sync(0xffffffffu, tma::mbar_wait(&tfull[buf], (nt >> 1) & 1, a.wait_ns))) {
        s_fail = 1;
        break;
      }
      fence_after();
      const int z = tile / a.tiles_z, k = tile - z * a.tiles_z;
      constexpr int K16 = NT / 16;
      uint32_t acc[T][K16][16];
#pragma unroll
      for (int j = 0; j < T; ++j)
#pragma unroll
        for (int k16 = 0; k16 < K16; ++k16)
          tmem_ld16_async(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)((buf * T + j) * NT + k16 * 16), acc[j][k16]);
      tmem_ld_wait();
#pragma unroll
      for (int j = 0; j < T; ++j)
#pragma unroll
        for (int k16 = 0; k16 < K16; ++k16) tmem_use16(acc[j][k16]);
      // tensor memory is free for the tile after next before anything is stored
      fence_before();
      __syncwarp();
      if ((tid & 31) == 0) mbar_arrive(&tempty[buf]);
#pragma unroll
      for (int j = 0; j < T; ++j) {
        const int f = (k * T + j) * 128 + tid;  // flattened over rows y of px columns
        const int y = f / g.px, x = f - y * g.px - 1;
        const bool live = y < g.n1 && x >= 0 && x < g.n2;
        float* const out = a.y + ((long long)z * g.n1 + y) * g.n2 + x;
        if (live) {
#pragma unroll
          for (int k16 = 0; k16 < K16; ++k16)
#pragma unroll
            for (int i = 0; i < 16; ++i) {
              const int o = k16 * 16 + i;
              const float q = __uint_as_float(acc[j][k16][i]) + bias[o];
              if (o < a.O) out[(long long)o * V] = q > 0.0f ? q : a.slope * q;
            }
        }
      }
    }
  }
  fence_before();
  __syncthreads();
  if (s_fail) {
    if (tid == 0 && a.err) atomicExch(a.err, 1);
    // an epilogue that gave up no longer waits for the accumulators' commits:
    // the last of each has arrived before the CTA leaves
    for (int b = 0; b < 2; ++b) {
      const int cnt = (commits + 1 - b) >> 1;
      if (cnt > 0) tma::mbar_wait(&tfull[b], (cnt - 1) & 1);
    }
  }
  __syncwarp();
  if (warp == 0) {
    fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ncols) : "memory");
  }
}

// ----------------------------------------------------------------------------
// weight gradient: dW[o][c][t] = sum_v gy[o](v) x[c](v + t), db[o] = sum_v gy[o](v)
// ----------------------------------------------------------------------------
// One MMA contracts 16 voxels: A is 128 rows = blocks of 8 channels at a
// constant distance in shared memory -- [half 2][dz 3][block 2] of a 16-channel
// chunk of x, then a block whose first channel is 1 (its row sums gy) -- at
// the shift dy, B is three copies of gy (zero padding), shifted by dx, each the
// two halves of 16 output channels; both have the channel as the contiguous
// index.  The accumulator of a shift holds all four products of halves.  A CTA walks a range of
// kWgK-voxel tiles and adds its accumulators to float32 registers after every
// tile, so that the tensor core's own accumulation stays short.
constexpr int kWgK = 256;
constexpr int kWgThreads = 128;
constexpr int kWgRows = 16;      // blocks addressed by an M = 128 operand
struct WgradArgs {
  PlaneGeom g;
  const uint4* x;              // planes of the layer's input (periodic padding)
  int nblk;                    // its blocks per half
  const uint4* gy;             // planes of gy with zero padding
  int oblk;                    // blocks per half (even)
  int O, C;
  int slices;                  // CTAs along the voxels
  int sy;                      // rows' distance in the shared tile: min(px, kWgK)
  long long vox;               // padded voxels from one before the first interior one to one after the last
  float* part;                 // [slice][chunk][shift 9][128 rows][O padded]
  int* err;
  unsigned long long wait_ns;
};
__host__ __device__ inline uint32_t wg_plane_bytes(int sy) { return (uint32_t)(2 * sy + kWgK) * 16; }
// 13 blocks, then gy; an M = 128 operand addresses 16 blocks (what the last
// three hold only reaches unused rows of the accumulator)
inline size_t wg_smem(int sy, int no) {
  const size_t p = wg_plane_bytes(sy), all = 13 * p + 6 * (size_t)no / 8 * kWgK * 16;
  return (all > kWgRows * p ? all : kWgRows * p) + 128;
}
// kind::f16, D float32, A and B bfloat16, both with the M / N index contiguous
__host__ __device__ constexpr uint32_t wg_instr_desc(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
}

// NO: output channels of the CTA's columns, both halves are 2 NO columns.
template <int NO> __global__ void __launch_bounds__(kWgThreads) k_wgrad_planes(WgradArgs a) {
  extern __shared__ __align__(1024) unsigned char smem[];
  __shared__ uint64_t full, done;
  __shared__ uint32_t tmem_slot;
  __shared__ volatile int s_fail;
  const int tid = threadIdx.x, warp = tid >> 5;
  const PlaneGeom& g = a.g;
  const uint32_t P = wg_plane_bytes(a.sy);
  unsigned char* const gys = smem + 13 * (size_t)P;
  constexpr int N = 6 * NO;    // [dx 3][half 2][NO]
  const int ck = blockIdx.y, ob0 = blockIdx.z * (NO / 8);
  const int sl = blockIdx.x;
  uint32_t ncols = 32;
  while (ncols < 3u * N) ncols <<= 1;
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tma::saddr(&tmem_slot)),
                 "r"(ncols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  // block 12: a one in the first channel
  for (uint32_t i = tid; i < P / 16; i += kWgThreads)
    reinterpret_cast<uint4*>(smem + 12 * (size_t)P)[i] = make_uint4(0x3F80u, 0u, 0u, 0u);
  if (tid == 0) {
    tma::mbar_init(&full, 1);
    tma::mbar_init(&done, 1);
    tma::fence_barrier_init();
    s_fail = 0;
  }
  tma::fence_proxy_async();
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = tmem_slot;
  const long long plane0 = (long long)g.py * g.px;
  const long long first = plane0 + g.px;  // one before the first interior voxel (gy shifted by dx = 1 starts there)
  const long long ntile = (a.vox + kWgK - 1) / kWgK;
  const long long t0 = ntile * sl / a.slices, t1 = ntile * (sl + 1) / a.slices;
  const uint32_t gbytes = N / 8 * kWgK * 16;
  float acc[9][NO];
#pragma unroll
  for (int s = 0; s < 9; ++s)
#pragma unroll
    for (int o = 0; o < NO; ++o) acc[s][o] = 0.0f;
  int it = 0;
  for (long long t = t0; t < t1; ++t, ++it) {
    if (tid == 0) {
      const long long f = first + t * kWgK;
      tma::mbar_arrive_expect_tx(&full, 12 * P + gbytes);
      for (int h = 0; h < 2; ++h)
        for (int dz = 0; dz < 3; ++dz)
          for (int cb = 0; cb < 2; ++cb) {
            const uint4* const src = a.x + kPlaneFront + ((long long)h * a.nblk + 2 * ck + cb) * g.stride + f +
                                     (dz - 1) * plane0 - g.px;
            unsigned char* const d = smem + (size_t)((h * 3 + dz) * 2 + cb) * P;
            if (a.sy == g.px) {
              tma::bulk_load(d, src, P, &full);
            } else {
              for (int dy = 0; dy < 3; ++dy)
                tma::bulk_load(d + (uint32_t)dy * a.sy * 16, src + (long long)dy * g.px, (uint32_t)a.sy * 16, &full);
            }
          }
      for (int dx = 0; dx < 3; ++dx)  // gy(f - (dx - 1))
        for (int h = 0; h < 2; ++h)
          for (int ob = 0; ob < NO / 8; ++ob)
            tma::bulk_load(gys + (size_t)((dx * 2 + h) * (NO / 8) + ob) * kWgK * 16,
                           a.gy + kPlaneFront + ((long long)h * a.oblk + ob0 + ob) * g.stride + f + 1 - dx, kWgK * 16,
                           &full);
      if (!tma::mbar_wait(&full, it & 1, a.wait_ns)) {
        tma::mbar_wait(&full, it & 1);  // the copies end before the CTA leaves
        s_fail = 1;
      } else {
        fence_after();
        const uint64_t bd0 = plane_desc(tma::saddr(gys), 128, kWgK * 16);
        uint64_t ad[3];
#pragma unroll
        for (int dy = 0; dy < 3; ++dy) ad[dy] = plane_desc(tma::saddr(smem) + (uint32_t)(dy * a.sy) * 16, 128, P);
        for (int k = 0; k < kWgK / 16; ++k) {
          // unswizzled, M / N contiguous: 8-channel blocks P (kWgK * 16) apart, 8-voxel groups 128 bytes apart
          const uint64_t bd = desc_at(bd0, k * 256);
#pragma unroll
          for (int dy = 0; dy < 3; ++dy)
            mma(tmem + (uint32_t)dy * N, desc_at(ad[dy], k * 256), bd, wg_instr_desc(N), k > 0 ? 1u : 0u);
        }
        commit(&done);
        if (!tma::mbar_wait(&done, it & 1, a.wait_ns)) {
          tma::mbar_wait(&done, it & 1);
          s_fail = 1;
        }
      }
    }
    __syncthreads();
    if (s_fail) break;
    fence_after();
    const uint32_t lane_base = tmem + ((uint32_t)(warp * 32) << 16);
#pragma unroll
    for (int s = 0; s < 9; ++s) {
#pragma unroll
      for (int c0 = 0; c0 < NO; c0 += 16) {
        float hi[16], lo[16];
        tmem_ld16(lane_base + (uint32_t)(s * 2 * NO + c0), hi);  // s = dy * 3 + dx
        tmem_ld16(lane_base + (uint32_t)(s * 2 * NO + NO + c0), lo);
#pragma unroll
        for (int i = 0; i < 16; ++i) acc[s][c0 + i] += hi[i] + lo[i];
      }
    }
    fence_before();
    __syncthreads();
  }
  if (!s_fail) {
    const int Op = a.oblk * 8, chunks = a.nblk / 2;
#pragma unroll
    for (int s = 0; s < 9; ++s) {
      float* const dst =
          a.part + ((((long long)sl * chunks + ck) * 9 + s) * 128 + tid) * Op + ob0 * 8;
#pragma unroll
      for (int o = 0; o < NO; ++o) dst[o] = acc[s][o];
    }
  } else if (tid == 0 && a.err) {
    atomicExch(a.err, 1);
  }
  __syncthreads();
  if (warp == 0) {
    fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ncols) : "memory");
  }
}

// gW[o][c][t] = sum over slices and halves; gb[o] from the row of ones.  Every
// layer in one launch (block row = layer).
struct WgradSumArgs {
  const float* part[kMaxConvLayers];
  float *gW[kMaxConvLayers], *gb[kMaxConvLayers];
  int O[kMaxConvLayers], C[kMaxConvLayers], slices[kMaxConvLayers];
};
__global__ void __launch_bounds__(128) k_wgrad_sum(WgradSumArgs a) {
  const int k = blockIdx.y, O = a.O[k], C = a.C[k], slices = a.slices[k];
  const int Op = (O + 15) / 16 * 16, chunks = (C + 15) / 16;
  const long long stride = (long long)chunks * 9 * 128 * Op;
  const int n = O * (C * 27 + 1);
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const int o = i % O;
    const int r = i / O;  // c * 27 + t, or C * 27 for the bias
    const bool is_bias = r == C * 27;
    const int c = is_bias ? 0 : r / 27, t = is_bias ? 13 : r - c * 27, dz = t / 9, sh = t - dz * 9;
    // row 96: the ones (any shift); else block (dz, c / 8 % 2) of the hi half, the lo half 48 rows on
    const int row = is_bias ? 96 : (dz * 2 + (c % 16) / 8) * 8 + c % 8;
    const float* p = a.part[k] + (((long long)(c / 16) * 9 + (is_bias ? 4 : sh)) * 128 + row) * Op + o;
    float v[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    int s = 0;
    for (; s + 4 <= slices; s += 4)
#pragma unroll
      for (int q = 0; q < 4; ++q) v[q] += is_bias ? p[(s + q) * stride] : p[(s + q) * stride] + p[(s + q) * stride + 48LL * Op];
    for (; s < slices; ++s) v[0] += is_bias ? p[s * stride] : p[s * stride] + p[s * stride + 48LL * Op];
    const float sum = (v[0] + v[1]) + (v[2] + v[3]);
    if (is_bias)
      a.gb[k][o] = sum;
    else
      a.gW[k][((long long)o * C + c) * 27 + t] = sum;
  }
}

}  // namespace tc
}  // namespace fh
