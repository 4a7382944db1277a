// fh_spectral.cuh -- the CG iteration of a refinement step in the frequency
// domain (float32; every refined solve, batch and all-loads solve).
//
// Residuals, directions and corrections of CG started as the refinement
// starts it are compatible zero-mean fields (Section 2.1): their spectra are
// v^(k) = u(k) psi(k) with the unit vector u = xi / |xi| and one complex
// scalar psi per frequency.  In this basis
//   A psi = psi + |xi| (xi . F[dL F^-1(u psi)]) / (xi . L0 . xi) / |N|,
// (v, w) = |N| sum_k conj(psi_v) psi_w, and the CG recurrences are those of
// the fields.  One vector costs one real scalar per node instead of d, and no
// vector is read or written in the real-space passes.  One iteration:
//
//   spec_inv  columns along axis 0: r -= alpha A p, x += alpha p, p = r + beta p,
//             (r, r); inverse FFT of (xi_0 g, xi_1 g) (2-D) or (xi_0 g, g)
//             (3-D) with g = p / |xi|.
//   spec_mid  3-D: inverse FFT along axis 1 of (v_0, xi_1 g, xi_2 g).
//   spec_row  lines: inverse FFT, tau = dL v at the nodes, forward FFT, in place.
//   spec_mid  3-D: forward FFT along axis 1, (tau_0, xi_1 tau_1 + xi_2 tau_2).
//   spec_fwd  columns along axis 0: forward FFT, projection, A p, (p, A p), (A p, A p),
//             (r, A p).
//   k_scal_spec  alpha, beta and the stopping tests from one reduction.
//
// The next (r, r) follows from the reductions of spec_fwd,
//   (r+, r+) = (r, r) - 2 alpha (r, A p) + alpha^2 (A p, A p),
// and the stored residual's own (r, r) replaces it one iteration later as the
// numerator of alpha, so rounding does not accumulate.  All three products are
// measured: the expansion is then within 1e-7 of the (r+, r+) of the stored
// residual (the rounding of its elements; contrast 10 to 1e4 in a float32
// model of the iteration), where (p, A p) in place of (r, A p), its value for a
// symmetric A in exact arithmetic, is 1e-6 off.
//
// The scalars of a solve are those of its fields times a power of two that
// brings the initial residual's norm to about 1 (psi_f, exact): psi is 1 / sqrt|N|
// of a field, and its squares would leave float32's range for loads of 1e-11.
//
// Memory moved per iteration in units of one real scalar per node: 18.25 in
// 2-D (update 7, spectra 8, projection 3, phase 1/4; 28.25 with the fields'
// passes), 30.25 in 3-D (54.25).
// Measured per iteration, against the passes on fields: 2187^2 168 -> 125 us
// (row 44, inv 42, fwd 38; 349 MB, 51 us at the copy rate), 243^3 with three
// loads 2.54 -> 1.46 ms (row 403, inv 287, mid 270 + 254, fwd 234; 5.2 GB,
// 0.76 ms at the copy rate).  Bound by the FFT stages' shared-memory
// round trips and barriers at 24 warps per SM (45 % of the issue slots); small
// grids (405x675: 25 us) by the length of one thread's chain per kernel.
//
// Spectra are stored line by line, S[line][k_last][channel] with k_last padded
// to Hp, so that the row pass, which reads and writes every line once, moves
// contiguous memory; the column passes read C frequencies (at least one
// 32-byte sector) of every line.  The scalar arrays are touched only by the
// column kernels and are stored tile by tile, [tile][i0][C].
#pragma once

#include "fh_kernels.cuh"

namespace fh {

struct SpecGeom {
  int C, csh;                  // frequencies per column tile (power of two)
  int Tt, Hp;                  // tiles; padded half spectrum Tt * C
  float invY[3], inv_nodes;
};

// Reference medium of one cell: xi . L0 . xi from its coefficients, and the
// factor of the projection.  float32: the kernels of an iteration do no
// float64 work per element or per thread (a warp's float64 instruction holds
// the pipe for 16 cycles; the conversions and the float64 block reductions of
// an earlier version kept that pipe 73 % busy in spec_fwd; sums are Sum3).
struct SpecMedium {
  float L00, s01, s02, L11, s12, L22;  // sij = L0ij + L0ji
  float scale;                         // 1 / (|N| l0) for isotropic L0, else 1 / |N|
  float iso;
};

struct SpecArgs {
  Geom g;
  SpecGeom sg;
  FFTPlan plan;                // along axis 0
  int tpc;                     // threads per column FFT
  int ss;                      // distance between columns in shared memory
  int nb_inner;                // 2-D: cells; 3-D: lines along axis 1
  int nl, three;               // loads; 3-D
  const float2* tw;
  float2* S;                   // two channels per load and frequency
  // scalar arrays per load, [tile][row along axis 0][C]
  float2* r[kMaxLoads];
  float2* p[kMaxLoads];
  float2* ap[kMaxLoads];
  float2* x[kMaxLoads];
  Scal* scal;
  // partial sums (Sum3), one per CTA: (p, A p) rows 0.., (A p, A p) rows kMaxLoads..,
  // (r, A p) rows 2 kMaxLoads.., (r, r) rows 3 kMaxLoads..
  float4* part;
  const SpecMedium* med;       // per cell
};

// ----------------------------------------------------------------------------
// sums over a CTA
// ----------------------------------------------------------------------------
// a + b = s + e exactly
__device__ __forceinline__ float two_sum(float a, float b, float& e) {
  const float s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
  return s;
}
// Sum held in three float32 parts s + c + r (the K-fold compensated summation
// of Ogita, Rump and Oishi with K = 3): more bits than float64, on the float32
// units.  A float64 instruction holds an SM's unit for 16 cycles per warp, and a
// tree of them at the end of every kernel is a chain that the next kernel waits
// for.
struct Sum3 {
  float s, c, r;
  __device__ __forceinline__ void low(float v) {
    float e;
    c = two_sum(c, v, e);
    r = __fadd_rn(r, e);
  }
  __device__ __forceinline__ void add(float vs, float vc, float vr) {
    float e;
    s = two_sum(s, vs, e);
    low(e);
    low(vc);
    r = __fadd_rn(r, vr);
  }
  // over groups of `width` lanes
  __device__ __forceinline__ void warp_sum(int width = 32) {
    for (int o = width >> 1; o > 0; o >>= 1)
      add(__shfl_down_sync(0xffffffffu, s, o), __shfl_down_sync(0xffffffffu, c, o), __shfl_down_sync(0xffffffffu, r, o));
  }
  __device__ __forceinline__ double get() const { return (double)s + ((double)c + (double)r); }
};
__device__ __forceinline__ float2 dot_parts(const DotAcc<float>& d) { return make_float2(d.s, -d.c); }

// Sums of `rows` rows of `count` values (a thread's two parts each) in shared
// memory, row k at src(k)[at(i)]; its sum goes to *out(k).  Call after a barrier
// behind the writes.  A row is summed by 32 lanes, or by 8 where a kernel carries several
// loads: there the CTAs are small and many, and the trees' instructions count
// more than the length of the chain (243^3, three loads: 644 -> 610 ms per tensor
// with that and the sums kept in the tile instead of behind it).
template <typename S, typename A, typename F>
__device__ __forceinline__ void rows_store(int rows, int count, int nl, S&& src, A&& at, F&& out) {
  const int width = nl > 1 ? 8 : 32, per = 32 / width;  // lanes per row, rows per warp
  const int lane = threadIdx.x & 31, sub = lane & (width - 1), nw = blockDim.x >> 5;
  for (int k0 = (threadIdx.x >> 5) * per; k0 < rows; k0 += nw * per) {
    const int k = k0 + lane / width;
    Sum3 t{0.0f, 0.0f, 0.0f};
    if (k < rows) {
      const float2* const row = src(k);
#pragma unroll 4
      for (int i = sub; i < count; i += width) {
        const float2 v = row[at(i)];
        t.add(v.x, v.y, 0.0f);
      }
    }
    t.warp_sum(width);
    if (sub == 0 && k < rows) *out(k) = make_float4(t.s, t.c, t.r, 0.0f);
  }
}

// Threads per sequence of a compile-time plan (27 values per thread), or the
// launch's count for run-time plans.
template <typename PS> __host__ __device__ constexpr int spec_plan_threads() {
  if constexpr (PlanLen<PS>::value > 0) {
    int t = 1;
    for (int i = 0; i < PS::S; ++i) {
      const int per = RegBudget<float>::value / PS::r[i];
      const int need = (PS::n / PS::r[i] + per - 1) / per;
      if (need > t) t = need;
    }
    return t;
  }
  return 0;
}
template <typename PS> __device__ __forceinline__ int spec_threads(int rt) {
  return PlanLen<PS>::value > 0 ? spec_plan_threads<PS>() : rt;
}

// Column FFTs of a tile stored column by column (column q at sm + q ss): the
// stage addresses of a compile-time plan are then constants, and ss >= n is
// chosen for the fewest bank conflicts (seq_stride).
template <bool INV, typename PS>
__device__ __forceinline__ void spec_col_fft(float2* sm, int ss, int n, int Q, const FFTPlan& plan, int tpc_rt,
                                             const float2* tw) {
  const int tpc = spec_threads<PS>(tpc_rt);
  const int q = threadIdx.x / tpc, u = threadIdx.x - q * tpc;
  fft_plan<INV, float, PS>(sm + (q < Q ? q : 0) * ss, 1, plan, q < Q ? u : n, tpc, tw);
}

// The scalars of one thread of a column kernel all belong to one frequency of
// the last axis (and of axis 1): what does not depend on the row is kept here.
struct SpecFreq {
  float invY0, c1, q1, scale, wgt;
  float L00, L01, L11;         // xi . L0 . xi = xi0 (L00 xi0 + L01) + L11
  int n, nyq;                  // axis-0 length, its Nyquist bin (-1: odd)
  bool dead, iso, zero0;       // no Green operator in this column; isotropic L0; row 0 is the zero frequency
  __device__ __forceinline__ void init(const SpecArgs& a, const SpecMedium& m, int n_, int kl, int i1) {
    const Geom& g = a.g;
    n = n_;
    nyq = (n_ & 1) ? -1 : n_ / 2;
    invY0 = a.sg.invY[0];
    const bool three = a.three;
    const int k1 = three ? signed_freq(i1, g.n[1]) : kl;
    const float xi1 = (float)k1 * a.sg.invY[1];
    const float xi2 = three ? (float)kl * a.sg.invY[2] : 0.0f;
    q1 = xi1 * xi1 + xi2 * xi2;
    c1 = three ? 1.0f : xi1;   // second channel: g (3-D) or xi_1 g (2-D)
    dead = kl >= g.H || nyquist_bin(kl, g.nlast) || (three && nyquist_bin(i1, g.n[1]));
    zero0 = k1 == 0 && kl == 0;
    wgt = kl == 0 ? 1.0f : 2.0f;  // half spectrum: k and -k
    iso = m.iso != 0.0f;
    scale = m.scale;
    L00 = m.L00;
    L01 = m.s01 * xi1 + m.s02 * xi2;
    L11 = xi1 * (m.L11 * xi1 + m.s12 * xi2) + m.L22 * xi2 * xi2;
  }
  __device__ __forceinline__ float xi0(int i) const { return (float)(i <= n / 2 ? i : i - n) * invY0; }
  // 1 / |xi|, zero where the Green operator is zero
  __device__ __forceinline__ float rnorm(int i, float x0) const {
    return dead || i == nyq || (i == 0 && zero0) ? 0.0f : rsqrtf(x0 * x0 + q1);
  }
  // 1 / (|xi|^2 rn), which takes xi . v back to psi where v = xi rn psi: the two
  // maps are inverse to each other to float32 rounding whatever the error of
  // rn is (rsqrtf's, squared, would be an error of the operator).  One Newton
  // step from rn; its defect |xi|^2 rn^2 - 1 is formed exactly.
  __device__ __forceinline__ float inverse(float x0, float rn) const {
    const float q = x0 * x0 + q1, t = q * rn;
    const float e = fmaf(t, rn, -1.0f) + fmaf(q, rn, -t) * rn;
    return rn == 0.0f ? 0.0f : fmaf(-rn, e, rn);
  }
  // 1 / (xi . L0 . xi rn) / |N|: the projection's factor
  __device__ __forceinline__ float project(float x0, float rn) const {
    if (iso) return inverse(x0, rn) * scale;
    return rn == 0.0f ? 0.0f : scale / ((x0 * (L00 * x0 + L01) + L11) * rn);
  }
};

// Tile of a column kernel: block index -> tile of frequencies and cell / line.
struct SpecTile {
  int t, inner, cell, slot;
  long long line0;             // line of row 0; row i is line line0 + i * step
  int step;
  long long sbase;             // first element of the tile in a scalar array
};
__device__ __forceinline__ SpecTile spec_tile(const SpecArgs& a, int n) {
  SpecTile s;
  const Geom& g = a.g;
  s.t = blockIdx.x / a.nb_inner;
  s.inner = blockIdx.x - s.t * a.nb_inner;
  s.cell = a.three ? 0 : s.inner;
  // partial sums of one cell are consecutive
  s.slot = a.three ? (int)blockIdx.x : s.cell * a.sg.Tt + s.t;
  s.line0 = a.three ? s.inner : (long long)s.cell * n;
  s.step = a.three ? g.n1 : 1;
  s.sbase = (long long)blockIdx.x * n * a.sg.C;
  return s;
}

// Rows i and words j of a tile row (wpr words) that one thread copies.
struct SpecWalk {
  int i, j, di, dj, wpr;
  __device__ __forceinline__ SpecWalk(int wpr_) : wpr(wpr_) {
    i = threadIdx.x / wpr;
    j = threadIdx.x - i * wpr;
    di = blockDim.x / wpr;
    dj = blockDim.x - di * wpr;
  }
  __device__ __forceinline__ void next() {
    i += di;
    j += dj;
    if (j >= wpr) {
      j -= wpr;
      ++i;
    }
  }
};

// Thread limits the column kernels are compiled for: 27 complex values per
// thread need ~80 registers.
template <typename PS> struct SpecBounds {
  static constexpr int threads = 768;
};

enum : int { kSpecUpdate = 0, kSpecFinish = 1 };   // spec_inv
enum : int { kSpecApply = 0, kSpecProject = 1 };   // spec_fwd

inline size_t spec_col_smem(int ss, int Q, int rows, int block) {
  return ((size_t)ss * Q + (size_t)rows * block) * sizeof(float2);
}

// kSpecUpdate: one CG update of the tile's scalars, then the inverse FFT of
// the new direction.  kSpecFinish: the inverse FFT of x + (owed step).
template <int MODE, typename PS = DynPlan>
__global__ void __launch_bounds__(SpecBounds<PS>::threads) k_spec_inv(SpecArgs a) {
  seq_begin();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2* sm = reinterpret_cast<float2*>(smem_raw);
  const int n = plan_len<PS>(a.plan), C = a.sg.C, csh = a.sg.csh, nl = a.nl;
  const int Q = 2 * nl * C;
  float2* const red = sm + (size_t)a.ss * Q;
  const SpecTile tl = spec_tile(a, n);
  Scal* const sc = a.scal + tl.cell * nl;
  if (MODE == kSpecUpdate && all_done(sc, nl)) return;
  // a thread holds two neighbouring frequencies (16-byte words)
  const int e = 2 * (threadIdx.x & (C / 2 - 1)), row0 = threadIdx.x >> (csh - 1), drow = blockDim.x >> (csh - 1);
  SpecFreq fq[2];
  fq[0].init(a, a.med[tl.cell], n, tl.t * C + e, tl.inner);
  fq[1].init(a, a.med[tl.cell], n, tl.t * C + e + 1, tl.inner);
  constexpr int kUnroll = 2;
  for (int l = 0; l < nl; ++l) {
    const Scal& s = sc[l];
    const bool fresh = s.iter == 0;
    const float al = MODE == kSpecUpdate || s.xpend ? s.alpha_f : 0.0f;
    const float be = s.beta_f;
    const bool live = MODE == kSpecUpdate ? s.done == kRunning : !fresh;
    const float back = s.psi_b;  // kSpecFinish: to the fields' scale
    float4* const r = reinterpret_cast<float4*>(a.r[l] + tl.sbase + e);
    float4* const p = reinterpret_cast<float4*>(a.p[l] + tl.sbase + e);
    float4* const x = reinterpret_cast<float4*>(a.x[l] + tl.sbase + e);
    const float4* const ap = reinterpret_cast<const float4*>(a.ap[l] + tl.sbase + e);
    float2* const ch = sm + (size_t)(e * nl + l) * 2 * a.ss;
    const int next = 2 * nl * a.ss;  // the second frequency's columns
    DotAcc<float> dot;
    for (int i0 = row0; i0 < n; i0 += kUnroll * drow) {
      float4 vr[kUnroll], vp[kUnroll], va[kUnroll], vx[kUnroll];
#pragma unroll
      for (int u = 0; u < kUnroll; ++u) {
        const int i = i0 + u * drow, k = i << (csh - 1);
        vr[u] = vp[u] = va[u] = vx[u] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (i < n && live) {
          // r and x are kept out of the way of what the next passes read again
          // (S, p, A p; r too is read by the projection, but storing it the
          // ordinary way made no difference: 2187^2 14.36 and 14.28 ms)
          if (MODE == kSpecUpdate) vr[u] = __ldcs(r + k);
          if (!fresh) {
            if (MODE == kSpecUpdate) va[u] = __ldg(ap + k);
            vp[u] = p[k];
            vx[u] = __ldcs(x + k);
          }
        }
      }
#pragma unroll
      for (int u = 0; u < kUnroll; ++u) {
        const int i = i0 + u * drow, k = i << (csh - 1);
        if (i >= n) continue;
        auto axpy = [](float4& y, float c, const float4& z) {
          y.x += c * z.x;
          y.y += c * z.y;
          y.z += c * z.z;
          y.w += c * z.w;
        };
        axpy(vx[u], al, vp[u]);
        float4 v = make_float4(back * vx[u].x, back * vx[u].y, back * vx[u].z, back * vx[u].w);
        if (MODE == kSpecUpdate) {
          axpy(vr[u], -al, va[u]);
          v = vr[u];
          axpy(v, be, vp[u]);
          if (live) {
            __stcs(r + k, vr[u]);
            p[k] = v;
            __stcs(x + k, vx[u]);
          }
          dot.add(fq[0].wgt * (vr[u].x * vr[u].x + vr[u].y * vr[u].y));
          dot.add(fq[1].wgt * (vr[u].z * vr[u].z + vr[u].w * vr[u].w));
        }
        const float x0 = fq[0].xi0(i);
        const float s0 = fq[0].rnorm(i, x0), s1 = fq[1].rnorm(i, x0);
        const float f0 = x0 * s0, g0 = fq[0].c1 * s0, f1 = x0 * s1, g1 = fq[1].c1 * s1;
        ch[i] = make_float2(f0 * v.x, f0 * v.y);
        ch[a.ss + i] = make_float2(g0 * v.x, g0 * v.y);
        ch[next + i] = make_float2(f1 * v.z, f1 * v.w);
        ch[next + a.ss + i] = make_float2(g1 * v.z, g1 * v.w);
      }
    }
    if (MODE == kSpecUpdate)
      red[l * blockDim.x + threadIdx.x] = dot_parts(dot);
  }
  __syncthreads();
  spec_col_fft<true, PS>(sm, a.ss, n, Q, a.plan, a.tpc, a.tw);
  const int wpr = nl * C;  // 16-byte words per row
  float4* const S = reinterpret_cast<float4*>(a.S) + (tl.line0 * a.sg.Hp + tl.t * C) * nl;
  const long long rs = (long long)tl.step * a.sg.Hp * nl;
  for (SpecWalk w(wpr); w.i < n; w.next()) {
    const float2 v0 = sm[2 * w.j * a.ss + w.i], v1 = sm[(2 * w.j + 1) * a.ss + w.i];
    S[w.i * rs + w.j] = make_float4(v0.x, v0.y, v1.x, v1.y);
  }
  if (MODE == kSpecUpdate)
    rows_store(
        nl, blockDim.x, nl, [&](int k) { return red + k * blockDim.x; }, [](int i) { return i; },
        [&](int k) { return a.part + (size_t)(3 * kMaxLoads + k) * gridDim.x + tl.slot; });
}

// kSpecApply: A p of the direction's tau spectrum, with (p, A p), (A p, A p) and (r, A p).
// kSpecProject: the scalars of a real residual field's spectrum into r.
template <int MODE, typename PS = DynPlan>
__global__ void __launch_bounds__(SpecBounds<PS>::threads) k_spec_fwd(SpecArgs a) {
  seq_begin();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2* sm = reinterpret_cast<float2*>(smem_raw);
  const int n = plan_len<PS>(a.plan), C = a.sg.C, csh = a.sg.csh, nl = a.nl;
  const int Q = 2 * nl * C;
  const SpecTile tl = spec_tile(a, n);
  Scal* const sc = a.scal + tl.cell * nl;
  if (MODE == kSpecApply && all_done(sc, nl)) return;
  const int e = 2 * (threadIdx.x & (C / 2 - 1)), row0 = threadIdx.x >> (csh - 1), drow = blockDim.x >> (csh - 1);
  constexpr int kUnroll = 4;
  {
    const int wpr = nl * C;
    const float4* const S = reinterpret_cast<const float4*>(a.S) + (tl.line0 * a.sg.Hp + tl.t * C) * nl;
    const long long rs = (long long)tl.step * a.sg.Hp * nl;
    SpecWalk w(wpr);
    while (w.i < n) {
      float4 buf[kUnroll];
      int at[kUnroll];
#pragma unroll
      for (int u = 0; u < kUnroll; ++u) {
        at[u] = w.i < n ? 2 * w.j * a.ss + w.i : -1;
        if (w.i < n) buf[u] = __ldg(S + w.i * rs + w.j);
        w.next();
      }
#pragma unroll
      for (int u = 0; u < kUnroll; ++u)
        if (at[u] >= 0) {
          sm[at[u]] = make_float2(buf[u].x, buf[u].y);
          sm[at[u] + a.ss] = make_float2(buf[u].z, buf[u].w);
        }
    }
  }
  __syncthreads();
  spec_col_fft<false, PS>(sm, a.ss, n, Q, a.plan, a.tpc, a.tw);
  SpecFreq fq[2];
  fq[0].init(a, a.med[tl.cell], n, tl.t * C + e, tl.inner);
  fq[1].init(a, a.med[tl.cell], n, tl.t * C + e + 1, tl.inner);
  for (int l = 0; l < nl; ++l) {
    const float toscale = a.sg.inv_nodes * sc[l].psi_f;  // kSpecProject
    DotAcc<float> d1, d2, d3;
    if (MODE == kSpecProject || sc[l].done == kRunning) {
      const float4* const p = reinterpret_cast<const float4*>(a.p[l] + tl.sbase + e);
      const float4* const r = reinterpret_cast<const float4*>(a.r[l] + tl.sbase + e);
      float4* const out = reinterpret_cast<float4*>((MODE == kSpecApply ? a.ap[l] : a.r[l]) + tl.sbase + e);
      const float2* const ch = sm + (size_t)(e * nl + l) * 2 * a.ss;
      const int next = 2 * nl * a.ss;
      constexpr int kUnrollA = 2;  // 4 spill
      for (int i0 = row0; i0 < n; i0 += kUnrollA * drow) {
        float4 vp[kUnrollA], vr[kUnrollA];
#pragma unroll
        for (int u = 0; u < kUnrollA; ++u) {
          const int i = i0 + u * drow;
          vp[u] = (MODE == kSpecApply && i < n) ? __ldg(p + (i << (csh - 1))) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
          vr[u] = (MODE == kSpecApply && i < n) ? __ldg(r + (i << (csh - 1))) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        }
#pragma unroll
        for (int u = 0; u < kUnrollA; ++u) {
          const int i = i0 + u * drow;
          if (i >= n) continue;
          const float x0 = fq[0].xi0(i);
          float2 y[2];
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const float2 v0 = ch[h * next + i], v1 = ch[h * next + a.ss + i];
            const float rn = fq[h].rnorm(i, x0);
            const float w = MODE == kSpecApply ? fq[h].project(x0, rn) : fq[h].inverse(x0, rn) * toscale;
            const float w0 = x0 * w, w1 = fq[h].c1 * w;
            y[h] = make_float2(w0 * v0.x + w1 * v1.x, w0 * v0.y + w1 * v1.y);
            if (MODE == kSpecApply) {
              const float2 q = h ? make_float2(vp[u].z, vp[u].w) : make_float2(vp[u].x, vp[u].y);
              const float2 rv = h ? make_float2(vr[u].z, vr[u].w) : make_float2(vr[u].x, vr[u].y);
              y[h].x += q.x;
              y[h].y += q.y;
              d1.add(fq[h].wgt * (q.x * y[h].x + q.y * y[h].y));
              d2.add(fq[h].wgt * (y[h].x * y[h].x + y[h].y * y[h].y));
              d3.add(fq[h].wgt * (rv.x * y[h].x + rv.y * y[h].y));
            }
          }
          out[i << (csh - 1)] = make_float4(y[0].x, y[0].y, y[1].x, y[1].y);
        }
      }
    }
    // the sums take the place of the thread's first row, which only it has read
    if (MODE == kSpecApply && row0 < n) {
      float2* const own = sm + (size_t)(e * nl + l) * 2 * a.ss + row0;
      own[0] = dot_parts(d1);
      own[a.ss] = dot_parts(d2);
      own[2 * nl * a.ss] = dot_parts(d3);
    }
  }
  if (MODE == kSpecApply) {
    __syncthreads();
    const int half = csh - 1, count = n << half < (int)blockDim.x ? n << half : (int)blockDim.x;
    rows_store(
        3 * nl, count, nl,
        [&](int k) {
          const int kind = k / nl;
          return sm + (k - kind * nl) * 2 * a.ss + (kind == 2 ? 2 * nl : kind) * a.ss;
        },
        [&](int i) { return 4 * nl * a.ss * (i & ((1 << half) - 1)) + (i >> half); },
        [&](int k) { return a.part + (size_t)(k / nl * kMaxLoads + k % nl) * gridDim.x + tl.slot; });
  }
}

// Green operator on a two-channel spectrum (the operator's product): forward
// FFT along axis 0, y^ = xi (xi . tau^) / (xi . L0 . xi) / |N|, inverse FFT.
// 3-D: two channels per frequency (xi_0 is the FFT axis, the other two
// components enter projected), 10 us on 63x135x105 where the three-channel
// pass took 21 us; 2-D 49 us on 2187^2, bound by the shared-memory stages.
template <typename PS = DynPlan>
__global__ void __launch_bounds__(SpecBounds<PS>::threads) k_spec_green(SpecArgs a) {
  seq_begin();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2* sm = reinterpret_cast<float2*>(smem_raw);
  const int n = plan_len<PS>(a.plan), C = a.sg.C, nl = a.nl;
  const int Q = 2 * nl * C, wpr = nl * C;
  const SpecTile tl = spec_tile(a, n);
  float4* const S = reinterpret_cast<float4*>(a.S) + (tl.line0 * a.sg.Hp + tl.t * C) * nl;
  const long long rs = (long long)tl.step * a.sg.Hp * nl;
  constexpr int kUnroll = 4;
  {
    SpecWalk w(wpr);
    while (w.i < n) {
      float4 buf[kUnroll];
      int at[kUnroll];
#pragma unroll
      for (int u = 0; u < kUnroll; ++u) {
        at[u] = w.i < n ? 2 * w.j * a.ss + w.i : -1;
        if (w.i < n) buf[u] = S[w.i * rs + w.j];
        w.next();
      }
#pragma unroll
      for (int u = 0; u < kUnroll; ++u)
        if (at[u] >= 0) {
          sm[at[u]] = make_float2(buf[u].x, buf[u].y);
          sm[at[u] + a.ss] = make_float2(buf[u].z, buf[u].w);
        }
    }
  }
  __syncthreads();
  spec_col_fft<false, PS>(sm, a.ss, n, Q, a.plan, a.tpc, a.tw);
  {
    const int csh = a.sg.csh;
    const int e = threadIdx.x & (C - 1), row0 = threadIdx.x >> csh, drow = blockDim.x >> csh;
    SpecFreq fq;
    fq.init(a, a.med[tl.cell], n, tl.t * C + e, tl.inner);
    const float c1 = fq.c1, L00 = fq.L00, L01 = fq.L01, L11 = fq.L11;
    for (int l = 0; l < nl; ++l) {
      float2* const ch = sm + (size_t)(e * nl + l) * 2 * a.ss;
      for (int i = row0; i < n; i += drow) {
        const float2 v0 = ch[i], v1 = ch[a.ss + i];
        const float x0 = fq.xi0(i);
        const bool zero = fq.dead || i == fq.nyq || (i == 0 && fq.zero0);
        const float f = zero ? 0.0f : a.sg.inv_nodes / (x0 * (L00 * x0 + L01) + L11);
        const float2 w = make_float2((x0 * v0.x + c1 * v1.x) * f, (x0 * v0.y + c1 * v1.y) * f);
        ch[i] = make_float2(x0 * w.x, x0 * w.y);
        ch[a.ss + i] = make_float2(c1 * w.x, c1 * w.y);
      }
    }
  }
  __syncthreads();
  spec_col_fft<true, PS>(sm, a.ss, n, Q, a.plan, a.tpc, a.tw);
  for (SpecWalk w(wpr); w.i < n; w.next()) {
    const float2 v0 = sm[2 * w.j * a.ss + w.i], v1 = sm[(2 * w.j + 1) * a.ss + w.i];
    S[w.i * rs + w.j] = make_float4(v0.x, v0.y, v1.x, v1.y);
  }
}

// ----------------------------------------------------------------------------
// 3-D: passes along axis 1 between the two-channel and the three-component
// spectra; one CTA per (tile, i0), rows of C frequencies.
// ----------------------------------------------------------------------------
struct SpecMidArgs {
  Geom g;
  SpecGeom sg;
  FFTPlan plan;                // along axis 1
  int tpc;
  int ss;                      // distance between columns in shared memory
  int nl;
  const float2* tw;
  float2* S2;                  // two channels per load
  float2* S3;                  // three components per load
  Scal* scal;                  // nullptr: never skipped
};

template <bool INV, typename PS = DynPlan>
__global__ void __launch_bounds__(SpecBounds<PS>::threads) k_spec_mid(SpecMidArgs a) {
  seq_begin();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2* sm = reinterpret_cast<float2*>(smem_raw);
  const Geom& g = a.g;
  const int n = plan_len<PS>(a.plan), C = a.sg.C, nl = a.nl;
  const int rc = C * nl;       // (frequency, load) pairs per row
  const int Q = 3 * rc;
  if (all_done(a.scal, nl)) return;
  const int t = blockIdx.x / g.n[0], i0 = blockIdx.x - t * g.n[0];
  const long long row0 = ((long long)i0 * n * a.sg.Hp + t * C) * nl;  // pairs
  const long long rs = (long long)a.sg.Hp * nl;
  float4* const S2 = reinterpret_cast<float4*>(a.S2) + row0;
  float2* const S3 = a.S3 + row0 * 3;
  const float invY1 = a.sg.invY[1], invY2 = a.sg.invY[2];
  constexpr int kUnroll = 4;
  if (INV) {
    SpecWalk w(rc);
    while (w.i < n) {
      float4 v[kUnroll];
      int wi[kUnroll], wj[kUnroll];
#pragma unroll
      for (int u = 0; u < kUnroll; ++u) {
        wi[u] = w.i;
        wj[u] = w.j;
        if (w.i < n) v[u] = S2[w.i * rs + w.j];
        w.next();
      }
#pragma unroll
      for (int u = 0; u < kUnroll; ++u) {
        if (wi[u] >= n) continue;
        const float xi1 = (float)signed_freq(wi[u], n) * invY1;
        const float xi2 = (float)(t * C + (nl == 1 ? wj[u] : wj[u] / 3)) * invY2;
        float2* d = sm + wj[u] * 3 * a.ss + wi[u];
        d[0] = make_float2(v[u].x, v[u].y);
        d[a.ss] = make_float2(xi1 * v[u].z, xi1 * v[u].w);
        d[2 * a.ss] = make_float2(xi2 * v[u].z, xi2 * v[u].w);
      }
    }
    __syncthreads();
    spec_col_fft<true, PS>(sm, a.ss, n, Q, a.plan, a.tpc, a.tw);
    for (SpecWalk o(Q); o.i < n; o.next()) S3[o.i * rs * 3 + o.j] = sm[o.j * a.ss + o.i];
  } else {
    SpecWalk w(Q);
    while (w.i < n) {
      float2 v[kUnroll];
      int at[kUnroll];
#pragma unroll
      for (int u = 0; u < kUnroll; ++u) {
        at[u] = w.i < n ? w.j * a.ss + w.i : -1;
        if (w.i < n) v[u] = S3[w.i * rs * 3 + w.j];
        w.next();
      }
#pragma unroll
      for (int u = 0; u < kUnroll; ++u)
        if (at[u] >= 0) sm[at[u]] = v[u];
    }
    __syncthreads();
    spec_col_fft<false, PS>(sm, a.ss, n, Q, a.plan, a.tpc, a.tw);
    for (SpecWalk o(rc); o.i < n; o.next()) {
      const float xi1 = (float)signed_freq(o.i, n) * invY1;
      const float xi2 = (float)(t * C + (nl == 1 ? o.j : o.j / 3)) * invY2;
      const float2* s = sm + o.j * 3 * a.ss + o.i;
      const float2 s0 = s[0], s1 = s[a.ss], s2 = s[2 * a.ss];
      S2[o.i * rs + o.j] = make_float4(s0.x, s0.y, xi1 * s1.x + xi2 * s2.x, xi1 * s1.y + xi2 * s2.y);
    }
  }
}

// ----------------------------------------------------------------------------
// row pass: inverse line FFTs, tau = dL v at the nodes, forward line FFTs
// ----------------------------------------------------------------------------
struct SpecRowArgs {
  Geom g;
  SpecGeom sg;
  FFTPlan plan;                // along the last axis
  int tpl;                     // threads per line FFT
  int lpc;                     // lines per CTA (3-D: even)
  int ss;                      // distance between sequences in shared memory
  const float2* tw;
  float2* S;                   // D components per load, in place
  const uint8_t* phase;
  const float* tab;            // per-phase tensors, or nullptr
  int nphase;
  const float* in[kMaxLoads];  // kSpecRowLoad, kSpecRowAdd: fields
  float* out[kMaxLoads];       // kSpecRowAdd: results (may be the fields)
  Scal* scal;
};

enum : int {
  kSpecRowTau = 0,   // S <- F[dL F^-1 S] along the lines
  kSpecRowLoad = 1,  // S <- F in, or F[tab in] when there is a table
  kSpecRowAdd = 2    // out = in + F^-1 S, or in + tab F^-1 S
};

// Complex sequences: 2-D, one per (line, load), its two components as real and
// imaginary part; 3-D, one per (pair of lines, load, component), the two lines
// as real and imaginary part (no channel is left unpaired).
// Thread and residency limits of the row kernels: 80 registers for the 27
// complex values of a thread of a compile-time plan; the run-time plans'
// kernels, which hold every radix twice, spill at 80.
constexpr int kSpecRowCtThreads = 192;
template <typename PS> struct SpecRowBounds {
  static constexpr int threads = PlanLen<PS>::value > 0 ? kSpecRowCtThreads : kRowMaxThreads;
  static constexpr int blocks = PlanLen<PS>::value > 0 ? 4 : 1;
};

inline size_t spec_row_smem(int d, int nl, int lpc, int n, int ss, int nphase) {
  const size_t nseq = d == 2 ? lpc * nl : lpc / 2 * d * nl;
  return (nseq * ss + 1) / 2 * 16 + (size_t)nphase * d * d * sizeof(float) + (size_t)lpc * n;
}

template <int D, int NL, int MODE, typename PS = DynPlan>
__global__ void __launch_bounds__(SpecRowBounds<PS>::threads, SpecRowBounds<PS>::blocks) k_spec_row(SpecRowArgs a) {
  seq_begin();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2* sm = reinterpret_cast<float2*>(smem_raw);
  const Geom& g = a.g;
  constexpr int M = D * NL;
  const int n = plan_len<PS>(a.plan);
  const int nthr = blockDim.x, tpl = spec_threads<PS>(a.tpl), lpc = a.lpc, H = g.H, Hp = a.sg.Hp, ss = a.ss;
  const int nseq = D == 2 ? lpc * NL : (lpc / 2) * M;
  const int line0 = blockIdx.x * lpc;
  const int cell = g.ncell > 1 ? line0 / g.lines_cell : 0;
  if (MODE == kSpecRowTau && all_done(a.scal + cell * NL, NL)) return;
  float* const stab = reinterpret_cast<float*>(sm + (((size_t)nseq * ss + 1) & ~(size_t)1));  // 16-byte aligned
  uint8_t* const sph = reinterpret_cast<uint8_t*>(stab + a.nphase * D * D);
  if (MODE == kSpecRowTau || a.tab != nullptr) {
    const float* const tabc = a.tab + (size_t)cell * g.tab_stride;
    for (int i = threadIdx.x; i < a.nphase * D * D; i += nthr) stab[i] = tabc[i];
    // phases of the CTA's lines (consecutive in the image)
    const int lines = g.nlines - line0 < lpc ? g.nlines - line0 : lpc;
    const uint8_t* const ph = a.phase + (long long)line0 * n;
    for (int i = threadIdx.x; i < lines * n; i += nthr) sph[i] = ph[i];
  }

  constexpr int kUnroll = 4;
  if (MODE != kSpecRowLoad) {
    // 1. full spectra of the packed sequences from the half spectra
    if constexpr (D == 2) {
      for (int ll = 0; ll < lpc; ++ll) {
        const bool ok = line0 + ll < g.nlines;
        const float4* const src = reinterpret_cast<const float4*>(a.S) + (long long)(line0 + ll) * Hp * NL;
        for (int w0 = threadIdx.x; w0 < H * NL; w0 += kUnroll * nthr) {
          float4 v[kUnroll];
#pragma unroll
          for (int u = 0; u < kUnroll; ++u) {
            const int w = w0 + u * nthr;
            v[u] = (ok && w < H * NL) ? src[w] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
          }
#pragma unroll
          for (int u = 0; u < kUnroll; ++u) {
            const int w = w0 + u * nthr;
            if (w >= H * NL) continue;
            const int kx = w / NL, l = w - kx * NL;
            float2* const seq = sm + (size_t)(ll * NL + l) * ss;
            if (kx == 0 || 2 * kx == n) {  // bins that are their own Hermitian partner
              seq[kx] = make_float2(v[u].x, v[u].z);
            } else {
              seq[kx] = make_float2(v[u].x - v[u].w, v[u].y + v[u].z);
              seq[n - kx] = make_float2(v[u].x + v[u].w, v[u].z - v[u].y);
            }
          }
        }
      }
    } else {
      const int nw = (H * M + 1) / 2;  // 16-byte words that hold the half spectrum (the line is padded)
      for (int lp = 0; lp < lpc / 2; ++lp) {
        const int line = line0 + 2 * lp;
        const float4* const srcA = reinterpret_cast<const float4*>(a.S + (long long)line * Hp * M);
        const float4* const srcB = srcA + (long long)Hp * M / 2;
        const bool okA = line < g.nlines, okB = line + 1 < g.nlines;
        for (int w0 = threadIdx.x; w0 < nw; w0 += kUnroll * nthr) {
          float4 va[kUnroll], vb[kUnroll];
#pragma unroll
          for (int u = 0; u < kUnroll; ++u) {
            const int w = w0 + u * nthr;
            va[u] = (okA && w < nw) ? srcA[w] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            vb[u] = (okB && w < nw) ? srcB[w] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
          }
#pragma unroll
          for (int u = 0; u < kUnroll; ++u) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const int c = 2 * (w0 + u * nthr) + h;
              const int kx = c / M, m = c - kx * M;
              if (kx >= H) continue;
              const float2 ya = h ? make_float2(va[u].z, va[u].w) : make_float2(va[u].x, va[u].y);
              const float2 yb = h ? make_float2(vb[u].z, vb[u].w) : make_float2(vb[u].x, vb[u].y);
              float2* const seq = sm + (size_t)(lp * M + m) * ss;
              if (kx == 0 || 2 * kx == n) {
                seq[kx] = make_float2(ya.x, yb.x);
              } else {
                seq[kx] = make_float2(ya.x - yb.y, ya.y + yb.x);
                seq[n - kx] = make_float2(ya.x + yb.y, yb.x - ya.y);
              }
            }
          }
        }
      }
    }
  } else {
    // 1. the fields' lines (polarised when there is a table) into the sequences
    if (a.tab != nullptr) __syncthreads();
    constexpr int kLines = D == 2 ? 1 : 2;   // lines packed into one sequence set
    constexpr int kUnrollF = 2;
    for (int lp = 0; lp < lpc / kLines; ++lp)
#pragma unroll
      for (int l = 0; l < NL; ++l) {
        const float* const src = a.in[l];
        for (int i0 = threadIdx.x; i0 < n; i0 += kUnrollF * nthr) {
          float v[kUnrollF][kLines][D];
#pragma unroll
          for (int u = 0; u < kUnrollF; ++u)
#pragma unroll
            for (int h = 0; h < kLines; ++h)
#pragma unroll
              for (int c = 0; c < D; ++c) {
                const int i = i0 + u * nthr, line = line0 + lp * kLines + h;
                v[u][h][c] = (i < n && line < g.nlines) ? __ldg(src + c * g.nodes + (long long)line * n + i) : 0.0f;
              }
#pragma unroll
          for (int u = 0; u < kUnrollF; ++u) {
            const int i = i0 + u * nthr;
            if (i >= n) continue;
            if (a.tab != nullptr) {
#pragma unroll
              for (int h = 0; h < kLines; ++h) {
                const int ll = lp * kLines + h;
                const float* const row = stab + (line0 + ll < g.nlines ? sph[ll * n + i] : 0) * (D * D);
                float t[D];
#pragma unroll
                for (int c = 0; c < D; ++c) {
                  t[c] = 0.0f;
#pragma unroll
                  for (int b2 = 0; b2 < D; ++b2) t[c] += row[c * D + b2] * v[u][h][b2];
                }
#pragma unroll
                for (int c = 0; c < D; ++c) v[u][h][c] = t[c];
              }
            }
            if constexpr (D == 2) {
              sm[(size_t)(lp * NL + l) * ss + i] = make_float2(v[u][0][0], v[u][0][1]);
            } else {
#pragma unroll
              for (int c = 0; c < D; ++c)
                sm[(size_t)(lp * M + l * D + c) * ss + i] = make_float2(v[u][0][c], v[u][kLines - 1][c]);
            }
          }
        }
      }
  }
  __syncthreads();

  const int s = threadIdx.x / tpl;
  const int u = s < nseq ? threadIdx.x - s * tpl : n;  // idle threads never touch smem
  float2* const seq = sm + (size_t)(s < nseq ? s : 0) * ss;
  if constexpr (MODE == kSpecRowLoad) {
    fft_plan<false, float, PS>(seq, 1, a.plan, u, tpl, a.tw);
  } else if constexpr (MODE == kSpecRowAdd) {
    fft_plan<true, float, PS>(seq, 1, a.plan, u, tpl, a.tw);
    constexpr int kUnrollF = 2;
    for (int ll = 0; ll < lpc; ++ll) {
      if (line0 + ll >= g.nlines) break;
      const long long lo = (long long)(line0 + ll) * n;
#pragma unroll
      for (int l = 0; l < NL; ++l)
        for (int i0 = threadIdx.x; i0 < n; i0 += kUnrollF * nthr) {
          float e[kUnrollF][D];
#pragma unroll
          for (int q = 0; q < kUnrollF; ++q)
#pragma unroll
            for (int c = 0; c < D; ++c) {
              const int i = i0 + q * nthr;
              e[q][c] = i < n ? a.in[l][c * g.nodes + lo + i] : 0.0f;
            }
#pragma unroll
          for (int q = 0; q < kUnrollF; ++q) {
            const int i = i0 + q * nthr;
            if (i >= n) continue;
            float y[D];
            if constexpr (D == 2) {
              const float2 v = sm[(size_t)(ll * NL + l) * ss + i];
              y[0] = v.x;
              y[1] = v.y;
            } else {
#pragma unroll
              for (int c = 0; c < D; ++c)
                y[c] = reinterpret_cast<const float*>(sm + (size_t)((ll / 2) * M + l * D + c) * ss + i)[ll & 1];
            }
            if (a.tab != nullptr) {
              const float* const row = stab + sph[ll * n + i] * (D * D);
              float t[D];
#pragma unroll
              for (int c = 0; c < D; ++c) {
                t[c] = 0.0f;
#pragma unroll
                for (int b2 = 0; b2 < D; ++b2) t[c] += row[c * D + b2] * y[b2];
              }
#pragma unroll
              for (int c = 0; c < D; ++c) y[c] = t[c];
            }
#pragma unroll
            for (int c = 0; c < D; ++c) a.out[l][c * g.nodes + lo + i] = e[q][c] + y[c];
          }
        }
    }
    return;
  } else if constexpr (D == 2) {
    // 2. both components of a load are in one sequence: the polarisation is
    // applied in registers between the last inverse and the first forward stage
    const int ll = s < nseq ? s / NL : 0;
    const uint8_t* const ph = sph + (line0 + ll < g.nlines ? ll : 0) * n;
    auto mid = [&](float2 v, int i, bool act) -> float2 {
      const float4 t = reinterpret_cast<const float4*>(stab)[act ? ph[i] : 0];
      return make_float2(t.x * v.x + t.y * v.y, t.z * v.x + t.w * v.y);
    };
    fft_mirror_plan<float, PS>(seq, 1, a.plan, u, tpl, a.tw, mid);
  } else {
    fft_plan<true, float, PS>(seq, 1, a.plan, u, tpl, a.tw);
    for (int lp = 0; lp < lpc / 2; ++lp) {
      if (line0 + 2 * lp >= g.nlines) break;
      const uint8_t* const pa = sph + 2 * lp * n;
      const uint8_t* const pb = line0 + 2 * lp + 1 < g.nlines ? pa + n : pa;
      float2* const base = sm + (size_t)lp * M * ss;
      for (int i = threadIdx.x; i < n; i += nthr) {
        const float* const ta = stab + pa[i] * 9;
        const float* const tb = stab + pb[i] * 9;
#pragma unroll
        for (int l = 0; l < NL; ++l) {
          float2 v[3];
#pragma unroll
          for (int c = 0; c < 3; ++c) v[c] = base[(l * 3 + c) * ss + i];
#pragma unroll
          for (int c = 0; c < 3; ++c)
            base[(l * 3 + c) * ss + i] = make_float2(ta[3 * c] * v[0].x + ta[3 * c + 1] * v[1].x + ta[3 * c + 2] * v[2].x,
                                                    tb[3 * c] * v[0].y + tb[3 * c + 1] * v[1].y + tb[3 * c + 2] * v[2].y);
        }
      }
    }
    __syncthreads();
    fft_plan<false, float, PS>(seq, 1, a.plan, u, tpl, a.tw);
  }

  // 3. half spectra of the two real channels of each sequence
  if constexpr (D == 2) {
    for (int ll = 0; ll < lpc; ++ll) {
      if (line0 + ll >= g.nlines) break;
      float4* const dst = reinterpret_cast<float4*>(a.S) + (long long)(line0 + ll) * Hp * NL;
      for (int w = threadIdx.x; w < Hp * NL; w += nthr) {
        const int kx = w / NL, l = w - kx * NL;
        float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (kx < H) {
          const float2* const sq = sm + (size_t)(ll * NL + l) * ss;
          const float2 z1 = sq[kx], z2 = sq[kx == 0 ? 0 : n - kx];
          v = make_float4(0.5f * (z1.x + z2.x), 0.5f * (z1.y - z2.y), 0.5f * (z1.y + z2.y), 0.5f * (z2.x - z1.x));
        }
        dst[w] = v;
      }
    }
  } else {
    for (int lp = 0; lp < lpc / 2; ++lp) {
      const int line = line0 + 2 * lp;
      if (line >= g.nlines) break;
      const bool okB = line + 1 < g.nlines;
      float4* const dstA = reinterpret_cast<float4*>(a.S + (long long)line * Hp * M);
      float4* const dstB = dstA + (long long)Hp * M / 2;
      for (int w = threadIdx.x; w < Hp * M / 2; w += nthr) {
        float4 va, vb;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int c = 2 * w + h;
          const int kx = c / M, m = c - kx * M;
          float2 ya = make_float2(0.0f, 0.0f), yb = ya;
          if (kx < H) {
            const float2* const sq = sm + (size_t)(lp * M + m) * ss;
            const float2 z1 = sq[kx], z2 = sq[kx == 0 ? 0 : n - kx];
            ya = make_float2(0.5f * (z1.x + z2.x), 0.5f * (z1.y - z2.y));
            yb = make_float2(0.5f * (z1.y + z2.y), 0.5f * (z2.x - z1.x));
          }
          if (h) {
            va.z = ya.x; va.w = ya.y; vb.z = yb.x; vb.w = yb.y;
          } else {
            va.x = ya.x; va.y = ya.y; vb.x = yb.x; vb.y = yb.y;
          }
        }
        dstA[w] = va;
        if (okB) dstB[w] = vb;
      }
    }
  }
}

// alpha, beta and the stopping tests of one iteration; nfac = nodes per cell
// ((v, w) = nfac psi_b^2 sum_k conj(psi_v) psi_w).  A step's x update is applied by
// the next spec_inv, so a stopping item leaves it owed (xpend).
constexpr int kSpecScalThreads = 512;
static __global__ void __launch_bounds__(kSpecScalThreads) k_scal_spec(Scal* scal, const float4* part, int np, int ncell,
                                                                       int nl, double nfac) {
  seq_begin();
  const ItemRef r = item_ref(np, ncell, nl);
  if (!r.valid) return;
  Scal& s = scal[r.item];
  // what thread 0 needs afterwards is loaded together with the partial sums
  const int done = s.done, iter = s.iter, max_iter = s.max_iter;
  const double b2 = s.b2, tol2 = s.tol2, ib2 = s.ib2, back = s.psi_b;
  // warp w sums a share of row w % 4
  constexpr int kRows = 4, kShares = kSpecScalThreads / 32 / kRows;
  __shared__ Sum3 red[kRows][kShares];
  __shared__ double tot[kRows], inv[kRows];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, row = warp % kRows, share = warp / kRows;
  Sum3 v{0.0f, 0.0f, 0.0f};
  {
    const float4* const p = part + (long long)(row * kMaxLoads + r.l) * np + (long long)r.cell * r.bpc;
#pragma unroll 4
    for (int i = share * 32 + lane; i < r.bpc; i += kShares * 32) {
      const float4 q = p[i];
      v.add(q.x, q.y, q.z);
    }
  }
  v.warp_sum();
  if (lane == 0) red[row][share] = v;
  __syncthreads();
  // each row's float64 value and reciprocal in a warp of its own: a float64
  // operation of one thread costs tens of cycles here, and every kernel of the
  // next iteration waits for this one
  if (warp < kRows && lane == 0) {
    for (int q = 1; q < kShares; ++q) v.add(red[warp][q].s, red[warp][q].c, red[warp][q].r);
    tot[warp] = nfac * back * back * v.get();
    inv[warp] = 1.0 / tot[warp];
  }
  __syncthreads();
  if (threadIdx.x != 0 || done != kRunning) return;
  const double den = tot[0], aa = tot[1], ra = tot[2], rr = tot[3];
  s.xpend = 0;
  s.den = den;
  if (!finite_d(den) || !finite_d(aa) || !finite_d(ra) || !finite_d(rr) || den <= 0.0) {
    s.done = kBreakdown;
    return;
  }
  const double alpha = rr * inv[0];
  s.alpha = alpha;
  s.alpha_f = (float)alpha;
  s.xpend = 1;
  // below 1e-8 of (r, r) the expansion is the rounding of its float32 products
  const double rr_new = fmax(rr + alpha * (alpha * aa - 2.0 * ra), 1e-8 * rr);
  const double beta = rr > 0.0 ? rr_new * inv[3] : 0.0;
  s.iter = iter + 1;
  s.beta_f = (float)beta;
  s.rr = rr_new;
  s.rel = sqrt(rr_new * ib2);
  record_hist(s);
  if (!finite_d(rr_new)) { s.done = kBreakdown; return; }
  if (rr_new <= tol2 * b2) { s.done = kConverged; return; }
  if (iter + 1 >= max_iter) { s.done = kCap; return; }
  if (stalled(s)) s.done = kStalled;
}

// Partial sums of |M u psi|^2 over the full spectrum (single-cell, one load):
// |N| psi_b^2 times their sum is |M v|^2 of the field v.
static __global__ void k_spec_matnorm2(SpecArgs a, Mat3 m, double* part) {
  const int n = a.plan.n, C = a.sg.C, csh = a.sg.csh;
  const SpecTile tl = spec_tile(a, n);
  const int e = threadIdx.x & (C - 1), kl = tl.t * C + e;
  SpecFreq fq;
  fq.init(a, a.med[0], n, kl, tl.inner);
  const float xi1 = (float)(a.three ? signed_freq(tl.inner, a.g.n[1]) : kl) * a.sg.invY[1];
  const float xi2 = a.three ? (float)kl * a.sg.invY[2] : 0.0f;
  DotAcc<float> dot;
  const float2* const p = a.p[0] + tl.sbase + e;
  for (int i = threadIdx.x >> csh; i < n; i += blockDim.x >> csh) {
    const float x0 = fq.xi0(i), rn = fq.rnorm(i, x0);
    const float xi[3] = {x0 * rn, xi1 * rn, xi2 * rn};
    float q = 0.0f;
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      float t = 0.0f;
#pragma unroll
      for (int c = 0; c < 3; ++c) t += (float)m.v[r * 3 + c] * xi[c];
      q += t * t;
    }
    const float2 v = p[i << csh];
    dot.add(q * (v.x * v.x + v.y * v.y));
  }
  double acc[1] = {fq.wgt * dot.get()};
  block_reduce_store<1>(acc, 1, part, gridDim.x, blockIdx.x);
}

}  // namespace fh
