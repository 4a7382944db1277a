// fh_launch.cuh -- per (precision, dimension, load count) launch table.
// The pass kernels are templates over D (2 or 3) and NL (loads per launch);
// each combination is compiled in its own translation unit and reached
// through a table of host function pointers.
#pragma once

#include "fh_kernels.cuh"
#include "fh_spectral.cuh"

namespace fh {

struct Launch {
  int grid = 0, block = 0;
  size_t smem = 0;
  bool chain = false;  // seq_launch: one of the kernels of an iteration
};

// Launch of a kernel that starts with seq_begin().  In a chain the kernel's
// launch does not wait for the one before it to drain; its CTAs wait for that
// (and for its writes) in seq_begin(), so stream order is kept.  An iteration
// of 4 to 10 short kernels gains 2 to 4 % (405x675 refined 8.19 -> 7.85 ms,
// 81^2 float64 CG 1.44 -> 1.41 ms); single products gain nothing and launch
// plainly.  Letting the next kernel's CTAs in before this one's have ended was
// worse on small grids (405x675: 9.73 ms, 255^2 BiCG 10.6 instead of
// 9.9 ms): they take the SMs that are free, two to an SM, and leave the others
// idle.
template <typename... P, typename... A>
inline void seq_launch(void (*kernel)(P...), const Launch& L, size_t smem, cudaStream_t st, const A&... args) {
  if (!L.chain) {
    kernel<<<L.grid, L.block, smem, st>>>(args...);
    return;
  }
  cudaLaunchConfig_t c = {};
  c.gridDim = dim3((unsigned)L.grid);
  c.blockDim = dim3((unsigned)L.block);
  c.dynamicSmemBytes = smem;
  c.stream = st;
  cudaLaunchAttribute at = {};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  c.attrs = &at;
  c.numAttrs = 1;
  cudaLaunchKernelEx(&c, kernel, P(args)...);
}
// The scalar kernels of an iteration.
inline Launch chain_launch(int grid, int block) {
  Launch L;
  L.grid = grid;
  L.block = block;
  L.chain = true;
  return L;
}

template <typename T>
struct LaunchTable {
  int D = 0, NL = 0;
  cudaError_t (*set_smem)(size_t row_smem, size_t col0_smem, size_t col1_smem) = nullptr;
  cudaError_t (*row_fwd)(int pro, const Launch&, const RowArgs<T>&, cudaStream_t) = nullptr;
  cudaError_t (*row_inv)(int epi, const Launch&, const RowArgs<T>&, cudaStream_t) = nullptr;
  cudaError_t (*col)(int mode, const Launch&, const ColArgs<T>&, cudaStream_t) = nullptr;
  // persistent bulk-copy Green pass (2-D only; nullptr otherwise)
  cudaError_t (*col_pipe)(const Launch&, const ColArgs<T>&, cudaStream_t) = nullptr;
  cudaError_t (*set_smem_pipe)(size_t bytes) = nullptr;
  cudaError_t (*occupancy_pipe)(int block, size_t smem, int* per_sm) = nullptr;
  // 2-D float64 Green pass in double-float arithmetic (the refinement
  // residual); tw_df is the axis-0 twiddle table as complex double-floats.
  // nullptr for float and for 3-D.
  cudaError_t (*col_df)(const Launch&, const ColArgs<T>&, const void* tw_df, cudaStream_t) = nullptr;
  cudaError_t (*cg_update)(const Launch&, const VecArgs<T>&, cudaStream_t) = nullptr;
  cudaError_t (*cg_flush)(const Launch&, const VecArgs<T>&, cudaStream_t) = nullptr;
  cudaError_t (*bicg_update)(const Launch&, const VecArgs<T>&, cudaStream_t) = nullptr;
  cudaError_t (*current_sum)(const Launch&, const T*, const uint8_t*, const double*, long long nodes,
                             int ncell, long long cell_nodes, int tab_stride, double*,
                             cudaStream_t) = nullptr;
  cudaError_t (*matnorm2)(const Launch&, const T*, long long nodes, int ncell, long long cell_nodes,
                          const Mat3&, double*, cudaStream_t) = nullptr;
  // Length of the compile-time FFT plan that every pass kernel of a CG
  // iteration (direction pass, A p pass, Green pass and, in 3-D, the
  // middle-axis passes) runs for these plans and launch shapes, or 0 when at
  // least one of them runs a run-time-plan kernel.
  int (*ct_plan)(const FFTPlan& prow, const Launch& row, const FFTPlan& pc0, const Launch& col0,
                 const FFTPlan& pc1, const Launch& col1) = nullptr;
};

// Launchers of the frequency-domain CG iteration (fh_spectral.cuh, float32;
// fh_spec_*.cu).  *_smem raise the shared-memory limit of the kernels these
// arguments run; *_ct: does a compile-time plan kernel run the iteration's
// pass with this plan and launch?
cudaError_t spec_inv(int mode, const Launch&, const SpecArgs&, cudaStream_t);
cudaError_t spec_fwd(int mode, const Launch&, const SpecArgs&, cudaStream_t);
cudaError_t spec_green(const Launch&, const SpecArgs&, cudaStream_t);
cudaError_t spec_col_set_smem(const SpecArgs&, size_t bytes);
bool spec_col_ct(const FFTPlan&);
cudaError_t spec_mid(bool inv, const Launch&, const SpecMidArgs&, cudaStream_t);
cudaError_t spec_mid_set_smem(const SpecMidArgs&, size_t bytes);
bool spec_mid_ct(const FFTPlan&);
cudaError_t spec_row_d2(int mode, const Launch&, const SpecRowArgs&, cudaStream_t);
cudaError_t spec_row_d3(int mode, const Launch&, const SpecRowArgs&, cudaStream_t);
cudaError_t spec_row_d2_set_smem(const SpecRowArgs&, const Launch&);
cudaError_t spec_row_d3_set_smem(const SpecRowArgs&, const Launch&);
bool spec_row_d2_ct(const FFTPlan&, const Launch&);
bool spec_row_d3_ct(const FFTPlan&, const Launch&);

// Supported (D, NL): (2, 1), (2, 2), (3, 1), (3, 3).
LaunchTable<float> launch_table_f32_d2(int nl);
LaunchTable<float> launch_table_f32_d3(int nl);
LaunchTable<double> launch_table_f64_d2(int nl);
LaunchTable<double> launch_table_f64_d3(int nl);

template <typename T> LaunchTable<T> launch_table(int d, int nl);
template <> inline LaunchTable<float> launch_table<float>(int d, int nl) {
  return d == 2 ? launch_table_f32_d2(nl) : launch_table_f32_d3(nl);
}
template <> inline LaunchTable<double> launch_table<double>(int d, int nl) {
  return d == 2 ? launch_table_f64_d2(nl) : launch_table_f64_d3(nl);
}

}  // namespace fh
