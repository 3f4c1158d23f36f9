// Host launchers of the chirp transforms (czt_kernel.cuh).  Not a standalone
// header: phi_ops.cu includes it inside its host-side anonymous namespace,
// after fft_launch.cuh.
#pragma once

template <int kLog>
int czt_pass_log(Plan& p, FftPass pass, const int32_t* stacks, int n, const float* x_in,
                 float2* grids, float* x_out, int accumulate, cudaStream_t s) {
  constexpr int row_threads = fft_row_threads<kLog>(), col_threads = czt_col_threads<kLog>();
  constexpr size_t row_smem = sizeof(float2) * fft_rows<kLog>() * fft_row_elems<kLog>();
  constexpr size_t col_smem = sizeof(float2) * czt_cols<kLog>() * czt_col_elems<kLog>();
  const int N = p.N;
  const dim3 rows(n, (N + fft_rows<kLog>() - 1) / fft_rows<kLog>());
  const dim3 cols((2 * N + czt_cols<kLog>() - 1) / czt_cols<kLog>(), n);
  const auto* omn = static_cast<const typename PixelPhase<float>::omn*>(p.omn_pix);
  const float* corr = static_cast<const float*>(p.corr_pix);
  const float2* tab = static_cast<const float2*>(p.fft_tab);
  switch (pass) {
    case kFftRowsForward:
      czt_rows_forward_kernel<kLog><<<rows, row_threads, row_smem, s>>>(x_in, omn, corr, p.wbar_dev,
                                                                        stacks, tab, N, grids);
      break;
    case kFftColsForward:
      czt_cols_forward_kernel<kLog><<<cols, col_threads, col_smem, s>>>(tab, N, grids);
      break;
    case kFftColsAdjoint:
      czt_cols_adjoint_kernel<kLog><<<cols, col_threads, col_smem, s>>>(tab, N, grids);
      break;
    case kFftRowsAdjoint: {
      const int groups = std::min(n, czt_adjoint_groups<kLog>());
      czt_rows_adjoint_kernel<kLog><<<rows.y, groups * row_threads, groups * row_smem, s>>>(
          grids, omn, corr, p.wbar_dev, stacks, n, tab, N, x_out, accumulate);
      break;
    }
  }
  PHI_CUDA_TRY(cudaGetLastError());
  return PHI_OK;
}

int czt_pass(Plan& p, FftPass pass, const int32_t* stacks, int n, const float* x_in, float2* grids,
             float* x_out, int accumulate, cudaStream_t s) {
  switch (p.czt_log) {
    case 10: return czt_pass_log<10>(p, pass, stacks, n, x_in, grids, x_out, accumulate, s);
    case 11: return czt_pass_log<11>(p, pass, stacks, n, x_in, grids, x_out, accumulate, s);
    default: return czt_pass_log<12>(p, pass, stacks, n, x_in, grids, x_out, accumulate, s);
  }
}

// The plan's table, and the column kernels' shared memory limits (fixed per
// kernel, the same for every plan).
template <int kLog>
int czt_setup_log(Plan& p, cudaStream_t s) {
  constexpr int M = 1 << kLog, roots = czt_roots(kLog);
  const int N = p.N;
  float2* tab = static_cast<float2*>(p.fft_tab);
  float2* c = tab + roots;
  float2* spec = c + 2 * N;
  double* cosm = reinterpret_cast<double*>(spec + M);
  double2* chirp = reinterpret_cast<double2*>(cosm + M);
  fft_table_kernel<float, float2><<<(roots + 255) / 256, 256, 0, s>>>(kLog, tab);
  czt_factors_kernel<<<(M + 127) / 128, 128, 0, s>>>(N, M, c, cosm, chirp);
  czt_spectrum_kernel<<<M, 128, 0, s>>>(N, M, cosm, chirp, spec);
  PHI_CUDA_TRY(cudaGetLastError());
  const cudaFuncAttribute a = cudaFuncAttributeMaxDynamicSharedMemorySize;
  const int col = static_cast<int>(sizeof(float2) * czt_cols<kLog>() * czt_col_elems<kLog>());
  PHI_CUDA_TRY(cudaFuncSetAttribute(czt_cols_forward_kernel<kLog>, a, col));
  PHI_CUDA_TRY(cudaFuncSetAttribute(czt_cols_adjoint_kernel<kLog>, a, col));
  return PHI_OK;
}
int czt_setup(Plan& p, cudaStream_t s) {
  switch (p.czt_log) {
    case 10: return czt_setup_log<10>(p, s);
    case 11: return czt_setup_log<11>(p, s);
    default: return czt_setup_log<12>(p, s);
  }
}
