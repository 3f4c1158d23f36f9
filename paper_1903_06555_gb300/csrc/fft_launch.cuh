// Host launchers of the two-pass transforms (fft_kernel.cuh).  Not a
// standalone header: phi_ops.cu includes it inside its host-side anonymous
// namespace, after PHI_TRY_ST.
#pragma once

enum FftPass { kFftRowsForward, kFftColsForward, kFftColsAdjoint, kFftRowsAdjoint };

template <typename T, typename C, int kLog>
int fft_pass_log(Plan& p, FftPass pass, const int32_t* stacks, int n, const T* x_in, C* grids,
                 T* x_out, int accumulate, cudaStream_t s) {
  constexpr int N = 1 << kLog;
  constexpr int row_threads = fft_row_threads<kLog>(), col_threads = fft_col_threads<kLog, T>();
  constexpr size_t row_smem = sizeof(C) * fft_rows<kLog>() * fft_row_elems<kLog>();
  constexpr size_t col_smem = sizeof(C) * fft_cols<kLog, T>() * fft_col_elems<kLog, T>();
  const dim3 rows(n, N / fft_rows<kLog>()), cols(2 * N / fft_cols<kLog, T>(), n);
  const auto* omn = static_cast<const typename PixelPhase<T>::omn*>(p.omn_pix);
  const T* corr = static_cast<const T*>(p.corr_pix);
  const C* tab = static_cast<const C*>(p.fft_tab);
  switch (pass) {
    case kFftRowsForward:
      fft_rows_forward_kernel<T, C, kLog><<<rows, row_threads, row_smem, s>>>(
          x_in, omn, corr, p.wbar_dev, stacks, tab, grids);
      break;
    case kFftColsForward:
      fft_cols_forward_kernel<T, C, kLog><<<cols, col_threads, col_smem, s>>>(tab, grids);
      break;
    case kFftColsAdjoint:
      fft_cols_adjoint_kernel<T, C, kLog><<<cols, col_threads, col_smem, s>>>(tab, grids);
      break;
    case kFftRowsAdjoint:
      fft_rows_adjoint_kernel<T, C, kLog><<<rows.y, row_threads, row_smem, s>>>(
          grids, omn, corr, p.wbar_dev, stacks, n, tab, x_out, accumulate);
      break;
  }
  PHI_CUDA_TRY(cudaGetLastError());
  return PHI_OK;
}

template <typename T, typename C>
int fft_pass(Plan& p, FftPass pass, const int32_t* stacks, int n, const T* x_in, C* grids,
             T* x_out, int accumulate, cudaStream_t s) {
  switch (p.fft_log) {
    case 6: return fft_pass_log<T, C, 6>(p, pass, stacks, n, x_in, grids, x_out, accumulate, s);
    case 7: return fft_pass_log<T, C, 7>(p, pass, stacks, n, x_in, grids, x_out, accumulate, s);
    case 8: return fft_pass_log<T, C, 8>(p, pass, stacks, n, x_in, grids, x_out, accumulate, s);
    case 9: return fft_pass_log<T, C, 9>(p, pass, stacks, n, x_in, grids, x_out, accumulate, s);
    case 10: return fft_pass_log<T, C, 10>(p, pass, stacks, n, x_in, grids, x_out, accumulate, s);
    default: return fft_pass_log<T, C, 11>(p, pass, stacks, n, x_in, grids, x_out, accumulate, s);
  }
}

// Dynamic shared memory limits (fixed per kernel, the same for every plan).
template <typename T, typename C, int kLog>
int set_fft_smem_log() {
  const cudaFuncAttribute a = cudaFuncAttributeMaxDynamicSharedMemorySize;
  const int row = static_cast<int>(sizeof(C) * fft_rows<kLog>() * fft_row_elems<kLog>());
  const int col = static_cast<int>(sizeof(C) * fft_cols<kLog, T>() * fft_col_elems<kLog, T>());
  PHI_CUDA_TRY(cudaFuncSetAttribute(fft_rows_forward_kernel<T, C, kLog>, a, row));
  PHI_CUDA_TRY(cudaFuncSetAttribute(fft_rows_adjoint_kernel<T, C, kLog>, a, row));
  PHI_CUDA_TRY(cudaFuncSetAttribute(fft_cols_forward_kernel<T, C, kLog>, a, col));
  PHI_CUDA_TRY(cudaFuncSetAttribute(fft_cols_adjoint_kernel<T, C, kLog>, a, col));
  return PHI_OK;
}
template <typename T, typename C>
int set_fft_smem() {
  PHI_TRY_ST((set_fft_smem_log<T, C, 6>()));
  PHI_TRY_ST((set_fft_smem_log<T, C, 7>()));
  PHI_TRY_ST((set_fft_smem_log<T, C, 8>()));
  PHI_TRY_ST((set_fft_smem_log<T, C, 9>()));
  PHI_TRY_ST((set_fft_smem_log<T, C, 10>()));
  PHI_TRY_ST((set_fft_smem_log<T, C, 11>()));
  return PHI_OK;
}
