// Host launchers of the two-pass transforms (fft_kernel.cuh).  Not a
// standalone header: phi_ops.cu includes it inside its host-side anonymous
// namespace, after PHI_TRY_ST.
#pragma once

enum FftPass { kFftRowsForward, kFftColsForward, kFftColsAdjoint, kFftRowsAdjoint };

// Shared memory of a column block: two tile buffers, the exchange, and room
// to align them.
template <typename T, typename C, int kLog>
constexpr size_t fft_col_smem() {
  return 128 + sizeof(C) * fft_cols<kLog, T>() *
                   (2 * (size_t(1) << kLog) + fft_col_elems<kLog, T>());
}

// The tensor maps of the plan's grids (fft_kernel.cuh says what they show).
template <typename T, typename C, int kLog>
int fft_make_maps_log(Plan& p) {
  constexpr uint64_t N = uint64_t(1) << kLog, row = 2 * N * sizeof(C);
  constexpr uint32_t kBox = N < 256 ? N : 256;
  constexpr uint32_t unit = sizeof(C) / 8;   // 8-byte elements per grid value
  void* fn = nullptr;
  cudaDriverEntryPointQueryResult found;
  PHI_CUDA_TRY(cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000,
                                                cudaEnableDefault, &found));
  if (found != cudaDriverEntryPointSuccess || !fn) return PHI_ERR_CUDA;
  typedef CUresult (*Encode)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                             const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                             const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                             CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
  auto encode = [&](CUtensorMap* map, int rank, const cuuint64_t* dims, const cuuint64_t* strides,
                    const cuuint32_t* box) {
    const cuuint32_t one[4] = {1, 1, 1, 1};
    return reinterpret_cast<Encode>(fn)(
               map, CU_TENSOR_MAP_DATA_TYPE_FLOAT64, rank, p.grid, dims, strides, box, one,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
               CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS
               ? PHI_OK
               : PHI_ERR_CUDA;
  };
  const uint64_t grids = static_cast<uint64_t>(p.group);
  const cuuint64_t idims[3] = {2 * N * unit, N, grids}, istr[2] = {row, 2 * N * row};
  const cuuint32_t ibox[3] = {fft_cols<kLog, T>() * unit, kBox, 1};
  PHI_TRY_ST(encode(&p.fft_maps.image, 3, idims, istr, ibox));
  const cuuint64_t hdims[4] = {2 * N * unit, N, 2, grids};
  const cuuint64_t hstr[3] = {2 * row, row, 2 * N * row};
  const cuuint32_t hbox[4] = {fft_cols<kLog, T>() * unit, kBox, 1, 1};
  return encode(&p.fft_maps.half, 4, hdims, hstr, hbox);
}

template <typename T, typename C, int kLog>
int fft_pass_log(Plan& p, FftPass pass, const int32_t* stacks, int n, const T* x_in, C* grids,
                 T* x_out, int accumulate, cudaStream_t s) {
  constexpr int N = 1 << kLog;
  constexpr int row_threads = fft_row_threads<kLog>(), col_threads = fft_col_threads<kLog, T>();
  constexpr size_t row_smem = sizeof(C) * fft_rows<kLog>() * fft_row_elems<kLog>();
  constexpr size_t col_smem = fft_col_smem<T, C, kLog>();
  const dim3 rows(n, N / fft_rows<kLog>());
  const int tiles = 2 * N / fft_cols<kLog, T>() * n;
  int* timeout = reinterpret_cast<int*>(p.counters + p.K + 4);
  auto cols = [&](auto kernel) {   // as many blocks as run at once, and no more than tiles
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, col_threads, col_smem) !=
            cudaSuccess ||
        per_sm < 1)
      per_sm = 1;
    return std::min(tiles, per_sm * p.num_sms);
  };
  const auto* omn = static_cast<const typename PixelPhase<T>::omn*>(p.omn_pix);
  const T* corr = static_cast<const T*>(p.corr_pix);
  const C* tab = static_cast<const C*>(p.fft_tab);
  switch (pass) {
    case kFftRowsForward:
      fft_rows_forward_kernel<T, C, kLog><<<rows, row_threads, row_smem, s>>>(
          x_in, omn, corr, p.wbar_dev, stacks, tab, grids);
      break;
    case kFftColsForward:
      fft_cols_forward_kernel<T, C, kLog>
          <<<cols(fft_cols_forward_kernel<T, C, kLog>), col_threads, col_smem, s>>>(
              tab, p.fft_maps, grids, tiles, p.fft_wait_limit, timeout);
      break;
    case kFftColsAdjoint:
      fft_cols_adjoint_kernel<T, C, kLog>
          <<<cols(fft_cols_adjoint_kernel<T, C, kLog>), col_threads, col_smem, s>>>(
              tab, p.fft_maps, grids, tiles, p.fft_wait_limit, timeout);
      break;
    case kFftRowsAdjoint: {
      // sets of threads for the stacks while the sets of all blocks fit the
      // chip at once (12 warps per SM of 170 registers)
      int groups = 1;
      while (2 * groups <= fft_adjoint_groups<kLog, T>() && groups < n &&
             2 * groups * rows.y * (row_threads / 32) <= static_cast<unsigned>(12 * p.num_sms))
        groups *= 2;
      constexpr bool split = fft_adjoint_groups<kLog, T>() > 1;
      auto kernel = groups > 1 ? fft_rows_adjoint_kernel<T, C, kLog, split>
                               : fft_rows_adjoint_kernel<T, C, kLog, false>;
      kernel<<<rows.y, groups * row_threads, groups * row_smem, s>>>(
          grids, omn, corr, p.wbar_dev, stacks, n, tab, x_out, accumulate);
      break;
    }
  }
  PHI_CUDA_TRY(cudaGetLastError());
  return PHI_OK;
}

// call(log2 N as a constant) for the plan's size: 2^6 .. 2^11 in FP32, 2^9 ..
// 2^11 in FP64 (fft_log).
template <typename T, typename F>
int fft_dispatch(const Plan& p, F call) {
  if constexpr (sizeof(T) == 4) {
    switch (p.fft_log) {
      case 6: return call(std::integral_constant<int, 6>());
      case 7: return call(std::integral_constant<int, 7>());
      case 8: return call(std::integral_constant<int, 8>());
    }
  }
  switch (p.fft_log) {
    case 9: return call(std::integral_constant<int, 9>());
    case 10: return call(std::integral_constant<int, 10>());
    default: return call(std::integral_constant<int, 11>());
  }
}

template <typename T, typename C>
int fft_pass(Plan& p, FftPass pass, const int32_t* stacks, int n, const T* x_in, C* grids,
             T* x_out, int accumulate, cudaStream_t s) {
  return fft_dispatch<T>(p, [&](auto log) {
    return fft_pass_log<T, C, log.value>(p, pass, stacks, n, x_in, grids, x_out, accumulate, s);
  });
}

// Dynamic shared memory limits (fixed per kernel, the same for every plan) and
// the plan's tensor maps.
template <typename T, typename C, int kLog>
int fft_setup_log(Plan& p) {
  const cudaFuncAttribute a = cudaFuncAttributeMaxDynamicSharedMemorySize;
  const int row = static_cast<int>(sizeof(C) * fft_rows<kLog>() * fft_row_elems<kLog>());
  const int col = static_cast<int>(fft_col_smem<T, C, kLog>());
  PHI_CUDA_TRY(cudaFuncSetAttribute(fft_rows_forward_kernel<T, C, kLog>, a, row));
  constexpr int groups = fft_adjoint_groups<kLog, T>();
  PHI_CUDA_TRY(cudaFuncSetAttribute(fft_rows_adjoint_kernel<T, C, kLog, false>, a, row));
  if (groups > 1)
    PHI_CUDA_TRY(cudaFuncSetAttribute(fft_rows_adjoint_kernel<T, C, kLog, (groups > 1)>, a,
                                      groups * row));
  PHI_CUDA_TRY(cudaFuncSetAttribute(fft_cols_forward_kernel<T, C, kLog>, a, col));
  PHI_CUDA_TRY(cudaFuncSetAttribute(fft_cols_adjoint_kernel<T, C, kLog>, a, col));
  return fft_make_maps_log<T, C, kLog>(p);
}
template <typename T, typename C>
int fft_setup(Plan& p) {
  return fft_dispatch<T>(p, [&](auto log) { return fft_setup_log<T, C, log.value>(p); });
}
