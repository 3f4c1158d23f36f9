// Host side of the sampled quadrature (series_kernel.cuh).  Not a standalone
// header: phi_ops.cu includes it inside its host-side anonymous namespace,
// after queue_batch.
#pragma once

template <typename T, typename C>
SeriesView<T> series_view(const Plan& p, int g) {
  SeriesView<T> v;
  v.j0 = static_cast<const double*>(p.series_j0);
  v.tiles_a = static_cast<const uint4*>(p.series_j0);
  v.nodes = p.series_nodes;
  v.stride = p.series_stride;
  v.tiles = p.series_stride / kSeriesTile;
  v.max_panels = p.series_max_panels;
  v.max_intervals = p.series_max_intervals;
  v.support = p.d.support;
  v.inv_delta = static_cast<T>(4.0 * p.R);
  v.inv_delta_f = static_cast<float>(4.0 * p.R);
  v.inv_cycles = p.series_inv_cycles;
  v.tol = static_cast<T>(p.d.quad_abs_tol);
  v.retry = p.retry;
  v.n_retry = p.retry_counters + 2 * g;
  return v;
}

// The smallest absolute tolerance the estimate can meet: FP32 panel sums
// carry about 1e-7 of rounding, FP64 ones 1e-15.
template <typename T>
constexpr double series_least_tol() { return sizeof(T) == 4 ? 2.5e-7 : 1e-14; }

// Whether visibilities of supports up to jw may fail on their a-priori panels.
// Evaluated in 64 bits for supports J of 2 to 64 pixels, oversampling 1.25 to
// 3, windows of 0.25 to 1 cycles, offsets from 0 to those of J_w up to J + 60
// and tolerances from these limits to 1e-6 (FP64 1e-12), those that do have
// few panels for their J, nearly filled: at most J / 4 panels in FP32 (1 below
// 8) and J / 2 in FP64, of 0.7 of the a-priori width and more (FP32, J <= 4:
// 0.87; FP64 0.6, but for J = 2 at 1e-14).  With one panel more all but one of
// 28,000 combinations pass.
template <typename T>
bool series_may_fail(const Plan& p, int jw) {
  const bool f64 = sizeof(T) == 8;
  const int J = p.d.support, most = f64 ? std::max(2, J / 2) : std::max(1, J / 4);
  const double least = f64 ? 0.6 : J <= 4 ? 0.85 : 0.7;
  for (int w = J; w <= jw; w += 2) {
    const double want = p.R * (w * 0.70710678 + 0.5 * (w - J)) * p.series_inv_cycles;
    const double n = std::max(1.0, std::ceil(want));
    if (n > most) break;
    if (want > least * n) return true;
  }
  return false;
}

// J0 table for the panel counts and supports of this plan.  Panels no wider
// than the automatic width, so that a plan with wide panels of its own still
// passes the estimate.
template <typename T, typename C>
int build_series_tables_t(Plan& p, cudaStream_t s) {
  if (p.n_kept == 0 || p.d.quad_abs_tol < series_least_tol<T>()) return PHI_OK;
  p.series_inv_cycles =
      static_cast<float>(1.0 / std::min(p.cycles_per_panel, p.auto_cycles_per_panel));
  int panels = 1, intervals = 1;
  const float inv_delta = static_cast<float>(4.0 * p.R);
  // nothing to gain where no visibility fits the tables (the launch that finds
  // it out took 1.5% of the radial series' time at J_w 66 to 76, alpha 1.5)
  int least = p.d.support;
  if (p.d.support_rule == PHI_SUPPORT_STACK) {
    least = p.max_jw;
    for (int k = 0; k < p.K; ++k)
      if (p.stack_jw[k] > 0) least = std::min(least, p.stack_jw[k]);
  }
  if (series_intervals(least, inv_delta) > kSeriesMaxSamples - SeriesN<T>::half) return PHI_OK;
  for (int k = 0; k < p.K; ++k) {
    if (p.stack_jw[k] == 0) continue;
    intervals = std::max(intervals, series_intervals(p.stack_jw[k], inv_delta));
    panels = std::max(panels, series_panels(p.stack_jw[k], p.d.support, static_cast<float>(p.R),
                                            static_cast<float>(p.c_support), p.series_inv_cycles,
                                            static_cast<float>(p.stack_maxabs[k])));
  }
  p.series_again = series_may_fail<T>(p, p.max_jw);
  if (p.series_again) ++panels;
  p.series_max_panels = std::min(panels, kSeriesMaxPanels);
  p.series_max_intervals = std::min(intervals, kSeriesMaxSamples - SeriesN<T>::half);
  const int grain = sizeof(T) == 4 ? kSeriesTile : 32;   // samples of a tile, of a warp
  const int stride = (p.series_max_intervals + SeriesN<T>::half + grain - 1) / grain * grain;
  const int64_t rows = panel_table_offset(p.series_max_panels + 1);
  const int panel_rows = series_panel_base(p.series_max_panels + 1);
  const size_t table = sizeof(T) == 4 ? sizeof(uint4) * 128 * panel_rows * (stride / kSeriesTile)
                                      : sizeof(double) * rows * stride;
  void* raw = nullptr;
  PHI_CUDA_TRY(cudaMalloc(&raw, table));
  p.series_j0 = raw;
  p.device_bytes += static_cast<int64_t>(table);
  if (sizeof(T) == 4) {
    const size_t bytes = sizeof(float4) * 32 * panel_rows;
    PHI_CUDA_TRY(cudaMalloc(&raw, bytes));
    p.series_nodes = static_cast<float4*>(raw);
    p.device_bytes += static_cast<int64_t>(bytes);
  }
  PHI_CUDA_TRY(cudaMalloc(&raw, sizeof(uint32_t) * p.n_kept));
  p.retry = static_cast<uint32_t*>(raw);
  p.device_bytes += static_cast<int64_t>(sizeof(uint32_t) * p.n_kept);
  const int64_t items = sizeof(T) == 4 ? int64_t(panel_rows) * (stride / kSeriesTile) * 64
                                       : rows * stride;
  const int blocks = static_cast<int>(std::min<int64_t>((items + 127) / 128, p.num_sms * 16));
  if (sizeof(T) == 4)
    series_tile_kernel<<<blocks, 128, 0, s>>>(panel_rows, stride / kSeriesTile, p.node_omn,
                                              static_cast<const float*>(p.node_hk),
                                              static_cast<uint4*>(p.series_j0), p.series_nodes);
  else
    series_table_kernel<<<blocks, 128, 0, s>>>(rows, stride, static_cast<double*>(p.series_j0));
  PHI_CUDA_TRY(cudaGetLastError());
  p.series_stride = stride;
  return PHI_OK;
}

// Block shape: as many warps per block (at most 8) as keep the most warps
// resident, each with its own samples and polynomials and `extra` bytes; no
// warps when one does not fit.
struct SeriesShape {
  int warps = 0, blocks = 0, batch = 1;
  size_t smem = 0;
};
template <typename T, typename C, typename K>
int series_shape(const Plan& p, K kernel, int64_t n, size_t extra, SeriesShape& sh) {
  const size_t per_warp = series_warp_bytes<T>(p.series_stride, p.series_max_intervals) + extra;
  int dev = 0, optin = 0, per_sm_smem = 0, reserved = 0;
  PHI_CUDA_TRY(cudaGetDevice(&dev));
  PHI_CUDA_TRY(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
  PHI_CUDA_TRY(cudaDeviceGetAttribute(&per_sm_smem, cudaDevAttrMaxSharedMemoryPerMultiprocessor,
                                      dev));
  PHI_CUDA_TRY(cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev));
  int best = 0;
  for (int w = 1; w <= kVisThreads / 32; ++w) {
    const size_t blk = per_warp * w;
    if (blk > static_cast<size_t>(optin)) break;
    const int resident = w * static_cast<int>(per_sm_smem / (blk + reserved));
    if (resident >= best) {
      best = resident;
      sh.warps = w;
    }
  }
  if (sh.warps == 0) return PHI_OK;
  sh.smem = per_warp * sh.warps;
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, 32 * sh.warps, sh.smem) !=
          cudaSuccess ||
      per_sm < 1)
    per_sm = 1;
  sh.blocks = per_sm * p.num_sms;
  // FP32 samples the visibilities of a batch four at a time: batches of a
  // multiple of four once there are several to a warp, smaller ones before
  // that, so that every warp has work
  const int64_t warps = static_cast<int64_t>(sh.blocks) * sh.warps;
  sh.batch = queue_batch(n, warps);
  if (SeriesVis<T>::n > 1) {
    if (sh.batch < 4)
      sh.batch = static_cast<int>(std::min<int64_t>(4, std::max<int64_t>(1, n / (2 * warps))));
    else
      sh.batch = sh.batch / 4 * 4;
  }
  return PHI_OK;
}

// The fused kernel over nk records (the plan's records from b0 on).
template <typename T, typename C, bool kGrid>
int launch_series(Plan& p, int g, const VisRec<T>* recs, int64_t b0, int64_t nk, const C* grids_in,
                  C* grids_out, const C* vis_in, C* vis_out, cudaStream_t s) {
  SeriesShape sh;
  constexpr bool f64 = sizeof(T) == 8;
  auto kernel = p.series_again ? vis_series_kernel<T, C, kGrid, true>
                               : vis_series_kernel<T, C, kGrid, f64>;
  PHI_TRY_ST((series_shape<T, C>(p, kernel, nk, 0, sh)));
  if (sh.warps == 0) return PHI_ERR_SUPPORT;   // not reached: one warp takes 31 KB at most
  kernel<<<sh.blocks, 32 * sh.warps, sh.smem, s>>>(
      recs, p.perm + b0, nk, grids_in, grids_out, vis_in, vis_out, p.quad(),
      series_view<T, C>(p, g), p.stack_slot_dev, p.counters + g, p.counters + p.K, sh.batch);
  PHI_CUDA_TRY(cudaGetLastError());
  return PHI_OK;
}
