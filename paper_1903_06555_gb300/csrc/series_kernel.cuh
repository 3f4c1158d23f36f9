// The quadrature with its taps' J0 factors interpolated in rho.  Not a
// standalone header: phi_ops.cu includes it inside namespace phi, after the
// quadrature, tap and work-queue pieces it uses.
//
// All J_w^2 taps of a visibility share the Gauss-Kronrod nodes r_j and their
// values h_j; they differ only in J0(2 pi rho r_j), a function of rho that is
// even and band-limited to R cycles per grid pixel.  So the sums over the
// nodes -- the Kronrod sums of every panel, and their differences from the
// embedded Gauss sums -- are formed at the samples rho_i = i / (4 R), twice
// the rate the sampling theorem asks for, with J0(2 pi rho_i r_j) = J0(pi i
// (2 p + 1 + x_k) / (4 P)) read from a table (it depends on the panel count P
// alone), and every tap's value is interpolated from the samples around it:
// per sample interval a polynomial in t = 2 (4 R rho - p) - 1, its
// coefficients the least-squares weights of series_fit.py (5.9e-8 at the
// band's edge in FP32, 1.2e-15 in FP64).  It is the same sum over the same
// nodes for every tap, in another order: per visibility 31 P (4 R rho_max +
// 10) products and a short polynomial per tap in place of 31 P J_w^2 Bessel
// functions.
//
// Tolerance.  The estimate E = sum over panels |K31 - G15| is formed at every
// sample.  Each panel's difference is band-limited like the kernel, and a
// function sampled at twice its Nyquist rate is bounded between the samples
// by 1 / cos(pi / 4) = 1.42 times its largest sample, so a visibility whose
// samples satisfy 1.5 E <= quad_abs_tol has every tap within the tolerance.
// The a-priori panels follow the support (the corner of the box and the
// largest |dw| the support covers), which leaves E two orders below 1e-6 at
// 6 cycles per panel.  A visibility that fails -- or needs more panels or
// samples than the tables hold -- is put on a list, and the kernel that
// integrates each tap by itself (vis_kernel and its companions), with its
// refinement and its count of unconverged taps, takes that list.
//
// Measured on the MWA-like snapshot (1.92M visibilities, J_w 26-40, FP32):
// 9.7 ms per degrid or grid launch where the per-tap kernel takes 63 and the
// 16-point radial series 18.6, and 3.9e-7 from the 64-bit operator (per tap
// 5.4e-7, radial series 9e-7: the table's J0 is rounded once, the per-tap
// kernel's polynomial and hardware cosine are not).  FP64 at 1e-12 (5,000
// visibilities, J_w 26): 1.0 ms, per tap 39 ms.  Bound: the shared-memory
// pipe (81% busy: four 16-byte entries per tap) and issue (70%).
#pragma once

#include "series_coef.cuh"

// Sample pairs and polynomial terms of the interpolation (series_fit.py).
template <typename T> struct SeriesN;
template <> struct SeriesN<float> { static constexpr int half = 10, terms = 8; };
template <> struct SeriesN<double> { static constexpr int half = 20, terms = 14; };

// Most samples per visibility (four per lane) and panels the tables hold.
constexpr int kSeriesMaxSamples = 128;
constexpr int kSeriesMaxPanels = 32;

// Sample intervals that cover the box of support J: its farthest tap lies
// within J / sqrt(2) of the visibility.
__host__ __device__ inline int series_intervals(int J, float inv_delta) {
  return static_cast<int>(static_cast<float>(J) * 0.70710678f * inv_delta) + 1;
}

// A-priori panels of a visibility: as initial_panels, for the corner of its
// box and the larger of its |dw| and the |dw| its support was sized for, so
// that visibilities of one support share their panels.
__host__ __device__ inline int series_panels(int J, int support, float Rf, float chirp_coeff,
                                             float inv_cycles, float adw) {
  const float chirp = fmaxf(adw * chirp_coeff, 0.5f * static_cast<float>(J - support));
  return panel_count_for(Rf * fmaf(static_cast<float>(J), 0.70710678f, chirp) * inv_cycles);
}

// J0(2 pi rho_i r_j) for sample i of panel-table row j: rows as the node
// tables (31 P rows for every panel count P), `stride` samples each; and, for
// FP32, each row's 1 - n(r_j) as the sum of two floats.
template <typename T>
__global__ void series_table_kernel(const double* __restrict__ omn, int64_t rows, int stride,
                                    T* __restrict__ j0_out, float2* __restrict__ omn2) {
  const int64_t total = rows * stride;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t row = e / stride;
    const int i = static_cast<int>(e - row * stride);
    int P = 1;
    while (panel_table_offset(P + 1) <= row) ++P;
    const int64_t local = row - panel_table_offset(P);
    const int p = static_cast<int>(local / kNodes), k = static_cast<int>(local % kNodes);
    j0_out[e] = static_cast<T>(j0(kPi * i * (2.0 * p + 1.0 + gk_node(k)) / (4.0 * P)));
    if (omn2 && i == 0) {
      const double v = omn[row];
      const float hi = static_cast<float>(v);
      omn2[row] = make_float2(hi, static_cast<float>(v - hi));
    }
  }
}

// Values of one node for the NV visibilities a warp samples together.
template <typename C, int NV> struct __align__(16) NodePack { C v[NV]; };

// e^{2 pi i dw (1 - n)}: FP32 forms the phase with dw and 1 - n as sums of
// two floats each (48 bits; the FP64 unit would take as long as the whole
// sampling), FP64 directly.
struct PhaseF {
  float hi, lo;
  __device__ __forceinline__ explicit PhaseF(double dw) {
    hi = static_cast<float>(dw);
    lo = static_cast<float>(dw - static_cast<double>(hi));
  }
  __device__ __forceinline__ float2 operator()(float2 omn) const {
    const float p = __fmul_rn(hi, omn.x);
    float e = fmaf(hi, omn.x, -p);
    e = fmaf(hi, omn.y, e);
    e = fmaf(lo, omn.x, e);
    float sn, cs;
    sincospif(2.0f * ((p - rintf(p)) + e), &sn, &cs);
    return make_float2(cs, sn);
  }
};
struct PhaseD {
  double dw;
  __device__ __forceinline__ explicit PhaseD(double w) : dw(w) {}
  __device__ __forceinline__ double2 operator()(double omn) const {
    double t = dw * omn;
    t -= rint(t);
    double sn, cs;
    sincospi(2.0 * t, &sn, &cs);
    return make_double2(cs, sn);
  }
};
template <typename T> struct PhaseOf;
template <> struct PhaseOf<float> { typedef PhaseF type; };
template <> struct PhaseOf<double> { typedef PhaseD type; };

// acc += J h for a real J.
__device__ __forceinline__ void rmad(float2& acc, float J, const float2& h) {
  acc = __ffma2_rn(make_float2(J, J), h, acc);
}
__device__ __forceinline__ void rmad(double2& acc, double J, const double2& h) {
  acc.x = fma(J, h.x, acc.x);
  acc.y = fma(J, h.y, acc.y);
}

// Kernel samples 0 .. 32 NS - 1 of NV visibilities with the same panel count
// P into smp (visibility v at smp + v * stride); ok[v]: the estimate passes at
// every sample of the box (sample intervals 0 .. NP - 1).  Per panel the
// lanes build its 31 node values (nk: Kronrod, ng: the 15 odd nodes with
// their Gauss weights), then each takes NS samples and walks the nodes, one
// table row per node; the NV visibilities share the row's loads.
template <typename T, typename C, int NV, int NS>
__device__ __forceinline__ void series_sample(NodePack<C, NV>* nk, NodePack<C, NV>* ng, C* smp,
                                              const SeriesView<T>& sv, const QuadParams& q,
                                              int P, const double (&dw)[NV], int NP,
                                              bool (&ok)[NV], int lane) {
  typedef typename PhaseOf<T>::type Phase;
  C K[NV][NS];
  T err[NV][NS];
#pragma unroll
  for (int v = 0; v < NV; ++v)
#pragma unroll
    for (int s = 0; s < NS; ++s) {
      K[v][s] = cmake<C>(0.0, 0.0);
      err[v][s] = T(0);
    }
  const int stride = sv.stride;
  const int64_t row0 = panel_table_offset(P);
  const T* __restrict__ tj = sv.j0 + row0 * stride + lane;
  for (int p = 0; p < P; ++p) {
    if (lane < kNodes) {
      const int64_t j = row0 + kNodes * p + lane;
      const T hk = static_cast<const T*>(q.node_hk)[j];
      T hg = static_cast<const T*>(q.node_hd)[j];
      if (sizeof(T) == 8) hg = hk - hg;   // the FP64 table holds the difference
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        C e;
        if constexpr (sizeof(T) == 4)
          e = Phase(dw[v])(sv.omn2[j]);
        else
          e = Phase(dw[v])(q.node_omn[j]);
        C h;
        h.x = hk * e.x;
        h.y = hk * e.y;
        nk[lane].v[v] = h;
        if (lane & 1) {
          h.x = hg * e.x;
          h.y = hg * e.y;
          ng[lane >> 1].v[v] = h;
        }
      }
    }
    __syncwarp();
    C A[NV][NS], G[NV][NS];
#pragma unroll
    for (int v = 0; v < NV; ++v)
#pragma unroll
      for (int s = 0; s < NS; ++s) A[v][s] = G[v][s] = cmake<C>(0.0, 0.0);
#pragma unroll 5
    for (int k = 0; k < (kNodes - 1) / 2; ++k) {
      const NodePack<C, NV> h0 = nk[2 * k], h1 = nk[2 * k + 1], g1 = ng[k];
#pragma unroll
      for (int s = 0; s < NS; ++s) {
        const T J0 = tj[32 * s], J1 = tj[stride + 32 * s];
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          rmad(A[v][s], J0, h0.v[v]);
          rmad(A[v][s], J1, h1.v[v]);
          rmad(G[v][s], J1, g1.v[v]);
        }
      }
      tj += 2 * stride;
    }
    {
      const NodePack<C, NV> h0 = nk[kNodes - 1];
#pragma unroll
      for (int s = 0; s < NS; ++s) {
        const T J0 = tj[32 * s];
#pragma unroll
        for (int v = 0; v < NV; ++v) rmad(A[v][s], J0, h0.v[v]);
      }
      tj += stride;
    }
#pragma unroll
    for (int v = 0; v < NV; ++v)
#pragma unroll
      for (int s = 0; s < NS; ++s) {
        K[v][s].x += A[v][s].x;
        K[v][s].y += A[v][s].y;
        const T dr = A[v][s].x - G[v][s].x, di = A[v][s].y - G[v][s].y;
        err[v][s] += est_sqrt(dr * dr + di * di);
      }
    __syncwarp();   // the node values are rewritten by the next panel
  }
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    bool good = true;
#pragma unroll
    for (int s = 0; s < NS; ++s) {
      smp[v * stride + 32 * s + lane] = K[v][s];
      if (32 * s + lane <= NP) good = good && T(1.5) * err[v][s] <= sv.tol;   // NaN fails
    }
    ok[v] = __all_sync(0xffffffffu, good);
  }
  __syncwarp();
}

// Where interval p's polynomial lies in an array of 16-byte entries: skewed
// by one entry in eight, so that intervals a stride of 1 or 2 apart (the taps
// of a row, from its middle to its ends) fall on different banks.
__device__ __forceinline__ int series_slot(int p) { return p + (p >> 3); }

// The polynomials of intervals 0 .. NP - 1 from the samples, two complex
// terms (FP32) or one (FP64) to a 16-byte entry, entry k of interval p at
// coef[k * slots + series_slot(p)].  One interval per lane.
__device__ __forceinline__ void series_polynomials(const float2* smp, float4* coef, int slots,
                                                   int NP, int lane) {
  constexpr int H = SeriesN<float>::half, M = SeriesN<float>::terms;
  for (int p = lane; p < NP; p += 32) {
    float2 c[M];
#pragma unroll
    for (int m = 0; m < M; ++m) c[m] = make_float2(0.f, 0.f);
#pragma unroll
    for (int d = 0; d < H; ++d) {
      const float2 lo = smp[abs(p - d)], hi = smp[p + 1 + d];
      const float2 sum = __fadd2_rn(hi, lo);
      const float2 dif = __fadd2_rn(hi, make_float2(-lo.x, -lo.y));
#pragma unroll
      for (int m = 0; m < M; ++m) c[m] = __ffma2_rn(c_series_f[m][d], (m & 1) ? dif : sum, c[m]);
    }
#pragma unroll
    for (int k = 0; k < M / 2; ++k)
      coef[k * slots + series_slot(p)] =
          make_float4(c[2 * k].x, c[2 * k].y, c[2 * k + 1].x, c[2 * k + 1].y);
  }
  __syncwarp();
}
__device__ __forceinline__ void series_polynomials(const double2* smp, double2* coef, int slots,
                                                   int NP, int lane) {
  constexpr int H = SeriesN<double>::half, M = SeriesN<double>::terms;
  for (int p = lane; p < NP; p += 32) {
    double2 c[M];
#pragma unroll
    for (int m = 0; m < M; ++m) c[m] = make_double2(0.0, 0.0);
#pragma unroll 2
    for (int d = 0; d < H; ++d) {
      const double2 lo = smp[abs(p - d)], hi = smp[p + 1 + d];
      const double2 sum = make_double2(hi.x + lo.x, hi.y + lo.y);
      const double2 dif = make_double2(hi.x - lo.x, hi.y - lo.y);
#pragma unroll
      for (int m = 0; m < M; ++m) {
        const double2 f = (m & 1) ? dif : sum;
        c[m].x = fma(c_series_d[m][d], f.x, c[m].x);
        c[m].y = fma(c_series_d[m][d], f.y, c[m].y);
      }
    }
#pragma unroll
    for (int k = 0; k < M; ++k) coef[k * slots + series_slot(p)] = c[k];
  }
  __syncwarp();
}

// [GC] at rho from the polynomials (last = NP - 1; a rho at the far end that
// rounds past it extrapolates the last interval).
__device__ __forceinline__ float2 series_eval(const float4* coef, int slots, int last,
                                              float last_f, float inv_delta, float rho) {
  int ip;
  float fr;
  table_index(rho * inv_delta, last, last_f, ip, fr);
  const float t = fmaf(2.0f, fr, -1.0f);
  const float2 t2 = make_float2(t, t);
  const float4* e = coef + series_slot(ip);
  float4 a = e[3 * slots];
  float2 k = __ffma2_rn(make_float2(a.z, a.w), t2, make_float2(a.x, a.y));
#pragma unroll
  for (int j = 2; j >= 0; --j) {
    a = e[j * slots];
    k = __ffma2_rn(k, t2, make_float2(a.z, a.w));
    k = __ffma2_rn(k, t2, make_float2(a.x, a.y));
  }
  return k;
}
__device__ __forceinline__ double2 series_eval(const double2* coef, int slots, int last,
                                               double last_f, double inv_delta, double rho) {
  int ip;
  double fr;
  table_index(rho * inv_delta, last, last_f, ip, fr);
  const double t = fma(2.0, fr, -1.0);
  const double2* e = coef + series_slot(ip);
  constexpr int M = SeriesN<double>::terms;
  double2 k = e[(M - 1) * slots];
#pragma unroll
  for (int j = M - 2; j >= 0; --j) {
    const double2 a = e[j * slots];
    k.x = fma(k.x, t, a.x);
    k.y = fma(k.y, t, a.y);
  }
  return k;
}

// One warp's shared memory: the node values, the samples, the polynomials.
template <typename T> struct SeriesEntry;
template <> struct SeriesEntry<float> { typedef float4 type; static constexpr int per_term = 2; };
template <> struct SeriesEntry<double> { typedef double2 type; static constexpr int per_term = 1; };
constexpr int kSeriesNodeBytes = 768;
__host__ __device__ inline int series_slots(int NP) { return NP + NP / 8 + 1; }
template <typename T>
__host__ __device__ inline int series_warp_bytes(int stride, int NP) {
  // FP32 samples two visibilities together while they fit two per lane
  const int vis = sizeof(T) == 4 && stride <= 64 ? 2 : 1;
  return kSeriesNodeBytes + vis * stride * 2 * static_cast<int>(sizeof(T)) +
         16 * series_slots(NP) * SeriesN<T>::terms / SeriesEntry<T>::per_term;
}

// A warp's view of its shared memory.
template <typename T, typename C>
struct SeriesWarp {
  typedef typename SeriesEntry<T>::type Entry;
  unsigned char* nodes;
  C* smp;
  Entry* coef;
  int slots;
  __device__ __forceinline__ SeriesWarp(unsigned char* base, const SeriesView<T>& sv) {
    const int vis = sizeof(T) == 4 && sv.stride <= 64 ? 2 : 1;
    nodes = base;
    smp = reinterpret_cast<C*>(base + kSeriesNodeBytes);
    coef = reinterpret_cast<Entry*>(smp + vis * sv.stride);
    slots = series_slots(sv.max_intervals);
  }

  template <int NV, int NS>
  __device__ __forceinline__ void sample_as(const SeriesView<T>& sv, const QuadParams& q, int P,
                                            const double (&dw)[NV], int NP, bool (&ok)[NV],
                                            int lane) {
    NodePack<C, NV>* nk = reinterpret_cast<NodePack<C, NV>*>(nodes);
    series_sample<T, C, NV, NS>(nk, nk + kNodes, smp, sv, q, P, dw, NP, ok, lane);
  }
  // NV visibilities' samples; as many per lane as the box needs.
  template <int NV>
  __device__ __forceinline__ void sample(const SeriesView<T>& sv, const QuadParams& q, int P,
                                         const double (&dw)[NV], int NP, bool (&ok)[NV],
                                         int lane) {
    const int need = NP + SeriesN<T>::half;
    if (need <= 32) return sample_as<NV, 1>(sv, q, P, dw, NP, ok, lane);
    if (NV == 2 || need <= 64) return sample_as<NV, 2>(sv, q, P, dw, NP, ok, lane);
    if constexpr (NV == 1) {
      if (need <= 96) return sample_as<NV, 3>(sv, q, P, dw, NP, ok, lane);
      return sample_as<NV, 4>(sv, q, P, dw, NP, ok, lane);
    }
  }
  __device__ __forceinline__ void polynomials(int v, const SeriesView<T>& sv, int NP, int lane) {
    series_polynomials(smp + v * sv.stride, coef, slots, NP, lane);
  }
};

// Takes the next visibility of the queue, and with it the one after it when
// the two can be sampled together (FP32, same support and panels, both
// claimed in this batch); false at the end.  A visibility beyond the tables
// goes to the retry list and the next is taken.
template <typename T>
__device__ __forceinline__ bool series_take(WarpQueue& wq, unsigned long long* head,
                                            unsigned long long batch, int64_t n,
                                            const VisRec<T>* __restrict__ recs,
                                            const SeriesView<T>& sv, const QuadParams& q,
                                            int lane, VisRec<T>& r0, VisRec<T>& r1,
                                            unsigned long long& i0, int& nv, int& P, int& NP) {
  while (wq.take(head, batch, n, lane, i0)) {
    r0 = recs[i0];
    P = series_panels(r0.jw, sv.support, q.Rf, q.chirp_coeff, sv.inv_cycles,
                      static_cast<float>(fabs(r0.dw)));
    NP = series_intervals(r0.jw, sv.inv_delta_f);
    if (P > sv.max_panels || NP > sv.max_intervals) {
      if (lane == 0) sv.retry[atomicAdd(sv.n_retry, 1ULL)] = static_cast<uint32_t>(i0);
      continue;
    }
    nv = 1;
    if (sizeof(T) == 4 && sv.stride <= 64 && wq.next < wq.stop) {
      r1 = recs[wq.next];
      if (r1.jw == r0.jw && series_panels(r1.jw, sv.support, q.Rf, q.chirp_coeff, sv.inv_cycles,
                                          static_cast<float>(fabs(r1.dw))) == P) {
        ++wq.next;
        nv = 2;
      }
    }
    return true;
  }
  return false;
}

// Samples the taken visibilities (bit v of the result: visibility v passes);
// those that do not go to the retry list.
template <typename T, typename C>
__device__ __forceinline__ int series_sample_taken(SeriesWarp<T, C>& w, const SeriesView<T>& sv,
                                                   const QuadParams& q, const VisRec<T>& r0,
                                                   const VisRec<T>& r1, unsigned long long i0,
                                                   int nv, int P, int NP, int lane) {
  int pass = 0;
  bool pair = false;
  if constexpr (sizeof(T) == 4) {
    if (nv == 2) {
      const double dw[2] = {r0.dw, r1.dw};
      bool ok[2];
      w.template sample<2>(sv, q, P, dw, NP, ok, lane);
      pass = (ok[0] ? 1 : 0) | (ok[1] ? 2 : 0);
      pair = true;
    }
  }
  if (!pair) {
    const double dw[1] = {r0.dw};
    bool ok[1];
    w.template sample<1>(sv, q, P, dw, NP, ok, lane);
    pass = ok[0] ? 1 : 0;
  }
  if (lane < nv && !((pass >> lane) & 1))
    sv.retry[atomicAdd(sv.n_retry, 1ULL)] = static_cast<uint32_t>(i0) + lane;
  return pass;
}

// The taps of one visibility in raster order, 32 at a time, tap t = b J_w + a
// advanced by 32 per step without a division.  kContig: the box lies inside
// the grid without wrapping and `grid` points at its first cell; otherwise
// `grid` is the stack's grid and each tap wraps its own indices.
template <bool kContig, bool kGrid, typename T, typename C>
__device__ __forceinline__ void series_taps(const SeriesWarp<T, C>& w, const VisRec<T>& r,
                                            int NP, T inv_delta, int npad,
                                            const C* __restrict__ grid_in, C* grid_out,
                                            const FixedGrid& fx, const C& yv, C& acc, int lane) {
  const int Jw = r.jw, half = Jw / 2, ntap = Jw * Jw;
  const int last = NP - 1;
  const T last_f = static_cast<T>(last);
  int a = lane % Jw, b = lane / Jw;
  const int step_b = 32 / Jw, step_a = 32 % Jw;
  // the tap's cell offsets as (exact) floating integers: no conversion per
  // tap, and one rounding in each distance
  T fa = static_cast<T>(a - half + 1), fb = static_cast<T>(b - half + 1);
  const T fstep_a = static_cast<T>(step_a), fstep_b = static_cast<T>(step_b);
  const T fJw = static_cast<T>(Jw);
  int off = b * npad + a;
  const int step_off = step_b * npad + step_a, carry_off = npad - Jw;
#pragma unroll 2
  for (int t0 = 0; t0 < ntap; t0 += 32) {
    const T du_ = r.fu - fa, dv_ = r.fv - fb;
    const C K = series_eval(w.coef, w.slots, last, last_f, inv_delta, sqrt(du_ * du_ + dv_ * dv_));
    int64_t gi;
    if (kContig) {
      gi = off;
    } else {
      gi = static_cast<int64_t>(wrap_index(r.bv + b - half + 1, npad)) * npad +
           wrap_index(r.bu + a - half + 1, npad);
    }
    if (t0 + lane < ntap) apply_tap<C, kGrid>(K, gi, yv, grid_in, grid_out, fx, acc);
    a += step_a;
    b += step_b;
    fa += fstep_a;
    fb += fstep_b;
    off += step_off;
    if (a >= Jw) {
      a -= Jw;
      ++b;
      fa -= fJw;
      fb += T(1);
      off += carry_off;
    }
  }
}

// Degrid / grid of visibilities [0, n): one warp per visibility (sampling two
// at a time in FP32), taken from the work queue.
template <typename T, typename C, bool kGrid>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 4 : 2)
    vis_series_kernel(const VisRec<T>* __restrict__ recs, const uint32_t* __restrict__ perm,
                      int64_t n, const C* __restrict__ grid_in, C* grid_out,
                      const C* __restrict__ vis_in, C* __restrict__ vis_out, QuadParams q,
                      SeriesView<T> sv, const int32_t* __restrict__ stack_slot,
                      unsigned long long* head, unsigned long long* stats, int batch) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int lane = threadIdx.x & 31;
  SeriesWarp<T, C> w(smem_raw + (threadIdx.x >> 5) *
                                    series_warp_bytes<T>(sv.stride, sv.max_intervals), sv);
  unsigned long long my_taps = 0, my_nodes = 0;
  const int npad = q.npad;
  WarpQueue wq;
  unsigned long long i0;
  VisRec<T> r[2];
  int nv, P, NP;
  while (series_take<T>(wq, head, static_cast<unsigned long long>(batch), n, recs, sv, q, lane,
                        r[0], r[1], i0, nv, P, NP)) {
    const int pass = series_sample_taken<T, C>(w, sv, q, r[0], r[1], i0, nv, P, NP, lane);
#pragma unroll 1
    for (int v = 0; v < nv; ++v) {
      if (!((pass >> v) & 1)) continue;
      const VisRec<T> rv = v ? r[1] : r[0];
      w.polynomials(v, sv, NP, lane);
      const int64_t gbase = static_cast<int64_t>(stack_slot[rv.stack]) * npad * npad;
      const uint32_t pm = perm[i0 + v];
      const C yv = kGrid ? load_visibility<T, C>(vis_in, pm, static_cast<T>(rv.weight))
                         : cmake<C>(0.0, 0.0);
      C acc = cmake<C>(0.0, 0.0);
      const int half = rv.jw / 2;
      const int u0 = wrap_index(rv.bu - half + 1, npad), v0 = wrap_index(rv.bv - half + 1, npad);
      if (u0 + rv.jw <= npad && v0 + rv.jw <= npad) {
        const int64_t o0 = gbase + static_cast<int64_t>(v0) * npad + u0;
        series_taps<true, kGrid>(w, rv, NP, sv.inv_delta, npad, kGrid ? nullptr : grid_in + o0,
                                 kGrid ? grid_out + o0 : nullptr, fixed_offset(q.fx, o0), yv,
                                 acc, lane);
      } else {
        series_taps<false, kGrid>(w, rv, NP, sv.inv_delta, npad,
                                  kGrid ? nullptr : grid_in + gbase,
                                  kGrid ? grid_out + gbase : nullptr, fixed_offset(q.fx, gbase),
                                  yv, acc, lane);
      }
      if (lane == 0) {
        my_taps += static_cast<unsigned long long>(rv.jw * rv.jw);
        my_nodes += static_cast<unsigned long long>((NP + 1) * kNodes * P);
      }
      if (!kGrid) store_visibility<T, C>(acc, static_cast<T>(rv.weight), pm, vis_out, lane);
      __syncwarp();   // the polynomials are rewritten for the next visibility
    }
  }
  flush_counts(stats, 0, my_taps, my_nodes, lane);
}

// The J_w x J_w kernel box of each of records [0, n) into boxes[i * jmax^2],
// row-major with row length J_w (pass 1 of the two-pass DDE convolution).
template <typename T, typename C>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 4 : 2)
    dde_box_series_kernel(const VisRec<T>* __restrict__ recs, int64_t n, C* __restrict__ boxes,
                          int jmax, QuadParams q, SeriesView<T> sv, unsigned long long* head,
                          unsigned long long* stats, int batch) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int lane = threadIdx.x & 31;
  SeriesWarp<T, C> w(smem_raw + (threadIdx.x >> 5) *
                                    series_warp_bytes<T>(sv.stride, sv.max_intervals), sv);
  unsigned long long my_nodes = 0;
  WarpQueue wq;
  unsigned long long i0;
  VisRec<T> r[2];
  int nv, P, NP;
  while (series_take<T>(wq, head, static_cast<unsigned long long>(batch), n, recs, sv, q, lane,
                        r[0], r[1], i0, nv, P, NP)) {
    const int pass = series_sample_taken<T, C>(w, sv, q, r[0], r[1], i0, nv, P, NP, lane);
#pragma unroll 1
    for (int v = 0; v < nv; ++v) {
      if (!((pass >> v) & 1)) continue;
      const VisRec<T> rv = v ? r[1] : r[0];
      w.polynomials(v, sv, NP, lane);
      const int Jw = rv.jw, half = Jw / 2, ntap = Jw * Jw;
      C* box = boxes + static_cast<int64_t>(i0 + v) * jmax * jmax;
      int a = lane % Jw, b = lane / Jw;
      const int step_b = 32 / Jw, step_a = 32 % Jw;
      for (int t = lane; t < ntap; t += 32) {
        const T du_ = rv.fu - static_cast<T>(a - half + 1);
        const T dv_ = rv.fv - static_cast<T>(b - half + 1);
        box[t] = series_eval(w.coef, w.slots, NP - 1, static_cast<T>(NP - 1), sv.inv_delta,
                             sqrt(du_ * du_ + dv_ * dv_));
        a += step_a;
        b += step_b;
        if (a >= Jw) {
          a -= Jw;
          ++b;
        }
      }
      if (lane == 0) my_nodes += static_cast<unsigned long long>((NP + 1) * kNodes * P);
      __syncwarp();
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) my_nodes += __shfl_xor_sync(0xffffffffu, my_nodes, o);
  if (lane == 0 && my_nodes) atomicAdd(stats + 3, my_nodes);
}
