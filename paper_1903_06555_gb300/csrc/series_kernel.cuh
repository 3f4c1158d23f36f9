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
// Tolerance.  The estimate E = sum over panels |K31 - G15| is formed at the
// samples within the box, and a visibility is settled if 1.5 E <= quad_abs_tol
// at all of them.  That is an estimate of the taps' E, as G15 against K31 is
// one of their error, not a bound: were the samples of the whole line tested,
// no tap's E could exceed 1 / cos(pi / 4) = 1.42 times the largest (each
// panel's difference is band-limited like the kernel and sampled at twice its
// Nyquist rate; one sum of the panels with the phases that align them at the
// tap is too), but those beyond the box, which the interpolation reads (9; FP64
// 19) and the panels are not sized for, are not.  Of 3,400 random supports,
// windows, oversamplings, offsets and tolerances whose samples passed,
// evaluated in 64 bits, no tap's E exceeded 0.63 of the tolerance.  The taps'
// values do not depend on it: the sums over the nodes are band-limited by
// construction, whatever their error against the integral.
// The a-priori panels follow the support (the corner of the box and the
// largest |dw| the support covers), which leaves E two orders below 1e-6 at
// 6 cycles per panel for the default support.  A visibility that fails -- or
// needs more panels or samples than the tables hold -- is put on a list, and
// the kernel that integrates each tap by itself (vis_kernel and its
// companions), with its refinement and its count of unconverged taps, takes
// that list.
//
// FP32 makes the sums on the tensor cores (series_tile_kernel says how the
// operands are split), four visibilities of one panel count to a warp: 1.3 ms
// of the snapshot's launch where one FP32 product per lane took 3.9 (two
// table loads and two broadcasts per node and pair of visibilities).  FP64
// walks the nodes, one sample per lane.
//
// Measured on the MWA-like snapshot (1.92M visibilities, J_w 26-40, FP32):
// 5.4 ms per degrid or grid launch where the per-tap kernel takes 63 and the
// 16-point radial series 18.6, and 4.2e-7 from the 64-bit operator (per tap
// 5.5e-7, radial series 9e-7: the table's J0 is rounded once, the per-tap
// kernel's polynomial and hardware cosine are not).  Of the 5.4 ms the taps
// take 3.3, the polynomials 0.8.  FP64 at 1e-12 (5,000 visibilities, J_w 26):
// 0.93 ms, per tap 39 ms.  Bound: the shared-memory pipe (80% busy; 16 of
// the 21 wavefronts per 32 taps read the polynomials) and issue (67%); FP64 its
// FP64 unit.  24 warps of 80 registers per SM: 32 of 64 spill (5.5 ms), 16
// of 128 hide less (6.6 ms).
#pragma once

#include "series_coef.cuh"

// Sample pairs and polynomial terms of the interpolation (series_fit.py).
template <typename T> struct SeriesN;
template <> struct SeriesN<float> { static constexpr int half = 10, terms = 8; };
template <> struct SeriesN<double> { static constexpr int half = 20, terms = 14; };

// Gauss over Kronrod weight at the odd nodes (position kk: node 2 kk + 1).
__constant__ float c_series_ratio[16] = {
#define PHI_RATIO(k) static_cast<float>(gk_gw(2 * (k) + 1) / gk_wk(2 * (k) + 1))
    PHI_RATIO(0), PHI_RATIO(1), PHI_RATIO(2), PHI_RATIO(3), PHI_RATIO(4),
    PHI_RATIO(5), PHI_RATIO(6), PHI_RATIO(7), PHI_RATIO(8), PHI_RATIO(9),
    PHI_RATIO(10), PHI_RATIO(11), PHI_RATIO(12), PHI_RATIO(13), PHI_RATIO(14), 0.0f
#undef PHI_RATIO
};

// Most samples per visibility and panels the tables hold.
constexpr int kSeriesMaxSamples = 128;
constexpr int kSeriesMaxPanels = 32;

// Sample intervals that cover the box of support J: its farthest tap lies
// within J / sqrt(2) of the visibility (the margin covers the rounding of
// every distance formed in FP32, so no tap falls past the last interval).
__host__ __device__ inline int series_intervals(int J, float inv_delta) {
  return static_cast<int>(static_cast<float>(J) * 0.70710678f * inv_delta + 1e-3f) + 1;
}

// A-priori panels of a visibility: as initial_panels, for the corner of its
// box and the larger of its |dw| and the |dw| its support was sized for, so
// that visibilities of one support share their panels.
__host__ __device__ inline int series_panels(int J, int support, float Rf, float chirp_coeff,
                                             float inv_cycles, float adw) {
  const float chirp = fmaxf(adw * chirp_coeff, 0.5f * static_cast<float>(J - support));
  return panel_count_for(Rf * fmaf(static_cast<float>(J), 0.70710678f, chirp) * inv_cycles);
}

// FP64: J0(2 pi rho_i r_j) for sample i of panel-table row j: rows as the
// node tables (31 P rows for every panel count P), `stride` samples each.
__global__ void series_table_kernel(int64_t rows, int stride, double* __restrict__ j0_out) {
  const int64_t total = rows * stride;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t row = e / stride;
    const int i = static_cast<int>(e - row * stride);
    int P = 1;
    while (panel_table_offset(P + 1) <= row) ++P;
    const int64_t local = row - panel_table_offset(P);
    const int p = static_cast<int>(local / kNodes), k = static_cast<int>(local % kNodes);
    j0_out[e] = j0(kPi * i * (2.0 * p + 1.0 + gk_node(k)) / (4.0 * P));
  }
}

// FP32: the sums over the nodes are matrix products, samples x nodes times
// nodes x (visibility, real or imaginary), on the tensor cores: m16n8k16 with
// FP16 operands and FP32 accumulation, each factor split into two halves
// (hi + lo, 22 bits) and the three products that matter taken -- per product
// 2^-23 of its size, as one FP32 rounding.  A panel's nodes make two steps of
// 16: the 15 Gauss nodes (odd) with a zero, then the 16 Kronrod-only ones, so
// that the Gauss sum takes the first step's J0 with its own weights.
// Fragments of m16n8k16: lane = 4 g + t holds A rows g, g + 8 at k = 2 t,
// 2 t + 1, 2 t + 8, 2 t + 9, B column g at the same k, C rows g, g + 8 at
// columns 2 t, 2 t + 1.
constexpr float kSeriesScaleA = 64.0f;     // J0, h scaled clear of FP16's subnormals
constexpr float kSeriesScaleB = 4096.0f;
constexpr int kSeriesTile = 16;            // samples per A tile
__host__ __device__ inline int series_fragment_k(int t, int e) { return 2 * t + (e & 1) + 8 * (e >> 1); }
// Node of position kk of a step (0: Gauss nodes, 1: the others); 31: none.
__host__ __device__ inline int series_step_node(int step, int kk) {
  return step ? 2 * kk : (kk < 15 ? 2 * kk + 1 : kNodes);
}
// Panels before those of the P-panel partition.
__host__ __device__ inline int series_panel_base(int P) { return P * (P - 1) / 2; }

// The A tiles of every panel of partitions 1 .. Pmax, [panel][tile][step][hi,
// lo][lane] of four registers, and the node table [panel][step][kk] = {1 - n
// as two floats, Kronrod weight times 2 pi h g r (scaled), 0}.
__global__ void series_tile_kernel(int panels, int tiles, const double* __restrict__ omn,
                                   const float* __restrict__ hk, uint4* __restrict__ a_out,
                                   float4* __restrict__ node_out) {
  const int total = panels * tiles * 2 * 32;
  for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < total; x += gridDim.x * blockDim.x) {
    const int lane = x & 31, step = (x >> 5) & 1, tile = (x >> 6) % tiles, row = (x >> 6) / tiles;
    int P = 1;
    while (series_panel_base(P + 1) <= row) ++P;
    const int p = row - series_panel_base(P);
    const int g = lane >> 2, t = lane & 3;
    unsigned hi[4], lo[4];
    for (int r = 0; r < 4; ++r) {          // a0: (g, low k), a1: (g + 8, low), a2, a3: high k
      const int i = kSeriesTile * tile + g + 8 * (r & 1);
      __half h[2], l[2];
      for (int c = 0; c < 2; ++c) {
        const int k = series_step_node(step, series_fragment_k(t, c + 2 * (r >> 1)));
        const float v = k < kNodes ? static_cast<float>(kSeriesScaleA *
                                         j0(kPi * i * (2.0 * p + 1.0 + gk_node(k)) / (4.0 * P)))
                                   : 0.0f;
        h[c] = __float2half_rn(v);
        l[c] = __float2half_rn(v - __half2float(h[c]));
      }
      hi[r] = __half_as_ushort(h[0]) | (static_cast<unsigned>(__half_as_ushort(h[1])) << 16);
      lo[r] = __half_as_ushort(l[0]) | (static_cast<unsigned>(__half_as_ushort(l[1])) << 16);
    }
    uint4* out = a_out + (static_cast<int64_t>(row * tiles + tile) * 2 + step) * 64 + lane;
    out[0] = make_uint4(hi[0], hi[1], hi[2], hi[3]);
    out[32] = make_uint4(lo[0], lo[1], lo[2], lo[3]);
    if (tile == 0 && lane < 16) {
      const int k = series_step_node(step, lane);
      float4 n = make_float4(0.f, 0.f, 0.f, 0.f);
      if (k < kNodes) {
        const int64_t j = panel_table_offset(P) + kNodes * p + k;
        const float o = static_cast<float>(omn[j]);
        n = make_float4(o, static_cast<float>(omn[j] - o), kSeriesScaleB * hk[j], 0.f);
      }
      node_out[(row * 2 + step) * 16 + lane] = n;
    }
  }
}

__device__ __forceinline__ void series_mma(float (&c)[4], const uint4& a, const unsigned (&b)[2]) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b[0]), "r"(b[1]));
}
// c += (a_hi + a_lo)(b_hi + b_lo) without the product of the two low parts.
struct SeriesB { unsigned hi[2], lo[2]; };
__device__ __forceinline__ void series_mma3(float (&c)[4], const uint4& ah, const uint4& al,
                                            const SeriesB& b) {
  series_mma(c, al, b.hi);
  series_mma(c, ah, b.lo);
  series_mma(c, ah, b.hi);
}
// Four values (fragment positions e = 0..3) split into the two halves.
__device__ __forceinline__ SeriesB series_split(const float (&v)[4]) {
  SeriesB b;
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const __half2 h = __floats2half2_rn(v[2 * i], v[2 * i + 1]);
    const float2 f = __half22float2(h);
    const __half2 l = __floats2half2_rn(v[2 * i] - f.x, v[2 * i + 1] - f.y);
    b.hi[i] = *reinterpret_cast<const unsigned*>(&h);
    b.lo[i] = *reinterpret_cast<const unsigned*>(&l);
  }
  return b;
}

// FP32: samples 16 m0 .. 16 (m0 + MT) - 1 of the four visibilities whose
// offsets dw this lane's B column takes part in (column g: visibility g / 2,
// real or imaginary part; a visibility that is not there has dw = 0 and is
// ignored) into smp (visibility v at smp + v * vstride, its first samples also
// mirrored to negative rho).  Returns whether the estimate passes at this
// lane's samples 0 .. NP of visibility t = lane % 4, NP that visibility's (-1:
// it keeps the samples it has).  Every column is computed alike, so a
// visibility's samples do not depend on what it is sampled with.
template <int MT, bool kAgain>
__device__ __forceinline__ bool series_sample_f32(float2* smp, int vstride,
                                                  const SeriesView<float>& sv, int P,
                                                  const PhaseF& phase, int m0, int NP, int lane) {
  const int g = lane >> 2, t = lane & 3, comp = g & 1;
  float K[MT][4], err[MT][2], ratio[4];
#pragma unroll
  for (int m = 0; m < MT; ++m) {
#pragma unroll
    for (int i = 0; i < 4; ++i) K[m][i] = 0.f;
    err[m][0] = err[m][1] = 0.f;
  }
#pragma unroll
  for (int e = 0; e < 4; ++e)   // Gauss over Kronrod weight of the first step's nodes
    ratio[e] = c_series_ratio[series_fragment_k(t, e)];
  const int row = series_panel_base(P);
  const float4* __restrict__ nodes = sv.nodes + (row * 2 + comp) * 16;
  const uint4* __restrict__ at =
      sv.tiles_a + (static_cast<int64_t>(row) * sv.tiles + m0) * 128 + lane;
  for (int p = 0; p < P; ++p, nodes += 32, at += sv.tiles * 128) {
    // the lane evaluates the four nodes of step `comp`; its partner (the
    // other part of the same visibility) those of the other step
    float mine[4], theirs[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const float4 nd = nodes[series_fragment_k(t, e)];
      const float2 cs = phase(nd.x, nd.y);
      mine[e] = nd.z * (comp ? cs.y : cs.x);
      theirs[e] = __shfl_xor_sync(0xffffffffu, nd.z * (comp ? cs.x : cs.y), 4);
    }
    float first[4], second[4], gauss[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      first[e] = comp ? theirs[e] : mine[e];
      second[e] = comp ? mine[e] : theirs[e];
      gauss[e] = ratio[e] * first[e];
    }
    const SeriesB b0 = series_split(first), b1 = series_split(second), bg = series_split(gauss);
#pragma unroll
    for (int m = 0; m < MT; ++m) {
      const uint4 h0 = at[m * 128], l0 = at[m * 128 + 32];
      const uint4 h1 = at[m * 128 + 64], l1 = at[m * 128 + 96];
      float A[4] = {0.f, 0.f, 0.f, 0.f}, G[4] = {0.f, 0.f, 0.f, 0.f};
      series_mma3(A, h0, l0, b0);
      series_mma3(G, h0, l0, bg);
      series_mma3(A, h1, l1, b1);
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const float dr = A[2 * i] - G[2 * i], di = A[2 * i + 1] - G[2 * i + 1];
        err[m][i] += est_sqrt(dr * dr + di * di);
        K[m][2 * i] += A[2 * i];
        K[m][2 * i + 1] += A[2 * i + 1];
      }
    }
  }
  constexpr float kUnscale = 1.0f / (kSeriesScaleA * kSeriesScaleB);
  bool good = true;
  smp += t * vstride;
#pragma unroll
  for (int m = 0; m < MT; ++m)
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int s = kSeriesTile * (m0 + m) + g + 8 * i;
      const float2 k = make_float2(kUnscale * K[m][2 * i], kUnscale * K[m][2 * i + 1]);
      if (!kAgain || NP >= 0) {
        smp[s] = k;
        if (m == 0 && m0 == 0 && s < SeriesN<float>::half) smp[-s] = k;   // even in rho
      }
      if (s <= NP) good = good && 1.5f * kUnscale * err[m][i] <= sv.tol;   // NaN fails
    }
  return good;
}

// FP64: samples 0 .. 32 NS - 1 of one visibility into smp; whether the
// estimate passes at samples 0 .. NP.  Per panel the lanes build its 31 node
// values (nk: Kronrod, ng: the 15 odd nodes with their Gauss weights), then
// each takes NS samples and walks the nodes, one table row per node.
template <int NS>
__device__ __forceinline__ bool series_sample_f64(double2* nk, double2* smp,
                                                  const SeriesView<double>& sv,
                                                  const QuadParams& q, int P, double dw, int NP,
                                                  int lane) {
  double2* ng = nk + kNodes;
  double2 K[NS];
  double err[NS];
#pragma unroll
  for (int s = 0; s < NS; ++s) {
    K[s] = make_double2(0.0, 0.0);
    err[s] = 0.0;
  }
  const int stride = sv.stride;
  const int64_t row0 = panel_table_offset(P);
  const double* __restrict__ tj = sv.j0 + row0 * stride + lane;
  for (int p = 0; p < P; ++p) {
    if (lane < kNodes) {
      const int64_t j = row0 + kNodes * p + lane;
      const double hk = static_cast<const double*>(q.node_hk)[j];
      const double hg = hk - static_cast<const double*>(q.node_hd)[j];   // the table: difference
      double t = dw * q.node_omn[j];
      t -= rint(t);
      double sn, cs;
      sincospi(2.0 * t, &sn, &cs);
      nk[lane] = make_double2(hk * cs, hk * sn);
      if (lane & 1) ng[lane >> 1] = make_double2(hg * cs, hg * sn);
    }
    __syncwarp();
    double2 A[NS], G[NS];
#pragma unroll
    for (int s = 0; s < NS; ++s) A[s] = G[s] = make_double2(0.0, 0.0);
    auto mad = [](double2& acc, double J, const double2& h) {
      acc.x = fma(J, h.x, acc.x);
      acc.y = fma(J, h.y, acc.y);
    };
#pragma unroll 5
    for (int k = 0; k < (kNodes - 1) / 2; ++k) {
      const double2 h0 = nk[2 * k], h1 = nk[2 * k + 1], g1 = ng[k];
#pragma unroll
      for (int s = 0; s < NS; ++s) {
        const double J0 = tj[32 * s], J1 = tj[stride + 32 * s];
        mad(A[s], J0, h0);
        mad(A[s], J1, h1);
        mad(G[s], J1, g1);
      }
      tj += 2 * stride;
    }
#pragma unroll
    for (int s = 0; s < NS; ++s) mad(A[s], tj[32 * s], nk[kNodes - 1]);
    tj += stride;
#pragma unroll
    for (int s = 0; s < NS; ++s) {
      K[s].x += A[s].x;
      K[s].y += A[s].y;
      const double dr = A[s].x - G[s].x, di = A[s].y - G[s].y;
      err[s] += est_sqrt(dr * dr + di * di);
    }
    __syncwarp();   // the node values are rewritten by the next panel
  }
  bool good = true;
#pragma unroll
  for (int s = 0; s < NS; ++s) {
    smp[32 * s + lane] = K[s];
    if (32 * s + lane <= NP) good = good && 1.5 * err[s] <= sv.tol;   // NaN fails
  }
  return good;
}

// FP64: where interval p's polynomial lies in an array of 16-byte entries,
// skewed by one entry in eight, so that intervals a stride of 1 or 2 apart
// (the taps of a row, from its middle to its ends) fall on different banks.
__device__ __forceinline__ int series_slot(int p) { return p + (p >> 3); }

// The polynomials of intervals 0 .. NP - 1 from the samples, term m of
// interval p at coef[m * slots + p] (FP64: + series_slot(p)).  One interval
// per lane.
__device__ __forceinline__ void series_polynomials(const float2* smp, float2* coef, int slots,
                                                   int NP, int lane) {
  constexpr int H = SeriesN<float>::half, M = SeriesN<float>::terms;
  for (int p = lane; p < NP; p += 32) {
    float2 c[M];
#pragma unroll
    for (int m = 0; m < M; ++m) c[m] = make_float2(0.f, 0.f);
#pragma unroll
    for (int d = 0; d < H; ++d) {
      const float2 lo = smp[p - d], hi = smp[p + 1 + d];
      const float2 sum = __fadd2_rn(hi, lo);
      const float2 dif = __ffma2_rn(lo, make_float2(-1.f, -1.f), hi);
#pragma unroll
      for (int m = 0; m < M; ++m) c[m] = __ffma2_rn(c_series_f[m][d], (m & 1) ? dif : sum, c[m]);
    }
#pragma unroll
    for (int m = 0; m < M; ++m) coef[m * slots + p] = c[m];
  }
  __syncwarp();
}
// (FP64: a lane takes the real or the imaginary part of an interval, so that
// fewer lanes of its FP64 unit idle in the last round.)
__device__ __forceinline__ void series_polynomials(const double2* smp, double2* coef, int slots,
                                                   int NP, int lane) {
  constexpr int H = SeriesN<double>::half, M = SeriesN<double>::terms;
  const double* part = reinterpret_cast<const double*>(smp) + (lane & 1);
  double* out = reinterpret_cast<double*>(coef) + (lane & 1);
  for (int p = lane >> 1; p < NP; p += 16) {
    double c[M];
#pragma unroll
    for (int m = 0; m < M; ++m) c[m] = 0.0;
#pragma unroll 4
    for (int d = 0; d < H; ++d) {
      const double lo = part[2 * abs(p - d)], hi = part[2 * (p + 1 + d)];
      const double sum = hi + lo, dif = hi - lo;
#pragma unroll
      for (int m = 0; m < M; ++m) c[m] = fma(c_series_d[m][d], (m & 1) ? dif : sum, c[m]);
    }
#pragma unroll
    for (int m = 0; m < M; ++m) out[2 * (m * slots + series_slot(p))] = c[m];
  }
  __syncwarp();
}

// The hardware square root (relative error about 2^-23, as the rounding of
// the squared distance itself).
__device__ __forceinline__ float series_sqrt(float x) {
  float y;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// [GC] at squared distance rho2 from the polynomials: interval ip = floor of
// s = 4 R rho by the rounding of s - 1/2 to an integer (as table_index; an
// exact integer s may fall to either neighbour, whose polynomials meet
// there), then the polynomial at t = 2 (s - ip) - 1.
__device__ __forceinline__ float2 series_horner(const float2* e, int slots, float t) {
  const float2 t2 = make_float2(t, t);
  constexpr int M = SeriesN<float>::terms;
  float2 k = e[(M - 1) * slots];
#pragma unroll
  for (int m = M - 2; m >= 0; --m) k = __ffma2_rn(k, t2, e[m * slots]);
  return k;
}
__device__ __forceinline__ float2 series_eval(const float2* coef, int slots, float inv_delta,
                                              float rho2) {
  const float big = 12582912.0f;                      // 1.5 * 2^23
  const float rho = series_sqrt(rho2);
  const float u = fmaf(rho, inv_delta, -0.5f) + big;
  const float f = u - big;
  const float t = fmaf(2.0f * inv_delta, rho, fmaf(-2.0f, f, -1.0f));
  return series_horner(coef + (__float_as_int(u) - __float_as_int(big)), slots, t);
}
// The same at two distances, the address arithmetic in paired FP32.
__device__ __forceinline__ void series_eval2(const float2* coef, int slots, float inv_delta,
                                             float2 rho2, float2& k0, float2& k1) {
  const float big = 12582912.0f;
  const float2 rho = make_float2(series_sqrt(rho2.x), series_sqrt(rho2.y));
  const float2 u = __fadd2_rn(__ffma2_rn(rho, make_float2(inv_delta, inv_delta),
                                         make_float2(-0.5f, -0.5f)), make_float2(big, big));
  const float2 f = __fadd2_rn(u, make_float2(-big, -big));
  const float2 t = __ffma2_rn(rho, make_float2(2.0f * inv_delta, 2.0f * inv_delta),
                              __ffma2_rn(f, make_float2(-2.f, -2.f), make_float2(-1.f, -1.f)));
  k0 = series_horner(coef + (__float_as_int(u.x) - __float_as_int(big)), slots, t.x);
  k1 = series_horner(coef + (__float_as_int(u.y) - __float_as_int(big)), slots, t.y);
}
__device__ __forceinline__ double2 series_eval(const double2* coef, int slots, double inv_delta,
                                               double rho2) {
  const double s = sqrt(rho2) * inv_delta;
  const int ip = static_cast<int>(s);
  const double t = fma(2.0, s - static_cast<double>(ip), -1.0);
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
// Slots per term: in FP32 64 or 128, as immediate offsets in the tap loop; in
// FP64 the skewed intervals.
template <typename T>
__host__ __device__ inline int series_slots(int NP) {
  return sizeof(T) == 4 ? (NP <= 64 ? 64 : 128) : NP + NP / 8 + 1;
}
// Visibilities sampled together, and the distance of their samples (FP32:
// room for the mirrored ones before each, and 4 more than a multiple of 16,
// so that a store of 8 samples of 4 visibilities is free of bank conflicts).
template <typename T> struct SeriesVis { static constexpr int n = sizeof(T) == 4 ? 4 : 1; };
template <typename T>
__host__ __device__ inline int series_vstride(int stride) {
  return sizeof(T) == 4 ? (stride + 15) / 16 * 16 + 20 : stride;
}
constexpr int kSeriesMirror = 16;       // FP32: first sample's place
constexpr int kSeriesNodeBytes = 768;   // FP64: node values of one panel
template <typename T>
__host__ __device__ inline int series_warp_bytes(int stride, int NP) {
  return (sizeof(T) == 4 ? 0 : kSeriesNodeBytes) +
         2 * static_cast<int>(sizeof(T)) * (SeriesVis<T>::n * series_vstride<T>(stride) +
                                            series_slots<T>(NP) * SeriesN<T>::terms);
}

// A warp's view of its shared memory.
template <typename T, typename C>
struct SeriesWarp {
  C* smp;
  C* coef;
  int slots, vstride;
  __device__ __forceinline__ SeriesWarp(unsigned char* base, const SeriesView<T>& sv) {
    vstride = series_vstride<T>(sv.stride);
    C* first = reinterpret_cast<C*>(base + (sizeof(T) == 4 ? 0 : kSeriesNodeBytes));
    coef = first + SeriesVis<T>::n * vstride;
    smp = first + (sizeof(T) == 4 ? kSeriesMirror : 0);
    slots = series_slots<T>(sv.max_intervals);
  }
  __device__ __forceinline__ void polynomials(int v, int NP, int lane) {
    series_polynomials(smp + v * vstride, coef, slots, NP, lane);
  }
};

// Samples of the taken visibilities (the lane's dw: FP32 the one of its B
// column, FP64 the visibility's; NP: intervals of visibility lane % 4, or -1
// for one that keeps the samples it has, top: the most of any); bit v of the
// result: visibility v passes.
template <bool kAgain>
__device__ __forceinline__ int series_sample(SeriesWarp<float, float2>& w,
                                             const SeriesView<float>& sv, const QuadParams&,
                                             int P, double dw, int NP, int top, int lane) {
  const PhaseF phase(dw);
  int tiles = (top + SeriesN<float>::half + kSeriesTile - 1) / kSeriesTile;
  bool good = true;
  int m0 = 0;
  for (; tiles > 4; tiles -= 4, m0 += 4)
    good = series_sample_f32<4, kAgain>(w.smp, w.vstride, sv, P, phase, m0, NP, lane) && good;
  if (tiles == 4)
    good = series_sample_f32<4, kAgain>(w.smp, w.vstride, sv, P, phase, m0, NP, lane) && good;
  else if (tiles == 3)
    good = series_sample_f32<3, kAgain>(w.smp, w.vstride, sv, P, phase, m0, NP, lane) && good;
  else if (tiles == 2)
    good = series_sample_f32<2, kAgain>(w.smp, w.vstride, sv, P, phase, m0, NP, lane) && good;
  else
    good = series_sample_f32<1, kAgain>(w.smp, w.vstride, sv, P, phase, m0, NP, lane) && good;
  const unsigned bad = __ballot_sync(0xffffffffu, !good);
  __syncwarp();
  int pass = 0;
#pragma unroll
  for (int v = 0; v < 4; ++v) pass |= (bad & (0x11111111u << v)) ? 0 : 1 << v;
  return pass;
}
template <bool kAgain>
__device__ __forceinline__ int series_sample(SeriesWarp<double, double2>& w,
                                             const SeriesView<double>& sv, const QuadParams& q,
                                             int P, double dw, int NP, int, int lane) {
  double2* nk = reinterpret_cast<double2*>(reinterpret_cast<unsigned char*>(w.smp) -
                                           kSeriesNodeBytes);
  const int need = NP + SeriesN<double>::half;
  bool good;
  if (need <= 32) good = series_sample_f64<1>(nk, w.smp, sv, q, P, dw, NP, lane);
  else if (need <= 64) good = series_sample_f64<2>(nk, w.smp, sv, q, P, dw, NP, lane);
  else if (need <= 96) good = series_sample_f64<3>(nk, w.smp, sv, q, P, dw, NP, lane);
  else good = series_sample_f64<4>(nk, w.smp, sv, q, P, dw, NP, lane);
  good = __all_sync(0xffffffffu, good);
  __syncwarp();
  return good ? 1 : 0;
}

// Takes the next visibility of the queue and, in FP32, up to three more with
// the same panels behind it in this batch; samples them, and puts those that
// fail on the retry list.  A visibility beyond the tables goes to the list
// at once.  False at the end.
//
// kAgain: one whose estimate fails is first sampled again on one panel more, if
// the tables go so far.  At some supports every visibility fails on the
// a-priori panels: where the taper is narrow against the first of them (12
// pixels of support, J_w 14, one panel of 5.4 cycles: 1.5 E = 8e-6).  One panel
// more brings E down by two orders and more; the list would take the whole
// observation (20,000 such visibilities: 212 us by the list, 72 sampled again;
// the per-tap kernel by itself 195).  FP32 plans without such supports take
// the kernels without it (its registers spill, 1% of the snapshot's time).
template <bool kAgain, typename T, typename C>
__device__ __forceinline__ bool series_take(SeriesWarp<T, C>& w, WarpQueue& wq,
                                            unsigned long long* head, unsigned long long batch,
                                            int64_t n, const VisRec<T>* __restrict__ recs,
                                            const SeriesView<T>& sv, const QuadParams& q,
                                            int lane, unsigned long long& i0, int& nv, int& pass,
                                            int& P, unsigned long long& nodes) {
  constexpr int NV = SeriesVis<T>::n;
  while (wq.take(head, batch, n, lane, i0)) {
    // the lane's candidate: FP32 the visibility of its B column
    const int v = NV > 1 ? lane >> 3 : 0;
    const bool there = i0 + v < wq.stop;
    const VisRec<T>* r = recs + (there ? i0 + v : i0);
    const double dw = r->dw;
    const int myNP = series_intervals(r->jw, sv.inv_delta_f);
    const int myP = series_panels(r->jw, sv.support, q.Rf, q.chirp_coeff, sv.inv_cycles,
                                  static_cast<float>(fabs(dw)));
    const bool fits = there && myP <= sv.max_panels && myNP <= sv.max_intervals;
    P = __shfl_sync(0xffffffffu, myP, 0);
    const unsigned alike = __ballot_sync(0xffffffffu, fits && myP == P);
    if (!(alike & 1)) {
      if (lane == 0) sv.retry[atomicAdd(sv.n_retry, 1ULL)] = static_cast<uint32_t>(i0);
      continue;
    }
    nv = 1;
    while (nv < NV && ((alike >> (8 * nv)) & 1)) ++nv;
    wq.next = i0 + nv;
    const int own = v < nv ? myNP : 0;
    const int top = __reduce_max_sync(0xffffffffu, own);
    // intervals of the visibility whose sums this lane will hold
    int NP = __shfl_sync(0xffffffffu, own, NV > 1 ? 8 * (lane & 3) : 0);
    if constexpr (kAgain) {
      pass = 0;
#pragma unroll 1
      for (int p = P, last = min(P + 1, sv.max_panels);; ++p) {
        // evaluations, counted by one lane of each visibility's columns
        if (v < nv && (lane & (NV > 1 ? 7 : 31)) == 0 && !((pass >> v) & 1))
          nodes += (myNP + 1) * kNodes * p;
        pass |= series_sample<kAgain>(w, sv, q, p, v < nv ? dw : 0.0, NP, top, lane);
        if (p >= last || !(~pass & ((1 << nv) - 1))) break;
        if (NV > 1 && ((pass >> (lane & 3)) & 1)) NP = -1;
      }
    } else {   // counted with the taps
      pass = series_sample<kAgain>(w, sv, q, P, v < nv ? dw : 0.0, NP, top, lane);
    }
    if (lane < nv && !((pass >> lane) & 1))
      sv.retry[atomicAdd(sv.n_retry, 1ULL)] = static_cast<uint32_t>(i0) + lane;
    return true;
  }
  return false;
}

// The taps of one visibility.  kContig: the box lies inside the grid without
// wrapping and `grid` points at its first cell; otherwise `grid` is the
// stack's grid and each tap wraps its own indices.  kSlots: the polynomials'
// slots per term when known at compile time (0: w.slots).  Columns advance
// without a division, the offsets kept as (exact) floating integers: no
// conversion per tap, one rounding in each distance.
//
// FP32: bands of four rows, 16 columns at a time, two vertical neighbours
// per lane (supports are even; their distances in paired arithmetic); the
// lanes of a half-warp hold 8 columns of two such pairs, whose intervals --
// two per column at most -- are 16 neighbouring ones, so that its 8-byte
// loads of a term meet no bank twice (16 columns of one row would: 27 against
// 20 shared-memory wavefronts per 32 taps).
template <bool kContig, bool kGrid, int kSlots>
__device__ __forceinline__ void series_taps(const SeriesWarp<float, float2>& w,
                                            const VisRec<float>& r, float inv_delta, int npad,
                                            const float2* __restrict__ grid_in, float2* grid_out,
                                            const FixedGrid& fx, const float2& yv, float2& acc,
                                            int lane) {
  const int Jw = r.jw, half = Jw / 2;
  const int items = Jw * ((Jw + 3) / 4);           // columns of all bands, one after another
  const int slots = kSlots ? kSlots : w.slots;
  const int c = (lane & 7) | ((lane & 16) >> 1);   // column within the step
  int a = c % Jw, b = 4 * (c / Jw) + 2 * ((lane >> 3) & 1);
  const int step_b = 4 * (16 / Jw), step_a = 16 % Jw;
  const float fu = r.fu, fv = r.fv;
  // minus the offsets of column a and row b
  float na = static_cast<float>(half - 1 - a), nb = static_cast<float>(half - 1 - b);
  const float fstep_a = static_cast<float>(step_a), fstep_b = static_cast<float>(step_b);
  const float fJw = static_cast<float>(Jw), fend = static_cast<float>(-half);
  int off = b * npad + a;
  const int step_off = step_b * npad + step_a, carry_off = 4 * npad - Jw;
#pragma unroll 1
  for (int x = c; x - c < items; x += 16) {
    // the last step may run past the last band, the last band past the box
    if (x < items && nb > fend) {
      const float du_ = fu + na, d2 = du_ * du_;
      const float2 dv_ = __fadd2_rn(make_float2(fv, fv), make_float2(nb, nb - 1.0f));
      float2 k0, k1;
      series_eval2(w.coef, slots, inv_delta, __ffma2_rn(dv_, dv_, make_float2(d2, d2)), k0, k1);
      int64_t g0, g1;
      if (kContig) {
        g0 = off;
        g1 = off + npad;
      } else {
        const int row = r.bv - static_cast<int>(nb), col = wrap_index(r.bu - static_cast<int>(na), npad);
        g0 = static_cast<int64_t>(wrap_index(row, npad)) * npad + col;
        g1 = static_cast<int64_t>(wrap_index(row + 1, npad)) * npad + col;
      }
      apply_tap<float2, kGrid>(k0, g0, yv, grid_in, grid_out, fx, acc);
      apply_tap<float2, kGrid>(k1, g1, yv, grid_in, grid_out, fx, acc);
    }
    na -= fstep_a;
    nb -= fstep_b;
    off += step_off;
    if (na < fend) {
      na += fJw;
      nb -= 4.0f;
      off += carry_off;
    }
  }
}
// FP64: raster order, 32 taps at a time.
template <bool kContig, bool kGrid, int kSlots>
__device__ __forceinline__ void series_taps(const SeriesWarp<double, double2>& w,
                                            const VisRec<double>& r, double inv_delta, int npad,
                                            const double2* __restrict__ grid_in,
                                            double2* grid_out, const FixedGrid& fx,
                                            const double2& yv, double2& acc, int lane) {
  const int Jw = r.jw, half = Jw / 2, ntap = Jw * Jw;
  int a = lane % Jw, b = lane / Jw;
  const int step_b = 32 / Jw, step_a = 32 % Jw;
  for (int t = lane; t < ntap; t += 32) {
    const double du_ = r.fu - static_cast<double>(a - half + 1);
    const double dv_ = r.fv - static_cast<double>(b - half + 1);
    const double2 k = series_eval(w.coef, w.slots, inv_delta, du_ * du_ + dv_ * dv_);
    const int64_t gi = kContig ? static_cast<int64_t>(b * npad + a)
                               : static_cast<int64_t>(wrap_index(r.bv + b - half + 1, npad)) * npad +
                                     wrap_index(r.bu + a - half + 1, npad);
    apply_tap<double2, kGrid>(k, gi, yv, grid_in, grid_out, fx, acc);
    a += step_a;
    b += step_b;
    if (a >= Jw) {
      a -= Jw;
      ++b;
    }
  }
}

// Degrid / grid of visibilities [0, n): one warp per visibility (sampling
// four at a time in FP32), taken from the work queue.
template <typename T, typename C, bool kGrid, bool kAgain>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 3 : 2)
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
  int nv, pass, P;
  while (series_take<kAgain, T, C>(w, wq, head, static_cast<unsigned long long>(batch), n, recs,
                                   sv, q, lane, i0, nv, pass, P, my_nodes)) {
#pragma unroll 1
    for (int v = 0; v < nv; ++v) {
      if (!((pass >> v) & 1)) continue;
      const VisRec<T> rv = recs[i0 + v];
      const int NP = series_intervals(rv.jw, sv.inv_delta_f);
      w.polynomials(v, NP, lane);
      const int64_t gbase = static_cast<int64_t>(stack_slot[rv.stack]) * npad * npad;
      const uint32_t pm = perm[i0 + v];
      const C yv = kGrid ? load_visibility<T, C>(vis_in, pm, static_cast<T>(rv.weight))
                         : cmake<C>(0.0, 0.0);
      C acc = cmake<C>(0.0, 0.0);
      const int half = rv.jw / 2;
      const int u0 = wrap_index(rv.bu - half + 1, npad), v0 = wrap_index(rv.bv - half + 1, npad);
      if (u0 + rv.jw <= npad && v0 + rv.jw <= npad) {
        const int64_t o0 = gbase + static_cast<int64_t>(v0) * npad + u0;
        const C* gin = kGrid ? nullptr : grid_in + o0;
        C* gout = kGrid ? grid_out + o0 : nullptr;
        const FixedGrid fx = fixed_offset(q.fx, o0);
        if (sizeof(T) == 4 && w.slots == 64)
          series_taps<true, kGrid, 64>(w, rv, sv.inv_delta, npad, gin, gout, fx, yv, acc, lane);
        else
          series_taps<true, kGrid, 0>(w, rv, sv.inv_delta, npad, gin, gout, fx, yv, acc, lane);
      } else {
        series_taps<false, kGrid, 0>(w, rv, sv.inv_delta, npad,
                                     kGrid ? nullptr : grid_in + gbase,
                                     kGrid ? grid_out + gbase : nullptr,
                                     fixed_offset(q.fx, gbase), yv, acc, lane);
      }
      if (lane == 0) {
        my_taps += static_cast<unsigned long long>(rv.jw * rv.jw);
        if (!kAgain) my_nodes += static_cast<unsigned long long>((NP + 1) * kNodes * P);
      }
      if (!kGrid) store_visibility<T, C>(acc, static_cast<T>(rv.weight), pm, vis_out, lane);
      __syncwarp();   // the polynomials are rewritten for the next visibility
    }
  }
  flush_counts(stats, 0, my_taps, my_nodes, lane);
}
