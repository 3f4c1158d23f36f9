// The two passes of fft_kernel.cuh for images of other sizes, up to N = 2046
// pixels padded to 2 N, FP32.  Not a standalone header: phi_ops.cu includes
// it inside namespace phi, after fft_kernel.cuh.
//
// As there, a 2 N-point transform of N values is two N-point ones.  Each is a
// convolution with a chirp (Bluestein 1970): with c[n] = e^{-i pi n^2 / N},
//
//   sum_n x[n] e^{-2 pi i n k / N} = c[k] sum_n (x[n] c[n]) conj(c[k - n]),
//
// cyclic of length M = 2^l >= 2 N - 1 through the radix-16 transforms: M-point
// forward, times the chirp's spectrum (in double precision, then rounded),
// M-point inverse.  n^2 mod 2 N is exact, so the factors are good to rounding
// at every n.  Inputs and wanted outputs fill at most half of M: the thread's
// first 8 of 16 values.
//
// Bound: the exchanges through shared memory, like fft_kernel.cuh's, at four
// times the length per point, and spills: czt_forward holds the input, both
// halves of the output and the 16 working values (152 to 432 bytes a thread at
// 128 registers; the adjoint, which takes the halves in turn, 4 to 152): 8 grids of 3972^2, forward 2.94 ms, adjoint 3.11
// (image steps and cuFFT 5.62 and 5.50), 3.4e-7 and 3.2e-7 from 64 bits (5.2e-7
// and 4.6e-7).
#pragma once

// log2 M when the chirp transforms take the plan's grid, or 0.  The library's
// time depends on the largest prime factor of N.  Forward and adjoint of 8
// stacks, library against these, in ms: 71 and less, none to 1.5 times gained
// (1136 = 16 * 71: 2.5 and 3.0); 73 to 127, 1.3 to 2.3 times (498 = 6 * 83:
// 0.76 and 0.34, 1356 = 12 * 113: 5.9 and 3.7); above, where it convolves too,
// 1.04 to 1.85 times (1402 = 2 * 701: 4.0 and 3.8, 1986 = 6 * 331: 11.1 and
// 6.1), but for images of 608 to 840 pixels, whose rows leave the second wave
// of blocks nearly empty (668 = 4 * 167, adjoint: 0.42 and 0.46).  N must fill
// M's half (524 = 4 * 131, just past 512: 0.56 and 0.57), and below 380 pixels
// the adjoint's rows are too few for the chip (302: 0.106 and 0.107).
__host__ inline int czt_log(int N, int npad, bool f64) {
  if (f64 || npad != 2 * N || N < 380 || N >= 2048) return 0;
  int prime = 1;
  for (int r = N, q = 2; r > 1; q = q == 2 ? 3 : q + 2)
    for (; r % q == 0; r /= q) prime = q;
  if (prime <= 71 || (prime > 127 && N > 608 && N < 840)) return 0;
  int l = 10;
  while ((1 << l) < 2 * N - 1) ++l;
  return 64 * N >= 17 * (1 << l) ? l : 0;
}

// Complex values of the plan's table: the roots of the M-point transforms,
// c[n] and c[n] W^n' (n' the pixel's offset, W = e^{-2 pi i / 2N}), the
// chirp's spectrum over M; then doubles to form it: cos(2 pi k / M), conj(c).
__host__ __device__ constexpr int czt_roots(int log) { return fft_table_size(1 << log); }
__host__ __device__ constexpr int czt_table_size(int N, int log) {
  return czt_roots(log) + 2 * N + (1 << log) + (1 << log) + 2 * N;
}
__global__ void czt_factors_kernel(int N, int M, float2* __restrict__ c, double* __restrict__ cosm,
                                   double2* __restrict__ chirp) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < M) cosm[i] = cospi(2.0 * i / M);
  if (i >= N) return;
  // the phases in units of pi / N, exact: n^2, and n' more
  const int sq = static_cast<int>(static_cast<int64_t>(i) * i % (2 * N));
  const int off = i < N / 2 ? i : i - N;
  double sn, cs;
  sincospi(static_cast<double>(sq) / N, &sn, &cs);
  chirp[i] = make_double2(cs, sn);
  c[i] = cmake<float2>(cs, -sn);
  sincospi(static_cast<double>((sq + off + 2 * N) % (2 * N)) / N, &sn, &cs);
  c[N + i] = cmake<float2>(cs, -sn);
}
// spec[k] = 1 / M sum over |n| < N of conj(c[n]) e^{-2 pi i n k / M}: one block per k.
__global__ void __launch_bounds__(128) czt_spectrum_kernel(int N, int M,
                                                           const double* __restrict__ cosm,
                                                           const double2* __restrict__ chirp,
                                                           float2* __restrict__ spec) {
  __shared__ double2 part[4];
  double2 s = make_double2(0.0, 0.0);
  for (int n = 1 + threadIdx.x; n < N; n += blockDim.x) {
    const double w = 2.0 * cosm[static_cast<int>(static_cast<unsigned>(n) * blockIdx.x & (M - 1u))];
    s.x = fma(w, chirp[n].x, s.x);
    s.y = fma(w, chirp[n].y, s.y);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    s.x += __shfl_xor_sync(0xffffffffu, s.x, o);
    s.y += __shfl_xor_sync(0xffffffffu, s.y, o);
  }
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0)
    spec[blockIdx.x] = cmake<float2>((1.0 + part[0].x + part[1].x + part[2].x + part[3].x) / M,
                                     (part[0].y + part[1].y + part[2].y + part[3].y) / M);
}

// Columns per block of the column passes (512 threads), and the memory of one.
template <int kLog> __host__ __device__ constexpr int czt_cols() { return 1 << (13 - kLog); }
template <int kLog> __host__ __device__ constexpr int czt_col_elems() {
  return fft_pad(1 << kLog) + 16 / czt_cols<kLog>();
}
template <int kLog> __host__ __device__ constexpr int czt_col_threads() {
  return czt_cols<kLog>() * (1 << (kLog - 4));
}

// Thread j's values m < 8, n = j + m M / 16 < N, times in[n]: convolved with
// the chirp.  The caller multiplies the results by their own factors.
template <int kLog>
__device__ __forceinline__ void czt_points(float2 (&v)[16], const float2 (&x)[8],
                                           const float2* __restrict__ in, int N, float2* sh, int j,
                                           const float2* __restrict__ tab,
                                           const float2* __restrict__ spec) {
  constexpr int TPM = 1 << (kLog - 4);
#pragma unroll
  for (int m = 0; m < 8; ++m) {
    const int n = j + m * TPM;
    v[m] = n < N ? fft_mul(x[m], in[n]) : make_float2(0.0f, 0.0f);
    v[m + 8] = make_float2(0.0f, 0.0f);
  }
  fft_points<kLog, -1>(v, sh, j, tab);
#pragma unroll
  for (int m = 0; m < 16; ++m) v[m] = fft_mul(v[m], spec[j + m * TPM]);
  fft_points<kLog, 1>(v, sh, j, tab);
}

// x's N-point transforms: X[2 n] in `even`, X[2 n + 1] in `odd`.
template <int kLog>
__device__ __forceinline__ void czt_forward(const float2 (&x)[8], float2 (&even)[8],
                                            float2 (&odd)[8], const float2* __restrict__ c, int N,
                                            float2* sh, int j, const float2* __restrict__ tab,
                                            const float2* __restrict__ spec) {
  constexpr int TPM = 1 << (kLog - 4);
  float2 v[16];
  czt_points<kLog>(v, x, c, N, sh, j, tab, spec);
#pragma unroll
  for (int m = 0; m < 8; ++m) even[m] = v[m];
  czt_points<kLog>(v, x, c + N, N, sh, j, tab, spec);
#pragma unroll
  for (int m = 0; m < 8; ++m) {
    const int n = min(j + m * TPM, N - 1);
    even[m] = fft_mul(even[m], c[n]);
    odd[m] = fft_mul(v[m], c[n]);
  }
}
// The adjoint: the conjugate of the transforms of the conjugated even and odd
// values, which load(parity, n) gives.
template <int kLog, typename F>
__device__ __forceinline__ void czt_adjoint(float2 (&out)[8], F load, const float2* __restrict__ c,
                                            int N, float2* sh, int j,
                                            const float2* __restrict__ tab,
                                            const float2* __restrict__ spec) {
  constexpr int TPM = 1 << (kLog - 4);
#pragma unroll 1
  for (int parity = 0; parity < 2; ++parity) {
    float2 x[8], v[16];
#pragma unroll
    for (int m = 0; m < 8; ++m) {
      const int n = j + m * TPM;
      x[m] = n < N ? load(parity, n) : make_float2(0.0f, 0.0f);
      x[m].y = -x[m].y;
    }
    czt_points<kLog>(v, x, c, N, sh, j, tab, spec);
#pragma unroll
    for (int m = 0; m < 8; ++m) {
      float2 r = fft_mul(v[m], c[parity * N + min(j + m * TPM, N - 1)]);
      r.y = -r.y;
      out[m] = parity ? fft_add(out[m], r) : r;
    }
  }
}

template <int kLog>
__global__ void __launch_bounds__(fft_row_threads<kLog>(), 512 / fft_row_threads<kLog>())
    czt_rows_forward_kernel(const float* __restrict__ x,
                            const typename PixelPhase<float>::omn* __restrict__ omn,
                            const float* __restrict__ corr, const double* __restrict__ wbar,
                            const int32_t* __restrict__ stacks, const float2* __restrict__ tab,
                            int N, float2* __restrict__ grids) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int TPM = 1 << (kLog - 4);
  const float2* c = tab + czt_roots(kLog);
  const int j = threadIdx.x % TPM, rl = threadIdx.x / TPM;
  float2* sh = reinterpret_cast<float2*>(smem_raw) + rl * fft_row_elems<kLog>();
  const int row = blockIdx.y * fft_rows<kLog>() + rl;
  const PixelPhase<float> phase(wbar[stacks[blockIdx.x]]);
  float2 in[8], even[8], odd[8];
#pragma unroll
  for (int m = 0; m < 8; ++m) {
    const int n = j + m * TPM;
    in[m] = make_float2(0.0f, 0.0f);
    if (n < N && row < N) {
      const int64_t at = static_cast<int64_t>(row) * N + (n < N / 2 ? n + N / 2 : n - N / 2);
      const float2 e = phase(omn[at]);
      const float v = x[at] * corr[at];
      in[m] = make_float2(v * e.x, v * e.y);
    }
  }
  czt_forward<kLog>(in, even, odd, c, N, sh, j, tab, c + 2 * N);
  float4* out = reinterpret_cast<float4*>(grids + (static_cast<int64_t>(blockIdx.x) * 2 * N + row) * 2 * N);
#pragma unroll
  for (int m = 0; m < 8; ++m) {
    const int n = j + m * TPM;
    if (n < N && row < N) out[n] = make_float4(even[m].x, even[m].y, odd[m].x, odd[m].y);
  }
}

// In place, rows 0 .. N - 1 to rows 0 .. 2 N - 1: every value of a column has
// been read when the first is written.
template <int kLog>
__global__ void __launch_bounds__(czt_col_threads<kLog>())
    czt_cols_forward_kernel(const float2* __restrict__ tab, int N, float2* __restrict__ grids) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int TPM = 1 << (kLog - 4), NC = czt_cols<kLog>();
  const float2* c = tab + czt_roots(kLog);
  const int cl = threadIdx.x % NC, j = threadIdx.x / NC, col = blockIdx.x * NC + cl;
  float2* sh = reinterpret_cast<float2*>(smem_raw) + cl * czt_col_elems<kLog>();
  float2* g = grids + static_cast<int64_t>(blockIdx.y) * 4 * N * N + col;
  float2 in[8], even[8], odd[8];
#pragma unroll
  for (int m = 0; m < 8; ++m) {
    const int n = j + m * TPM;
    in[m] = n < N && col < 2 * N
                ? g[static_cast<int64_t>(n < N / 2 ? n + N / 2 : n - N / 2) * 2 * N]
                : make_float2(0.0f, 0.0f);
  }
  czt_forward<kLog>(in, even, odd, c, N, sh, j, tab, c + 2 * N);
#pragma unroll
  for (int m = 0; m < 8; ++m) {
    const int n = j + m * TPM;
    if (n < N && col < 2 * N) {
      g[static_cast<int64_t>(2 * n) * 2 * N] = even[m];
      g[static_cast<int64_t>(2 * n + 1) * 2 * N] = odd[m];
    }
  }
}

// In place, rows 0 .. 2 N - 1 to rows 0 .. N - 1.
template <int kLog>
__global__ void __launch_bounds__(czt_col_threads<kLog>())
    czt_cols_adjoint_kernel(const float2* __restrict__ tab, int N, float2* __restrict__ grids) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int TPM = 1 << (kLog - 4), NC = czt_cols<kLog>();
  const float2* c = tab + czt_roots(kLog);
  const int cl = threadIdx.x % NC, j = threadIdx.x / NC, col = blockIdx.x * NC + cl;
  float2* sh = reinterpret_cast<float2*>(smem_raw) + cl * czt_col_elems<kLog>();
  float2* g = grids + static_cast<int64_t>(blockIdx.y) * 4 * N * N + col;
  float2 out[8];
  czt_adjoint<kLog>(
      out,
      [&](int parity, int n) {
        return col < 2 * N ? g[static_cast<int64_t>(2 * n + parity) * 2 * N] : make_float2(0.0f, 0.0f);
      },
      c, N, sh, j, tab, c + 2 * N);
#pragma unroll
  for (int m = 0; m < 8; ++m) {
    const int n = j + m * TPM;
    if (n < N && col < 2 * N)
      g[static_cast<int64_t>(n < N / 2 ? n + N / 2 : n - N / 2) * 2 * N] = out[m];
  }
}

// As fft_rows_adjoint_kernel, the stacks over two sets of threads where the
// rows of M = 1024 (380 to 512 pixels) fill a third of the chip: 50 stacks of
// 394^2 440 us with one set, 292 with two (the whole call 1031 and 885, by the
// library's transforms 1006); 24 of 498^2 264 and 188.
template <int kLog> __host__ __device__ constexpr int czt_adjoint_groups() { return kLog == 10 ? 2 : 1; }
template <int kLog>
__global__ void __launch_bounds__(fft_row_threads<kLog>() * czt_adjoint_groups<kLog>(),
                                  512 / (fft_row_threads<kLog>() * czt_adjoint_groups<kLog>()))
    czt_rows_adjoint_kernel(const float2* __restrict__ grids,
                            const typename PixelPhase<float>::omn* __restrict__ omn,
                            const float* __restrict__ corr, const double* __restrict__ wbar,
                            const int32_t* __restrict__ stacks, int nslots,
                            const float2* __restrict__ tab, int N, float* __restrict__ x,
                            int accumulate) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int TPM = 1 << (kLog - 4), kThreads = fft_row_threads<kLog>();
  constexpr bool kSplit = czt_adjoint_groups<kLog>() > 1;
  static_assert(fft_rows<kLog>() == 1 && czt_adjoint_groups<kLog>() <= 2, "one row, two sets at most");
  const float2* c = tab + czt_roots(kLog);
  const int groups = kSplit ? blockDim.x / kThreads : 1;
  const int group = kSplit ? threadIdx.x / kThreads : 0, j = threadIdx.x % kThreads;
  float2* sh = reinterpret_cast<float2*>(smem_raw) + group * fft_row_elems<kLog>();
  const int row = blockIdx.x;
  float acc[8];
#pragma unroll
  for (int m = 0; m < 8; ++m) acc[m] = 0.0f;
#pragma unroll 1
  for (int s0 = 0; s0 < nslots; s0 += groups) {
    const int sl = s0 + group;
    const bool on = !kSplit || sl < nslots;   // the other set keeps step at the barriers
    const PixelPhase<float> phase(wbar[stacks[on ? sl : 0]]);
    const float2* src = grids + (static_cast<int64_t>(on ? sl : 0) * 2 * N + row) * 2 * N;
    float2 out[8];
    czt_adjoint<kLog>(
        out, [&](int parity, int n) { return src[2 * n + parity]; }, c, N, sh, j, tab, c + 2 * N);
#pragma unroll
    for (int m = 0; m < 8; ++m) {
      const int n = j + m * TPM;
      if (n < N && on) {
        const float2 e = phase(omn[static_cast<int64_t>(row) * N + (n < N / 2 ? n + N / 2 : n - N / 2)]);
        acc[m] += e.x * out[m].x + e.y * out[m].y;
      }
    }
  }
  if (kSplit && groups > 1) {   // the second set's sums, over the exchange
    float* part = reinterpret_cast<float*>(smem_raw);
    __syncthreads();
    if (group) {
#pragma unroll
      for (int m = 0; m < 8; ++m) part[m * kThreads + j] = acc[m];
    }
    __syncthreads();
    if (group) return;
#pragma unroll
    for (int m = 0; m < 8; ++m) acc[m] += part[m * kThreads + j];
  }
#pragma unroll
  for (int m = 0; m < 8; ++m) {
    const int n = j + m * TPM;
    if (n < N) {
      const int64_t at = static_cast<int64_t>(row) * N + (n < N / 2 ? n + N / 2 : n - N / 2);
      const float v = corr[at] * acc[m];
      x[at] = accumulate ? x[at] + v : v;
    }
  }
}
