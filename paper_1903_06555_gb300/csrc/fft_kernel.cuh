// Image-domain steps and FFTs in two passes for the common grids: images of
// N = 2^6 .. 2^11 pixels padded to 2 N.  Not a standalone header: phi_ops.cu
// includes it inside namespace phi.
//
// Only N of the 2 N rows and columns of the padded image hold pixels, so in
// each direction the 2 N-point transform is two N-point ones.  With n' =
// -N/2 .. N/2 - 1 the pixel's offset and W = e^{-2 pi i / 2N}:
//
//   forward  X[2 k + e] = sum_n' (x[n'] W^{e n'}) e^{-2 pi i n' k / N},  e = 0, 1
//   adjoint  x[n'] = sum_k X[2k] e^{2 pi i n' k / N}
//                    + W^{-n'} sum_k X[2k + 1] e^{2 pi i n' k / N}
//
// Forward: the row pass applies S~_k to an image row and writes its 2 N
// columns (row p of the image to row p of the grid), the column pass turns
// the N rows into 2 N in place.  Adjoint: the column pass turns 2 N rows into
// N, the row pass transforms them, applies conj(S~_k), sums over the group's
// stacks and writes the image.  Against separate steps around a library FFT
// the zero half is neither written, transformed nor read: 2 N^2 grid values
// of 8 bytes in and out per stack and direction in place of 5 of prep (write)
// and the FFT's two passes: 8 stacks of 4096^2 in
// FP32, forward 0.73 ms (prep 0.24 and cuFFT 1.01), adjoint 0.73 ms (cuFFT
// 1.03 and the image step 0.11), and no library workspace (1 GiB).  Bound: the
// column passes by the latency of their exchanges (16 warps per SM; 3 TB/s),
// the row passes by shared memory (75%).  Tried for the column passes:
// persistent blocks with the next tile by cp.async (0.54 and 0.60 ms against
// 0.53), 2 columns in place of 4 (0.73), 64 registers (0.83, spills).
//
// An N-point transform runs over N / 16 threads of 16 values each, in radix-16
// Stockham steps and a last one of radix N / 16^k, exchanged through shared
// memory (one value in nine left free: power-of-two strides then meet no bank
// twice).  A butterfly's twiddles are products of its 1st, 2nd, 4th and 8th
// powers, which lie in a table per step, neighbouring threads' side by side
// (gathered from one table of W^k they took 16 wavefronts a load).
#pragma once

constexpr int kFftMinLog = 6, kFftMaxLog = 11;

// log2 N when the two-pass transforms take the plan's grid, or 0.  FP64 from
// N = 512 on (six stacks of 512^2: 0.76 ms, separate steps 1.11); below, its
// few rows fill too little of the chip's FP64 units (128^2: 0.080 against
// 0.050 ms).
__host__ inline int fft_log(int N, int npad, bool f64) {
  if (npad != 2 * N) return 0;
  for (int l = f64 ? 9 : kFftMinLog; l <= kFftMaxLog; ++l)
    if (N == 1 << l) return l;
  return 0;
}

// Roots of unity: W^k = e^{-2 pi i k / 2N} for k < 2 N; then for the steps
// after the first, with Ns = 16 and 256 points done and radix R, e^{-2 pi i
// 2^q k / (Ns R)}, k < Ns, q = 0 .. 3.
__host__ __device__ constexpr int fft_step_radix(int log, int done) {
  return log - done >= 4 ? 16 : 1 << (log - done);
}
__host__ __device__ constexpr int fft_step_table(int N, int done) { return 2 * N + (done == 4 ? 0 : 64); }
__host__ __device__ constexpr int fft_table_size(int N) { return 2 * N + 64 + 1024; }
template <typename T, typename C>
__global__ void fft_table_kernel(int log, C* __restrict__ w) {
  const int N = 1 << log;
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= fft_table_size(N)) return;
  double turns;
  if (k < 2 * N) {
    turns = static_cast<double>(k) / (2 * N);
  } else {
    const int e = k - 2 * N, done = e < 64 ? 4 : 8, Ns = 1 << done;
    const int i = done == 4 ? e : e - 64;
    const int R = log > done ? fft_step_radix(log, done) : 1;
    turns = static_cast<double>((1 << (i / Ns)) * (i % Ns)) / (static_cast<double>(Ns) * R);
  }
  double sn, cs;
  sincospi(-2.0 * turns, &sn, &cs);
  w[k] = cmake<C>(cs, sn);
}

template <typename C>
__device__ __forceinline__ C fft_add(const C& a, const C& b) {
  C r;
  r.x = a.x + b.x;
  r.y = a.y + b.y;
  return r;
}
template <typename C>
__device__ __forceinline__ C fft_sub(const C& a, const C& b) {
  C r;
  r.x = a.x - b.x;
  r.y = a.y - b.y;
  return r;
}
template <typename C>
__device__ __forceinline__ C fft_mul(const C& a, const C& b) {
  C r;
  r.x = fma(a.x, b.x, -(a.y * b.y));
  r.y = fma(a.x, b.y, a.y * b.x);
  return r;
}
// a times e^{kSign i pi / 2}
template <int kSign, typename C>
__device__ __forceinline__ C fft_turn(const C& a) {
  C r;
  r.x = kSign > 0 ? -a.y : a.y;
  r.y = kSign > 0 ? a.x : -a.x;
  return r;
}
// w or its conjugate (the table holds the forward roots).
template <int kSign, typename C>
__device__ __forceinline__ C fft_root(const C& w) {
  C r = w;
  if (kSign > 0) r.y = -r.y;
  return r;
}

template <int kSign, typename C>
__device__ __forceinline__ void fft_radix2(C& a, C& b) {
  const C s = fft_add(a, b), d = fft_sub(a, b);
  a = s;
  b = d;
}
template <int kSign, typename C>
__device__ __forceinline__ void fft_radix4(C& a, C& b, C& c, C& d) {
  const C s0 = fft_add(a, c), s1 = fft_sub(a, c), s2 = fft_add(b, d);
  const C s3 = fft_turn<kSign>(fft_sub(b, d));
  a = fft_add(s0, s2);
  b = fft_add(s1, s3);
  c = fft_sub(s0, s2);
  d = fft_sub(s1, s3);
}
// a times e^{kSign 2 pi i k / 16}
template <int kSign, int k, typename C>
__device__ __forceinline__ C fft_turn16(const C& a) {
  typedef decltype(a.x + a.x) T;
  if constexpr (k == 0) return a;
  if constexpr (k == 4) return fft_turn<kSign>(a);
  constexpr double c1 = 0.92387953251128675613, s1 = 0.38268343236508977173,
                   r2 = 0.70710678118654752440;
  constexpr double cs = k == 1 ? c1 : k == 2 ? r2 : k == 3 ? s1 : k == 6 ? -r2 : k == 9 ? -c1 : 0.0;
  constexpr double sn = k == 1 ? s1 : k == 2 ? r2 : k == 3 ? c1 : k == 6 ? r2 : k == 9 ? -s1 : 0.0;
  C w;
  w.x = static_cast<T>(cs);
  w.y = static_cast<T>(kSign * sn);
  return fft_mul(a, w);
}

// R-point transform of v[0], v[st], ..; the result X[i] is at v[st pos(i)].
template <int R> __device__ __forceinline__ constexpr int fft_pos(int i) {
  return R == 16 ? 4 * (i & 3) + (i >> 2) : R == 8 ? 2 * (i & 3) + (i >> 2) : i;
}
template <int R, int kSign, int st, typename C>
__device__ __forceinline__ void fft_radix(C* v) {
  if constexpr (R == 2) {
    fft_radix2<kSign>(v[0], v[st]);
  } else if constexpr (R == 4) {
    fft_radix4<kSign>(v[0], v[st], v[2 * st], v[3 * st]);
  } else if constexpr (R == 8) {
    // n = 2 n1 + n2, k = k1 + 4 k2
    fft_radix4<kSign>(v[0], v[2 * st], v[4 * st], v[6 * st]);
    fft_radix4<kSign>(v[st], v[3 * st], v[5 * st], v[7 * st]);
    v[3 * st] = fft_turn16<kSign, 2>(v[3 * st]);
    v[5 * st] = fft_turn16<kSign, 4>(v[5 * st]);
    v[7 * st] = fft_turn16<kSign, 6>(v[7 * st]);
#pragma unroll
    for (int k = 0; k < 4; ++k) fft_radix2<kSign>(v[2 * k * st], v[(2 * k + 1) * st]);
  } else {
    static_assert(R == 16, "radix");
    // n = 4 n1 + n2, k = k1 + 4 k2
#pragma unroll
    for (int n = 0; n < 4; ++n) fft_radix4<kSign>(v[n * st], v[(4 + n) * st], v[(8 + n) * st], v[(12 + n) * st]);
    v[5 * st] = fft_turn16<kSign, 1>(v[5 * st]);
    v[6 * st] = fft_turn16<kSign, 2>(v[6 * st]);
    v[7 * st] = fft_turn16<kSign, 3>(v[7 * st]);
    v[9 * st] = fft_turn16<kSign, 2>(v[9 * st]);
    v[10 * st] = fft_turn16<kSign, 4>(v[10 * st]);
    v[11 * st] = fft_turn16<kSign, 6>(v[11 * st]);
    v[13 * st] = fft_turn16<kSign, 3>(v[13 * st]);
    v[14 * st] = fft_turn16<kSign, 6>(v[14 * st]);
    v[15 * st] = fft_turn16<kSign, 9>(v[15 * st]);
#pragma unroll
    for (int k = 0; k < 4; ++k)
      fft_radix4<kSign>(v[4 * k * st], v[(4 * k + 1) * st], v[(4 * k + 2) * st], v[(4 * k + 3) * st]);
  }
}

__host__ __device__ constexpr int fft_pad(int i) { return i + (i >> 3); }

// One Stockham step: thread j of N / 16 holds values m = 0 .. 15 at positions
// j + m N / 16, 16 / R butterflies of R; after it the values go to `sh` in
// the order of the next step (or stay, in order, after the last).
template <int kLog, int kDone, int kSign, typename C>
__device__ __forceinline__ void fft_steps(C (&v)[16], C* sh, int j, const C* __restrict__ tab) {
  constexpr int N = 1 << kLog, Ns = 1 << kDone;
  constexpr int R = kLog - kDone >= 4 ? 16 : 1 << (kLog - kDone);
  constexpr int B = 16 / R;                    // butterflies per thread
#pragma unroll
  for (int b = 0; b < B; ++b) {
    const int jb = j + b * (N / 16);
    if constexpr (kDone > 0) {
      const C* __restrict__ t = tab + fft_step_table(N, kDone) + (jb & (Ns - 1));
      const C w1 = fft_root<kSign>(t[0]);
      v[b + B] = fft_mul(v[b + B], w1);
      if constexpr (R >= 4) {
        const C w2 = fft_root<kSign>(t[Ns]);
        const C w3 = fft_mul(w1, w2);
        v[b + 2 * B] = fft_mul(v[b + 2 * B], w2);
        v[b + 3 * B] = fft_mul(v[b + 3 * B], w3);
        if constexpr (R >= 8) {
          const C w4 = fft_root<kSign>(t[2 * Ns]);
          v[b + 4 * B] = fft_mul(v[b + 4 * B], w4);
          v[b + 5 * B] = fft_mul(v[b + 5 * B], fft_mul(w4, w1));
          v[b + 6 * B] = fft_mul(v[b + 6 * B], fft_mul(w4, w2));
          v[b + 7 * B] = fft_mul(v[b + 7 * B], fft_mul(w4, w3));
          if constexpr (R >= 16) {
            const C w8 = fft_root<kSign>(t[3 * Ns]);
            v[8] = fft_mul(v[8], w8);
            v[9] = fft_mul(v[9], fft_mul(w8, w1));
            v[10] = fft_mul(v[10], fft_mul(w8, w2));
            v[11] = fft_mul(v[11], fft_mul(w8, w3));
            const C w12 = fft_mul(w8, w4);
            v[12] = fft_mul(v[12], w12);
            v[13] = fft_mul(v[13], fft_mul(w12, w1));
            v[14] = fft_mul(v[14], fft_mul(w12, w2));
            v[15] = fft_mul(v[15], fft_mul(w12, w3));
          }
        }
      }
    }
    fft_radix<R, kSign, B>(v + b);
  }
  if constexpr ((1 << kDone) * R == N) {
    C o[16];
#pragma unroll
    for (int b = 0; b < B; ++b)
#pragma unroll
      for (int i = 0; i < R; ++i) o[b + i * B] = v[b + fft_pos<R>(i) * B];
#pragma unroll
    for (int m = 0; m < 16; ++m) v[m] = o[m];
  } else {
    __syncthreads();                           // the last reads of sh are done
#pragma unroll
    for (int b = 0; b < B; ++b) {
      const int jb = j + b * (N / 16);
      const int base = (jb & ~(Ns - 1)) * R + (jb & (Ns - 1));
#pragma unroll
      for (int i = 0; i < R; ++i) sh[fft_pad(base + i * Ns)] = v[b + fft_pos<R>(i) * B];
    }
    __syncthreads();
#pragma unroll
    for (int m = 0; m < 16; ++m) v[m] = sh[fft_pad(j + m * (N / 16))];
    fft_steps<kLog, kDone + 4, kSign>(v, sh, j, tab);
  }
}
template <int kLog, int kSign, typename C>
__device__ __forceinline__ void fft_points(C (&v)[16], C* sh, int j, const C* __restrict__ tab) {
  fft_steps<kLog, 0, kSign>(v, sh, j, tab);
}

// Shared memory of one transform; rows per block of the row passes (a warp
// at least, and no more than that: small images have few rows); columns
// per block of the column passes (32 bytes of a row at N = 2048, 128 at most:
// neighbouring blocks share their lines in L2), each with 16 / C values more,
// so that the columns of a half-warp meet no bank twice.
template <int kLog> __host__ __device__ constexpr int fft_row_elems() { return fft_pad(1 << kLog); }
template <int kLog> __host__ __device__ constexpr int fft_rows() { return kLog >= 9 ? 1 : 1 << (9 - kLog); }
template <int kLog, typename T> __host__ __device__ constexpr int fft_cols() {
  return (kLog >= 9 ? 1 << (13 - kLog) : 16) * 4 / static_cast<int>(sizeof(T));
}
template <int kLog, typename T> __host__ __device__ constexpr int fft_col_elems() {
  return fft_pad(1 << kLog) + (fft_cols<kLog, T>() >= 16 ? 1 : 16 / fft_cols<kLog, T>());
}
template <int kLog> __host__ __device__ constexpr int fft_row_threads() {
  return fft_rows<kLog>() * (1 << (kLog - 4));
}
template <int kLog, typename T> __host__ __device__ constexpr int fft_col_threads() {
  return fft_cols<kLog, T>() * (1 << (kLog - 4));
}

// Row pass of the forward transform: image row p times S~_k into row p of
// the stack's grid.  The stacks of a row run next to one another (blockIdx.x),
// so that the pixel tables come from memory once.
template <typename T, typename C, int kLog>
__global__ void __launch_bounds__(fft_row_threads<kLog>(), (sizeof(T) == 4 ? 512 : 256) / fft_row_threads<kLog>())
    fft_rows_forward_kernel(const T* __restrict__ x,
                            const typename PixelPhase<T>::omn* __restrict__ omn,
                            const T* __restrict__ corr, const double* __restrict__ wbar,
                            const int32_t* __restrict__ stacks, const C* __restrict__ tab,
                            C* __restrict__ grids) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  struct __align__(2 * sizeof(C)) Pair { C c[2]; };
  constexpr int N = 1 << kLog, TPR = N / 16;
  const int j = threadIdx.x % TPR, rl = threadIdx.x / TPR;
  C* sh = reinterpret_cast<C*>(smem_raw) + rl * fft_row_elems<kLog>();
  const int row = blockIdx.y * fft_rows<kLog>() + rl;
  const PixelPhase<T> phase(wbar[stacks[blockIdx.x]]);
  const int64_t pix = static_cast<int64_t>(row) * N;
  C in[16], even[16];
#pragma unroll
  for (int m = 0; m < 16; ++m) {
    const int n = j + m * TPR;
    const int64_t at = pix + (n ^ (N / 2));    // pixel (n + N / 2) mod N
    const C e = phase(omn[at]);
    const T v = x[at] * corr[at];
    in[m].x = v * e.x;
    in[m].y = v * e.y;
    even[m] = in[m];
  }
  fft_points<kLog, -1>(even, sh, j, tab);
#pragma unroll
  for (int m = 0; m < 16; ++m) {
    const int n = j + m * TPR;
    in[m] = fft_mul(in[m], tab[n < N / 2 ? n : n + N]);
  }
  fft_points<kLog, -1>(in, sh, j, tab);
  Pair* out = reinterpret_cast<Pair*>(grids + (static_cast<int64_t>(blockIdx.x) * 2 * N + row) * 2 * N);
#pragma unroll
  for (int m = 0; m < 16; ++m) {
    Pair o;
    o.c[0] = even[m];
    o.c[1] = in[m];
    out[j + m * TPR] = o;
  }
}

// Column pass of the forward transform, in place: rows 0 .. N - 1 (image rows)
// to rows 0 .. 2 N - 1 of the transform.
template <typename T, typename C, int kLog>
__global__ void __launch_bounds__(fft_col_threads<kLog, T>(),
                                  (sizeof(T) == 4 ? 512 : 256) / fft_col_threads<kLog, T>())
    fft_cols_forward_kernel(const C* __restrict__ tab, C* grids) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int N = 1 << kLog, TPC = N / 16, NC = fft_cols<kLog, T>();
  const int c = threadIdx.x % NC, j = threadIdx.x / NC;
  C* sh = reinterpret_cast<C*>(smem_raw) + c * fft_col_elems<kLog, T>();
  C* col = grids + static_cast<int64_t>(blockIdx.y) * 4 * N * N + blockIdx.x * NC + c;
  C in[16], v[16];
#pragma unroll
  for (int m = 0; m < 16; ++m) {
    const int n = j + m * TPC;
    in[m] = col[static_cast<int64_t>(n ^ (N / 2)) * 2 * N];
    v[m] = in[m];
  }
  fft_points<kLog, -1>(v, sh, j, tab);
  // every row of these columns has been read once the block has passed its
  // first exchange, which precedes this point for all of its threads
#pragma unroll
  for (int m = 0; m < 16; ++m) col[static_cast<int64_t>(j + m * TPC) * 4 * N] = v[m];
#pragma unroll
  for (int m = 0; m < 16; ++m) {
    const int n = j + m * TPC;
    in[m] = fft_mul(in[m], tab[n < N / 2 ? n : n + N]);
  }
  fft_points<kLog, -1>(in, sh, j, tab);
#pragma unroll
  for (int m = 0; m < 16; ++m) col[static_cast<int64_t>(j + m * TPC) * 4 * N + 2 * N] = in[m];
}

// Column pass of the adjoint, in place: 2 N rows to rows 0 .. N - 1 (image rows).
template <typename T, typename C, int kLog>
__global__ void __launch_bounds__(fft_col_threads<kLog, T>(),
                                  (sizeof(T) == 4 ? 512 : 256) / fft_col_threads<kLog, T>())
    fft_cols_adjoint_kernel(const C* __restrict__ tab, C* grids) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int N = 1 << kLog, TPC = N / 16, NC = fft_cols<kLog, T>();
  const int c = threadIdx.x % NC, j = threadIdx.x / NC;
  C* sh = reinterpret_cast<C*>(smem_raw) + c * fft_col_elems<kLog, T>();
  C* col = grids + static_cast<int64_t>(blockIdx.y) * 4 * N * N + blockIdx.x * NC + c;
  C even[16], v[16];
#pragma unroll
  for (int m = 0; m < 16; ++m) even[m] = col[static_cast<int64_t>(j + m * TPC) * 4 * N];
#pragma unroll
  for (int m = 0; m < 16; ++m) v[m] = col[static_cast<int64_t>(j + m * TPC) * 4 * N + 2 * N];
  fft_points<kLog, 1>(even, sh, j, tab);
  fft_points<kLog, 1>(v, sh, j, tab);
  // (both sets of rows were read before the first exchange)
#pragma unroll
  for (int m = 0; m < 16; ++m) {
    const int n = j + m * TPC;
    const C o = fft_add(even[m], fft_mul(v[m], fft_root<1>(tab[n < N / 2 ? n : n + N])));
    col[static_cast<int64_t>(n ^ (N / 2)) * 2 * N] = o;
  }
}

// Row pass of the adjoint: row p of every grid of the group, times conj(S~_k),
// real part, summed over the stacks into image row p.
template <typename T, typename C, int kLog>
__global__ void __launch_bounds__(fft_row_threads<kLog>(), (sizeof(T) == 4 ? 384 : 256) / fft_row_threads<kLog>())
    fft_rows_adjoint_kernel(const C* __restrict__ grids,
                            const typename PixelPhase<T>::omn* __restrict__ omn,
                            const T* __restrict__ corr, const double* __restrict__ wbar,
                            const int32_t* __restrict__ stacks, int nslots,
                            const C* __restrict__ tab, T* __restrict__ x, int accumulate) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  struct __align__(2 * sizeof(C)) Pair { C c[2]; };
  constexpr int N = 1 << kLog, TPR = N / 16;
  const int j = threadIdx.x % TPR, rl = threadIdx.x / TPR;
  C* sh = reinterpret_cast<C*>(smem_raw) + rl * fft_row_elems<kLog>();
  const int row = blockIdx.x * fft_rows<kLog>() + rl;
  const int64_t pix = static_cast<int64_t>(row) * N;
  T acc[16];
#pragma unroll
  for (int m = 0; m < 16; ++m) acc[m] = T(0);
#pragma unroll 1
  for (int sl = 0; sl < nslots; ++sl) {
    const PixelPhase<T> phase(wbar[stacks[sl]]);
    const Pair* src = reinterpret_cast<const Pair*>(
        grids + (static_cast<int64_t>(sl) * 2 * N + row) * 2 * N);
    C even[16], odd[16];
#pragma unroll
    for (int m = 0; m < 16; ++m) {
      const Pair p = src[j + m * TPR];
      even[m] = p.c[0];
      odd[m] = p.c[1];
    }
    fft_points<kLog, 1>(even, sh, j, tab);
    fft_points<kLog, 1>(odd, sh, j, tab);
#pragma unroll
    for (int m = 0; m < 16; ++m) {
      const int n = j + m * TPR;
      const C g = fft_add(even[m], fft_mul(odd[m], fft_root<1>(tab[n < N / 2 ? n : n + N])));
      const C e = phase(omn[pix + (n ^ (N / 2))]);
      acc[m] += e.x * g.x + e.y * g.y;
    }
  }
#pragma unroll
  for (int m = 0; m < 16; ++m) {
    const int64_t at = pix + ((j + m * TPR) ^ (N / 2));
    const T v = corr[at] * acc[m];
    x[at] = accumulate ? x[at] + v : v;
  }
}
