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
// in and out per stack and direction, where the image step's write and the
// library's two passes over the padded grid moved 5 times that.  8 stacks of
// 4096^2 in FP32: forward 0.57 ms (image step 0.24 and cuFFT 1.01), adjoint
// 0.56 ms (cuFFT 1.03 and image step 0.11), and no library workspace (1 GiB).
// Bound: the exchanges (the row passes keep the shared-memory pipe 70-78%
// busy, the column passes 50-57% with 16 warps per SM); DRAM at 4.1-4.3 TB/s
// in the column passes.  Tried for them: tiles by cp.async into two buffers
// (0.54 and 0.60 ms), by plain loads and stores 4 columns wide (0.53), 2
// columns (0.73), 64 registers (0.83, spills).
//
// An N-point transform runs over N / 16 threads of 16 values each, in radix-16
// Stockham steps and a last one of radix N / 16^k, exchanged through shared
// memory (one value in nine left free: power-of-two strides then meet no bank
// twice).  A butterfly's twiddles are products of its 1st, 2nd, 4th and 8th
// powers, which lie in a table per step, neighbouring threads' side by side
// (gathered from one table of W^k they took 16 wavefronts a load).
#pragma once

constexpr int kFftMinLog = 6, kFftMinLog64 = 9, kFftMaxLog = 11;

// log2 N when the two-pass transforms take the plan's grid, or 0.  FP64 from
// N = 512 on (six stacks of 512^2: 0.76 ms, separate steps 1.11); below, its
// few rows fill too little of the chip's FP64 units (128^2: 0.080 against
// 0.050 ms).
__host__ inline int fft_log(int N, int npad, bool f64) {
  if (npad != 2 * N) return 0;
  for (int l = f64 ? kFftMinLog64 : kFftMinLog; l <= kFftMaxLog; ++l)
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
// per tile of the column passes (32 bytes of a row at N = 2048, 128 at most),
// each column's exchange memory with 16 / C values more, so that the columns
// of a half-warp meet no bank twice.
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

// The column passes move their tiles (fft_cols columns of one grid) by TMA:
// N rows of a tile at a time into shared memory, [row][column], and results
// out of it, while the tile before is transformed.  A tile's rows are 32 to
// 128 bytes long and a grid row apart, so that loads and stores by the
// threads cost the shared-memory pipe one wavefront for each row of a warp's
// request: 0.53 ms for 8 grids of 4096^2, more than half of it that, against
// 0.38 (forward) and 0.37 (adjoint).  One block per SM, tiles in turn.
//
// The tensor maps (fft_maps): `image` the rows 0 .. N - 1 of every grid,
// [grid][row][column]; `half` all 2 N rows, [grid][row mod 2][row / 2][column].
// Boxes of fft_cols columns and min(N, 256) rows.
__device__ __forceinline__ unsigned fft_smem_addr(const void* p) {
  return static_cast<unsigned>(__cvta_generic_to_shared(p));
}
// TMA boxes start on 128-byte boundaries of shared memory.
__device__ __forceinline__ unsigned char* fft_aligned(unsigned char* p) {
  return p + ((128u - fft_smem_addr(p)) & 127u);
}
__device__ __forceinline__ void fft_bar_init(unsigned long long* bar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(fft_smem_addr(bar)) : "memory");
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void fft_bar_expect(unsigned long long* bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(fft_smem_addr(bar)),
               "r"(bytes)
               : "memory");
}
// Waits for the phase of the given parity, polling `limit` times at most; false
// if it did not complete.
constexpr int kFftWaitLimit = 1 << 20;   // polls of about a microsecond each
__device__ __forceinline__ bool fft_bar_wait(unsigned long long* bar, unsigned parity, int limit) {
  for (int i = 0; i < limit; ++i) {
    unsigned done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, 1000;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(fft_smem_addr(bar)), "r"(parity)
        : "memory");
    if (done) return true;
  }
  return false;
}
// What a block does about the tiles it will not transform, after its copies
// have been waited for: it records that it gave up, and every row of those
// tiles that the next pass reads becomes NaN, so that no result computed from
// them passes for a value.
template <typename T, typename C, int N, int NC>
__device__ __noinline__ void fft_give_up(C* __restrict__ grids, int rows, int tile, int tiles,
                                         int* __restrict__ timeout) {
  constexpr int kTiles = 2 * N / NC;
  if (threadIdx.x == 0) *timeout = 1;
  C nan;
  nan.x = nan.y = static_cast<T>(NAN);
  for (; tile < tiles; tile += gridDim.x) {
    C* g = grids + static_cast<int64_t>(tile / kTiles) * 4 * N * N + tile % kTiles * NC;
    for (int i = threadIdx.x; i < rows * NC; i += blockDim.x)
      g[static_cast<int64_t>(i / NC) * 2 * N + i % NC] = nan;
  }
}
// N rows of a tile into buf: rows of the image map, or rows of one parity of
// the half map (one thread).
template <typename C, int N, int NC, bool kHalf>
__device__ __forceinline__ void fft_tile_load(C* buf, const FftMaps* maps, int col, int parity,
                                              int grid, unsigned long long* bar) {
  constexpr int kBox = N < 256 ? N : 256;
  fft_bar_expect(bar, static_cast<unsigned>(sizeof(C)) * N * NC);
  // columns in 8-byte units
  const int x = col * static_cast<int>(sizeof(C) / 8);
#pragma unroll 1
  for (int r = 0; r < N; r += kBox) {
    const unsigned dst = fft_smem_addr(buf + r * NC);
    if (kHalf)
      asm volatile(
          "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], "
          "[%1, {%2, %3, %4, %5}], [%6];" ::"r"(dst),
          "l"(&maps->half), "r"(x), "r"(r), "r"(parity), "r"(grid), "r"(fft_smem_addr(bar))
          : "memory");
    else
      asm volatile(
          "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], "
          "[%1, {%2, %3, %4}], [%5];" ::"r"(dst),
          "l"(&maps->image), "r"(x), "r"(r), "r"(grid), "r"(fft_smem_addr(bar))
          : "memory");
  }
}
// The same rows from buf to the grid (one thread, after fft_publish).
template <typename C, int N, int NC, bool kHalf>
__device__ __forceinline__ void fft_tile_store(const C* buf, const FftMaps* maps, int col,
                                               int parity, int grid) {
  constexpr int kBox = N < 256 ? N : 256;
  const int x = col * static_cast<int>(sizeof(C) / 8);
#pragma unroll 1
  for (int r = 0; r < N; r += kBox) {
    const unsigned src = fft_smem_addr(buf + r * NC);
    if (kHalf)
      asm volatile(
          "cp.async.bulk.tensor.4d.global.shared::cta.bulk_group [%0, {%1, %2, %3, %4}], [%5];" ::"l"(
              &maps->half),
          "r"(x), "r"(r), "r"(parity), "r"(grid), "r"(src)
          : "memory");
    else
      asm volatile(
          "cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%0, {%1, %2, %3}], [%4];" ::"l"(
              &maps->image),
          "r"(x), "r"(r), "r"(grid), "r"(src)
          : "memory");
  }
  asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}
__device__ __forceinline__ void fft_stores_read() {   // their source may be rewritten
  asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
}
__device__ __forceinline__ void fft_stores_done() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
// Makes this thread's writes to shared memory visible to the TMA unit.
__device__ __forceinline__ void fft_publish() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// Column pass of the forward transform, in place: rows 0 .. N - 1 (image
// rows) to rows 0 .. 2 N - 1 of the transform, even ones first.
template <typename T, typename C, int kLog>
__global__ void __launch_bounds__(fft_col_threads<kLog, T>())
    fft_cols_forward_kernel(const C* __restrict__ tab, const __grid_constant__ FftMaps maps,
                            C* __restrict__ grids, int tiles, int limit,
                            int* __restrict__ timeout) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ __align__(8) unsigned long long bar;
  // a thread's wait ran out, read after the next barrier (__syncthreads_or, as
  // in the adjoint, spills here)
  __shared__ int failed;
  constexpr int N = 1 << kLog, TPC = N / 16, NC = fft_cols<kLog, T>(), kTiles = 2 * N / NC;
  const int c = threadIdx.x % NC, j = threadIdx.x / NC;
  C* in = reinterpret_cast<C*>(fft_aligned(smem_raw));
  C* out = in + N * NC;
  C* sh = out + N * NC + c * fft_col_elems<kLog, T>();
  const bool lead = threadIdx.x == 0;
  if (lead) {
    failed = 0;
    fft_bar_init(&bar);
    fft_tile_load<C, N, NC, false>(in, &maps, blockIdx.x % kTiles * NC, 0, blockIdx.x / kTiles, &bar);
  }
  __syncthreads();
  unsigned parity = 0;
  int tile = blockIdx.x;
  for (; tile < tiles; tile += gridDim.x, parity ^= 1) {
    const int col = tile % kTiles * NC, grid = tile / kTiles, next = tile + gridDim.x;
    if (!fft_bar_wait(&bar, parity, limit)) failed = 1;
    C v[16];
#pragma unroll
    for (int m = 0; m < 16; ++m) v[m] = in[((j + m * TPC) ^ (N / 2)) * NC + c];
    fft_points<kLog, -1>(v, sh, j, tab);
    if (lead) fft_stores_read();
    __syncthreads();
    if (failed) break;   // the whole block; the tile's load is the one copy in flight
#pragma unroll
    for (int m = 0; m < 16; ++m) out[(j + m * TPC) * NC + c] = v[m];
    fft_publish();
    __syncthreads();
    if (lead) fft_tile_store<C, N, NC, true>(out, &maps, col, 0, grid);
#pragma unroll
    for (int m = 0; m < 16; ++m) {
      const int n = j + m * TPC;
      v[m] = fft_mul(in[(n ^ (N / 2)) * NC + c], tab[n < N / 2 ? n : n + N]);
    }
    __syncthreads();   // the tile has been read
    if (lead && next < tiles)
      fft_tile_load<C, N, NC, false>(in, &maps, next % kTiles * NC, 0, next / kTiles, &bar);
    fft_points<kLog, -1>(v, sh, j, tab);
    if (lead) fft_stores_read();
    __syncthreads();
#pragma unroll
    for (int m = 0; m < 16; ++m) out[(j + m * TPC) * NC + c] = v[m];
    fft_publish();
    __syncthreads();
    if (lead) fft_tile_store<C, N, NC, true>(out, &maps, col, 1, grid);
  }
  if (failed) {
    if (lead) fft_bar_wait(&bar, parity, kFftWaitLimit);
    __syncthreads();
    fft_give_up<T, C, N, NC>(grids, 2 * N, tile, tiles, timeout);
  }
  if (lead) fft_stores_done();
}

// Column pass of the adjoint, in place: 2 N rows to rows 0 .. N - 1 (image
// rows).  One buffer for the even rows and one for the odd, each refilled as
// soon as it has been read; the results leave from the exchange's memory (from
// the even rows' buffer, which then waited for them: 0.52 ms).
template <typename T, typename C, int kLog>
__global__ void __launch_bounds__(fft_col_threads<kLog, T>())
    fft_cols_adjoint_kernel(const C* __restrict__ tab, const __grid_constant__ FftMaps maps,
                            C* __restrict__ grids, int tiles, int limit,
                            int* __restrict__ timeout) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ __align__(8) unsigned long long bars[2];
  constexpr int N = 1 << kLog, TPC = N / 16, NC = fft_cols<kLog, T>(), kTiles = 2 * N / NC;
  const int c = threadIdx.x % NC, j = threadIdx.x / NC;
  C* buf = reinterpret_cast<C*>(fft_aligned(smem_raw));   // even rows
  C* buf1 = buf + N * NC;                                 // odd rows
  C* out = buf1 + N * NC;                                 // results, over the exchange
  C* sh = out + c * fft_col_elems<kLog, T>();
  const bool lead = threadIdx.x == 0;
  if (lead) {
    fft_bar_init(&bars[0]);
    fft_bar_init(&bars[1]);
    const int col = blockIdx.x % kTiles * NC, grid = blockIdx.x / kTiles;
    fft_tile_load<C, N, NC, true>(buf, &maps, col, 0, grid, &bars[0]);
    fft_tile_load<C, N, NC, true>(buf1, &maps, col, 1, grid, &bars[1]);
  }
  __syncthreads();
  unsigned parity = 0;
  int tile = blockIdx.x;
  // leaves; parity0: of the load last sent to the even rows' buffer (one load
  // may be in flight to each)
  auto give_up = [&](unsigned parity0) {
    if (lead) {
      fft_bar_wait(&bars[0], parity0, kFftWaitLimit);
      fft_bar_wait(&bars[1], parity, kFftWaitLimit);
    }
    __syncthreads();
    fft_give_up<T, C, N, NC>(grids, N, tile, tiles, timeout);
  };
  for (; tile < tiles; tile += gridDim.x, parity ^= 1) {
    const int col = tile % kTiles * NC, grid = tile / kTiles, next = tile + gridDim.x;
    C even[16], v[16];
    bool late = !fft_bar_wait(&bars[0], parity, limit);
#pragma unroll
    for (int m = 0; m < 16; ++m) even[m] = buf[(j + m * TPC) * NC + c];
    if (lead) fft_stores_read();   // the exchange's memory is free again
    if (__syncthreads_or(late)) {  // and the even rows have been read
      give_up(parity);             // the whole block
      break;
    }
    if (lead && next < tiles)
      fft_tile_load<C, N, NC, true>(buf, &maps, next % kTiles * NC, 0, next / kTiles, &bars[0]);
    fft_points<kLog, 1>(even, sh, j, tab);
    late = !fft_bar_wait(&bars[1], parity, limit);
#pragma unroll
    for (int m = 0; m < 16; ++m) v[m] = buf1[(j + m * TPC) * NC + c];
    if (__syncthreads_or(late)) {  // the odd rows have been read
      give_up(next < tiles ? parity ^ 1 : parity);
      break;
    }
    if (lead && next < tiles)
      fft_tile_load<C, N, NC, true>(buf1, &maps, next % kTiles * NC, 1, next / kTiles, &bars[1]);
    fft_points<kLog, 1>(v, sh, j, tab);
    __syncthreads();               // the last exchange has been read
#pragma unroll
    for (int m = 0; m < 16; ++m) {
      const int n = j + m * TPC;
      out[(n ^ (N / 2)) * NC + c] =
          fft_add(even[m], fft_mul(v[m], fft_root<1>(tab[n < N / 2 ? n : n + N])));
    }
    fft_publish();
    __syncthreads();
    if (lead) fft_tile_store<C, N, NC, false>(out, &maps, col, 0, grid);
  }
  if (lead) fft_stores_done();
}

// Row pass of the adjoint: row p of every grid of the group, times conj(S~_k),
// real part, summed over the stacks into image row p.  One block per row (or
// rows: fft_rows); where the rows of a small image leave the chip idle the
// stacks are split over `groups` sets of threads of the block (set g takes
// stacks g, g + groups, ...), whose sums are added in the order of the sets.
// Serial over the stacks, one warp for 8 rows of 64^2 took 1.4 us a stack (24
// stacks 38.7 us, with the sets 15.5; 126 177 and 55; 128^2, 24 stacks, 42.6
// and 14.7), and the whole adjoint call was slower than by the library's
// transforms from 12 stacks of 64^2 and 4 of 128^2 on.  Images of 512^2 and
// more have rows enough (and spill with two sets).
template <int kLog, typename T> __host__ __device__ constexpr int fft_adjoint_groups() {
  return sizeof(T) == 4 && kLog <= 8 ? 8 : 1;
}
template <typename T, typename C, int kLog, bool kSplit>
__global__ void __launch_bounds__(fft_row_threads<kLog>() * (kSplit ? fft_adjoint_groups<kLog, T>() : 1),
                                  kSplit ? 1 : (sizeof(T) == 4 ? 384 : 256) / fft_row_threads<kLog>())
    fft_rows_adjoint_kernel(const C* __restrict__ grids,
                            const typename PixelPhase<T>::omn* __restrict__ omn,
                            const T* __restrict__ corr, const double* __restrict__ wbar,
                            const int32_t* __restrict__ stacks, int nslots,
                            const C* __restrict__ tab, T* __restrict__ x, int accumulate) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  struct __align__(2 * sizeof(C)) Pair { C c[2]; };
  constexpr int N = 1 << kLog, TPR = N / 16, kThreads = fft_row_threads<kLog>();
  const int groups = kSplit ? static_cast<int>(blockDim.x) / kThreads : 1;
  const int group = kSplit ? static_cast<int>(threadIdx.x) / kThreads : 0;
  const int t = kSplit ? static_cast<int>(threadIdx.x) % kThreads : static_cast<int>(threadIdx.x);
  const int j = t % TPR, rl = t / TPR;
  C* sh = reinterpret_cast<C*>(smem_raw) + (group * fft_rows<kLog>() + rl) * fft_row_elems<kLog>();
  const int row = blockIdx.x * fft_rows<kLog>() + rl;
  const int64_t pix = static_cast<int64_t>(row) * N;
  T acc[16];
#pragma unroll
  for (int m = 0; m < 16; ++m) acc[m] = T(0);
#pragma unroll 1
  for (int s0 = 0; s0 < nslots; s0 += groups) {
    const int sl = s0 + group;
    const bool on = !kSplit || sl < nslots;   // the others keep step at the block's barriers
    const PixelPhase<T> phase(wbar[stacks[on ? sl : 0]]);
    const Pair* src = reinterpret_cast<const Pair*>(
        grids + (static_cast<int64_t>(on ? sl : 0) * 2 * N + row) * 2 * N);
    C even[16], odd[16];
#pragma unroll
    for (int m = 0; m < 16; ++m) {
      const Pair p = src[j + m * TPR];
      even[m] = p.c[0];
      odd[m] = p.c[1];
    }
    fft_points<kLog, 1>(even, sh, j, tab);
    fft_points<kLog, 1>(odd, sh, j, tab);
    if (on) {
#pragma unroll
      for (int m = 0; m < 16; ++m) {
        const int n = j + m * TPR;
        const C g = fft_add(even[m], fft_mul(odd[m], fft_root<1>(tab[n < N / 2 ? n : n + N])));
        const C e = phase(omn[pix + (n ^ (N / 2))]);
        acc[m] += e.x * g.x + e.y * g.y;
      }
    }
  }
  auto put = [&](int m, T sum) {
    const int64_t at = pix + ((j + m * TPR) ^ (N / 2));
    const T v = corr[at] * sum;
    x[at] = accumulate ? x[at] + v : v;
  };
  if (!kSplit) {
#pragma unroll
    for (int m = 0; m < 16; ++m) put(m, acc[m]);
    return;
  }
  // [set][m][thread], over the exchange; the first set adds and stores (all
  // sixteen loads of corr at once; a few m to each set, in turn, took 2 us more)
  T* part = reinterpret_cast<T*>(smem_raw);
  static_assert(16 * kThreads * sizeof(T) <= sizeof(C) * fft_rows<kLog>() * fft_row_elems<kLog>(),
                "a set's sums must fit its exchange memory");
  __syncthreads();
#pragma unroll
  for (int m = 0; m < 16; ++m) part[(group * 16 + m) * kThreads + t] = acc[m];
  __syncthreads();
  if (group) return;
  for (int g = 1; g < groups; ++g)
#pragma unroll
    for (int m = 0; m < 16; ++m) acc[m] += part[(g * 16 + m) * kThreads + t];
#pragma unroll
  for (int m = 0; m < 16; ++m) put(m, acc[m]);
}
