// FP32 sgemv, y := alpha op(A) x + beta y (BLAS convention): the Level-2
// operation the paper names as the weak point of its HPL run (Section IV-C,
// V).  Memory-bound: every element of A is read once from HBM, in coalesced
// order, with several independent loads in flight per thread.
//
//   op(A) = A   ("N"): a thread owns four rows and runs over a share of a
//               slice of the columns; x comes through shared memory.  y_i
//               needs the whole row, so when the rows alone give too few
//               blocks the columns are cut into slices whose partial sums a
//               second kernel adds in a fixed order.
//   op(A) = A^T ("T"): a block owns four columns j and runs over a slice of
//               the rows (consecutive rows of a column are consecutive in
//               memory); each x_i is read once for the four columns, and the
//               block's threads are combined in a fixed order.
//
// What bounds both is memory: enough bytes have to be in flight (128 a thread,
// 16-byte loads where every column starts on 16 bytes) in long pieces of a
// column.  Measured on GB300 at 16384^2 (1.07 GB), back to back: N 179.6 ->
// 154 us (7.0 TB/s), T 186 -> 148 us; with ld + 1, N 175 -> 172, T 186 ->
// 164; a y of 300 from 12000 columns 22.6 -> 10.4 us (the slices' sums spread
// over eight threads a row, and that kernel launched ahead).
// Every sum is formed in the same order on every run (no atomics).
#include "internal.h"

namespace gbg {
namespace {

constexpr int kGemvThreads = 256;   // "T"
constexpr int kGemvNThreads = 512;  // "N"
constexpr int kXChunk = 1024;  // x values staged in shared memory at a time ("N")
constexpr int kTCols = 4;      // columns per block ("T")

// Element e of a BLAS vector of length len with increment inc (inc < 0: the
// vector runs backwards from the end of the storage).
__device__ __forceinline__ int64_t vec_index(int64_t e, int64_t len, int64_t inc) {
  return inc > 0 ? e * inc : (len - 1 - e) * (-inc);
}

// Partial (or final) y_i over columns [j0, j1) of 4 RT rows.  A thread takes
// four rows of a share of the columns, eight columns at a time, all 32 loads
// (VEC, columns that start on 16 bytes: 8 loads of 16 bytes, of neighbouring
// rows) issued before the first is used; the shares are added in order.
template <bool VEC, int RT>
__global__ void __launch_bounds__(kGemvNThreads, 2) gemv_n_kernel(int64_t m, int64_t n, const float* __restrict__ A,
                                                                  int64_t lda, const float* __restrict__ x,
                                                                  int64_t incx, int64_t slice,
                                                                  float* __restrict__ partial, float alpha,
                                                                  float beta, float* __restrict__ y, int64_t incy) {
  constexpr int U = 8;                     // columns per step
  constexpr int G = kGemvNThreads / RT;    // column shares
  __shared__ float xs[kXChunk];
  __shared__ float red[G][4 * RT];
  const int rt = threadIdx.x % RT, g = threadIdx.x / RT;
  constexpr int VS = VEC ? 1 : RT;         // between a thread's rows
  const int r0 = VEC ? 4 * rt : rt;        // its first row in the block
  const int64_t i = (int64_t)blockIdx.x * (4 * RT) + r0;
  const int64_t j0 = (int64_t)blockIdx.y * slice;
  const int64_t j1 = (j0 + slice < n) ? j0 + slice : n;
  const int rows = i >= m ? 0 : (m - i - 1) / VS + 1 < 4 ? (int)((m - i - 1) / VS + 1) : 4;  // that exist
  const float* a = A + (rows ? i : 0);
  float sum[4] = {0.f, 0.f, 0.f, 0.f};  // of sums of 32 columns: shorter chains than one sum's, less rounding
  for (int64_t jc = j0; jc < j1; jc += kXChunk) {
    const int nj = (int)((j1 - jc < kXChunk) ? j1 - jc : kXChunk);
    __syncthreads();  // the previous chunk is no longer read
    for (int t = threadIdx.x; t < nj; t += kGemvNThreads) xs[t] = x[vec_index(jc + t, n, incx)];
    __syncthreads();
    const int per = (nj + G - 1) / G;
    int t = g * per;
    const int te = min(nj, t + per);
    const float* col = a + (jc + t) * lda;
    if (rows == 0) continue;
    float acc[4][2];
#pragma unroll
    for (int v = 0; v < 4; ++v) acc[v][0] = acc[v][1] = 0.f;
    for (int step = 1; t < te; t += U, col += U * lda, ++step) {
      const int cnt = te - t;  // columns left: the same for a whole share
      float w[U][4];
      if (rows == 4 && cnt >= U) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
          if constexpr (VEC) {
            const float4 f = __ldg(reinterpret_cast<const float4*>(col + u * lda));
            w[u][0] = f.x; w[u][1] = f.y; w[u][2] = f.z; w[u][3] = f.w;
          } else {
#pragma unroll
            for (int v = 0; v < 4; ++v) w[u][v] = __ldg(col + u * lda + v * VS);
          }
        }
      } else if (VEC && rows == 4) {  // the last columns
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
          const float4 f = u < cnt ? __ldg(reinterpret_cast<const float4*>(col + u * lda)) : zero;
          w[u][0] = f.x; w[u][1] = f.y; w[u][2] = f.z; w[u][3] = f.w;
        }
      } else {  // the last columns, or the last rows
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
          for (int v = 0; v < 4; ++v) w[u][v] = (u < cnt && v < rows) ? __ldg(col + u * lda + v * VS) : 0.f;
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (u < cnt)
#pragma unroll
          for (int v = 0; v < 4; ++v) acc[v][u & 1] = fmaf(w[u][v], xs[t + u], acc[v][u & 1]);
      if ((step & 3) == 0 || t + U >= te) {
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          sum[v] += acc[v][0] + acc[v][1];
          acc[v][0] = acc[v][1] = 0.f;
        }
      }
    }
  }
#pragma unroll
  for (int v = 0; v < 4; ++v) red[g][r0 + v * VS] = sum[v];
  __syncthreads();
  for (int q = threadIdx.x; q < 4 * RT; q += kGemvNThreads) {
    const int64_t r = (int64_t)blockIdx.x * (4 * RT) + q;
    if (r >= m) return;
    float s = red[0][q];
#pragma unroll
    for (int k = 1; k < G; ++k) s += red[k][q];
    if (partial) {
      partial[(int64_t)blockIdx.y * m + r] = s;
    } else {
      float* yi = y + vec_index(r, m, incy);
      *yi = (beta != 0.f) ? fmaf(alpha, s, beta * *yi) : alpha * s;
    }
  }
}

// Partial (or final) y_j for columns j .. j+3 over rows [i0, i1) (i0 a
// multiple of 4).  V = 4 (columns that start on 16 bytes): four rows a thread
// and load, U = 2 loads of each column in flight; V = 1: U = 4 (or 2, with more
// blocks on an SM) loads of 4 bytes of each column in flight.
template <int V, int U>
__global__ void __launch_bounds__(kGemvThreads, V == 4 ? 3 : U == 4 ? 4 : 6)
    gemv_t_kernel(int64_t m, int64_t n, const float* __restrict__ A, int64_t lda, const float* __restrict__ x,
                  int64_t incx, int64_t slice, float* __restrict__ partial, float alpha, float beta,
                  float* __restrict__ y, int64_t incy) {
  constexpr int ACC = V == 4 ? 4 : 2;    // sums per column
  __shared__ float red[kTCols][kGemvThreads / 32];
  const int64_t jb = (int64_t)blockIdx.x * kTCols;
  const int64_t i0 = (int64_t)blockIdx.y * slice;
  const int64_t i1 = (i0 + slice < m) ? i0 + slice : m;
  const int nc = (int)((n - jb < kTCols) ? n - jb : kTCols);
  const float* col[kTCols];  // the columns past n read the first one and are not stored
#pragma unroll
  for (int c = 0; c < kTCols; ++c) col[c] = A + (jb + (c < nc ? c : 0)) * lda;
  float acc[kTCols][ACC];
#pragma unroll
  for (int c = 0; c < kTCols; ++c)
#pragma unroll
    for (int u = 0; u < ACC; ++u) acc[c][u] = 0.f;
  constexpr int64_t step = (int64_t)V * kGemvThreads;
  int64_t i = i0 + V * threadIdx.x;
  for (; i < i1; i += U * step) {
    float w[U][kTCols][V], xv[U][V];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t r = i + u * step;
      const bool full = r + V <= i1;  // by step: of the last rows most threads still have four
#pragma unroll
      for (int c = 0; c < kTCols; ++c) {
        if (V == 4 && full) {
          const float4 f = __ldg(reinterpret_cast<const float4*>(col[c] + r));
          w[u][c][0] = f.x; w[u][c][V / 2 - V / 4] = f.y; w[u][c][V / 2] = f.z; w[u][c][V - 1] = f.w;
        } else {
#pragma unroll
          for (int v = 0; v < V; ++v) w[u][c][v] = (full || r + v < i1) ? __ldg(col[c] + r + v) : 0.f;
        }
      }
#pragma unroll
      for (int v = 0; v < V; ++v) xv[u][v] = (full || r + v < i1) ? x[vec_index(r + v, m, incx)] : 0.f;
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int c = 0; c < kTCols; ++c)
#pragma unroll
        for (int v = 0; v < V; ++v) {
          const int t = V == 4 ? v : u % ACC;
          acc[c][t] = fmaf(w[u][c][v], xv[u][v], acc[c][t]);
        }
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int c = 0; c < kTCols; ++c) {
    float v = acc[c][0] + acc[c][1];
    if constexpr (ACC == 4) v += acc[c][2] + acc[c][3];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    if (lane == 0) red[c][warp] = v;
  }
  __syncthreads();
  if (threadIdx.x < nc) {
    const int c = threadIdx.x;
    float s = 0.f;
#pragma unroll
    for (int w = 0; w < kGemvThreads / 32; ++w) s += red[c][w];
    const int64_t j = jb + c;
    if (partial) {
      partial[(int64_t)blockIdx.y * n + j] = s;
    } else {
      float* yj = y + vec_index(j, n, incy);
      *yj = (beta != 0.f) ? fmaf(alpha, s, beta * *yj) : alpha * s;
    }
  }
}

// y_t := alpha sum_s partial[s][t] + beta y_t; with nslice 0, y_t := beta y_t
// (alpha == 0).  A block takes 32 rows at a time, eight threads a row (every
// eighth slice each, then the eight sums in order): the slices of a short y
// are hundreds.
__global__ void __launch_bounds__(256) gemv_finish_kernel(int64_t len, int nslice, const float* __restrict__ partial,
                                                          float alpha, float beta, float* __restrict__ y,
                                                          int64_t incy) {
  __shared__ float red[8][32];
  const int lane = threadIdx.x & 31, g = threadIdx.x >> 5;
  asm volatile("griddepcontrol.wait;" ::: "memory");  // the partial sums (launched ahead of their end)
  for (int64_t t0 = (int64_t)blockIdx.x * 32; t0 < len; t0 += (int64_t)gridDim.x * 32) {
    const int64_t t = t0 + lane;
    float s = 0.f;
    if (t < len) {
#pragma unroll 8
      for (int k = g; k < nslice; k += 8) s += partial[(int64_t)k * len + t];
    }
    red[g][lane] = s;
    __syncthreads();
    if (g == 0 && t < len) {
      float* yt = y + vec_index(t, len, incy);
      if (nslice == 0) {
        *yt = (beta == 0.f) ? 0.f : beta * *yt;
      } else {
#pragma unroll
        for (int k = 1; k < 8; ++k) s += red[k][lane];
        *yt = (beta != 0.f) ? fmaf(alpha, s, beta * *yt) : alpha * s;
      }
    }
    __syncthreads();
  }
}

cudaError_t launch_finish(int64_t len, int nslice, const float* partial, float alpha, float beta, float* y,
                          int64_t incy, int num_sms, bool dependent, cudaStream_t s) {
  const int64_t cap = (int64_t)(num_sms > 0 ? num_sms : 148) * 8, blocks = (len + 31) / 32;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(blocks < cap ? blocks : cap));
  cfg.blockDim = dim3(256);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = dependent ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, gemv_finish_kernel, len, nslice, partial, alpha, beta, y, incy);
}

int64_t ceil_div(int64_t a, int64_t b) { return (a + b - 1) / b; }

}  // namespace

int64_t gemv_slices(bool trans, int64_t m, int64_t n, int num_sms) {
  const int64_t want = 4 * (int64_t)num_sms;  // blocks to cover the SMs
  if (!trans) {
    const int64_t rb = ceil_div(m, 256);
    int64_t s = ceil_div(want, rb);
    const int64_t cap = ceil_div(n, 32);  // at least 32 columns a slice
    if (s > cap) s = cap;
    if (s > 65535) s = 65535;
    return s < 1 ? 1 : s;
  }
  const int64_t cb = ceil_div(n, kTCols);
  int64_t s = ceil_div(want, cb);
  const int64_t cap = ceil_div(m, 2048);  // at least 2048 rows a slice
  if (s > cap) s = cap;
  if (s > 65535) s = 65535;
  return s < 1 ? 1 : s;
}

cudaError_t launch_gemv(bool trans, int64_t m, int64_t n, float alpha, const float* A, int64_t lda, const float* x,
                        int64_t incx, float beta, float* y, int64_t incy, int64_t slices, float* partial,
                        int num_sms, cudaStream_t s) {
  const int64_t len_y = trans ? n : m;
  if (len_y <= 0) return cudaSuccess;
  if (alpha == 0.f || (trans ? m : n) == 0) {
    return launch_finish(len_y, 0, nullptr, alpha, beta, y, incy, num_sms, false, s);
  }
  if (slices > 1 && !partial) return cudaErrorInvalidValue;
  float* part = slices > 1 ? partial : nullptr;
  const bool vec = (lda & 3) == 0 && (reinterpret_cast<uintptr_t>(A) & 15) == 0;  // every column 16-byte aligned
  if (!trans) {
    const int64_t slice = ceil_div(n, slices);
    // Rows per block (4 rt): with aligned columns as many as can be, for the
    // memory's sake (16384^2, from cold: 1024 rows 173 us, 512 rows 197, one
    // row a thread 195); with others 256 (ld + 1: 185 us, 512 rows 201, one row
    // a thread 193); 512 for the few rows of a short y, 256 below; 512 where a
    // slice has too few columns for two shares (16384 x 20: 4.6 us, with 1024
    // rows 6.0).
    const int rt = m <= 256 ? 64 : m <= 1024 ? 128 : vec ? (slice <= 64 ? 128 : 256) : 64;
    const dim3 grid((unsigned)ceil_div(m, 4 * rt), (unsigned)ceil_div(n, slice));
    if (ceil_div(m, 4 * rt) > 0x7FFFFFFF) return cudaErrorInvalidConfiguration;
    auto kernel = vec ? (rt == 64    ? gemv_n_kernel<true, 64>
                         : rt == 128 ? gemv_n_kernel<true, 128>
                                     : gemv_n_kernel<true, 256>)
                      : (rt == 64 ? gemv_n_kernel<false, 64> : gemv_n_kernel<false, 128>);
    kernel<<<grid, kGemvNThreads, 0, s>>>(m, n, A, lda, x, incx, slice, part, alpha, beta, y, incy);
    slices = grid.y;
  } else {
    const int64_t slice = ceil_div(ceil_div(m, slices), 4) * 4;
    const dim3 grid((unsigned)ceil_div(n, kTCols), (unsigned)ceil_div(m, slice));
    if (ceil_div(n, kTCols) > 0x7FFFFFFF) return cudaErrorInvalidConfiguration;
    // Four rows a thread from 4096 on (16384^2 148 against 164 us): below, their
    // steps are few and long (1025 x 4096: 8.5 against 6.5 us, 1500 x 16384 29.4
    // against 26.5).  Two loads of 4 bytes in flight, but more blocks on an SM,
    // below 1024 rows, where a step is all (300 x 12000: 8.4 us, four rows a
    // thread 9.6), below 2048 with many rounds of blocks (1500 x 16384: 23.3),
    // and where a second round would be nearly empty (4097 x 2500, ld + 1: 12.5
    // against 14.5).
    const int64_t blocks = (int64_t)grid.x * grid.y;
    const bool two = slice < 1024 || (slice < 2048 && blocks > 16 * num_sms) ||
                     (!vec && slice > 4096 && blocks > 4 * num_sms && blocks <= 6 * num_sms);
    auto kernel = two ? gemv_t_kernel<1, 2> : vec && slice > 4096 ? gemv_t_kernel<4, 2> : gemv_t_kernel<1, 4>;
    kernel<<<grid, kGemvThreads, 0, s>>>(m, n, A, lda, x, incx, slice, part, alpha, beta, y, incy);
    slices = grid.y;
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess || !part) return e;
  return launch_finish(len_y, (int)slices, part, alpha, beta, y, incy, num_sms, true, s);
}

}  // namespace gbg
