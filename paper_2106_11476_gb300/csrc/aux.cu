// Source injection, sensor recording, field copies, the field scan and the self-test of
// the bounded wait (sm_103a).
#include <algorithm>

#include "async.cuh"
#include "fw2_prep.cuh"

namespace fw2 {

namespace {

// One thread per distinct target cell: the entries feeding it are summed in
// a fixed order, so repeated runs give identical results (no atomics).
__global__ void inject_kernel(float *field, const long long *tgt, const int *off, const int *col,
                              const float *row, int n_tgt) {
  const int u = blockIdx.x * blockDim.x + threadIdx.x;
  if (u >= n_tgt) return;
  float s = 0.f;
  for (int e = off[u]; e < off[u + 1]; ++e) s += __ldg(row + col[e]);
  field[tgt[u]] += s;
}

// One thread per sensor group: mean of p over the group's cells.
__global__ void record_kernel(const float *p, const long long *cell, const int *off, int n_groups,
                              float *out) {
  const int g = blockIdx.x * blockDim.x + threadIdx.x;
  if (g >= n_groups) return;
  const int b = off[g], e = off[g + 1];
  float s = 0.f;
  for (int i = b; i < e; ++i) s += p[cell[i]];
  out[g] = e > b ? s / (float)(e - b) : 0.f;
}

// max |x| over the valid cells, non-finite values count as +inf.  Each block
// reduces in shared memory and folds its result into *out_bits with an
// integer atomicMax (non-negative floats order like their bit patterns).
__global__ void absmax_kernel(const float *f, int nx, int pitch, long long rows, unsigned int *out_bits) {
  __shared__ float red[256];
  float m = 0.f;
  const long long n = rows * (long long)nx;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n;
       t += (long long)gridDim.x * blockDim.x) {
    const long long r = t / nx;
    const int i = (int)(t - r * nx);
    const float v = fabsf(f[r * pitch + i]);
    m = isfinite(v) ? fmaxf(m, v) : __int_as_float(0x7f800000);
  }
  red[threadIdx.x] = m;
  __syncthreads();
  for (int s = 128; s > 0; s >>= 1) {
    if (threadIdx.x < s) red[threadIdx.x] = fmaxf(red[threadIdx.x], red[threadIdx.x + s]);
    __syncthreads();
  }
  if (threadIdx.x == 0) atomicMax(out_bits, __float_as_uint(red[0]));
}

}  // namespace

namespace {

// Rows of a field between the pitched cell layout and a dense buffer: one
// warp per segment of kSeg values of a row, blockIdx.y the array (mechanism).
// Bound by HBM (read and write once).  cudaMemcpy2DAsync moved the 19 state
// arrays of 2048 x 1024 cells at 1.3 TB/s and a small field in 13 us.  V =
// float4 where the dense rows are 16-byte aligned too, else float.
constexpr int kSeg = 1024;
template <typename V>
__global__ void __launch_bounds__(256) copy_rows_kernel(float *dst, long long dst_row, long long dst_arr,
                                                        const float *src, long long src_row, long long src_arr,
                                                        int nx, long long rows) {
  constexpr int kE = sizeof(V) / 4, kUnroll = 4;
  const int lane = threadIdx.x & 31, segs = (nx + kSeg - 1) / kSeg;
  const long long items = rows * segs;
  dst += blockIdx.y * dst_arr;
  src += blockIdx.y * src_arr;
  for (long long it = blockIdx.x * 8ll + (threadIdx.x >> 5); it < items; it += gridDim.x * 8ll) {
    const long long r = segs == 1 ? it : it / segs;
    const int x0 = (int)(it - r * segs) * kSeg, n = (min(kSeg, nx - x0) + kE - 1) / kE;
    V *d = reinterpret_cast<V *>(dst + r * dst_row + x0);
    const V *s = reinterpret_cast<const V *>(src + r * src_row + x0);
    for (int i = lane; i < n; i += 32 * kUnroll) {
      V v[kUnroll];
#pragma unroll
      for (int m = 0; m < kUnroll; ++m)
        if (i + 32 * m < n) v[m] = __ldcs(s + i + 32 * m);
#pragma unroll
      for (int m = 0; m < kUnroll; ++m)
        if (i + 32 * m < n) __stcs(d + i + 32 * m, v[m]);
    }
  }
}

}  // namespace

cudaError_t launch_copy_rows(float *dst, long long dst_row, long long dst_arr, const float *src, long long src_row,
                             long long src_arr, int nx, long long rows, int arrays, cudaStream_t s) {
  if (rows <= 0 || arrays <= 0) return cudaSuccess;
  const long long items = rows * ((nx + kSeg - 1) / kSeg);
  const dim3 grid((unsigned)std::min<long long>((items + 7) / 8, 152 * 16), (unsigned)arrays);
  const auto aligned = [](const float *p, long long row, long long arr) {
    return reinterpret_cast<uintptr_t>(p) % 16 == 0 && row % 4 == 0 && arr % 4 == 0;
  };
  if (nx % 4 == 0 && aligned(dst, dst_row, dst_arr) && aligned(src, src_row, src_arr))
    copy_rows_kernel<float4><<<grid, 256, 0, s>>>(dst, dst_row, dst_arr, src, src_row, src_arr, nx, rows);
  else
    copy_rows_kernel<float><<<grid, 256, 0, s>>>(dst, dst_row, dst_arr, src, src_row, src_arr, nx, rows);
  return cudaGetLastError();
}

cudaError_t launch_inject(float *field, const long long *tgt, const int *off, const int *col,
                          const float *row, int n_tgt, cudaStream_t s) {
  if (n_tgt <= 0) return cudaSuccess;
  inject_kernel<<<(n_tgt + 127) / 128, 128, 0, s>>>(field, tgt, off, col, row, n_tgt);
  return cudaGetLastError();
}

cudaError_t launch_record(const float *p, const long long *cell, const int *off, int n_groups,
                          float *out, cudaStream_t s) {
  if (n_groups <= 0) return cudaSuccess;
  record_kernel<<<(n_groups + 127) / 128, 128, 0, s>>>(p, cell, off, n_groups, out);
  return cudaGetLastError();
}

cudaError_t launch_absmax(const float *f, int nx, int pitch, long long rows, unsigned int *out_bits,
                          cudaStream_t s) {
  long long n = rows * (long long)nx;
  long long blocks = (n + 255) / 256;
  if (blocks > 152 * 8) blocks = 152 * 8;
  if (blocks < 1) blocks = 1;
  absmax_kernel<<<(int)blocks, 256, 0, s>>>(f, nx, pitch, rows, out_bits);
  return cudaGetLastError();
}

namespace {
// one thread waits on an mbarrier that never completes (count 1, no arrival)
__global__ void bounded_wait_kernel(unsigned long long limit_ns, int *timed_out) {
  __shared__ __align__(8) uint64_t bar;
  mbar_init(&bar, 1);
  fence_mbarrier_init();
  *timed_out = mbar_wait_bounded(&bar, 0, limit_ns) ? 0 : 1;
}
// one block: a barrier that it completes, then one that it does not
__global__ void grid_barrier_kernel(unsigned long long limit_ns, unsigned long long *words) {
  unsigned int *status = reinterpret_cast<unsigned int *>(words + 1);
  GridBarrier gb;
  gb.init(words);
  gb.arrive();
  const bool passed = gb.wait(nullptr, limit_ns);
  gb.target += gridDim.x;
  status[1] = passed && !gb.wait(status, limit_ns) ? 1 : 0;
}
}  // namespace

cudaError_t launch_grid_barrier_selftest(unsigned long long limit_ns, unsigned long long *words) {
  grid_barrier_kernel<<<1, 1>>>(limit_ns, words);
  return cudaGetLastError();
}

cudaError_t launch_bounded_wait_selftest(unsigned long long limit_ns, int *timed_out) {
  bounded_wait_kernel<<<1, 1>>>(limit_ns, timed_out);
  return cudaGetLastError();
}

}  // namespace fw2
