// spmv.cu -- y = (H + shift I) v for the scene's BSR Hessian (the product a
// Newton driver's conjugate-gradient solve needs; the paper minimises with
// projected Newton, App. A).  Vectors are [3][n] SoA.
//
// G lanes share a block row, each taking every G-th 3x3 block.  Bound by the
// FP64 pipe and the L1's sectors: nine fused multiply-adds and twelve loads a
// block, 1.7M blocks of a pleated 256x256 sheet are 24 us of FP64 and 19 us of
// HBM at their rates.  Against one lane per row (G = 1) four lanes read blocks
// that lie side by side, and a warp waits for the longest of 8 rows instead of
// 32; more lanes would spend the FP64 pipe on idle slots and on the sums
// across lanes (a full warp instruction each).  Few rows leave the chip idle
// and wait for one lane's chain of loads, so G grows until the lanes fill it.
// One lane per row -> G: pleated 256x256 70 -> 53 us and 200x200 63 -> 38 (4),
// pleated 97x97 53 -> 16 (32), two layers of 144 vertices with rows of a hundred
// blocks and more 73 -> 6 (32), 64 rod scenes (1.1M rows, most of them short)
// 273 -> 238 (4).
#include "scene.cuh"

namespace {

template <int G>
__global__ void __launch_bounds__(CB_THREADS) k_bsr_spmv(int n, const int32_t* __restrict__ row_ptr,
                                                         const int32_t* __restrict__ col,
                                                         const double* __restrict__ val, const double* __restrict__ v,
                                                         double shift, double* __restrict__ y) {
  const int64_t t = (int64_t)blockIdx.x * CB_THREADS + threadIdx.x;
  const int r = (int)(t / G), l = (int)(t % G);
  double y0 = 0.0, y1 = 0.0, y2 = 0.0;
  if (r < n) {
    const int end = row_ptr[r + 1];
    auto add = [&](int k, int c) {
      const double* b = val + 9 * (size_t)k;
      const double v0 = v[c], v1 = v[(size_t)n + c], v2 = v[2 * (size_t)n + c];
      y0 = fma(b[2], v2, fma(b[1], v1, fma(b[0], v0, y0)));
      y1 = fma(b[5], v2, fma(b[4], v1, fma(b[3], v0, y1)));
      y2 = fma(b[8], v2, fma(b[7], v1, fma(b[6], v0, y2)));
    };
    int k = row_ptr[r] + l;
    for (; k + G < end; k += 2 * G) {  // two blocks at once: their loads overlap
      const int c0 = col[k], c1 = col[k + G];
      add(k, c0);
      add(k + G, c1);
    }
    if (k < end) add(k, col[k]);
  }
  // sum over the G lanes, the three components spread over lanes 0, 2 and 1 of each four on the way
  const unsigned full = 0xffffffffu;
  const bool odd = l & 1, up = l & 2;
  const double s0 = __shfl_xor_sync(full, odd ? y0 : y2, 1), s1 = __shfl_xor_sync(full, y1, 1);
  const double a = (odd ? y2 : y0) + s0, b = y1 + s1;
  double s = (up ? b : a) + __shfl_xor_sync(full, up ? a : b, 2);
#pragma unroll
  for (int o = 4; o < G; o <<= 1) s += __shfl_xor_sync(full, s, o);
  if (r < n && l < 3) {
    const size_t i = (size_t)(l == 0 ? 0 : 3 - l) * n + r;
    y[i] = fma(shift, v[i], s);
  }
}

}  // namespace
extern "C" cb_status cb_bsr_spmv(cb_scene* s, const double* v, double* y, double shift, void* stream) {
  if (!s || !v || !y || v == y) return CB_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  s->last_stream = st;
  if (s->n == 0) return CB_OK;
  if (!s->bsr_row.p) return CB_ERR_ARG;  // no barrier_eval / barrier_energy yet
  // lanes per row: 4, more while that leaves an SM with fewer than 1,024 threads
  const int64_t n = s->n, fill = (int64_t)s->n_sms * 1024;
  const int g = n * 4 >= fill ? 4 : (n * 8 >= fill ? 8 : (n * 16 >= fill ? 16 : 32));
  auto* f = g == 4 ? k_bsr_spmv<4> : (g == 8 ? k_bsr_spmv<8> : (g == 16 ? k_bsr_spmv<16> : k_bsr_spmv<32>));
  // an empty matrix (no active pair) still has row_ptr: zeros
  f<<<cb_grid(n * g), CB_THREADS, 0, cb_count(st)>>>(s->n, (const int32_t*)s->bsr_row.p, (const int32_t*)s->bsr_col.p,
                                                     (const double*)s->bsr_val.p, v, shift, y);
  CB_CUDA(cudaGetLastError());
  return CB_OK;
}
