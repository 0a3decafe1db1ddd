// Exact squared Euclidean distance transform of one raster per problem, shared by the skeleton
// initialisation (distance to the nearest outside pixel) and the quality metrics (distance to the
// nearest object pixel): a column pass (rows to the nearest site of the same column), then per row
// the minimum over the columns k of (j - k)^2 + g(k)^2.  Integers throughout.
#pragma once
#include "internal.h"

namespace collage {

constexpr int kEdtCols = 8;         // columns per block: one 32-byte sector of a float row
constexpr int kEdtThreads = 1024;   // 8 columns x 128 runs of 8 rows
constexpr int kEdtRowThreads = 128;
constexpr unsigned short kEdtNone = 0xffff;   // no site in this column
constexpr unsigned kEdtFar2 = 0x7fffffffu;    // its square: above 2 (32768 - 1)^2, any real distance

// Dynamic shared memory of the passes for the largest side.
inline size_t edt_col_smem(int max_res) {
  return (size_t)((max_res + 31) / 32) * kEdtCols * (sizeof(unsigned) + 2 * sizeof(int));
}
inline size_t edt_row_smem(int max_res) { return sizeof(unsigned) * (size_t)max_res; }
// The limit a kernel needs for more than the default 48 KB, at `used` of at most `most` bytes.  It is an
// attribute of the function on the device, common to all threads and handles: always the most, so that no
// call lowers it between another's setting and its launch.
template <class Kernel>
inline cudaError_t edt_smem_limit(Kernel* kernel, size_t used, size_t most) {
  if (used <= 48 * 1024) return cudaSuccess;
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
}
constexpr int kEdtMaxRes = 32768;

// Column pass, one block per strip of kEdtCols columns.  Each thread reads 8 rows of a column as
// independent loads into one byte of the column's site bits; two short scans over the 32-row words
// (up and down) then give every word the nearest site beyond it, and each pixel's answer is a leading-
// or trailing-bit count in its word.  Bound by the latency of two rounds of loads; one thread walking a
// whole column was a chain of `res` dependent rows on res / 128 blocks (1024^2, cold: 250 us for the
// float raster, 608 us for the byte mask; 12 us now).  With `border` the rows -1 and res count as sites.
// Site: callable, whether the pixel at a global index is a site.
template <class Site>
__global__ void __launch_bounds__(kEdtThreads) k_edt_cols(Dev d, Site site, unsigned short* g, int border) {
  extern __shared__ unsigned s_words[];
  const int p = blockIdx.y, res = d.prob_res[p];
  const int c = threadIdx.x % kEdtCols, k = blockIdx.x * kEdtCols + c;
  if ((int)blockIdx.x * kEdtCols >= res) return;
  const int W = (res + 31) / 32;
  int* s_up = reinterpret_cast<int*>(s_words + W * kEdtCols);
  int* s_down = s_up + W * kEdtCols;
  const long long pb = d.prob_pix_base[p] + k;
  for (int b = threadIdx.x / kEdtCols; b < 4 * W; b += kEdtThreads / kEdtCols) {
    unsigned m = 0u;
    if (k < res) {
#pragma unroll
      for (int r = 0; r < 8; ++r) {
        const int i = b * 8 + r;
        if (i < res && site(pb + (long long)i * res)) m |= 1u << r;
      }
    }
    reinterpret_cast<unsigned char*>(s_words)[((b >> 2) * kEdtCols + c) * 4 + (b & 3)] = (unsigned char)m;
  }
  __syncthreads();
  constexpr int kBeyond = 1 << 17;  // farther than any row
  if (threadIdx.x < kEdtCols) {
    int last = border ? -1 : -kBeyond;  // the last site above word w
    for (int w = 0; w < W; ++w) {
      s_up[w * kEdtCols + c] = last;
      const unsigned m = s_words[w * kEdtCols + c];
      if (m) last = w * 32 + 31 - __clz((int)m);
    }
  } else if (threadIdx.x >= 32 && threadIdx.x < 32 + kEdtCols) {
    int next = border ? res : 2 * kBeyond;  // the first site below word w
    for (int w = W - 1; w >= 0; --w) {
      s_down[w * kEdtCols + c] = next;
      const unsigned m = s_words[w * kEdtCols + c];
      if (m) next = w * 32 + __ffs((int)m) - 1;
    }
  }
  __syncthreads();
  if (k >= res) return;
  for (int b = threadIdx.x / kEdtCols; b < 4 * W; b += kEdtThreads / kEdtCols) {
    const int w = b >> 2;
    const unsigned m = s_words[w * kEdtCols + c];
    const int up = s_up[w * kEdtCols + c], down = s_down[w * kEdtCols + c];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int r = (b & 3) * 8 + u, i = w * 32 + r;
      if (i >= res) break;
      const unsigned above = m & (0xffffffffu >> (31 - r)), below = m >> r;
      const int last = above ? w * 32 + 31 - __clz((int)above) : up;
      const int next = below ? i + __ffs((int)below) - 1 : down;
      const int dist = min(i - last, next - i);
      g[pb + (long long)i * res] = dist < kBeyond / 2 ? (unsigned short)dist : kEdtNone;
    }
  }
}

// The row's squared column distances into shared memory.
__device__ __forceinline__ void edt_stage_row(const unsigned short* grow, int res, unsigned* s_g2) {
  for (int k = threadIdx.x; k < res; k += kEdtRowThreads) {
    const unsigned v = grow[k];
    s_g2[k] = v == kEdtNone ? kEdtFar2 : v * v;
  }
}

// min over the columns k of (j - k)^2 + g(k)^2, no larger than `best`: outwards from j, stopping once
// the column offset alone reaches the minimum.  A pixel at distance D from its site visits D columns
// a side, where a scan of every column visits `res` of them (1024^2, the annulus, whose distances
// average 72 px: 27 us, issue-bound, against 545 us).  A column index clamped to the row's end stands
// for an offset no smaller than its own, so it can not undercut the minimum.
__device__ __forceinline__ unsigned edt_search(const unsigned* s_g2, int res, int j, unsigned best) {
  best = min(best, s_g2[j]);
  const int kmax = max(j, res - 1 - j);
  for (int k = 1; k <= kmax && (unsigned)(k * k) < best; k += 4) {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const unsigned kk = (unsigned)(k + u);
      best = min(best, kk * kk + min(s_g2[max(j - (k + u), 0)], s_g2[min(j + k + u, res - 1)]));
    }
  }
  return best;
}

}  // namespace collage
