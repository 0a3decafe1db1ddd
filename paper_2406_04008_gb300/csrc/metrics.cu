// Quality metrics of a collage (Sec. 6, "Metrics of Collage Quality", and the layout
// non-uniformity of the uniformity ablation, Sec. 6.1), computed on the device from a render pass
// at the current params.
//
// A pixel is object where O = 1 - Ihat >= 1/2, shape where the container coverage is >= 1/2, and
// overlap where at least two elements have sd >= 0 (c_i >= 1/2).  Per problem: LC = object pixels
// inside the shape / shape pixels, OO = overlap pixels / shape pixels, EA = object pixels outside
// the shape / shape pixels, and L-nU = the mean, over the non-object shape pixels, of the squared
// distance (unit coordinates) from the pixel centre to the nearest object pixel centre.  All
// counts and squared distances are integers, summed exactly.
#include "collage.h"
#include "edt.h"
#include "internal.h"

namespace collage {

constexpr int kMetWarps = 4;

struct ObjectSite {
  const uint8_t* obj;
  __device__ __forceinline__ bool operator()(long long pix) const { return obj[pix] != 0; }
};

// Counts per problem: cnt[4p + 0] object in shape, [1] shape, [2] overlap, [3] object outside the
// shape; obj[pix] = 1 for an object pixel.  One tile per warp.
template <int T>
__global__ void __launch_bounds__(kMetWarps * 32) k_metric_counts(Dev d, uint8_t* obj, unsigned long long* cnt) {
  constexpr int NP = T * T, PPL = NP / 32;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int tile = blockIdx.x * kMetWarps + wid; tile < d.total_tiles; tile += gridDim.x * kMetWarps) {
    int p = 0, lo = 0, hi = d.n_probs - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (d.prob_tile_base[mid] <= tile) lo = mid;
      else hi = mid - 1;
    }
    p = lo;
    const int lt = tile - d.prob_tile_base[p], ntx = d.prob_ntx[p], res = d.prob_res[p];
    const int tx = lt % ntx, ty = lt / ntx;
    const long long pixbase = d.prob_pix_base[p];
    const int m = d.tile_m[tile];
    const uint2* list = d.tile_list + (size_t)tile * d.tile_cap;
    unsigned c_in = 0, c_shape = 0, c_over = 0, c_out = 0;
#pragma unroll
    for (int k = 0; k < PPL; ++k) {
      const int local = lane + 32 * k;
      const int X = tx * T + local % T, Y = ty * T + local / T;
      bool valid = X < res && Y < res, o = false, sh = false, ov = false;
      if (valid) {
        const long long pix = pixbase + (long long)Y * res + X;
        int n_in = 0;
        for (int i = 0; i < m && n_in < 2; ++i) {
          const unsigned e = list[i].x, cls = e >> kSlotBits;
          if (cls == kPairIn) n_in += 1;
          else if (cls == kPairNear && d.saved[(size_t)(e & kSlotMask) * NP + local].x >= 0.0f) n_in += 1;
        }
        o = d.img_I[pix] <= 0.5f;
        sh = d.covc[pix] >= 0.5f;
        ov = n_in >= 2;
        obj[pix] = o ? 1 : 0;
      }
      c_in += __popc(__ballot_sync(0xffffffffu, o && sh));
      c_shape += __popc(__ballot_sync(0xffffffffu, sh));
      c_over += __popc(__ballot_sync(0xffffffffu, ov));
      c_out += __popc(__ballot_sync(0xffffffffu, o && !sh));
    }
    if (lane == 0) {
      if (c_in) atomicAdd(&cnt[4 * p + 0], (unsigned long long)c_in);
      if (c_shape) atomicAdd(&cnt[4 * p + 1], (unsigned long long)c_shape);
      if (c_over) atomicAdd(&cnt[4 * p + 2], (unsigned long long)c_over);
      if (c_out) atomicAdd(&cnt[4 * p + 3], (unsigned long long)c_out);
    }
  }
}

// Row pass, one row per block: for each non-object shape pixel the squared distance to the nearest
// object pixel; the row's sum goes to sums[p] (exact 64-bit integers).
__global__ void __launch_bounds__(kEdtRowThreads) k_metric_rows(Dev d, const unsigned short* g, unsigned long long* sums) {
  extern __shared__ unsigned s_g2[];
  const int p = blockIdx.y, i = blockIdx.x, res = d.prob_res[p];
  if (i >= res) return;
  const long long rowb = d.prob_pix_base[p] + (long long)i * res;
  edt_stage_row(g + rowb, res, s_g2);
  __syncthreads();
  unsigned long long acc = 0;
  for (int j = threadIdx.x; j < res; j += kEdtRowThreads) {
    // (an object pixel is its column's own site)
    if (s_g2[j] == 0u || !(d.covc[rowb + j] >= 0.5f)) continue;
    const unsigned best = edt_search(s_g2, res, j, kEdtFar2);
    if (best < kEdtFar2) acc += best;
  }
  for (int o = 16; o; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0 && acc) atomicAdd(&sums[p], acc);
}

cudaError_t launch_metrics(const Dev& d, cudaStream_t s, uint8_t* obj, unsigned short* gcol,
                           unsigned long long* cnt, unsigned long long* sums, int max_res) {
  cudaError_t e = cudaMemsetAsync(cnt, 0, sizeof(unsigned long long) * 4 * d.n_probs, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(sums, 0, sizeof(unsigned long long) * d.n_probs, s);
  const size_t cs = edt_col_smem(max_res), rs = edt_row_smem(max_res);
  if (e == cudaSuccess) e = edt_smem_limit(k_edt_cols<ObjectSite>, cs, edt_col_smem(kEdtMaxRes));
  if (e == cudaSuccess) e = edt_smem_limit(k_metric_rows, rs, edt_row_smem(kEdtMaxRes));
  if (e != cudaSuccess) return e;
  const int tgrid = (d.total_tiles + kMetWarps - 1) / kMetWarps;
  if (d.tile == 8) k_metric_counts<8><<<tgrid, kMetWarps * 32, 0, s>>>(d, obj, cnt);
  else if (d.tile == 16) k_metric_counts<16><<<tgrid, kMetWarps * 32, 0, s>>>(d, obj, cnt);
  else return cudaErrorInvalidValue;
  k_edt_cols<<<dim3((max_res + kEdtCols - 1) / kEdtCols, d.n_probs), kEdtThreads, cs, s>>>(
      d, ObjectSite{obj}, gcol, 0);
  k_metric_rows<<<dim3(max_res, d.n_probs), kEdtRowThreads, rs, s>>>(d, gcol, sums);
  return cudaGetLastError();
}

}  // namespace collage
