// Tile rasteriser (forward), its adjoint, and the container raster.
//
// Coverage of element i at pixel p is c = S(sd / rho) with sd the signed distance (winding number
// for the sign, positive inside; hw - d for open strokes) and S(x) = (1 + x)^2 (2 - x) / 4 on
// [-1, 1] (the same cubic as 1/2 + 3x/4 - x^3/4, written in factored form so that 1 - S(x) =
// S(-x) keeps full relative precision near x = 1).  This is the anti-aliased, differentiable
// rasteriser the method builds on (Sec. 3 "Differentiable Rendering"); the composites and
// per-pixel losses are those of Sec. 4.2 (Eqs. 5, 6 and the force term of Sec. 5).
//
// Precision: each element's vertices are stored relative to its translation, in pixels, and the
// pixel is brought into that frame as (p - t_hi) - t_lo, so every FP32 quantity is a few tens of
// pixels at most and the signed distance carries an error of ~1e-6 px at any grid size.
//
// The forward pass saves, for every (tile, element) pair and pixel of the tile, the signed
// distance and the closest segment; the adjoint reads them back instead of repeating the segment
// loop, so only one pass over the pixel-segment pairs happens per iteration.  Pixels farther than
// the coverage margin from the outline carry sd = +-1e30 (saturated coverage, no gradient).
#include <cfloat>
#include <type_traits>

#include "arith.h"
#include "internal.h"

namespace collage {

__device__ __forceinline__ float Sfun(float x) {
  x = fminf(fmaxf(x, -1.0f), 1.0f);
  const float a = 1.0f + x;
  return 0.25f * a * a * (2.0f - x);
}
__device__ __forceinline__ float dSfun(float x) {
  x = fminf(fmaxf(x, -1.0f), 1.0f);
  return 0.75f * (1.0f - x) * (1.0f + x);
}

__device__ __forceinline__ int find_prob(const int* base, int P, int tile) {
  int lo = 0, hi = P - 1;  // last p with base[p] <= tile
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (base[mid] <= tile) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// Distance / winding update of one point against one staged segment (a, a + e) whose end point
// has y = b_y.  Winding: the segment crosses the +x ray from the point when the two end points lie
// on different sides of it (half-open in y); cross(e, w) > 0 puts the crossing right of the point
// for an upward segment, < 0 for a downward one.
struct SegQuery {
  float best;  // squared distance
  int idx;
  int wn;
};

__device__ __forceinline__ void seg_update(SegQuery& Q, float dx, float dy, float4 s, float2 s2,
                                           int j, bool winding) {
  const float wx = dx - s.x, wy = dy - s.y;
  const float t = __saturatef((wx * s.z + wy * s.w) * s2.y);
  const float qx = fmaf(-t, s.z, wx), qy = fmaf(-t, s.w, wy);
  const float d2 = fmaf(qx, qx, qy * qy);
  if (d2 < Q.best) {
    Q.best = d2;
    Q.idx = j;
  }
  if (winding) {
    const bool a_le = wy >= 0.0f;         // a.y <= p.y
    const bool b_le = dy - s2.x >= 0.0f;  // b.y <= p.y
    const float cr = s.z * wy - s.w * wx;
    if (a_le && !b_le && cr > 0.0f) Q.wn += 1;
    if (!a_le && b_le && cr < 0.0f) Q.wn -= 1;
  }
}

constexpr int kSegCap = 1024;   // container segments staged per chunk
constexpr int kRowCross = 16;   // crossings listed per pixel row of an emission chunk
constexpr int kPairWarps = 4;   // units per block of the adjoint (one per warp)
constexpr float kFar = 1e30f;   // |sd| of a pixel farther than the coverage margin

// Winding number of a point (element frame) over every segment of an outline: the crossing test of
// the per-row lists below applied to all segments (for rows that cross the outline too often).
__device__ __noinline__ int winding_all(const Dev& d, int v0, int ns, float px, float py) {
  int w = 0;
  for (int j = 0; j < ns; ++j) {
    const float4 sa = d.segA[v0 + j];
    const float wy = py - sa.y;
    const bool a_le = wy >= 0.0f, b_le = py - d.segB[v0 + j].x >= 0.0f;
    if (a_le != b_le && px < fmaf(wy, d.segS[v0 + j], sa.x)) w += a_le ? 1 : -1;
  }
  return w;
}

// ------------------------------------------------------------------------------------------------
// Emission and signed distances, one (element, chunk) work item per block at a time.  A chunk is a
// square of up to kChunkPx x kChunkPx pixels of the element's tile rectangle (8 x 8 tiles of 8 px,
// 4 x 4 of 16 px); the transform kernel lists every element's chunks.  Per chunk the block
//  1. takes the pair slot of each of its tiles (the element's slots follow its tile rectangle
//     row-major from the base the transform allocated) and records it in the tile's list (a
//     list beyond its capacity latches a status bit: the host grows the lists and runs again);
//  2. passes once over the element's segments, staging them in shared memory by index: a segment
//     whose box meets a unit's pixel-centre box grown by the coverage margin m = rho + pad
//     (+ stroke half-width) (+ 0.06 px of slack) is near that unit (a bit per segment and unit);
//     units are the 64 pixels a warp takes at once: a tile of 8 x 8, or four rows of a tile of 16 x 16;
//     for every pixel row of the chunk that a segment crosses (half-open in y, on the dy the
//     pixels form) the crossing x is listed for the row, or, when it lies right of every pixel of
//     the chunk, added to the row's backdrop (+1 upward, -1 downward);
//  3. classifies the tiles: a tile that no segment is near has saturated coverage on every pixel
//     (0 or 1, as the winding number of its first pixel says) and needs no per-pixel work;
//  4. its warps take the near tiles' units one at a time: per pixel, the minimum squared distance over
//     the unit's near segments in index order (the lowest index wins ties, as the oracle's scan
//     does); winding = row backdrop + listed crossings right of the pixel (a row with more than
//     kRowCross crossings tests every segment); sd = +-distance within the margin, else +-1e30
//     (saturated); the (sd, closest segment) record is saved and units with a non-saturated pixel
//     are listed for the adjoint.
// Outlines of more than kStageSegs segments are not staged: their tiles test every segment's box
// on the fly, reading the outline from global memory.
// A pixel beyond the margin from every segment near its unit is beyond it from all segments (the
// near test is conservative), so the distance minimum over the near ones is exact wherever it
// matters, and the winding counts every crossing right of the pixel exactly once.
// ------------------------------------------------------------------------------------------------
constexpr int kStageSegs = 512;   // outline segments staged in shared memory
constexpr int kLiveBatch = 32;

// Units (T x 64 / T pixels) of the chunk whose grown pixel-centre box a segment's box [x0, x1] x [y0, y1]
// (absolute px) meets: columns [*c0, *c1], rows [*r0, *r1] relative to the chunk's first unit (ux0, uy0),
// clipped to it.
template <int T>
__device__ __forceinline__ void seg_units(float x0, float x1, float y0, float y1, float m, int ux0, int uy0,
                                          int cuw, int cuh, int* c0, int* c1, int* r0, int* r1) {
  constexpr float W = (float)T, iW = 1.0f / W, H = 64.0f / W, iH = 1.0f / H;  // powers of two: exact
  *c0 = max((int)floorf((x0 - m - (W - 0.5f)) * iW) + 1 - ux0, 0);
  *c1 = min((int)floorf((x1 + m - 0.5f) * iW) - ux0, cuw - 1);
  *r0 = max((int)floorf((y0 - m - (H - 0.5f)) * iH) + 1 - uy0, 0);
  *r1 = min((int)floorf((y1 + m - 0.5f) * iH) - uy0, cuh - 1);
}

// Squared distance from (dx, dy) to the segment a + u e, u in [0, 1], with f = e / |e|^2 (the
// clamped parameter is then a dot product): the operations of the oracle's closest-point rule.
__device__ __forceinline__ float seg_d2(float dx, float dy, float4 s, float2 f) {
  const float wx = dx - s.x, wy = dy - s.y;
  const float t = __saturatef(fmaf(wy, f.y, wx * f.x));
  const float qx = fmaf(-t, s.z, wx), qy = fmaf(-t, s.w, wy);
  return fmaf(qx, qx, qy * qy);
}

// NT threads per block (128 or 256, the autotuner's choice); registers capped so that 1024 threads are
// resident per SM.  Bound by issue slots and by the latency of each chunk's phases.  (With 16-px tiles a
// warp used to take a whole tile, eight pixels a lane, 114 registers, and tested every segment near the
// tile at each of them: 120 elements at 200^2 28 us, 22.6 now; 64 collages at 8-px tiles, by
// the same code, 251 -> 235.)
template <int T, int NT>
__global__ void __launch_bounds__(NT, 1024 / NT) k_raster_chunks(Dev d, int n_sm) {
  const int first = first_item(d.slots, n_sm);
  pdl_enter();
  constexpr int CW = kChunkPx / T, NCT = CW * CW, NP = T * T, UNITS = NP / 64, UH = 64 / T;
  constexpr int NCU = NCT * UNITS;  // units of a chunk
  constexpr int ROWS = kChunkPx, MW = kStageSegs / 32;
  __shared__ float4 s_seg[kStageSegs];  // start (px, relative to the translation), direction
  __shared__ float2 s_f[kStageSegs];    // direction / |direction|^2
  __shared__ unsigned s_mask[NCU][MW];  // bit j of unit k: segment j is near unit k
  __shared__ int s_slot[NCT];           // pair slot of each tile (-1: void)
  __shared__ unsigned char s_tn[NCT];   // some segment is near the tile
  __shared__ int2 s_unit[NCU];          // the near tiles' units: (pair slot | unit in the tile << kSlotBits,
                                        //   unit | column << 8 | row << 16)
  __shared__ int2 s_row[ROWS];          // per pixel row: (crossings right of every pixel, listed)
  __shared__ float2 s_rx[ROWS][kRowCross];  // listed crossings: (x, +1 upward / -1 downward)
  __shared__ int s_nt, s_take;
  __shared__ int s_next[2];
  __shared__ int4 s_live[kLiveBatch];
  __shared__ int s_nlive;
  const float inv_rho = 1.0f / d.L.rho_px, pad = d.L.pad_px;
  const int tid = threadIdx.x, lane = tid & 31;
  const int n_heavy = d.chunk_count[0], n_chunks = n_heavy + d.chunk_count[1];
  if (blockIdx.x == 0 && tid == 0) {
    // the transform has completed: its slot count becomes the iteration's pair count, its
    // pending-step flag is spent, and the composite's fullest-tile maximum starts over
    *d.total_pairs = *d.pair_need;
    *d.pair_need = 0;
    *d.tile_max = 0;
    *d.pending = 0;
  }
  // the slots are void when the pairs exceed the capacity (the transform latched it)
  for (int i = (*d.status & kStatusOverflow) ? n_chunks : first, it = 0; i < n_chunks; ++it) {
    if (tid == 0) {
      // chunks beyond the grid are taken by an atomic count (none when the grid covers them all)
      s_next[it & 1] = n_chunks > (int)gridDim.x ? (int)gridDim.x + atomicAdd(&d.work[0], 1) : n_chunks;
      s_nlive = 0;
      s_take = 0;
    }
    const int li = i < n_heavy ? i : d.list_cap - 1 - (i - n_heavy);
    if (!in_bounds(d, li >= 0 && li < d.list_cap)) break;
    const int4 rec = d.near_list[li];
    const int g = rec.x, tx0 = rec.y & 0xffff, ty0 = rec.y >> 16, p = rec.z;
    if (!in_bounds(d, g >= 0 && g < d.n_elems && p >= 0 && p < d.n_probs)) break;
    const int4 r = d.rect[g];
    const int cs = min(d.chunk_tiles, CW);
    const int ctw = min(cs, r.z - tx0 + 1), cth = min(cs, r.w - ty0 + 1), nct = ctw * cth;
    const int res = d.prob_res[p], ntx = d.prob_ntx[p], tb = d.prob_tile_base[p];
    const int v0 = d.elem_voff[g], nv = d.elem_voff[g + 1] - v0;
    const bool closed = d.elem_closed[g] != 0;
    const int ns = closed ? nv : nv - 1;
    const bool staged = ns <= kStageSegs;
    const int mw = staged ? (ns + 31) >> 5 : 0;
    // 1. pair slots and their places in the tiles' lists (the entries are written once the tiles are
    // classified, when the counts taken here have long arrived); cleared marks and row lists
    int place = -1;
    if (tid < NCT) {
      int slot = -1;
      const int t = tb + (ty0 + tid / ctw) * ntx + tx0 + tid % ctw;
      if (tid < nct && in_bounds(d, t >= tb && t < d.prob_tile_base[p + 1])) {
        const int u = d.elem_pbase[g] + (ty0 + tid / ctw - r.y) * (r.z - r.x + 1) + tx0 + tid % ctw - r.x;
        if (in_bounds(d, u >= 0 && u < d.cap)) {
          slot = u;
          place = atomicAdd(&d.tile_n[t], 1);
        }
      }
      s_slot[tid] = slot;
      s_tn[tid] = 0;
    }
    for (int q = tid; q < nct * UNITS * mw; q += NT) s_mask[q / mw][q % mw] = 0u;
    for (int q = tid; q < ROWS; q += NT) s_row[q] = make_int2(0, 0);
    const float4 tp = d.tpx[g];
    const float hwpx = closed ? 0.0f : d.elem_hw[g] * (float)res;
    const float mrg = d.L.rho_px + pad + hwpx, mrg2 = mrg * mrg;
    const float tpx = tp.x + tp.z, tpy = tp.y + tp.w;
    const int X0 = tx0 * T, Y0 = ty0 * T, ncol = ctw * T, nrow = cth * T;
    // the chunk's pixel-centre box in the element frame, as the pixels form dx and dy
    const float min_dx = ((float)X0 + 0.5f - tp.x) - tp.z;
    const float max_dx = ((float)(X0 + ncol - 1) + 0.5f - tp.x) - tp.z;
    const float sl = mrg + 0.06f, rsl = 0.02f + 5e-7f * fabsf(tpy);  // slack of the near test, of the rows
    const int ux0 = tx0, uy0 = ty0 * UNITS, cuh = cth * UNITS;  // (a unit is as wide as a tile)
    __syncthreads();
    // 2. one pass over the segments: staging, the units they are near, row crossings
    if (ns > kStageSegs && tid == 0 && d.paths) atomicAdd(&d.paths[1], 1ull);
    for (int j = tid; j < ns; j += NT) {
      const float4 sa = d.segA[v0 + j];
      const float2 sb = d.segB[v0 + j];
      if (staged) {
        s_seg[j] = sa;
        s_f[j] = make_float2(sa.z * sb.y, sa.w * sb.y);
      }
      const float bx = sa.x + sa.z, by = sb.x;
      const float x0 = fminf(sa.x, bx), x1 = fmaxf(sa.x, bx), y0 = fminf(sa.y, by), y1 = fmaxf(sa.y, by);
      int c0, c1, r0, r1;
      seg_units<T>(x0 + tpx, x1 + tpx, y0 + tpy, y1 + tpy, sl, ux0, uy0, ctw, cuh, &c0, &c1, &r0, &r1);
      for (int rr = r0; rr <= r1; ++rr)
        for (int cc = c0; cc <= c1; ++cc) {
          if (!in_bounds(d, rr * ctw + cc < NCU)) continue;
          s_tn[rr / UNITS * ctw + cc] = 1;
          if (staged) atomicOr(&s_mask[rr * ctw + cc][j >> 5], 1u << (j & 31));
        }
      if (closed && y1 > y0 && x1 > min_dx) {  // crosses some row right of the first pixel column
        // candidate rows (with slack for the rounding of these sums; most segments of a curve cross one
        // row or none), then the exact half-open test
        const int q0 = max((int)ceilf(y0 + tpy - 0.5f - rsl) - Y0, 0);
        const int q1 = min((int)floorf(y1 + tpy - 0.5f + rsl) - Y0, nrow - 1);
        const float slope = d.segS[v0 + j];
        for (int q = q0; q <= q1; ++q) {
          if (!in_bounds(d, q < ROWS)) break;
          const float yr = ((float)(Y0 + q) + 0.5f - tp.y) - tp.w;
          const bool a_le = yr - sa.y >= 0.0f, b_le = yr - by >= 0.0f;
          if (a_le == b_le) continue;
          const float xc = fmaf(yr - sa.y, slope, sa.x);
          const int dir = a_le ? 1 : -1;
          if (xc > max_dx) {
            atomicAdd(&s_row[q].x, dir);  // right of every pixel of the row
          } else if (xc > min_dx) {
            const int k = atomicAdd(&s_row[q].y, 1);
            if (k < kRowCross) s_rx[q][k] = make_float2(xc, (float)dir);
          }
        }
      }
    }
    __syncthreads();
    // 3. classification; the near tiles in tile order
    if (tid < nct && s_slot[tid] >= 0) {
      const int slot = s_slot[tid];
      unsigned cls = kPairNear;
      if (!s_tn[tid]) {
        int w = 0;
        if (closed) {
          const int q = (tid / ctw) * T;
          const float dx0 = ((float)(X0 + (tid % ctw) * T) + 0.5f - tp.x) - tp.z;
          const int2 row = s_row[q];
          if (row.y <= kRowCross) {
            float wf = (float)row.x;
            for (int k = 0; k < row.y; ++k) {
              const float2 c = s_rx[q][k];
              if (dx0 < c.x) wf += c.y;
            }
            w = (int)wf;
          } else {
            w = winding_all(d, v0, ns, dx0, ((float)(Y0 + q) + 0.5f - tp.y) - tp.w);
          }
        }
        cls = w != 0 ? kPairIn : kPairOut;
        if (d.deterministic)
          for (int u = 0; u < UNITS; ++u) d.partial[(size_t)slot * UNITS + u] = make_float4(0.f, 0.f, 0.f, 0.f);
      }
      const int t = tb + (ty0 + tid / ctw) * ntx + tx0 + tid % ctw;
      const uint2 entry = make_uint2((unsigned)slot | cls << kSlotBits, (unsigned)g);
      if (place < d.tile_cap) d.tile_list[(size_t)t * d.tile_cap + place] = entry;
      else atomicOr(d.status, kStatusTileCap);
    }
    if (tid < 32) {  // warp 0: the near tiles' units, in order
      int n = 0;
      for (int k0 = 0; k0 < nct * UNITS; k0 += 32) {
        const int k = k0 + lane, ur = k / ctw, uc = k - ur * ctw, tl = ur / UNITS * ctw + uc;
        const bool nr = k < nct * UNITS && s_slot[tl] >= 0 && s_tn[tl];
        const unsigned bal = __ballot_sync(0xffffffffu, nr);
        if (nr)
          s_unit[n + __popc(bal & ((1u << lane) - 1u))] =
              make_int2(s_slot[tl] | (int)((unsigned)(ur % UNITS) << kSlotBits), k | uc << 8 | ur << 16);
        n += __popc(bal);
      }
      if (lane == 0) s_nt = n;
    }
    __syncthreads();
    const int nt = s_nt;
    // 4. the near tiles' units, one per warp at a time (the next one taken while this one is worked on)
    int ni = 0;
    if (lane == 0) ni = atomicAdd(&s_take, 1);
    ni = __shfl_sync(0xffffffffu, ni, 0);
    while (ni < nt) {
      int nn = 0;
      if (lane == 0) nn = atomicAdd(&s_take, 1);
      const int2 nti = s_unit[ni];
      const int k = nti.y & 0xff, kc = (nti.y >> 8) & 0xff, kr = nti.y >> 16;
      // the lane's pixels: rows q and q + 32 / T of the chunk, one column
      const int q = kr * UH + lane / T;
      const float dx = ((float)((tx0 + kc) * T + lane % T) + 0.5f - tp.x) - tp.z;
      float dy[2], best[2] = {FLT_MAX, FLT_MAX};
      int bidx[2] = {0, 0};
#pragma unroll
      for (int e = 0; e < 2; ++e) dy[e] = ((float)(Y0 + q + e * (32 / T)) + 0.5f - tp.y) - tp.w;
      if (staged) {
        for (int w = 0; w < mw; ++w) {
          unsigned bits = s_mask[k][w];
          while (bits) {
            const int j = w * 32 + __ffs(bits) - 1;  // in index order
            bits &= bits - 1u;
            const float4 sg = s_seg[j];
            const float2 f = s_f[j];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
              const float d2 = seg_d2(dx, dy[e], sg, f);
              if (d2 < best[e]) {
                best[e] = d2;
                bidx[e] = j;
              }
            }
          }
        }
      } else {
        // the unit's near segments by the same box test as the marks, from global memory
        for (int j = 0; j < ns; ++j) {
          const float4 s = d.segA[v0 + j];
          const float2 sb = d.segB[v0 + j];
          const float bx = s.x + s.z;
          int c0, c1, r0, r1;
          seg_units<T>(fminf(s.x, bx) + tpx, fmaxf(s.x, bx) + tpx, fminf(s.y, sb.x) + tpy,
                       fmaxf(s.y, sb.x) + tpy, sl, ux0, uy0, ctw, cuh, &c0, &c1, &r0, &r1);
          if (kc < c0 || kc > c1 || kr < r0 || kr > r1) continue;
          const float2 f = make_float2(s.z * sb.y, s.w * sb.y);
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const float d2 = seg_d2(dx, dy[e], s, f);
            if (d2 < best[e]) {
              best[e] = d2;
              bidx[e] = j;
            }
          }
        }
      }
      float2* sv = d.saved + (size_t)(nti.x & (int)kSlotMask) * NP + (unsigned)nti.x / (1u << kSlotBits) * 64 + lane;
      bool live = false;
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        // (outside the element's box the crossings cancel and the distance is beyond the margin; a
        // pixel beyond the image is never read)
        int w = 0;
        if (closed) {
          const int2 row = s_row[q + e * (32 / T)];
          if (row.y <= kRowCross) {
            float wf = (float)row.x;
            for (int c = 0; c < row.y; ++c) {
              const float2 cr = s_rx[q + e * (32 / T)][c];
              if (dx < cr.x) wf += cr.y;
            }
            w = (int)wf;
          } else {
            w = winding_all(d, v0, ns, dx, dy[e]);
          }
        }
        float sd = closed && w != 0 ? kFar : -kFar;
        if (best[e] < mrg2) {
          const float dist = sqrtf(best[e]);
          sd = closed ? (w != 0 ? dist : -dist) : hwpx - dist;
        }
        live |= fabsf(sd * inv_rho) < 1.0f || fabsf((sd + pad) * inv_rho) < 1.0f;
        sv[32 * e] = make_float2(sd, __int_as_float(bidx[e]));
      }
      if (d.paths && closed && lane < UH && s_row[kr * UH + lane].y > kRowCross) atomicAdd(&d.paths[0], 1ull);
      if (__any_sync(0xffffffffu, live)) {
        if (lane == 0) {
          const int4 lr = make_int4(nti.x, g, (tx0 + kc) | (ty0 + kr / UNITS) << 16, p);
          const int l = atomicAdd(&s_nlive, 1);
          if (l < kLiveBatch) {
            s_live[l] = lr;
          } else {
            const int at = atomicAdd(&d.work[1], 1);
            if (in_bounds(d, at < d.cap * UNITS)) d.live_list[at] = lr;
          }
        }
      } else if (lane == 0 && d.deterministic) {
        d.partial[(size_t)(nti.x & (int)kSlotMask) * UNITS + (unsigned)nti.x / (1u << kSlotBits)] =
            make_float4(0.f, 0.f, 0.f, 0.f);
      }
      ni = __shfl_sync(0xffffffffu, nn, 0);
    }
    __syncthreads();
    // the chunk's live units go out with one atomic
    if (tid < 32) {
      const int n = min(s_nlive, kLiveBatch);
      int at = 0;
      if (lane == 0 && n > 0) at = atomicAdd(&d.work[1], n);
      at = __shfl_sync(0xffffffffu, at, 0);
      if (lane < n && in_bounds(d, at + lane < d.cap * UNITS)) d.live_list[at + lane] = s_live[lane];
    }
    __syncthreads();  // s_live, s_nlive and the shared lists are reused by the next chunk
    i = s_next[it & 1];
  }
}

// ------------------------------------------------------------------------------------------------
// Composite, one unit of 64 pixels per warp: a tile of 8 x 8, or four rows of a tile of 16 x 16 (whose
// four units are the four warps of a block).  The tile's pairs with some coverage are ordered by
// element id (ids are unique in a tile, so an id's rank is the number of smaller ids; for up to 32
// pairs the lanes hold the ids and rank them by shuffles), then per pixel Ihat = prod(1 - c_i) and
// prod(1 - tau c_i^pad) over the pairs in that order, and the per-pixel loss terms (Eq. 5, Eq. 6
// surrogate, force), summed over the unit by a fixed shuffle tree.
//
// Bound by instructions and by the round trips of one tile after another, not by bytes.  So a warp takes
// a run of tiles at once, a tile per lane (C of them, launch_raster_fwd): the lanes find their tiles'
// places and read the counts and first entries together, and settle the tiles without coverage by
// themselves (their loss is a constant of the level); the others are taken one at a time, the next one's
// entries in flight.  A list entry carries the slot, its class and its element (no gather per pair).
// The images are written where a later kernel reads them: Ihat everywhere when the distribution term
// (or the metrics) follows, both where a pair is near (the adjoint's pixels).  64 collages, 27.6 Mpx,
// 431 k tiles, 170 k of them covered: 283 -> 172 us, of which 55 are the products, 43 the loss terms
// and sums, 41 the tiles without coverage; 5000 elements at 2048^2: 78 -> 72 us; 64 outlines at 256^2:
// 48 -> 34 us; 1000 elements at 1024^2: 18 us before and now, 8 of them the launch and the first reads.
// ------------------------------------------------------------------------------------------------
constexpr int kCompWarps = 4;
constexpr int kCompWide = 256;  // lists of up to this many covering pairs are ranked in shared memory

// A tile's place: origin in pixels (x | y << 16), side and first pixel of its problem.
struct TilePos {
  unsigned xy;
  int res;
  long long pix;
};
// The places of tiles base + lane (a lane beyond `count` repeats the last): the problem of the first, by
// one round of loads over the lanes for up to 1024 problems, then stepped to the lane's own.
__device__ __forceinline__ TilePos locate_tiles(const Dev& d, int base, int count, int T) {
  const int lane = threadIdx.x & 31, tile = base + min(lane, count - 1);
  int p = 0;
  if (d.n_probs > 1) {
    if (d.n_probs <= 1024) {
      p = -1;
      for (int i = 0; i < d.n_probs; i += 32)
        p += __popc(__ballot_sync(0xffffffffu, i + lane < d.n_probs && d.prob_tile_base[min(i + lane, d.n_probs)] <= base));
    } else {
      p = find_prob(d.prob_tile_base, d.n_probs, base);
    }
    while (p + 1 < d.n_probs && d.prob_tile_base[p + 1] <= tile) ++p;
  }
  const int lt = tile - d.prob_tile_base[p], ntx = d.prob_ntx[p];
  // lt / ntx by a float reciprocal, off by at most one (lt <= 2^24 is exact)
  int ty = (int)((float)lt * __frcp_rn((float)ntx));
  int tx = lt - ty * ntx;
  if (tx < 0) {
    ty -= 1;
    tx += ntx;
  } else if (tx >= ntx) {
    ty += 1;
    tx -= ntx;
  }
  return {(unsigned)(tx * T) | (unsigned)(ty * T) << 16, d.prob_res[p], d.prob_pix_base[p]};
}

// G pairs' records are read together: two where the tiles outnumber the warps and resident warps hide the
// reads, eight (with twice the registers) where each warp has one tile at most, so that a crowded tile's
// list is a shorter chain.  1000 elements, two -> eight: 20 -> 16 us at 128^2, 14 -> 12 at 256^2 (the whole
// iteration 68 -> 64 and 70 -> 66); 200 blobs at 512^2: 50.6 -> 49.3 an iteration; with more tiles than
// warps eight are slower, as fewer warps are resident (1000 elements at 1024^2: 87 -> 91, 64 collages: 863 ->
// 943).
constexpr int kCompWideGroup = 8;
template <int T, int G>
__global__ void __launch_bounds__(kCompWarps * 32, G == 2 ? 9 : 4) k_composite(Dev d, float* out_bw, float* out_tau,
                                                                              int flags, int C) {
  constexpr int UNITS = T * T / 64, NP = T * T, DY = 32 / T;
  __shared__ unsigned s_ord[kCompWarps][kCompWide];   // the covering pairs' slots and classes, in order
  __shared__ unsigned s_elem[kCompWarps][kCompWide];  // a long list's element ids, in list order
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int stride = (UNITS == 1 ? gridDim.x * kCompWarps : gridDim.x) * C;
  const int unit = UNITS == 1 ? 0 : wid;
  int base = (UNITS == 1 ? blockIdx.x * kCompWarps + wid : blockIdx.x) * C;
  // what the level switch wrote is read before the emission has completed
  TilePos pos{};
  float empty = 0.0f;
  auto place = [&]() {
    const int count = min(C, d.total_tiles - base);
    pos = locate_tiles(d, base, count, T);
    if ((flags & kCompLoss) && lane < count) empty = d.loss0[(base + lane) * UNITS + unit];
  };
  if (base < d.total_tiles) place();
  pdl_enter();
  if (blockIdx.x == 0)  // the emission has completed
    for (int i = threadIdx.x; i < kSlotInts; i += kCompWarps * 32) d.slots[i] = 0;
  if (blockIdx.x == 0 && threadIdx.x == 0) {  // the emission has completed: its work list is spent
    d.chunk_count[0] = d.chunk_count[1] = 0;
    d.work[0] = 0;
  }
  if (*d.status & kStatusNoBins) return;
  const float inv_rho = 1.0f / d.L.rho_px, pad = d.L.pad_px, tau = d.L.tau;
  unsigned* w_ord = s_ord[wid];
  unsigned* w_elem = s_elem[wid];
  const int ux = lane % T, uy = unit * (64 / T) + lane / T;  // the lane's first pixel in a tile; the
                                                             // second lies DY rows below
  int m_max = 0;  // the fullest list this warp saw (the host keeps the lists' capacity ahead of it)
  for (; base < d.total_tiles; base += stride) {
    // ---- the run's tiles, one per lane ----
    const bool mine = lane < C && base + lane < d.total_tiles;
    int n = 0;
    bool covered = false;
    if (mine) {
      n = d.tile_n[base + lane];
      const unsigned first = d.tile_list[(size_t)(base + lane) * d.tile_cap].x;  // used when n = 1
      if (!in_bounds(d, n >= 0 && n <= d.tile_cap)) n = 0;
      covered = n > 1 || (n == 1 && first >> kSlotBits != kPairOut);
      m_max = max(m_max, n);
    }
    if (UNITS > 1) __syncthreads();  // every unit has the tiles' counts
    if (mine && unit == 0) {  // for the next iteration, empty lists
      d.tile_n[base + lane] = 0;
      d.tile_m[base + lane] = n;
    }
    const unsigned todo0 = __ballot_sync(0xffffffffu, covered);
    auto tile_at = [&](int b) -> TilePos {
      return {__shfl_sync(0xffffffffu, pos.xy, b), __shfl_sync(0xffffffffu, pos.res, b),
              __shfl_sync(0xffffffffu, pos.pix, b)};
    };
    auto no_coverage = [&](const TilePos& at) {  // Ihat = 1, A_tau = 0
      const int X = (int)(at.xy & 0xffffu) + ux, Y = (int)(at.xy >> 16) + uy, off = Y * at.res + X;
      const bool in0 = X < at.res && Y < at.res, in1 = X < at.res && Y + DY < at.res;
      auto fill = [&](float* img, float v) {
        if (in0) img[at.pix + off] = v;
        if (in1) img[at.pix + off + DY * at.res] = v;
      };
      if (flags & kCompAllI) fill(d.img_I, 1.0f);
      if (out_bw) fill(out_bw, 1.0f);
      if (out_tau) fill(out_tau, 0.0f);
    };
    if ((flags & kCompLoss) && mine && !covered)
      d.lossA[(base + lane) * UNITS + unit] = make_float4(empty, 0.0f, 0.0f, 0.0f);
    if ((flags & kCompAllI) || out_bw || out_tau)
      for (unsigned b = __ballot_sync(0xffffffffu, mine) & ~todo0; b; b &= b - 1u) no_coverage(tile_at(__ffs((int)b) - 1));
    // ---- the covered ones, one at a time ----
    uint2 ent = make_uint2(0u, 0u);
    auto fetch = [&](int b) {  // for lane l, entry l of tile base + b (used only below the count)
      if (lane < d.tile_cap) ent = d.tile_list[(size_t)(base + b) * d.tile_cap + lane];
    };
    if (todo0) fetch(__ffs((int)todo0) - 1);
    for (unsigned todo = todo0; todo;) {
      const int b = __ffs((int)todo) - 1, cur = base + b;
      todo &= todo - 1u;
      const int m = __shfl_sync(0xffffffffu, n, b);
      const TilePos at = tile_at(b);
      const uint2 e0 = ent;
      if (todo) fetch(__ffs((int)todo) - 1);
      const int X = (int)(at.xy & 0xffffu) + ux, Y = (int)(at.xy >> 16) + uy, off = Y * at.res + X;
      const bool in0 = X < at.res && Y < at.res, in1 = X < at.res && Y + DY < at.res;
      // the covering pairs in element order: w_ord[0..na)
      const size_t lb = (size_t)cur * d.tile_cap;
      int na = 0;
      bool near = false, wide = false;
      __syncwarp();  // the previous tile's readers of this warp's lists are done
      if (m <= 32) {
        const unsigned cls = e0.x >> kSlotBits;
        const bool act = lane < m && cls != kPairOut;
        const unsigned bal = __ballot_sync(0xffffffffu, act);
        near = __any_sync(0xffffffffu, act && cls == kPairNear);
        na = __popc(bal);
        int r = 0;
        if (na > 1)
          for (unsigned q = bal; q; q &= q - 1u) r += __shfl_sync(0xffffffffu, e0.y, __ffs((int)q) - 1) < e0.y ? 1 : 0;
        if (act) w_ord[r] = e0.x;
      } else {
        if (lane == 0 && unit == 0 && d.paths) atomicAdd(&d.paths[2], 1ull);
        // the covering pairs' ids compacted into shared memory, then ranked against one another there
        // (one address for every lane); beyond kCompWide of them, ranked in global memory
        for (int i0 = 0; i0 < m; i0 += 32) {
          const uint2 e = i0 + lane < m ? d.tile_list[lb + i0 + lane] : make_uint2(0u, 0u);
          const unsigned cls = e.x >> kSlotBits;
          const bool act = i0 + lane < m && cls != kPairOut;
          const unsigned bal = __ballot_sync(0xffffffffu, act);
          near |= __any_sync(0xffffffffu, act && cls == kPairNear);
          const int k = na + __popc(bal & ((1u << lane) - 1u));
          if (act && k < kCompWide) w_elem[k] = e.y;
          na += __popc(bal);
        }
        __syncwarp();
        wide = na > kCompWide;
        unsigned* out = wide ? d.tile_sorted + lb : w_ord;
        for (int i = lane; i < m; i += 32) {
          const uint2 e = d.tile_list[lb + i];
          if (e.x >> kSlotBits == kPairOut) continue;
          int r = 0;
          if (!wide)
            for (int j = 0; j < na; ++j) r += w_elem[j] < e.y ? 1 : 0;
          else
            for (int j = 0; j < m; ++j) {
              const uint2 f = d.tile_list[lb + j];
              r += f.x >> kSlotBits != kPairOut && f.y < e.y ? 1 : 0;
            }
          out[r] = e.x;  // (the units of a tile write the same values to the global list)
        }
      }
      __syncwarp();  // the ordered list is visible to the whole warp
      if (na == 0) {  // every listed pair is outside
        no_coverage(at);
        if ((flags & kCompLoss) && lane == b) d.lossA[cur * UNITS + unit] = make_float4(empty, 0.0f, 0.0f, 0.0f);
        continue;
      }
      float cov[2] = {0.0f, 0.0f};
      if (flags & kCompLoss) {
        if (in0) cov[0] = d.covc[at.pix + off];
        if (in1) cov[1] = d.covc[at.pix + off + DY * at.res];
      }
      // products over the pairs in element order, in groups of G pairs whose signed
      // distances are read before any is used
      float keep[2] = {1.0f, 1.0f}, keept[2] = {1.0f, 1.0f};
      int nfull[2] = {0, 0}, npos[2] = {0, 0};  // pairs with c^pad = 1, with c^pad > 0
      const float2* sv = d.saved + unit * 64 + lane;
      for (int i0 = 0; i0 < na; i0 += G) {
        if (wide && i0 % kCompWide == 0) {  // the next stretch of a very long list
          __syncwarp();
          for (int i = lane; i < min(kCompWide, na - i0); i += 32) w_ord[i] = d.tile_sorted[lb + i0 + i];
          __syncwarp();
        }
        float sd[G][2];
        unsigned ent_u[G];
#pragma unroll
        for (int u = 0; u < G; ++u) {
          ent_u[u] = i0 + u < na ? w_ord[(i0 + u) % kCompWide] : kPairOut << kSlotBits;
          if (ent_u[u] >> kSlotBits == kPairNear) {
            const float2* rec = sv + (size_t)(ent_u[u] & kSlotMask) * NP;
            sd[u][0] = rec[0].x;
            sd[u][1] = rec[32].x;
          }
        }
#pragma unroll
        for (int u = 0; u < G; ++u) {
          const unsigned cls = ent_u[u] >> kSlotBits;  // (the same in every lane)
          if (cls == kPairNear) {
#pragma unroll
            for (int k = 0; k < 2; ++k) {
              const float omc = Sfun(-sd[u][k] * inv_rho), cp = Sfun((sd[u][k] + pad) * inv_rho);
              keep[k] *= omc;
              keept[k] *= 1.0f - tau * cp;
              nfull[k] += cp == 1.0f;
              npos[k] += cp > 0.0f;
            }
          } else if (cls == kPairIn) {  // c = c^pad = 1
#pragma unroll
            for (int k = 0; k < 2; ++k) {
              keep[k] = 0.0f;
              keept[k] *= 1.0f - tau;
              nfull[k] += 1;
              npos[k] += 1;
            }
          }
        }
      }
      const bool grad = (flags & kCompLoss) && near;  // the adjoint reads this unit's images
      float lc = 0.0f, lo = 0.0f, ld = 0.0f;
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        if (!(k ? in1 : in0)) continue;
        const int o = off + k * DY * at.res;
        const float ihat = keep[k];
        const float A = 1.0f - keept[k];
        if (flags & kCompLoss) {
          const float W = cov[k] >= 0.5f ? d.L.w_in : d.L.w_out;
          const float df = ihat - (1.0f - cov[k]);
          lc += W * df * df;
          // the kink of max(0, A - tau): one fully covering element gives A = tau exactly and any
          // other element with c^pad > 0 lifts A above it, by less than float can resolve when that
          // c^pad is tiny; so the side of the kink is taken from the counts in that case (exact)
          const bool over = nfull[k] >= 2 || (nfull[k] == 1 ? npos[k] > 1 : A > tau);
          lo += over ? fmaxf(A - tau, 0.0f) : 0.0f;
          // the downward potential 1 - y in pixels (exact), divided by the side once per unit
          const float fy = (float)(Y + k * DY) + 0.5f;
          ld += (1.0f - ihat) * (d.L.force_kind == 0
                                     ? (float)at.res - fy
                                     : force_potential(d.L, ((float)X + 0.5f) / (float)at.res, fy / (float)at.res));
          if (grad) d.img_Pt[at.pix + o] = over ? -keept[k] : keept[k];  // the sign: the side of the kink
        }
        if (grad || (flags & kCompAllI)) d.img_I[at.pix + o] = ihat;
        if (out_bw) out_bw[at.pix + o] = ihat;
        if (out_tau) out_tau[at.pix + o] = A;
      }
      if (flags & kCompLoss) {
        // fixed-order sums of the three partials, in one tree: after two steps lane l carries value
        // l / 8 (lc, lo, ld, none)
        const bool h = lane & 16, q = lane & 8;
        const float a = (h ? ld : lc) + __shfl_xor_sync(0xffffffffu, h ? lc : ld, 16);
        const float b2 = (h ? 0.0f : lo) + __shfl_xor_sync(0xffffffffu, h ? lo : 0.0f, 16);
        float v = (q ? b2 : a) + __shfl_xor_sync(0xffffffffu, q ? a : b2, 8);
        for (int o = 4; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 16 && d.L.force_kind == 0) v /= (float)at.res;
        if ((lane & 7) == 0) reinterpret_cast<float*>(d.lossA + cur * UNITS + unit)[lane >> 3] = v;
      }
    }
    if (base + stride < d.total_tiles) {
      base += stride;
      place();
      base -= stride;
    }
  }
  // (the host asks only whether a list passed 3/4 of the capacity)
  if (m_max * 4 > d.tile_cap * 3) atomicMax(d.tile_max, m_max);
}

// Per level: the containment loss of a unit that no element covers (Ihat = 1), summed as above.
template <int T>
__global__ void __launch_bounds__(kCompWarps * 32) k_empty_loss(Dev d) {
  constexpr int UNITS = T * T / 64, DY = 32 / T;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int u = blockIdx.x * kCompWarps + wid;
  if (u >= d.total_tiles * UNITS) return;
  const TilePos at = locate_tiles(d, u / UNITS, 1, T);
  const int X = (int)(at.xy & 0xffffu) + lane % T, Y = (int)(at.xy >> 16) + (u % UNITS) * (64 / T) + lane / T;
  float lc = 0.0f;
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    if (X >= at.res || Y + k * DY >= at.res) continue;
    const float cov = d.covc[at.pix + (long long)(Y + k * DY) * at.res + X];
    const float W = cov >= 0.5f ? d.L.w_in : d.L.w_out;
    const float df = 1.0f - (1.0f - cov);
    lc += W * df * df;
  }
  for (int o = 16; o; o >>= 1) lc += __shfl_xor_sync(0xffffffffu, lc, o);
  if (lane == 0) d.loss0[u] = lc;
}

// ------------------------------------------------------------------------------------------------
// Adjoint, one unit (64 pixels) of a (tile, element) pair per warp: dL/dIhat and dL/dA_tau per pixel,
// then the chain dL/dc -> dc/dsd -> dsd/d(closest segment) -> d/d(tx, ty, theta, s) of Eq. 2, reduced
// over the unit's pixels by a fixed shuffle tree and added to the element's gradient (or stored per unit).
// The grid's first blocks, one per problem or more, assemble the loss instead: its partials are complete,
// and the work (a read of 16 B per unit) fits beside the adjoint's round trips without a launch, a second
// stream and the two joins that the end of an iteration waited for.
// Where the distribution term's adjoint is the predecessor, what the kernels before that one wrote (the
// work list, the transforms, the saved distances and segments, the images, the loss partials) is read
// while it drains, from L2 (pdl_enter's second rule): 100 outlines at 1000^2 52.0 us an iteration instead of
// 55.2, 200 blobs at 512^2 43.1 instead of 45.7.
// ------------------------------------------------------------------------------------------------
__device__ __forceinline__ float warp_sum_f(float x) {
  for (int o = 16; o; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}
// Loss of one problem (Eq. 8) in parts of kLossUnits units or more, by its own size alone, so that it has the
// same bits in any batch: fixed-order float sums of a part's partials (eight strided accumulators per thread,
// then a shuffle tree within a warp; the sums over warps and parts, the means and the weighted total in float
// pairs), and the block that ends last adds the parts in order.  No FP64, which is slow on this part.  A block reads 1024 units in a round trip, and one block for the 16384 of a 1024^2 image ended 4 to 7
// us after the adjoint's others; in parts, summed before the predecessor has completed where that is the
// distribution term's adjoint, an iteration of 100 outlines at 1000^2 takes 56.4 us instead of 61.9, of 64
// outline fits at 256^2 96.5 instead of 99.3, of 5000 elements at 2048^2 370 instead of 373.
// Returns whether the problem has more than one part and this was one of them.
__device__ bool assemble_loss(const Dev& d, int p, int part, bool wait) {
  constexpr int NT = kPairWarps * 32, ACC = 8;
  __shared__ float s_red[4][kPairWarps];
  const int units = d.tile * d.tile / 64;
  int t0 = d.prob_tile_base[p] * units, t1 = d.prob_tile_base[p + 1] * units;
  const int parts = min(max((t1 - t0) / kLossUnits, 1), kLossParts);
  const float side = (float)d.prob_res[p];
  float np_lo;  // pixels: np + np_lo
  const float np = two_prod(side, side, np_lo), inv_np = div_normal(1.0f, np);
  if (wait) pdl_enter();  // the place is the level's: read before the predecessor has completed
  if (part >= parts) return false;
  if (parts > 1) {
    const int n = (t1 - t0 + parts - 1) / parts;
    t0 += part * n;
    t1 = min(t0 + n, t1);
  }
  float a[ACC] = {}, b[ACC] = {}, c[ACC] = {}, u[ACC] = {};
  for (int t = t0 + (int)threadIdx.x; t < t1; t += NT * ACC)
#pragma unroll
    for (int k = 0; k < ACC; ++k) {
      const float4 v = t + k * NT < t1 ? __ldcg(&d.lossA[t + k * NT]) : make_float4(0.f, 0.f, 0.f, 0.f);
      a[k] += v.x;
      b[k] += v.y;
      c[k] += v.z;
    }
  if (d.L.gamma != 0.0f && d.L.n_dil > 0) {
    int u0 = d.prob_dtile_base[p], u1 = d.prob_dtile_base[p + 1];
    if (parts > 1) {
      const int n = (u1 - u0 + parts - 1) / parts;
      u0 += part * n;
      u1 = min(u0 + n, u1);
    }
    for (int t = u0 + (int)threadIdx.x; t < u1; t += NT * ACC)
#pragma unroll
      for (int k = 0; k < ACC; ++k) u[k] += t + k * NT < u1 ? __ldcg(&d.lossU[t + k * NT]) : 0.0f;
  }
  auto sum = [](float (&x)[ACC]) {
    return warp_sum_f(((x[0] + x[1]) + (x[2] + x[3])) + ((x[4] + x[5]) + (x[6] + x[7])));
  };
  const float sa = sum(a), sb = sum(b), sc = sum(c), su = sum(u);
  const int w = threadIdx.x >> 5;
  if ((threadIdx.x & 31) == 0) {
    s_red[0][w] = sa;
    s_red[1][w] = sb;
    s_red[2][w] = sc;
    s_red[3][w] = su;
  }
  __syncthreads();
  if (w == 0) {  // from here on in float pairs, a sum on each of lanes 0..3, so that each term is rounded once
    const int lane = threadIdx.x & 31, k = lane & 3;
    FloatPair r{s_red[k][0], 0.0f};
    for (int i = 1; i < kPairWarps; ++i) r.add(s_red[k][i]);
    if (parts > 1) {
      float2* sums = d.loss_part + 4 * (size_t)p * kLossParts;
      if (lane < 4) __stcg(&sums[4 * part + k], make_float2(r.hi, r.lo));
      __threadfence();
      __syncwarp();
      int done = 0;
      if (lane == 0) done = atomicAdd(&d.loss_done[p], 1);
      if (__shfl_sync(0xffffffffu, done, 0) != parts - 1) return true;
      __threadfence();
      if (lane == 0) d.loss_done[p] = 0;
      r = {0.0f, 0.0f};
#pragma unroll 1  // (the kernel's code, fetched anew by each block, is what a small problem waits for)
      for (int i = 0; i < parts; ++i) {
        const float2 v = __ldcg(&sums[4 * i + k]);
        r.add(v.x);
        r.lo += v.y;
      }
    }
    FloatPair m = r;
    if (k != 3) {  // the mean over the pixels
      m.hi = r.hi * inv_np;
      m.lo = (fmaf(-m.hi, np, r.hi) + fmaf(-m.hi, np_lo, r.lo)) * inv_np;
    }
    FloatPair L{0.0f, 0.0f};  // the weighted total
    L.add_product(k == 0 ? d.L.alpha : k == 1 ? d.L.beta : k == 2 ? d.L.delta : d.L.gamma, m);
#pragma unroll
    for (int o = 1; o <= 2; o *= 2) {
      const float hi = __shfl_xor_sync(0xffffffffu, L.hi, o), lo = __shfl_xor_sync(0xffffffffu, L.lo, o);
      L.add(hi);
      L.lo += lo;
    }
    float* out = d.loss_terms + 5 * p;
    if (lane < 4) out[k ^ (k >> 1)] = m.value();  // containment, overlap, distribution, force
    if (lane == 0) out[4] = L.value();
  }
  return parts > 1;
}

// FIT: also dL/d(vertex) for outline fitting (d.fit).  RES: a grid of resident blocks (else a block per unit slot).
template <int T, bool FIT, bool RES>
__global__ void __launch_bounds__(kPairWarps * 32, FIT ? 7 : 8) k_raster_bwd(Dev d, int mark, int early, int n_loss) {
  constexpr int NP = T * T, UNITS = NP / 64, DY = 32 / T;
  if ((int)blockIdx.x < n_loss) {
    const bool ok = !(__ldcg(d.status) & kStatusNoBins);
    int p = blockIdx.x, part = 0, per = 1;  // blocks per problem
    if (n_loss > d.n_probs) {
      per = n_loss / d.n_probs;
      part = p / d.n_probs;
      p -= part * d.n_probs;
    }
    bool wait = !early;
    for (; ok && part < kLossParts && assemble_loss(d, p, part, wait); part += per) {
      wait = false;
      __syncthreads();
    }
    if (early || !ok) pdl_enter();
    if (ok && mark) mark_step_if_last(d);
    return;
  }
  const float inv_rho = 1.0f / d.L.rho_px, pad = d.L.pad_px, tau = d.L.tau;
  const bool use_u = d.L.gamma != 0.0f;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int stride = ((int)gridDim.x - n_loss) * kPairWarps;
  int i = ((int)blockIdx.x - n_loss) * kPairWarps + wid;
  // the status and the number of listed units (those without a gradient-carrying pixel are not listed): before
  // the wait from L2, by one thread of a block, and only in a grid of resident blocks.  (The words are the same
  // for all blocks: read from L2 by every warp of a block per unit slot, 1000 elements at 1024^2 took 148 us an
  // iteration, 113 after the wait through L1; 30 elements at 64^2 by every warp of 1216 blocks 36.0, 34.9 by one of
  // each.)
  int status, live;
  bool waited = !RES;
  if (RES) {
    __shared__ int2 s_head;
    if (threadIdx.x == 0) s_head = make_int2(__ldcg(d.status), __ldcg(&d.work[1]));
    __syncthreads();
    status = s_head.x;
    live = s_head.y;
  } else {
    pdl_enter();
    status = *d.status;
    live = d.work[1];
  }
  if (status & kStatusNoBins) {
    if (!waited) pdl_enter();
    return;
  }
  const int n_live = min(live, d.cap * UNITS);
  auto wait = [&]() {
    if (!waited) pdl_enter();
    waited = true;
  };
  int4 rec = i < n_live ? __ldcg(&d.live_list[i]) : make_int4(0, 0, 0, 0);
  for (; i < n_live; i += stride) {
    // the next unit's record is read while this one is worked on
    const int4 rec_next = i + stride < n_live ? __ldcg(&d.live_list[i + stride]) : rec;
    const int slot = rec.x & (int)kSlotMask, unit = (int)((unsigned)rec.x >> kSlotBits), g = rec.y, txy = rec.z, p = rec.w;
    if (!in_bounds(d, slot >= 0 && slot < d.cap && g >= 0 && g < d.n_elems && p >= 0 && p < d.n_probs)) {
      rec = rec_next;
      continue;
    }
    const int res = d.prob_res[p];
    const float inv_np = 1.0f / ((float)res * (float)res);
    const int v0 = d.elem_voff[g];
    const bool closed = d.elem_closed[g] != 0;
    const float4 tp = __ldcg(&d.tpx[g]);
    const float4 qg = __ldcg(&d.q[g]);
    const float s_inv = 1.0f / qg.w;
    // the lane's pixels: one column, rows Y and Y + DY
    const int X = (txy & 0xffff) * T + lane % T, Y = (txy >> 16) * T + unit * (64 / T) + lane / T;
    const long long pix0 = d.prob_pix_base[p] + (long long)Y * res + X;
    const float2* sv = d.saved + (size_t)slot * NP + unit * 64 + lane;
    // outline fitting: d(pixel)/d(local vertex) = s res R(theta), applied transposed below
    float fc = 0.0f, fs = 0.0f, sres = 0.0f;
    int nv = 0;
    if (FIT) {
      sincosf(qg.z, &fs, &fc);
      sres = qg.w * (float)res;
      nv = d.elem_voff[g + 1] - v0;
    }
    // every per-pixel input of the warp's pixels in one round of loads
    float2 srec[2];
    float ihat[2], pt_s[2], cov[2], gou[2];
    if (!early) wait();
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      srec[k] = make_float2(kFar, 0.0f);
      ihat[k] = pt_s[k] = cov[k] = gou[k] = 0.0f;
      if (X < res && Y + k * DY < res) {
        const long long pix = pix0 + k * DY * res;
        srec[k] = __ldcg(&sv[32 * k]);
        ihat[k] = __ldcg(&d.img_I[pix]);
        pt_s[k] = __ldcg(&d.img_Pt[pix]);
        cov[k] = d.covc[pix];
      }
    }
    // the closest segments of the pixels that may carry a gradient (never the out-of-range ones, whose
    // sd is 1e30), in flight before the weights are formed
    bool act[2];
    float4 sa[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const float sd = srec[k].x;
      act[k] = fabsf(sd * inv_rho) < 1.0f || fabsf((sd + pad) * inv_rho) < 1.0f;
      if (act[k] && !in_bounds(d, (unsigned)__float_as_int(srec[k].y) < (unsigned)(d.elem_voff[g + 1] - v0)))
        act[k] = false;
      if (act[k]) sa[k] = __ldcg(&d.segA[v0 + __float_as_int(srec[k].y)]);
    }
    wait();
    if (use_u)
#pragma unroll
      for (int k = 0; k < 2; ++k)
        if (act[k]) gou[k] = d.gOu[pix0 + k * DY * res];
    // dL/dsd per pixel
    float gsd[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const float sd = srec[k].x;
      const float x = sd * inv_rho, xp = (sd + pad) * inv_rho;
      gsd[k] = 0.0f;
      if (act[k]) {
        const float pt = fabsf(pt_s[k]);  // negative: the pixel is on the rising side of the Eq. 6 kink
        const float W = cov[k] >= 0.5f ? d.L.w_in : d.L.w_out;
        const float py = (float)(Y + k * DY) + 0.5f;
        // O = 1 - Ihat: the uniform and force terms enter dL/dIhat with a minus sign
        float gI = d.L.alpha * inv_np * 2.0f * W * (ihat[k] - (1.0f - cov[k])) - d.L.gamma * gou[k];
        if (d.L.delta != 0.0f)
          gI -= d.L.delta * inv_np * force_potential(d.L, ((float)X + 0.5f) / (float)res, py / (float)res);
        const float gA = pt_s[k] < 0.0f ? d.L.beta * inv_np : 0.0f;
        const float omc = Sfun(-x), cp = Sfun(xp);
        // dIhat/dc_i = -prod_{j != i}(1 - c_j) = -Ihat / (1 - c_i)   (0 when another c_j = 1)
        const float gc = omc > 0.0f ? div_normal(-gI * ihat[k], omc) : 0.0f;
        // dA/dc^pad_i = tau prod_{j != i}(1 - tau c^pad_j)
        const float gcp = div_normal(gA * tau * pt, 1.0f - tau * cp);
        gsd[k] = (gc * dSfun(x) + gcp * dSfun(xp)) * inv_rho;
      }
    }
    float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      if (gsd[k] == 0.0f) continue;
      const float sd = srec[k].x;
      const float dx = ((float)X + 0.5f - tp.x) - tp.z, dy = ((float)(Y + k * DY) + 0.5f - tp.y) - tp.w;
      const float ex = sa[k].z, ey = sa[k].w, ee = ex * ex + ey * ey;
      const float wx = dx - sa[k].x, wy = dy - sa[k].y;
      // (a segment shorter than 1e-19 px is its start point)
      const float u = ee >= FLT_MIN ? __saturatef(div_normal(wx * ex + wy * ey, ee)) : 0.0f;
      const float qx = fmaf(u, ex, sa[k].x), qy = fmaf(u, ey, sa[k].y);  // closest point, rel. to t
      // unit normal from the closest point towards the pixel: for a closest point inside the
      // segment it is the segment's perpendicular on the pixel's side (well conditioned even
      // when the pixel is almost on the outline); at an end point it is the direction to the pixel
      const bool inner = u > 0.0f && u < 1.0f;
      const float rx = dx - qx, ry = dy - qy, rr = rx * rx + ry * ry;
      const float nn = inner ? ee : rr;
      if (!(nn >= FLT_MIN)) continue;  // the pixel is the closest point
      const float ir = rsqrt_normal(nn), side = ex * wy - ey * wx >= 0.0f ? ir : -ir;
      const float nx = inner ? -ey * side : rx * ir, ny = inner ? ex * side : ry * ir;
      // sd = sig * dist (closed: sig = +-1 by the winding; open: sd = hw - dist, sig = -1)
      const float sig = closed ? (sd > 0.0f ? 1.0f : -1.0f) : -1.0f;
      const float gs = -sig * gsd[k];
      a0 += gs * nx * (float)res;              // d(dist)/dt = -n, t in unit coords
      a1 += gs * ny * (float)res;
      a2 += gs * (ny * qx - nx * qy);          // d(dist)/dtheta = -n . J q
      a3 += gs * (nx * qx + ny * qy) * s_inv;  // d(dist)/ds = -n . q / s
      if (FIT) {
        // d(dist)/d(end points) = -n (1 - u), -n u (the closest point moves with them), taken to
        // element-local unit coordinates
        const float gx = gs * nx, gy = gs * ny;
        const float lx = sres * (fc * gx + fs * gy), ly = sres * (fc * gy - fs * gx);
        const int j = __float_as_int(srec[k].y);
        const int ja = v0 + j, jb = v0 + (j + 1 == nv ? 0 : j + 1);
        atomicAdd(&d.dv[ja].x, lx * (1.0f - u));
        atomicAdd(&d.dv[ja].y, ly * (1.0f - u));
        atomicAdd(&d.dv[jb].x, lx * u);
        atomicAdd(&d.dv[jb].y, ly * u);
      }
    }
    // the four sums in one shuffle tree: after two steps lane l carries sum l / 8
    const bool h = lane & 16, q8 = lane & 8;
    const float b0 = (h ? a2 : a0) + __shfl_xor_sync(0xffffffffu, h ? a0 : a2, 16);
    const float b1 = (h ? a3 : a1) + __shfl_xor_sync(0xffffffffu, h ? a1 : a3, 16);
    float v = (q8 ? b1 : b0) + __shfl_xor_sync(0xffffffffu, q8 ? b0 : b1, 8);
    for (int o = 4; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((lane & 7) == 0) {
      if (d.deterministic) reinterpret_cast<float*>(d.partial + (size_t)slot * UNITS + unit)[lane >> 3] = v;
      else atomicAdd(d.dq + 4 * (size_t)g + (lane >> 3), (double)v);
    }
    rec = rec_next;
  }
  wait();
  if (mark) mark_step_if_last(d);
}

// ------------------------------------------------------------------------------------------------
// Container: coverage of every pixel by the container rings (nonzero rule), once per level.  One tile
// per block.  A ring segment matters to a tile if it comes within the coverage margin of the tile's
// pixel centres, or lies right of them at their height (the winding's ray runs to the right); any other
// is farther than the margin, where coverage saturates, and crosses no ray.  The block picks those by a
// float test with slack and brings only them into the tile's frame, in double and rounded once (FP64
// and the pixel-segment pairs bound the kernel when every segment was taken: 512 segments at 1024^2,
// 416 us, 45 now; 64 containers, 27.6 Mpx, 5.6 ms, 0.9 now).
// ------------------------------------------------------------------------------------------------
template <int T, int NT>
__global__ void __launch_bounds__(NT) k_container(Dev d) {
  constexpr int NP = T * T, PPT = NP / NT;
  __shared__ float4 s_seg[kSegCap];
  __shared__ float2 s_seg2[kSegCap];
  __shared__ int s_n;
  const float inv_rho = 1.0f / d.L.rho_px;
  for (int tile = blockIdx.x; tile < d.total_tiles; tile += gridDim.x) {
    const int p = find_prob(d.prob_tile_base, d.n_probs, tile);
    const int lt = tile - d.prob_tile_base[p], ntx = d.prob_ntx[p], res = d.prob_res[p];
    const int tx = lt % ntx, ty = lt / ntx;
    const double ox = (double)(tx * T), oy = (double)(ty * T);
    const float fres = (float)res;
    const float cx0 = (float)(tx * T) + 0.5f, cy0 = (float)(ty * T) + 0.5f, cy1 = cy0 + (float)(T - 1);
    SegQuery Q[PPT];
    float dx[PPT], dy[PPT];
#pragma unroll
    for (int k = 0; k < PPT; ++k) {
      const int local = threadIdx.x + k * NT;
      dx[k] = (float)(local % T) + 0.5f;
      dy[k] = (float)(local / T) + 0.5f;
      Q[k].best = FLT_MAX;
      Q[k].idx = 0;
      Q[k].wn = 0;
    }
    const int r0 = d.prob_ring_base[p], r1 = d.prob_ring_base[p + 1];
    for (int r = r0; r < r1; ++r) {
      const int b0 = d.ring_off[r], nv = d.ring_off[r + 1] - b0;
      for (int c0 = 0; c0 < nv; c0 += kSegCap) {
        const int cn = min(kSegCap, nv - c0);
        if (c0 > 0 && threadIdx.x == 0 && d.paths) atomicAdd(&d.paths[3], 1ull);
        if (threadIdx.x == 0) s_n = 0;
        __syncthreads();
        for (int j = threadIdx.x; j < cn; j += NT) {
          const int ai = b0 + c0 + j, bi = c0 + j + 1 == nv ? b0 : ai + 1;
          const float2 fa = d.ring_f[ai], fb = d.ring_f[bi];
          const float x1 = fmaxf(fa.x, fb.x) * fres, y0 = fminf(fa.y, fb.y) * fres, y1 = fmaxf(fa.y, fb.y) * fres;
          // the margin, and slack for the rounding of these floats
          const float m = d.L.rho_px + 0.06f + 4e-7f * fmaxf(fabsf(x1), fmaxf(fabsf(y0), fabsf(y1)));
          if (x1 + m < cx0 || y1 + m < cy0 || y0 - m > cy1) continue;
          const double ax = d.ring_pts[2 * ai] * res - ox, ay = d.ring_pts[2 * ai + 1] * res - oy;
          const double bx = d.ring_pts[2 * bi] * res - ox, by = d.ring_pts[2 * bi + 1] * res - oy;
          const float ex = (float)(bx - ax), ey = (float)(by - ay);
          const float ee = ex * ex + ey * ey;
          const int k = atomicAdd(&s_n, 1);  // (the order of the list does not matter)
          s_seg[k] = make_float4((float)ax, (float)ay, ex, ey);
          s_seg2[k] = make_float2((float)by, ee > 0.0f ? 1.0f / ee : 0.0f);
        }
        __syncthreads();
        const int n = s_n;
        for (int j = 0; j < n; ++j) {
          const float4 s = s_seg[j];
          const float2 s2 = s_seg2[j];
#pragma unroll
          for (int k = 0; k < PPT; ++k) seg_update(Q[k], dx[k], dy[k], s, s2, j, true);
        }
        __syncthreads();  // the list is refilled
      }
    }
#pragma unroll
    for (int k = 0; k < PPT; ++k) {
      const int local = threadIdx.x + k * NT;
      const int X = tx * T + local % T, Y = ty * T + local / T;
      if (X >= res || Y >= res) continue;
      const float dist = sqrtf(Q[k].best);
      const float sd = Q[k].wn != 0 ? dist : -dist;
      d.covc[d.prob_pix_base[p] + (long long)Y * res + X] = Sfun(sd * inv_rho);
    }
  }
}

// ------------------------------------------------------------------------------------------------
template <int T>
struct TileCfg;
template <>
struct TileCfg<8> {
  static constexpr int NT = 64;
};
template <>
struct TileCfg<16> {
  static constexpr int NT = 256;
};

template <int T>
static cudaError_t fwd_t(const Dev& d, cudaStream_t s, int pair_grid, int tile_grid, float* bw,
                         float* tau, int part, int flags) {

  cudaError_t e = cudaSuccess;
  // (with more chunks than blocks the first wave is all long outlines, and the rest are taken as blocks end)
  const int n_sm = d.few_chunks ? slot_sms(d, pair_grid, kSlotRanks) : 0;
  if (part & 1)
    e = d.emit_threads == 256 ? klaunch(d.pdl, k_raster_chunks<T, 256>, pair_grid, 256, 0, s, d, n_sm)
                              : klaunch(d.pdl, k_raster_chunks<T, 128>, pair_grid, 128, 0, s, d, n_sm);
  if (e == cudaSuccess && (part & 2)) {
    // tiles a warp takes at once: a power of two that leaves four resident waves of blocks, so that dense
    // and empty stretches even out; then one run per warp
    const int per_block = T == 8 ? kCompWarps : 1;
    int C = 1;
    while (C < 32 && 2ll * C * 4 * tile_grid * per_block <= d.total_tiles) C *= 2;
    const int grid = C > 1 ? (d.total_tiles + C * per_block - 1) / (C * per_block) : tile_grid;
    const bool few = d.total_tiles <= tile_grid * per_block;
    e = klaunch(d.pdl, few ? k_composite<T, kCompWideGroup> : k_composite<T, 2>, grid, kCompWarps * 32, 0, s, d, bw,
                tau, flags, C);
  }
  return e;
}

cudaError_t launch_raster_fwd(const Dev& d, cudaStream_t s, int pair_grid, int tile_grid,
                              float* out_bw, float* out_tau, int part, int flags) {
  switch (d.tile) {
    case 8: return fwd_t<8>(d, s, pair_grid, tile_grid, out_bw, out_tau, part, flags);
    case 16: return fwd_t<16>(d, s, pair_grid, tile_grid, out_bw, out_tau, part, flags);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_raster_bwd(const Dev& d, cudaStream_t s, int unit_grid, bool resident, bool mark_step) {
  // the loss blocks take the place of as many resident ones (at most half of them), so that none waits
  const int units = (int)min((long long)d.max_tiles * (d.tile * d.tile / 64), (long long)kLossUnits * kLossParts);
  // a block for each part of the largest problem, in a sixteenth of the resident blocks: more of them leave
  // the units' strided share to fewer warps (64 collages, an eighth and a half: 118.8 -> 122.9 and 190 us)
  const int lb = max(min(units / kLossUnits, unit_grid / (16 * d.n_probs)), 1);
  const int n_loss = d.n_probs * lb;
  const int grid = max(unit_grid - n_loss, (unit_grid + 1) / 2) + n_loss, mk = mark_step ? 1 : 0;
  const int early = d.L.gamma != 0.0f && d.L.n_dil > 0 ? 1 : 0;  // the predecessor is the distribution adjoint
  if (d.tile != 8 && d.tile != 16) return cudaErrorInvalidValue;
  auto kernel = [&](auto t, auto fit) {
    constexpr int T = decltype(t)::value;
    constexpr bool FIT = decltype(fit)::value;
    return resident ? k_raster_bwd<T, FIT, true> : k_raster_bwd<T, FIT, false>;
  };
  using std::false_type;
  using std::integral_constant;
  using std::true_type;
  const auto k = d.tile == 8 ? d.fit ? kernel(integral_constant<int, 8>{}, true_type{}) : kernel(integral_constant<int, 8>{}, false_type{})
                 : d.fit     ? kernel(integral_constant<int, 16>{}, true_type{})
                             : kernel(integral_constant<int, 16>{}, false_type{});
  return klaunch(d.pdl, k, grid, kPairWarps * 32, 0, s, d, mk, early, n_loss);
}

cudaError_t launch_container(const Dev& d, cudaStream_t s) {
  switch (d.tile) {
    case 8: k_container<8, TileCfg<8>::NT><<<d.total_tiles, TileCfg<8>::NT, 0, s>>>(d); break;
    case 16: k_container<16, TileCfg<16>::NT><<<d.total_tiles, TileCfg<16>::NT, 0, s>>>(d); break;
    default: return cudaErrorInvalidValue;
  }
  const int units = d.total_tiles * (d.tile * d.tile / 64), grid = (units + kCompWarps - 1) / kCompWarps;
  if (d.tile == 8) k_empty_loss<8><<<grid, kCompWarps * 32, 0, s>>>(d);
  else k_empty_loss<16><<<grid, kCompWarps * 32, 0, s>>>(d);
  return cudaGetLastError();
}

template <int T>
static void per_sm_t(int emit_threads, RasterOcc* o) {
  int a = 1, b = 1, c = 1;
  if (emit_threads == 256) cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, k_raster_chunks<T, 256>, 256, 0);
  else cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, k_raster_chunks<T, 128>, 128, 0);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_raster_bwd<T, false, true>, kPairWarps * 32, 0);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&c, k_composite<T, 2>, kCompWarps * 32, 0);
  o->fwd_per_sm = a > 0 ? a : 1;
  o->bwd_per_sm = b > 0 ? b : 1;
  o->tile_per_sm = c > 0 ? c : 1;
  o->bwd_pairs_per_block = kPairWarps;
  o->tiles_per_block = T == 8 ? kCompWarps : 1;
}

void raster_occupancy(int tile, int emit_threads, RasterOcc* o) {
  if (tile == 16) per_sm_t<16>(emit_threads, o);
  else per_sm_t<8>(emit_threads, o);
}

}  // namespace collage
