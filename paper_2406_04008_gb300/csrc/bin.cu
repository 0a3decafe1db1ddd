// Transform (Eq. 2) and tile binning.
//
// Binning: the transform kernel gives every element a block of consecutive pair slots, one per tile
// of its tile rectangle (one atomic per element; a total beyond the capacity latches the overflow
// bit before any pair is written), and lists every element's kChunkPx-square chunks of its
// rectangle; the emission (csrc/raster.cu, per chunk) records each (tile, element) pair's slot in
// its tile's list; the composite then orders each tile's short list by element id before using it,
// so every tile lists its elements in increasing order whatever the order of the atomics.  The tile rectangle follows a fixed float formula
// (bin_rect), so the bins are bit-exact against the oracle's rule.
#include "internal.h"
#include "trig.h"

namespace collage {

// Tile rectangle of one element, float arithmetic in a fixed order with explicit round-to-nearest
// intrinsics (no contraction):
//   R_px = (s * r_bin) * res, c = t * res, m = ((rho + pad) + hw * res) + 1,
//   [floor(((c - R_px) - m) / T), floor(((c + R_px) + m) / T)] clipped to the grid's tiles.
// The circle of radius s * r_bin about t holds the whole outline because r_bin bounds every
// control point and a Bezier curve stays inside the convex hull of its control points.
__device__ int4 bin_rect(float4 q, float rbin, float hw, int res, int T, float rho, float pad) {
  const float fres = (float)res;
  const float Rpx = __fmul_rn(__fmul_rn(q.w, rbin), fres);
  const float cx = __fmul_rn(q.x, fres), cy = __fmul_rn(q.y, fres);
  const float m = __fadd_rn(__fadd_rn(__fadd_rn(rho, pad), __fmul_rn(hw, fres)), 1.0f);
  const float x0 = __fsub_rn(__fsub_rn(cx, Rpx), m), x1 = __fadd_rn(__fadd_rn(cx, Rpx), m);
  const float y0 = __fsub_rn(__fsub_rn(cy, Rpx), m), y1 = __fadd_rn(__fadd_rn(cy, Rpx), m);
  const float fT = (float)T;
  const float fx0 = floorf(__fdiv_rn(x0, fT)), fx1 = floorf(__fdiv_rn(x1, fT));
  const float fy0 = floorf(__fdiv_rn(y0, fT)), fy1 = floorf(__fdiv_rn(y1, fT));
  const int nt = (res + T - 1) / T;
  const float lim = (float)(nt - 1);
  int4 r = make_int4(0, 0, -1, -1);
  if (!(fx1 >= 0.0f && fy1 >= 0.0f && fx0 <= lim && fy0 <= lim)) return r;  // also NaN
  r.x = fx0 < 0.0f ? 0 : (int)fx0;
  r.y = fy0 < 0.0f ? 0 : (int)fy0;
  r.z = fx1 > lim ? nt - 1 : (int)fx1;
  r.w = fy1 > lim ? nt - 1 : (int)fy1;
  return r;
}

// Vertex of an element relative to its translation, in pixels: (s res R(theta)) v.  The matrix is
// formed once per element as float hi + lo parts (csrc/trig.h); the per-vertex product uses
// error-free transformations in float (FMA two-product and Knuth's two-sum, as in Ogita, Rump &
// Oishi 2005), so the result is within about one float ulp of the exact value without FP64 work
// per vertex (FP64 throughput is low on this part).  Explicit round-to-nearest intrinsics keep the
// compiler from contracting the error terms away.  A segment's end point and the next segment's
// start point come from the same call, so they are bitwise equal (the winding test relies on it).
struct RotFF {
  float m[4][2];  // row-major 2x2, (hi, lo)
};

__device__ __forceinline__ float dot2_ff(const float (&a)[2], const float (&b)[2], float vx, float vy) {
  const float p1 = __fmul_rn(a[0], vx), e1 = __fmaf_rn(a[0], vx, -p1);
  const float p2 = __fmul_rn(b[0], vy), e2 = __fmaf_rn(b[0], vy, -p2);
  const float sum = __fadd_rn(p1, p2);
  const float bb = __fsub_rn(sum, p1);
  const float es = __fadd_rn(__fsub_rn(p1, __fsub_rn(sum, bb)), __fsub_rn(p2, bb));
  const float tail = __fmaf_rn(a[1], vx, __fmaf_rn(b[1], vy, __fadd_rn(__fadd_rn(e1, e2), es)));
  return __fadd_rn(sum, tail);
}

__device__ __forceinline__ float2 vertex_px(const float2 v, const RotFF& M) {
  return make_float2(dot2_ff(M.m[0], M.m[1], v.x, v.y), dot2_ff(M.m[2], M.m[3], v.x, v.y));
}

// E = 1 or 4 elements per block: the pending Adam step of the previous iteration, then segment records
// (start, direction, end y, 1/|e|^2) of the vertices relative to the translation, translation in
// pixels as a float hi/lo pair, tile rectangle, the element's pair slots and its emission chunks.
// In warp 0, eight lanes per element take the step (one parameter each of the first four, the two bias
// powers on different lanes) and form the rotation-scale matrix; one barrier separates the step from
// the vertices.  Lanes own consecutive vertices; a segment's end point is the next lane's start point,
// shuffled, so each vertex is transformed once.
// E = 1: warps 0..2 transform the vertices while warp 3 files the tile rectangle, the pair slots and
// the chunk list, which do not depend on the vertices: the shortest chain for one element.
// E = 4: each warp does both for one element, so that four elements share the step's instructions.  It is taken when the elements fill the device several times
// over (launch_transform), where issue slots rather than latency bound the kernel.
constexpr int kTfThreads = 128;
constexpr int kTfWideElems = 4096;  // elements from which a block takes four: the two forms meet here
                                    // (18 and 17.5 us; at 26 k elements four take 56 us, one 100)
constexpr int kTfVertexWarps = 3;
template <int E>
__global__ void __launch_bounds__(kTfThreads) k_transform(Dev d, int zero_grad, int follows) {
  static_assert(E == 1 || E == 4, "eight lanes per element in one warp, one warp per element or block");
  __shared__ RotFF s_rot[E];
  __shared__ float4 s_q[E];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int g = E == 1 ? blockIdx.x : min((int)blockIdx.x * E + wid, d.n_elems - 1);
  const bool live = E == 1 || (int)blockIdx.x * E + wid < d.n_elems;
  // what is written once, at create or per level, is read before the predecessor has completed
  // (a single problem's resolution is read without waiting for the element's problem index)
  const int p = d.n_probs == 1 ? 0 : d.elem_prob[g];
  const int res = d.prob_res[p];
  const int v0 = d.elem_voff[g], nv = d.elem_voff[g + 1] - v0;
  const bool closed = d.elem_closed[g] != 0;
  const float hw = closed ? 0.0f : d.elem_hw[g];
  const bool files = E == 4 || wid == kTfVertexWarps, verts = E == 4 || wid < kTfVertexWarps;
  constexpr int kStride = E == 4 ? 32 : kTfVertexWarps * 32;
  const int k_first = E == 4 ? lane : wid * 32 + lane;
  float rbin = 0.0f;
  float2 va0 = make_float2(0.f, 0.f), vb0 = make_float2(0.f, 0.f);
  auto first_vertices = [&]() {  // (written by calls that replace the outlines, and by each fitting iteration)
    if (files) rbin = d.elem_rbin[g];
    if (verts && k_first < nv) {
      va0 = d.vloc[v0 + k_first];
      if (lane == 31 || k_first + 1 == nv) vb0 = d.vloc[v0 + (k_first + 1 == nv ? 0 : k_first + 1)];
    }
  };
  const bool early = follows && !d.fit;
  if (early) first_vertices();
  pdl_enter();
  if (!early) first_vertices();
  if (blockIdx.x == 0 && threadIdx.x == 0) {  // this iteration's live pairs and finished gradient blocks
    d.work[1] = 0;
    d.work[3] = 0;
  }
  if (blockIdx.x == 0)  // the distribution term's blocks count themselves again while the composite runs
    for (int i = threadIdx.x; i < 2 * kSlotInts; i += kTfThreads) d.slots[kSlotInts + i] = 0;
  if (wid == 0) {
    const int e = E == 1 ? 0 : lane >> 3, k = lane & 3, ge = min((int)blockIdx.x * E + e, d.n_elems - 1);
    const bool writer = (E == 1 ? lane < 4 : (lane & 7) < 4) && (int)blockIdx.x * E + e < d.n_elems;
    const int re = E == 1 ? res : d.prob_res[d.n_probs == 1 ? 0 : d.elem_prob[ge]];
    float x = reinterpret_cast<const float*>(d.q + ge)[k];
    // the previous iteration's step (when the outlines are fitted the transforms stay fixed)
    const bool step = *d.pending && !d.fit;
    if (step) {
      float m = reinterpret_cast<const float*>(d.m + ge)[k], v = reinterpret_cast<const float*>(d.v + ge)[k];
      const float gr = (float)d.dq[4 * (size_t)ge + k];
      const bool tr = !d.trainable || reinterpret_cast<const unsigned char*>(d.trainable + ge)[k];
      const float pw = powf((lane & 4) ? d.b2 : d.b1, (float)*d.step);
      const AdamScale a = adam_scale(d, __shfl_sync(0xffffffffu, pw, 0), __shfl_sync(0xffffffffu, pw, 4));
      if (tr) adam_entry(d, a, gr, x, m, v);
      if (k == 3) x = fminf(fmaxf(x, d.s_min), d.s_max);
      if (writer) {
        reinterpret_cast<float*>(d.m + ge)[k] = m;
        reinterpret_cast<float*>(d.v + ge)[k] = v;
      }
    }
    // the host-buffer step: the caller's params replace the stepped ones (the moments keep the step)
    if (d.q_in) x = reinterpret_cast<const float*>(d.q_in + ge)[k];
    if (writer && (step || d.q_in)) reinterpret_cast<float*>(d.q + ge)[k] = x;
    const float z = __shfl_sync(0xffffffffu, x, 2, 4), sc = __shfl_sync(0xffffffffu, x, 3, 4);
    if (writer) {
      reinterpret_cast<float*>(&s_q[e])[k] = x;
      // entry k of s res [cos, -sin; sin, cos]
      const float f = k == 1 ? -sc : sc;
      if (fabsf(z) <= kTrigMax) trig_entry(z, k == 0 || k == 3, f, (float)re, d.trig, s_rot[e].m[k]);
      else trig_wide(z, k == 0 || k == 3, f, (float)re, s_rot[e].m[k]);
    }
  }
  __syncthreads();
  if (!live) return;
  const int slot = E == 1 ? 0 : wid;
  const float4 q = s_q[slot];
  int4 r = make_int4(0, 0, -1, -1);
  int nx = 0, ny = 0, cbase = 0;
  bool heavy = false;
  if (files) {
    // the tile rectangle, the pair slots and the emission's chunks (lane 0 takes the counts)
    const bool finite = isfinite(q.x) && isfinite(q.y) && isfinite(q.z) && isfinite(q.w) && q.w > 0.0f;
    if (finite) r = bin_rect(q, rbin, hw, res, d.tile, d.L.rho_px, d.L.pad_px);
    else if (lane == 0) atomicOr(d.status, kStatusBadParam);
    if (lane == 0) {
      d.rect[g] = r;
      if (zero_grad) {
        double2* dq = reinterpret_cast<double2*>(d.dq + 4 * (size_t)g);
        dq[0] = dq[1] = make_double2(0.0, 0.0);
      }
    }
    if (r.z >= r.x && r.w >= r.y) {
      // the pair slots of the rectangle; beyond the capacity the bins of the iteration are void
      const int n = (r.z - r.x + 1) * (r.w - r.y + 1);
      // the emission's work: the rectangle in chunks of kChunkPx / T tiles a side; chunks whose
      // segments x tiles exceed kHeavyChunk are listed from the front, the others from the back,
      // so that the emission takes the costliest first and none trails at the end
      const int cw = d.chunk_tiles;
      nx = (r.z - r.x) / cw + 1;
      ny = (r.w - r.y) / cw + 1;
      const int tiles = min(r.z - r.x + 1, cw) * min(r.w - r.y + 1, cw);
      heavy = nv * tiles > kHeavyChunk;
      if (lane == 0) {  // both counts taken at once (neither waits for the other's result)
        const int pbase = atomicAdd(d.pair_need, n);
        cbase = atomicAdd(d.chunk_count + (heavy ? 0 : 1), nx * ny);
        if (pbase > d.cap - n) atomicOr(d.status, kStatusOverflow);
        d.elem_pbase[g] = pbase;
      }
    }
  }
  auto file_chunks = [&]() {
    if (nx == 0) return;
    const int at0 = __shfl_sync(0xffffffffu, cbase, 0), cw = d.chunk_tiles;
    // (heavy + light chunks beyond the list mean more pairs than the capacity too: the iteration
    // overflows and the emission does not read the list; every write stays inside it)
    if (at0 + nx * ny <= d.list_cap)
      for (int c = lane; c < nx * ny; c += 32) {
        const int at = heavy ? at0 + c : d.list_cap - 1 - (at0 + c);
        d.near_list[at] = make_int4(g, (r.x + (c % nx) * cw) | ((r.y + (c / nx) * cw) << 16), p, 0);
      }
  };
  if (E == 1 && files) {
    file_chunks();
    return;  // no barrier follows for this warp
  }
  const RotFF rot = s_rot[slot];
  for (int k0 = E == 4 ? 0 : wid * 32; k0 < nv; k0 += kStride) {  // warp-uniform trip count
    const int k = k0 + lane;
    const bool first = k0 < kStride;
    float2 a = make_float2(0.f, 0.f);
    if (k < nv) a = vertex_px(first ? va0 : d.vloc[v0 + k], rot);
    float2 b;
    b.x = __shfl_down_sync(0xffffffffu, a.x, 1);
    b.y = __shfl_down_sync(0xffffffffu, a.y, 1);
    const int kb = k + 1 == nv ? 0 : k + 1;
    if (k < nv && (lane == 31 || k + 1 == nv)) b = vertex_px(first ? vb0 : d.vloc[v0 + kb], rot);
    if (k < nv) {
      float4 sa = make_float4(a.x, a.y, 0.f, 0.f);
      float2 sb = make_float2(a.y, 0.f);
      float slope = 0.0f;
      if (closed || k + 1 < nv) {
        const float ex = b.x - a.x, ey = b.y - a.y, ee = ex * ex + ey * ey;
        sa.z = ex;
        sa.w = ey;
        sb = make_float2(b.y, ee > 0.0f ? 1.0f / ee : 0.0f);
        slope = ey != 0.0f ? ex / ey : 0.0f;
      }
      d.segA[v0 + k] = sa;
      d.segB[v0 + k] = sb;
      d.segS[v0 + k] = slope;
    }
  }
  if (E == 4) file_chunks();
  if (E == 1 ? threadIdx.x == 0 : lane == 0) {
    float lx, ly;
    const float hx = two_prod(q.x, (float)res, lx), hy = two_prod(q.y, (float)res, ly);
    d.tpx[g] = make_float4(hx, hy, lx, ly);
  }
}

cudaError_t launch_transform(const Dev& d, cudaStream_t s, bool zero_grad, bool follows) {
  const int z = zero_grad ? 1 : 0, f = follows ? 1 : 0;
  if (d.n_elems >= kTfWideElems) return klaunch(d.pdl, k_transform<4>, (d.n_elems + 3) / 4, kTfThreads, 0, s, d, z, f);
  return klaunch(d.pdl, k_transform<1>, d.n_elems, kTfThreads, 0, s, d, z, f);
}

}  // namespace collage
