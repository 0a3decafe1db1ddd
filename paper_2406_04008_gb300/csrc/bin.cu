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
// formed in double once per element and split into float hi + lo parts; the per-vertex product uses
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

// Float pairs (hi + lo).  FP64 runs at 1/64 of the FP32 rate on this part, and one element's sine and
// cosine in double were a dependent chain of about a hundred such instructions: 2 us of the
// transform's 12 at 1000 elements, and most of its 100 at 26 k.  The pairs below carry 46
// bits (|error| <= 2^-46 over |angle| <= 8192, measured), past the 2^-24 to which a vertex is rounded.
// Sum a + b as hi + lo, exactly (Knuth); the second form needs |a| >= |b| or a = 0 (Dekker).
__device__ __forceinline__ float two_sum(float a, float b, float& lo) {
  const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
  lo = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
  return s;
}
__device__ __forceinline__ float fast_two_sum(float a, float b, float& lo) {
  const float s = __fadd_rn(a, b);
  lo = __fsub_rn(b, __fsub_rn(s, a));
  return s;
}
// Product a b as hi + lo, exactly (FMA).
__device__ __forceinline__ float two_prod(float a, float b, float& lo) {
  const float p = __fmul_rn(a, b);
  lo = __fmaf_rn(a, b, -p);
  return p;
}

// Sine and cosine of an angle |z| <= kTrigMax as unevaluated float pairs.  z = k (2 pi / 1024) + x with
// the step in three floats (Cody & Waite 1980) and the products and differences carried exactly, then
// the angle sum of the tabled sin, cos of k (2 pi / 1024) with sin x = x - x^3/6 + x^5/120 and
// cos x - 1 = -x^2/2 + x^4/24, |x| <= 0.0031, of which only the leading terms need the low part.
constexpr float kTrigMax = 8192.0f;
constexpr double kTrigStep = 6.283185307179586 / kTrigSteps;                // 2 pi / 1024
constexpr double kTrigStepLow = 2.4492935982947064e-16 / kTrigSteps;  // ... beyond a double
constexpr float kTrigC1 = (float)kTrigStep;
constexpr float kTrigC2 = (float)(kTrigStep - (double)kTrigC1);
constexpr float kTrigC3 = (float)(kTrigStep - (double)kTrigC1 - (double)kTrigC2 + kTrigStepLow);

// One of the pair: T + A x' + B y', with T, A the tabled values (hi, lo), x' = sin x (xh + xl) and
// y = cos x - 1 (yh + yl) multiplying T: sin(k + x) = S + C sin x + S (cos x - 1), and so on.
__device__ __forceinline__ float trig_sum(float th, float tl, float ah, float al, float xh, float xl, float yh,
                                          float yl, float& lo) {
  float e1, e2, f1, f2;
  const float p1 = two_prod(ah, xh, e1), p2 = two_prod(th, yh, e2);
  const float s1 = two_sum(th, p1, f1);
  const float s2 = two_sum(s1, p2, f2);
  const float rest = __fadd_rn(__fadd_rn(__fadd_rn(e1, e2), __fadd_rn(f1, f2)),
                               __fmaf_rn(ah, xl, __fmaf_rn(al, xh, __fmaf_rn(th, yl, __fmaf_rn(tl, yh, tl)))));
  return fast_two_sum(s2, rest, lo);
}

__device__ __forceinline__ void sincos_ff(float z, const float4* table, float (&s)[2], float (&c)[2]) {
  const float k = rintf(__fmul_rn(z, 1.0f / kTrigC1));
  const float4 t = table[(int)k & (kTrigSteps - 1)];  // sin hi, lo, cos hi, lo
  float e, q, b, dd;
  const float p = two_prod(k, kTrigC1, e);
  const float u = two_prod(k, kTrigC2, q);
  const float a1 = two_sum(__fsub_rn(z, p), -e, b);  // z - p is exact: p is within a factor 2 of z
  const float a2 = two_sum(a1, -u, dd);
  float xl;
  const float xh = fast_two_sum(a2, __fsub_rn(__fadd_rn(b, dd), __fmaf_rn(k, kTrigC3, q)), xl);
  float y2l;
  const float y2 = two_prod(xh, xh, y2l);
  y2l = __fmaf_rn(2.0f * xh, xl, y2l);
  // sin x beyond its leading term x, cos x - 1 beyond -x^2/2
  const float sl = __fmaf_rn(__fmul_rn(xh, y2), __fmaf_rn(y2, 1.0f / 120.0f, -1.0f / 6.0f), xl);
  const float yl = __fmaf_rn(__fmul_rn(y2, y2), 1.0f / 24.0f, -0.5f * y2l);
  s[0] = trig_sum(t.x, t.y, t.z, t.w, xh, sl, -0.5f * y2, yl, s[1]);
  c[0] = trig_sum(t.z, t.w, -t.x, -t.y, xh, sl, -0.5f * y2, yl, c[1]);
}

__device__ __noinline__ void sincos_wide(float z, float (&s)[2], float (&c)[2]) {  // any other angle
  double sn, cs;
  sincos((double)z, &sn, &cs);
  s[0] = (float)sn;
  s[1] = (float)(sn - (double)s[0]);
  c[0] = (float)cs;
  c[1] = (float)(cs - (double)c[0]);
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
      const float gr = reinterpret_cast<const float*>(d.dq + ge)[k];
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
      float s[2], c[2];
      if (fabsf(z) <= kTrigMax) sincos_ff(z, d.trig, s, c);
      else sincos_wide(z, s, c);
      // entry k of s res [cos, -sin; sin, cos]
      float th = k == 0 || k == 3 ? c[0] : s[0], tl = k == 0 || k == 3 ? c[1] : s[1];
      if (k == 1) {
        th = -th;
        tl = -tl;
      }
      float hl, pl, lo;
      const float hh = two_prod(sc, (float)re, hl), pp = two_prod(hh, th, pl);
      s_rot[e].m[k][0] = fast_two_sum(pp, __fadd_rn(pl, __fmaf_rn(hh, tl, __fmul_rn(hl, th))), lo);
      s_rot[e].m[k][1] = lo;
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
      if (zero_grad) d.dq[g] = make_float4(0.f, 0.f, 0.f, 0.f);
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

void trig_table(float4* t) {
  for (int k = 0; k < kTrigSteps; ++k) {
    const double a = k * (6.283185307179586 / kTrigSteps), s = sin(a), c = cos(a);
    t[k] = make_float4((float)s, (float)(s - (double)(float)s), (float)c, (float)(c - (double)(float)c));
  }
}

cudaError_t launch_transform(const Dev& d, cudaStream_t s, bool zero_grad, bool follows) {
  const int z = zero_grad ? 1 : 0, f = follows ? 1 : 0;
  if (d.n_elems >= kTfWideElems) return klaunch(d.pdl, k_transform<4>, (d.n_elems + 3) / 4, kTfThreads, 0, s, d, z, f);
  return klaunch(d.pdl, k_transform<1>, d.n_elems, kTfThreads, 0, s, d, z, f);
}

}  // namespace collage
