// Skeleton-based initialisation (Sec. 4.1): the medial axis of the container and its medial width
// (distance to the nearest boundary point), then the elements placed along the axis, larger ones
// where the width is larger.
//
// On the container raster of the current level (inside: coverage >= 1/2; the pixels one step beyond
// the image count as outside):
//  - D2(p): the squared distance, in pixels, from an inside pixel centre to the nearest outside pixel
//    centre (exact integers: a column pass, then per row the minimum over columns k of
//    (j - k)^2 + g(k)^2);
//  - the medial axis: the ridge of D2, the inside pixels that are a maximum of D2 along one of the
//    four lines through them (horizontal, vertical, the two diagonals): D2 >= both line neighbours
//    and > at least one (neighbours beyond the image count 0);
//  - placement, per problem: the elements in decreasing radius r = rbin s res (pixels; ties: lower
//    index first) each take the axis pixel of largest D2 (ties: lower pixel index) whose clearance
//    min_j (|p - c_j| - r_j) over the elements placed so far is >= r; if no axis pixel has that
//    clearance, the one of largest clearance.  Clearances are float32 with a fixed operation order,
//    so every decision is reproducible.  The element's translation becomes its pixel centre;
//    rotation and scale are kept.
#include <cfloat>
#include <type_traits>

#include "collage.h"
#include "edt.h"
#include "internal.h"

namespace collage {

struct OutsideSite {  // outside pixels of the container raster
  const float* covc;
  __device__ __forceinline__ bool operator()(long long pix) const { return !(covc[pix] >= 0.5f); }
};

// Row pass, one row per block: D2 = min over the columns k in [-1, res] of (j - k)^2 + g(k)^2, with
// g = 0 in the two columns beyond the image; 0 for outside pixels.
__global__ void __launch_bounds__(kEdtRowThreads) k_mat_rows(Dev d, const unsigned short* g, unsigned* d2) {
  extern __shared__ unsigned s_g2[];
  const int p = blockIdx.y, i = blockIdx.x, res = d.prob_res[p];
  if (i >= res) return;
  const long long rowb = d.prob_pix_base[p] + (long long)i * res;
  edt_stage_row(g + rowb, res, s_g2);
  __syncthreads();
  for (int j = threadIdx.x; j < res; j += kEdtRowThreads) {
    unsigned v = 0u;
    if (s_g2[j] != 0u) {  // an inside pixel (g = 0 is an outside pixel itself)
      const unsigned left = (unsigned)(j + 1) * (unsigned)(j + 1), right = (unsigned)(res - j) * (unsigned)(res - j);
      v = edt_search(s_g2, res, j, min(left, right));
    }
    d2[rowb + j] = v;
  }
}

// Medial axis test per pixel, one warp per 32 columns of a row; the axis pixels are appended to their
// problem's candidate list, packed x | y << 16, with one atomic per warp (in no particular order: the
// placement orders them by key).
constexpr int kAxisThreads = 128;
__global__ void __launch_bounds__(kAxisThreads) k_mat_axis(Dev d, const unsigned* d2, unsigned* cand, int* n_cand,
                                                           int* axis_out, float* width_out) {
  const int p = blockIdx.z, y = blockIdx.y, res = d.prob_res[p];
  const int x = blockIdx.x * kAxisThreads + threadIdx.x, lane = threadIdx.x & 31;
  if (y >= res || x - lane >= res) return;  // warp-uniform
  const long long pb = d.prob_pix_base[p];
  auto at = [&](int xx, int yy) -> unsigned {
    return xx < 0 || yy < 0 || xx >= res || yy >= res ? 0u : d2[pb + (long long)yy * res + xx];
  };
  const unsigned a = at(x, y);
  bool axis = false;
  if (a > 0) {
    const int dirs[4][2] = {{1, 0}, {0, 1}, {1, 1}, {1, -1}};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const unsigned u = at(x + dirs[k][0], y + dirs[k][1]), v = at(x - dirs[k][0], y - dirs[k][1]);
      axis |= a >= u && a >= v && (a > u || a > v);
    }
  }
  const unsigned bal = __ballot_sync(0xffffffffu, axis);
  if (bal != 0u) {
    int base = 0;
    if (lane == 0) base = atomicAdd(&n_cand[p], __popc(bal));
    base = __shfl_sync(0xffffffffu, base, 0);
    if (axis) cand[pb + base + __popc(bal & ((1u << lane) - 1u))] = (unsigned)x | (unsigned)y << 16;
  }
  if (x >= res) return;
  const long long pix = pb + (long long)y * res + x;
  if (axis_out) axis_out[pix] = axis ? 1 : 0;
  if (width_out) width_out[pix] = a > 0 ? sqrtf((float)a) : 0.0f;
}

// A float's bits as an unsigned key with the float's order (negative values included).
__device__ __forceinline__ unsigned ordered(float f) {
  const unsigned u = __float_as_uint(f);
  return u ^ ((unsigned)((int)u >> 31) | 0x80000000u);
}

// The warp's largest value (no NaN).
__device__ __forceinline__ float warp_maxf(float v) {
  float m;
  asm("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(m) : "f"(v));
  return m;
}

// The warp's largest (hi, lo) pair.
__device__ __forceinline__ void warp_max2(unsigned& hi, unsigned& lo) {
  const unsigned m = __reduce_max_sync(0xffffffffu, hi);
  lo = __reduce_max_sync(0xffffffffu, hi == m ? lo : 0u);
  hi = m;
}

// Greedy placement, one block per problem, or a cluster of eight where the axis pixels exceed one block's
// shared memory (kPlaceBlocks).  The elements' order is fixed before the first step
// (sorted by radius), and each step chooses one axis pixel (a candidate), so the steps are a serial
// chain: what bounds this kernel is the latency of one step, not the candidates' arithmetic.
//
// The candidates are sorted by cell of the raster and taken in groups of 32, each owned by one lane of
// one warp for the whole run.  A lane keeps its group's box, largest clearance, widest pixel with
// room, and the largest clearance among the wider ones without room.  A step then touches only the
// groups whose choice can have changed (12 of 500 on average for 1000 elements in the annulus at
// 1024^2):
//  - those the previous element's disk can reach: the distance from the disk's centre to the group's
//    box is below the group's largest clearance plus the disk's radius;
//  - those where a wider pixel gains room because the radius has shrunk.
// In a group the pixels are in order of their key (D2, then the lower pixel), so the widest with room
// is the first set bit of a ballot.  The warps' choices meet in one double-buffered exchange and one
// barrier a step, and every warp reduces them by itself.  1000 elements on 16 k candidates: 0.05 ms to
// sort and 0.45 us a step once the first disks are placed (eight clustered blocks that scanned every
// candidate at each step, with 64-bit shuffle reductions and a cluster barrier: 2.2 us a step).
// Sixteen warps: with 32 the barrier and the shared issue slots cost more than the fewer groups a
// warp looks at save.
constexpr int kPlaceThreads = 512;
constexpr int kPlaceWarps = kPlaceThreads / 32;
constexpr int kPlaceRankMax = 4096;        // elements sorted in shared memory (more: a reduction per step)
constexpr int kPlaceCells = 32;            // cells a side of the candidates' spatial order
constexpr int kPlaceFast = kPlaceThreads;  // groups kept one per lane, their pixels in shared memory
// Shared memory for the keys and the candidates.  (The cluster form's exchange takes 2 KB more.)
__host__ __device__ constexpr int place_smem(int blocks) { return (blocks == 1 ? 221 : 219) * 1024; }
// A problem whose candidates one block can not hold (14 to 16 k of them: the star from 1024^2 on, the disk
// and the annulus from 1100^2 on) is placed by a cluster of eight blocks, each with an eighth of the list:
// a step's choices meet in every block's shared memory behind one cluster barrier, a step of 1.0 us.  (By
// one block with the candidates in global memory a step took 3.3 us, more than the 2.2 us of a scan of every
// candidate: 1000 elements in the star at 1200^2 4.2 ms for the whole initialisation, 1.08 now.)
constexpr int kPlaceBlocks = 8;

__device__ __forceinline__ unsigned long long elem_key(const Dev& d, int e, float fres) {
  const float r = __fmul_rn(__fmul_rn(d.elem_rbin[e], d.q[e].w), fres);
  return ((unsigned long long)__float_as_uint(r) << 32) | (0xffffffffu - (unsigned)e);
}

__device__ __forceinline__ unsigned long long block_max(unsigned long long v, unsigned long long* s) {
  unsigned hi = (unsigned)(v >> 32), lo = (unsigned)v;
  warp_max2(hi, lo);
  __syncthreads();  // the previous reduction's readers are done
  if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = ((unsigned long long)hi << 32) | lo;
  __syncthreads();
  v = s[threadIdx.x % kPlaceWarps];
  hi = (unsigned)(v >> 32);
  lo = (unsigned)v;
  warp_max2(hi, lo);
  return ((unsigned long long)hi << 32) | lo;
}

// What a lane keeps of a group.  Its best pixel's key puts those with room before the others: 0xd0000000
// + D2 (below 2^28 for a side of at most 32768) with room, else the clearance's ordered bits, which are
// below 0xc8000000 for any distance on the raster (FLT_MAX, before the first disk, is held down to
// 0xcfffffff); the lower pixel wins ties (its complement is the larger).
struct PlaceGroup {
  float x0, x1, y0, y1;  // the box of its pixels
  float cl;              // the largest clearance
  float nx;              // the largest clearance among the pixels wider than the widest with room
  unsigned key, pix;     // the best pixel's key and its complement
};
constexpr unsigned kRoomKey = 0xd0000000u;

// ---- the cluster form ----
__device__ __forceinline__ unsigned cluster_rank() {
  unsigned r;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync() {  // every thread of every block, converged warps
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Into the same variable of block `rank`.
__device__ __forceinline__ void store_remote(uint2* at, unsigned rank, uint2 v) {
  unsigned a = (unsigned)__cvta_generic_to_shared(at), r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  asm volatile("st.shared::cluster.v2.u32 [%0], {%1, %2};" ::"r"(r), "r"(v.x), "r"(v.y) : "memory");
}

// FAST: the candidates in shared memory and at most one group per lane; else both in global memory.
// NB blocks place a problem together, each with its share of nc candidates, and take the same steps.
// ranked: the elements' order is in s_key; else each thread keeps the largest of every 512th element, and looks
// again when it is placed (5000 elements: 1.9 us a step; with a look at every element in each step 2.8).
template <bool FAST, int NB, bool ranked>
__device__ void place_steps(const Dev& d, int p, int nc, int ne, unsigned long long* s_key,
                            unsigned* cxy, float* ccl, const unsigned* cd2, PlaceGroup* groups, const unsigned* d2,
                            int* placed, unsigned long long* s_red, uint2 (*s_part)[NB * kPlaceWarps]) {
  const unsigned rank = NB > 1 ? cluster_rank() : 0u;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, ng = (nc + 31) / 32;
  const int res = d.prob_res[p], e0 = d.prob_elem_base[p];
  const long long pb = d.prob_pix_base[p];
  const float fres = (float)res;
  PlaceGroup own{};  // FAST: the lane's group (key 0 when it has none)
  const bool has_own = FAST && lane * kPlaceWarps + wid < ng;
  if (has_own) own = groups[lane * kPlaceWarps + wid];
  uint2 best = make_uint2(0u, 0u);  // the warp's best
  unsigned* s_key32 = reinterpret_cast<unsigned*>(s_key);  // (element, radius bits) of each step
  unsigned r_bits = ranked ? s_key32[1] : 0u;
  int px = 0, py = 0;  // the previous element's pixel and radius (none before the first step)
  float pr = -1.0f, r_last = 0.0f;
  unsigned long long ek = 0;  // not ranked: the thread's largest element not yet placed
  bool own_placed = true;
  for (int step = 0; step < ne; ++step) {
    unsigned e_inv = 0u;
    if (!ranked) {
      if (own_placed) {
        ek = 0;
        for (int i = tid; i < ne; i += kPlaceThreads) {
          if (placed[e0 + i]) continue;
          const unsigned long long k = elem_key(d, e0 + i, fres);
          ek = k > ek ? k : ek;
        }
      }
      const unsigned long long top = block_max(ek, s_red);
      r_bits = (unsigned)(top >> 32);
      e_inv = (unsigned)top;
      own_placed = top == ek;  // (the keys differ by the element)
      if (own_placed) placed[0xffffffffu - e_inv] = 1;
    }
    const float r = __uint_as_float(r_bits);
    // the groups' choices hold for radii that do not grow (the keys order the radii by their bits,
    // so a negative one precedes the positive ones)
    const bool all = (step == 0) | !(r <= r_last);
    r_last = r;
    const bool disk = pr >= 0.0f;
    const float fpx = (float)px, fpy = (float)py;
    // whether the previous disk reaches a group, or a wider pixel may have gained room (with a margin
    // for the rounding of the distances; the offsets are exact)
    auto changed = [&](const PlaceGroup& G) {
      const float dx = fmaxf(fmaxf(G.x0 - fpx, fpx - G.x1), 0.0f), dy = fmaxf(fmaxf(G.y0 - fpy, fpy - G.y1), 0.0f);
      const float t = fmaxf(G.cl + pr, 0.0f);
      const bool reach = fmaf(dx, dx, dy * dy) <= fmaf(t * t, 1.0001f, 1.0f);
      return (disk & reach) | all | !(r > G.nx);
    };
    // one group, by the whole warp: the disk into the clearances, then the group's choice, kept by the
    // lane whose group it is (`mine`); selects rather than branches, as a step is a chain of latencies
    auto look = [&](int gi, PlaceGroup& G, bool mine) {
      const int c = gi * 32 + lane;
      const bool in = FAST || c < nc;  // (in shared memory the last group is padded)
      const unsigned xy = in ? cxy[c] : 0xffffffffu;
      float v = in ? ccl[c] : -INFINITY;
      const int dx = (int)(xy & 0xffffu) - px, dy = (int)(xy >> 16) - py;
      const float dist = __fsub_rn(sqrtf(__int2float_rn(dx * dx + dy * dy)), pr);
      v = disk && dist < v ? dist : v;
      if (in) ccl[c] = v;
      const float top = warp_maxf(v);
      const unsigned fits = __ballot_sync(0xffffffffu, v >= r);
      unsigned key, pix;
      float nx = top;
      if (fits == 0u) {  // none has room: the largest clearance, the lowest pixel that has it
        pix = __reduce_max_sync(0xffffffffu, v == top ? ~xy : 0u);
        key = min(ordered(top), kRoomKey - 1u);
      } else {
        const int first = __ffs((int)fits) - 1;
        const unsigned fxy = __shfl_sync(0xffffffffu, xy, first);
        key = kRoomKey + (FAST ? cd2[gi * 32 + first] : d2[pb + (long long)(fxy >> 16) * res + (fxy & 0xffffu)]);
        pix = ~fxy;
        nx = warp_maxf(lane < first ? v : -INFINITY);  // (-inf, none wider: no radius asks for another look)
      }
      G.cl = mine ? top : G.cl;
      G.nx = mine ? nx : G.nx;
      G.key = mine ? key : G.key;
      G.pix = mine ? pix : G.pix;
    };
    if (FAST) {
      const unsigned todo0 = __ballot_sync(0xffffffffu, has_own & changed(own));
      for (unsigned todo = todo0; todo; todo &= todo - 1u) {
        const int b = __ffs((int)todo) - 1;
        look(b * kPlaceWarps + wid, own, lane == b);
      }
      if (todo0) {  // (else the warp's best stands)
        best = make_uint2(own.key, own.pix);
        warp_max2(best.x, best.y);
      }
    } else {
      best = make_uint2(0u, 0u);
      for (int g0 = wid; g0 < ng; g0 += kPlaceThreads) {
        const int gi = g0 + lane * kPlaceWarps;
        PlaceGroup G{};
        if (gi < ng) G = groups[gi];
        for (unsigned todo = __ballot_sync(0xffffffffu, gi < ng && changed(G)); todo; todo &= todo - 1u) {
          const int b = __ffs((int)todo) - 1;
          look(g0 + b * kPlaceWarps, G, lane == b);
          if (lane == b) groups[gi] = G;
        }
        if (gi < ng && (G.key > best.x || (G.key == best.x && G.pix > best.y))) best = make_uint2(G.key, G.pix);
      }
      warp_max2(best.x, best.y);
    }
    if (NB > 1) {
      if (lane < NB) store_remote(&s_part[step & 1][rank * kPlaceWarps + wid], (unsigned)lane, best);
    } else if (lane == 0) {
      s_part[step & 1][wid] = best;
    }
    if (ranked) r_bits = s_key32[2 * min(step + 1, ne - 1) + 1];  // the next step's radius
    // (the buffer is written again two steps on, after the next step's barrier)
    if (NB > 1) {
      __syncwarp();
      cluster_sync();
    } else {
      __syncthreads();
    }
    uint2 win = s_part[step & 1][lane % (NB * kPlaceWarps)];
#pragma unroll
    for (int i = 32; i < NB * kPlaceWarps; i += 32) {
      const uint2 o = s_part[step & 1][i + lane];
      if (o.x > win.x || (o.x == win.x && o.y > win.y)) win = o;
    }
    warp_max2(win.x, win.y);
    px = (int)(~win.y & 0xffffu);
    py = (int)(~win.y >> 16);
    pr = r;
    if (tid == 0) {
      if (ranked) {
        s_key32[2 * step + 1] = ~win.y;  // the pixel, beside the element
      } else if (rank == 0) {
        const int e = (int)(0xffffffffu - e_inv);
        d.q[e].x = __fdiv_rn(__fadd_rn((float)px, 0.5f), fres);
        d.q[e].y = __fdiv_rn(__fadd_rn((float)py, 0.5f), fres);
      }
    }
  }
}

// Whether the keys and nc candidates of a problem of ne elements fit one block's shared memory and lanes.
__host__ __device__ __forceinline__ bool place_fits(int nc, int ne, int smem, int* n_keys) {
  int nk = 0;  // keys, padded to a power of two
  if (ne <= kPlaceRankMax)
    for (nk = 1; nk < ne;) nk <<= 1;
  *n_keys = nk;
  const int ng = (nc + 31) / 32;
  return ng <= kPlaceFast && 8 * nk + ng * (32 * 12 + (int)sizeof(PlaceGroup)) <= smem;
}

// One problem, by the NB blocks of a cluster.
template <int NB>
__device__ void place(const Dev& d, int p, unsigned* cand, int n_cand, const unsigned* d2, unsigned* gxy, float* clear,
                      int* placed) {
  extern __shared__ __align__(16) unsigned char s_dyn[];
  __shared__ int s_cell[kPlaceCells * kPlaceCells];
  __shared__ int s_wsum[kPlaceWarps];
  __shared__ unsigned long long s_red[kPlaceWarps];
  __shared__ uint2 s_part[2][NB * kPlaceWarps];  // per step parity: each warp's best (key, pixel)
  static_assert(kPlaceCells * kPlaceCells == 2 * kPlaceThreads, "two cells per thread in the scan");
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int res = d.prob_res[p], e0 = d.prob_elem_base[p], ne = d.prob_elem_base[p + 1] - e0;
  const float fres = (float)res;
  // the block's share of the candidates, and its place in the arrays of them
  const int rank = NB > 1 ? (int)cluster_rank() : 0;
  const int c_lo = (int)((long long)n_cand * rank / NB), nc = (int)((long long)n_cand * (rank + 1) / NB) - c_lo;
  const long long pix0 = d.prob_pix_base[p], pb = pix0 + c_lo;
  int nk;
  const bool fast = place_fits((n_cand + NB - 1) / NB, ne, place_smem(NB), &nk);  // (the same in every block)
  // ---- the elements in placement order: decreasing key (radius bits, then the lower index) ----
  const bool ranked = ne <= kPlaceRankMax;
  unsigned long long* s_key = reinterpret_cast<unsigned long long*>(s_dyn);
  if (ranked) {
    for (int i = tid; i < nk; i += kPlaceThreads) s_key[i] = i < ne ? elem_key(d, e0 + i, fres) : 0ull;
    for (int k = 2; k <= nk; k <<= 1)
      for (int j = k >> 1; j > 0; j >>= 1) {
        __syncthreads();
        for (int i = tid; i < nk / 2; i += kPlaceThreads) {
          const int a = (i / j) * 2 * j + i % j, b = a + j;
          const unsigned long long x = s_key[a], y = s_key[b];
          if ((a & k) == 0 ? x < y : x > y) {
            s_key[a] = y;
            s_key[b] = x;
          }
        }
      }
  } else {
    for (int i = tid; i < ne; i += kPlaceThreads) placed[e0 + i] = 0;
  }
  // ---- the candidates by cell, and the groups ----
  const int ng = (nc + 31) / 32;
  unsigned char* s_cand = s_dyn + sizeof(unsigned long long) * nk;
  unsigned* cxy = fast ? reinterpret_cast<unsigned*>(s_cand) : gxy + pb;
  float* ccl = fast ? reinterpret_cast<float*>(s_cand) + 32 * ng : clear + pb;
  unsigned* cd2 = reinterpret_cast<unsigned*>(s_cand) + 64 * ng;  // in shared memory only
  // (the unsorted list is spent once the candidates are sorted: when they stay in global memory, which
  // takes thousands of them, its space then holds the groups, 8 words for 32 candidates)
  PlaceGroup* groups = fast ? reinterpret_cast<PlaceGroup*>(s_cand + 32 * 12 * ng)
                            : reinterpret_cast<PlaceGroup*>(cand + pb);
  int shift = 0;
  while (((res - 1) >> shift) >= kPlaceCells) ++shift;
  auto cell = [&](unsigned xy) {
    return (int)((xy >> 16) >> shift) * kPlaceCells + (int)((xy & 0xffffu) >> shift);
  };
  s_cell[2 * tid] = s_cell[2 * tid + 1] = 0;
  __syncthreads();
  for (int c = tid; c < nc; c += kPlaceThreads) atomicAdd(&s_cell[cell(cand[pb + c])], 1);
  __syncthreads();
  {  // exclusive scan of the cells' counts
    const int v0 = s_cell[2 * tid], v = v0 + s_cell[2 * tid + 1];
    int incl = v;
    for (int o = 1; o < 32; o <<= 1) {
      const int u = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += u;
    }
    if (lane == 31) s_wsum[wid] = incl;
    __syncthreads();
    int before = incl - v;
    for (int w = 0; w < wid; ++w) before += s_wsum[w];
    s_cell[2 * tid] = before;
    s_cell[2 * tid + 1] = before + v0;
  }
  __syncthreads();
  for (int c = tid; c < nc; c += kPlaceThreads) {
    const unsigned xy = cand[pb + c];
    cxy[atomicAdd(&s_cell[cell(xy)], 1)] = xy;
  }
  __syncthreads();
  for (int gi = wid; gi < ng; gi += kPlaceWarps) {
    const int c = gi * 32 + lane;
    unsigned xy = c < nc ? cxy[c] : 0xffffffffu;
    unsigned w = c < nc ? d2[pix0 + (long long)(xy >> 16) * res + (xy & 0xffffu)] : 0u;
    const unsigned x = xy & 0xffffu, y = xy >> 16;
    const unsigned x0 = __reduce_min_sync(0xffffffffu, x), x1 = __reduce_max_sync(0xffffffffu, c < nc ? x : 0u);
    const unsigned y0 = __reduce_min_sync(0xffffffffu, y), y1 = __reduce_max_sync(0xffffffffu, c < nc ? y : 0u);
    // bitonic sort of the lanes, decreasing D2, then increasing pixel (beyond the list: D2 = 0, last)
#pragma unroll
    for (int k = 2; k <= 32; k <<= 1)
#pragma unroll
      for (int j = k >> 1; j > 0; j >>= 1) {
        const unsigned wo = __shfl_xor_sync(0xffffffffu, w, j), xo = __shfl_xor_sync(0xffffffffu, xy, j);
        const bool before = w > wo || (w == wo && xy < xo);  // this lane's goes first
        const bool first = ((lane & j) == 0) == ((lane & k) == 0);
        if (first != before && (w != wo || xy != xo)) {
          w = wo;
          xy = xo;
        }
      }
    if (c < nc || fast) {  // (the padding of the last group: no pixel, never the best)
      cxy[c] = xy;
      ccl[c] = c < nc ? FLT_MAX : -INFINITY;
      if (fast) cd2[c] = w;
    }
    if (lane == 0) groups[gi] = PlaceGroup{(float)x0, (float)x1, (float)y0, (float)y1, FLT_MAX, FLT_MAX, 0u, 0u};
  }
  __syncthreads();
  if (NB > 1) cluster_sync();  // every block has started (before the first store into another's shared memory)
  auto steps = [&](auto in_smem, auto in_order) {  // (shared memory by its own addresses, not by generic ones)
    constexpr bool FAST = decltype(in_smem)::value, ORDER = decltype(in_order)::value;
    if constexpr (FAST)
      place_steps<true, NB, ORDER>(d, p, nc, ne, s_key, reinterpret_cast<unsigned*>(s_cand),
                                   reinterpret_cast<float*>(s_cand) + 32 * ng, cd2, groups, d2, placed, s_red, s_part);
    else
      place_steps<false, NB, ORDER>(d, p, nc, ne, s_key, gxy + pb, clear + pb, nullptr, groups, d2, placed, s_red, s_part);
  };
  using std::true_type;
  using std::false_type;
  if (fast && ranked) steps(true_type{}, true_type{});
  else if (fast) steps(true_type{}, false_type{});
  else if (NB > 1 && ranked) steps(false_type{}, true_type{});
  else if (NB > 1) steps(false_type{}, false_type{});
  if (!ranked || rank != 0) return;
  __syncthreads();
  for (int i = tid; i < ne; i += kPlaceThreads) {
    const unsigned xy = (unsigned)(s_key[i] >> 32);
    const int e = (int)(0xffffffffu - (unsigned)s_key[i]);
    d.q[e].x = __fdiv_rn(__fadd_rn((float)(xy & 0xffffu), 0.5f), fres);
    d.q[e].y = __fdiv_rn(__fadd_rn((float)(xy >> 16), 0.5f), fres);
  }
}

__global__ void __launch_bounds__(kPlaceThreads) k_mat_place(Dev d, unsigned* cand, const int* n_cand,
                                                             const unsigned* d2, int* placed) {
  pdl_enter();
  const int p = blockIdx.x, nc = n_cand[p];
  int nk;
  if (nc == 0 || !place_fits(nc, d.prob_elem_base[p + 1] - d.prob_elem_base[p], place_smem(1), &nk)) return;
  place<1>(d, p, cand, nc, d2, nullptr, nullptr, placed);
}
// The problems that the other kernel leaves, scheduled while that one runs.  (No inside pixel: the params
// stay.)
__global__ void __cluster_dims__(kPlaceBlocks) __launch_bounds__(kPlaceThreads)
    k_mat_place_wide(Dev d, unsigned* cand, const int* n_cand, const unsigned* d2, unsigned* gxy, float* clear,
                     int* placed) {
  pdl_enter();
  const int p = blockIdx.x / kPlaceBlocks, nc = n_cand[p];
  int nk;
  if (place_fits(nc, d.prob_elem_base[p + 1] - d.prob_elem_base[p], place_smem(1), &nk)) return;  // (the cluster's blocks agree)
  place<kPlaceBlocks>(d, p, cand, nc, d2, gxy, clear, placed);
}

cudaError_t prepare_mat_init() {
  cudaError_t e = cudaFuncSetAttribute(k_mat_place, cudaFuncAttributeMaxDynamicSharedMemorySize, place_smem(1));
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(k_mat_place_wide, cudaFuncAttributeMaxDynamicSharedMemorySize, place_smem(kPlaceBlocks));
}

cudaError_t launch_mat_init(const Dev& d, cudaStream_t s, int max_res, unsigned* g, unsigned* d2,
                            unsigned* cand, int* n_cand, float* clear, int* placed, int* axis_out,
                            float* width_out) {
  cudaError_t e = cudaMemsetAsync(n_cand, 0, sizeof(int) * d.n_probs, s);
  const size_t cs = edt_col_smem(max_res), rs = edt_row_smem(max_res);
  if (e == cudaSuccess) e = edt_smem_limit(k_edt_cols<OutsideSite>, cs, edt_col_smem(kEdtMaxRes));
  if (e == cudaSuccess) e = edt_smem_limit(k_mat_rows, rs, edt_row_smem(kEdtMaxRes));
  if (e != cudaSuccess) return e;
  unsigned short* gcol = reinterpret_cast<unsigned short*>(g);
  k_edt_cols<<<dim3((max_res + kEdtCols - 1) / kEdtCols, d.n_probs), kEdtThreads, cs, s>>>(
      d, OutsideSite{d.covc}, gcol, 1);
  k_mat_rows<<<dim3(max_res, d.n_probs), kEdtRowThreads, rs, s>>>(d, gcol, d2);
  k_mat_axis<<<dim3((max_res + kAxisThreads - 1) / kAxisThreads, max_res, d.n_probs), kAxisThreads, 0, s>>>(
      d, d2, cand, n_cand, axis_out, width_out);
  // g is free after the row pass: it holds the candidates' coordinates when they do not fit in
  // shared memory
  k_mat_place<<<d.n_probs, kPlaceThreads, place_smem(1), s>>>(d, cand, n_cand, d2, placed);
  int nk;  // (one block holds every problem's candidates, were all of its pixels on the axis)
  if ((e = cudaGetLastError()) != cudaSuccess ||
      (max_res <= 1024 && place_fits(max_res * max_res, kPlaceRankMax, place_smem(1), &nk)))
    return e;
  return klaunch(d.pdl, k_mat_place_wide, d.n_probs * kPlaceBlocks, kPlaceThreads, place_smem(kPlaceBlocks), s, d, cand,
                 n_cand, d2, g, clear, placed);
}

}  // namespace collage
