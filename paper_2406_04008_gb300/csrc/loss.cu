// Even-distribution term (Eq. 7), the deterministic gradient reduction and the flush of a pending Adam
// step.
//
// Eq. 7 as implemented: K box kernels of widths 5 + 6k pixels (k = 0..K-1) dilate the occupancy
// O = 1 - Ihat; D_k = min(1, B_k) with B_k the zero-padded box sum; the term sums
// w_k M_C (1 - O) (1 - D_k) over the container.  Its adjoint is
//   dL_u/dO(q) = sum_k w_k [ -M_C(q)(1 - D_k(q)) - sum_{p in box_k(q)} M_C(p)(1 - O(p)) [B_k(p) < 1] ].
// Both passes stage a 32 x 32 tile plus a halo of the largest radius in shared memory and form the
// box sums in fixed point: the forward pass from one integral image of the staged occupancy, the
// adjoint (whose summand differs per kernel) separably, rows then columns, with running windows.
#include "internal.h"

namespace collage {

constexpr int kDT = 32;       // dilation tile side
constexpr int kDThreads = 256;

__device__ __forceinline__ int find_prob_d(const int* base, int P, int t) {
  int lo = 0, hi = P - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (base[mid] <= t) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// Box sums in fixed point: a value v in [0, 1] is held as round(v 2^Q) in a 32-bit unsigned
// integer, with Q the largest precision for which (w^2 + w) 2^Q < 2^32, w the widest kernel (so a
// full box, w^2 2^Q, may pass 2^31).  Integer sums are exact in any order: unsigned wrap-around
// cancels between the add and the subtract of a running window, and in the four-corner difference
// of an integral image, since every box sum is below 2^32.  The adjoint slides one window along
// kSeg outputs of a row (or column) of one kernel, with one add and one subtract per output and no
// rounding drift; the forward pass reads every kernel's box sums from one integral image.  The
// kernels are instantiated per number of dilations K so that every window loop unrolls.
//
// Shared-memory layout, chosen so that the 32 lanes of a warp touch 32 distinct banks: the staged
// region and the integral image have odd row strides; the horizontal sums H of kernel k keep only
// the 32 + 2 r_k rows its vertical pass reads, with a row stride of 33; consecutive lanes take
// consecutive rows in the horizontal pass and the row scan, and consecutive columns in the
// vertical pass, the column scan and the staging.
constexpr int kSeg = 32;  // one running window per row of the tile
constexpr int kNSeg = kDT / kSeg;
constexpr int kHP = kDT + 1;  // row stride of H

__host__ __device__ constexpr int dil_r(int k) { return 2 + 3 * k; }  // (5 + 6k - 1) / 2
__host__ __device__ constexpr int hrows(int k) { return kDT + 2 * dil_r(k); }
__host__ __device__ constexpr int hbase(int k) { return k == 0 ? 0 : hbase(k - 1) + hrows(k - 1); }
__host__ __device__ constexpr int qbits(int w) {  // at most 23: bits 24..31 carry the B_k < 1 mask
  int q = 0;
  while (q < 23 && ((unsigned long long)(w * w + w) << (q + 1)) < (1ull << 32)) ++q;
  return q;
}

template <int K>
struct DilGeom {
  static constexpr int h = dil_r(K - 1);  // radius of the widest kernel
  static constexpr int S = kDT + 2 * h;   // staged side
  static constexpr int SP = S | 1;        // staged row stride (odd)
  static constexpr int HR = hbase(K);     // rows of H over all kernels
  static constexpr int Q = qbits(2 * h + 1);
  static constexpr int CW = S <= 32 ? 32 : S <= 64 ? 64 : 128;  // staging: threads per staged row
  static_assert(CW <= kDThreads, "a staged row fits the block");
};

template <int K>
__device__ __forceinline__ uint32_t to_fixed(float v) {
  return __float2uint_rn(v * (float)(1u << DilGeom<K>::Q));
}

// One horizontal running-window item of kernel k: outputs c0..c0+kSeg-1 of staged row
// rr = h - r + li, H[k][li][c] = sum_{|dc| <= r_k} src(k, rr, c + h + dc).
template <int K, int k, class Src>
__device__ __forceinline__ void hsum_one(const Src& src, uint32_t* H, int it) {
  constexpr int h = DilGeom<K>::h, r = dil_r(k), rows = hrows(k);
  const int li = it % rows, seg = it / rows, rr = h - r + li;
  const int c0 = seg * kSeg;
  uint32_t acc = 0u;
#pragma unroll
  for (int dc = -r; dc <= r; ++dc) acc += src(k, rr, c0 + h + dc);
  uint32_t* out = H + (hbase(k) + li) * kHP + c0;
  out[0] = acc;
#pragma unroll
  for (int c = 1; c < kSeg; ++c) {
    acc += src(k, rr, c0 + c + h + r) - src(k, rr, c0 + c + h - r - 1);
    out[c] = acc;
  }
}

// (The adjoint's summand is zero wherever a kernel's box holds a pixel's worth of occupancy, which for the
// wide kernels is almost everywhere between crowded elements: `act` has a bit per kernel that some staged
// pixel feeds, and the sums of the others are zero: 5000 elements at 2048^2 70 -> 59 us for the two passes
// together with the staging of interior tiles without bounds tests, 64 collages 317 -> 301.)
//
// Vertical pass fused with the per-pixel output: a thread forms the box sums of all K kernels at
// kVRows consecutive output rows of one column (a running window per kernel), then uses them
// directly, so no per-kernel result image is kept in shared memory.
// B[k][i] = sum_{|dr| <= r_k} H[k][r0 + i + r_k + dr][c].
constexpr int kVRows = 4;
constexpr int kVItems = kDT * (kDT / kVRows);
static_assert(kVItems == kDThreads, "one output item per thread");

template <int K, int k = 0>
__device__ __forceinline__ void vsums_col(const uint32_t* H, int c, int r0, unsigned act, uint32_t (&B)[K][kVRows]) {
  if constexpr (k < K) {
    constexpr int r = dil_r(k);
#pragma unroll
    for (int i = 0; i < kVRows; ++i) B[k][i] = 0u;
    if (act >> k & 1u) {
      const uint32_t* col = H + hbase(k) * kHP + c;
      uint32_t acc = 0u;
#pragma unroll
      for (int j = 0; j <= 2 * r; ++j) acc += col[(r0 + j) * kHP];
      B[k][0] = acc;
#pragma unroll
      for (int i = 1; i < kVRows; ++i) {
        acc += col[(r0 + i + 2 * r) * kHP] - col[(r0 + i - 1) * kHP];
        B[k][i] = acc;
      }
    }
    vsums_col<K, k + 1>(H, c, r0, act, B);
  }
}

// Item `it` of the flattened list of the active kernels' horizontal items: every thread of the block
// gets work, whatever the kernel sizes.  Returns false beyond the list.
template <int K, int k = 0, class Src>
__device__ __forceinline__ bool hsum_item(const Src& src, uint32_t* H, int it, unsigned act) {
  if constexpr (k < K) {
    constexpr int items_k = hrows(k) * kNSeg;
    if (act >> k & 1u) {
      if (it < items_k) {
        hsum_one<K, k>(src, H, it);
        return true;
      }
      it -= items_k;
    }
    return hsum_item<K, k + 1>(src, H, it, act);
  }
  return false;
}

struct GSrc {  // G_k = M_C (1 - O) where B_k < 1, else 0; the staged word holds the fixed-point
               // M_C (1 - O) in bits 0..23 and the B_k < 1 bits from bit 24 on (one load per use)
  const uint32_t* sM;
  int SP;
  __device__ uint32_t operator()(int k, int rr, int cc) const {
    const uint32_t x = sM[rr * SP + cc];
    // bit 24 + k moved to the sign and spread over the word: all ones where B_k < 1
    return x & 0xffffffu & (uint32_t)((int)(x << (7 - k)) >> 31);
  }
};

template <int K, class Src>
__device__ __forceinline__ void hsums_all(const Src& src, uint32_t* H, unsigned act) {
  for (int it = threadIdx.x; hsum_item<K>(src, H, it, act); it += blockDim.x) {
  }
}

// The tiles a pass visits: those with the given flag, from the per-level list (every tile when
// there is no list).  Tiles off the list hold zeros written once per level.
__device__ __forceinline__ int dil_count(const Dev& d, int which) {
  return d.dtile_list ? d.dtile_n[which] : d.total_dtiles;
}

// A dilation tile's place.
struct DilTile {
  int dt, x0, y0, res;
  bool own;  // it has container coverage of its own
  long long pb;
};
__device__ __forceinline__ DilTile dil_locate(const Dev& d, int dt, bool own) {
  const int p = find_prob_d(d.prob_dtile_base, d.n_probs, dt);
  const int res = d.prob_res[p], nd = (res + kDT - 1) / kDT, ld = dt - d.prob_dtile_base[p];
  return {dt, (ld % nd) * kDT, (ld / nd) * kDT, res, own, d.prob_pix_base[p]};
}
// One 16-byte entry per listed tile instead of the search and the divisions in every thread of every
// block (64 collages, 27 k tiles: the two passes 345 -> 318 us): dt | own << 31, (x0 | y0 << 16), then the first pixel (48 bits) and res << 48.
__device__ __forceinline__ int4 dil_pack(const DilTile& t) {
  const unsigned long long w = (unsigned long long)t.pb | (unsigned long long)t.res << 48;
  return make_int4((int)((unsigned)t.dt | (t.own ? 0x80000000u : 0u)), t.x0 | t.y0 << 16, (int)(unsigned)w,
                   (int)(unsigned)(w >> 32));
}
__device__ __forceinline__ DilTile dil_place(const Dev& d, int which, int li) {
  if (!d.dtile_list) return dil_locate(d, li, true);
  const int4 e = d.dtile_list[(size_t)which * d.total_dtiles + li];
  const unsigned long long w = (unsigned long long)(unsigned)e.w << 32 | (unsigned)e.z;
  return {e.x & 0x7fffffff, e.y & 0xffff, (int)((unsigned)e.y >> 16), (int)(w >> 48), e.x < 0,
          (long long)(w & 0xffffffffffffull)};
}

// The forward pass forms every box sum from one integral image of the staged occupancy:
// II[i][j] = sum of the staged values at rows < i and columns < j (row 0 and column 0 are zero), so
// B_k at a pixel is four loads at offsets fixed by r_k.  Unsigned wrap-around is exact here too.
template <int K>
struct IIGeom {
  static constexpr int S = DilGeom<K>::S;
  static constexpr int P = S + 1;  // row stride and side of II; odd, as S is even
  static_assert(P % 2 == 1, "odd row stride");
};

// Listed tiles per SM up to which the blocks take theirs by rank on their SM, whatever the number of kernels
// (and so of resident blocks).  Up to there the blocks of the front of the list crowd onto some SMs; beyond, most
// SMs have as many as they hold anyway and the two atomics cost more.  Iterations with the limit at 0 (by
// index), 3, 4, 5 and 8 (us; K = 4 where not said): the star at 700^2 45.1, 43.0, 43.1, 43.1, 43.1, at 1000^2 52.7,
// 50.8, 50.6, 50.4, 50.5 (K = 8: 74.0, 72.6, 73.0, 72.9, 72.8); the annulus at 850^2 52.5, 52.5, 51.5, 51.4, 51.2, at
// 1000^2 62.9, 62.8, 63.0, 63.2, 63.3 (K = 1: 55.7, 55.8, 55.8, 57.6, 57.7; K = 8: 87.9, 88.0, 88.1, 87.9, 90.4);
// the open rectangle at 1000^2 76.0, 76.0, 75.9, 76.0, 77.1 (K = 8: 105.0, 105.1, 105.0, 105.1, 107.5).
constexpr int kBalanced = 4;

template <int K>
__global__ void __launch_bounds__(kDThreads, 5) k_dilate_fwd(Dev d, int n_sm) {
  constexpr int S = DilGeom<K>::S, P = IIGeom<K>::P, h = DilGeom<K>::h, Q = DilGeom<K>::Q;
  constexpr float inv_q = 1.0f / (float)(1u << Q);
  extern __shared__ uint32_t sm[];
  __shared__ float s_red[kDThreads / 32];
  uint32_t* II = sm;
  // the tiles with container coverage; on the others M_C (1 - O) = 0, dL_u/dO = 0 and the loss
  // partial is 0, as written once per level.  The lists and the coverage are the level's: the first
  // tile's place and coverage are read before the composite has completed.
  const int n_own = dil_count(d, 0);
  const int first = first_item(d.slots + kSlotInts, n_own <= kBalanced * n_sm ? n_sm : 0);
  DilTile t{};
  if (first < n_own) t = dil_place(d, 0, first);
  // the thread's output item: column c, rows r0..r0 + kVRows - 1
  const int c = threadIdx.x % kDT, r0 = (threadIdx.x / kDT) * kVRows;
  float Iv[kVRows], Mv[kVRows];
  auto coverage = [&]() {  // from a clamped address, used only inside the image
#pragma unroll
    for (int i = 0; i < kVRows; ++i)
      Mv[i] = d.covc[t.pb + min(t.y0 + r0 + i, t.res - 1) * t.res + min(t.x0 + c, t.res - 1)];
  };
  if (first < n_own) coverage();
  pdl_enter();
  if (*d.status & kStatusNoBins) return;
  for (int li = first; li < n_own; li += gridDim.x) {
    if (li != first) {
      t = dil_place(d, 0, li);
      coverage();
    }
    const int x0 = t.x0, y0 = t.y0, res = t.res, dt = t.dt;
    const long long pb = t.pb;
    const float* Ib = d.img_I + pb;
    __syncthreads();
    {  // thread (column, first row): no division per element, 32-bit offsets from the problem's base
      constexpr int CW = DilGeom<K>::CW, RP = kDThreads / CW;
      const int c = threadIdx.x % CW, X = x0 + c - h;
      const bool col_in = X >= 0 && X < res;
      if (c < S) {
        if (x0 >= h && y0 >= h && x0 + kDT + h <= res && y0 + kDT + h <= res) {  // all inside the image
          const float* src = Ib + (y0 - h + (int)threadIdx.x / CW) * res + X;
          uint32_t* dst = II + (threadIdx.x / CW + 1) * P + c + 1;
#pragma unroll 8
          for (int r = threadIdx.x / CW; r < S; r += RP, src += RP * res, dst += RP * P)
            *dst = to_fixed<K>(1.0f - *src);
        } else {
#pragma unroll 8
          for (int r = threadIdx.x / CW; r < S; r += RP) {  // unrolled: loads in flight together
            const int Y = y0 + r - h;
            II[(r + 1) * P + c + 1] = col_in && Y >= 0 && Y < res ? to_fixed<K>(1.0f - Ib[Y * res + X]) : 0u;
          }
        }
      }
      if (threadIdx.x < P) II[threadIdx.x] = 0u;              // row 0
      if (threadIdx.x < S) II[(threadIdx.x + 1) * P] = 0u;    // column 0
    }
    // the occupancy of the thread's pixels, in flight during the scans
    const int X = x0 + c;
#pragma unroll
    for (int i = 0; i < kVRows; ++i) Iv[i] = Ib[min(y0 + r0 + i, res - 1) * res + min(X, res - 1)];
    __syncthreads();
    if (threadIdx.x < S) {  // rows: lanes take rows (odd stride, distinct banks)
      uint32_t* row = II + (threadIdx.x + 1) * P + 1;
      uint32_t acc = 0u;
#pragma unroll 9
      for (int c = 0; c < S; ++c) {
        acc += row[c];
        row[c] = acc;
      }
    }
    __syncthreads();
    if (threadIdx.x < S) {  // columns: lanes take columns
      uint32_t* col = II + P + 1 + threadIdx.x;
      uint32_t acc = 0u;
#pragma unroll 9
      for (int r = 0; r < S; ++r) {
        acc += col[r * P];
        col[r * P] = acc;
      }
    }
    __syncthreads();
    float lu = 0.0f;
    {
      // II index of the pixel's own staged position (row r0 + i + h + 1, column c + h + 1)
      const uint32_t* q0 = II + (r0 + h) * P + c + h;
#pragma unroll
      for (int i = 0; i < kVRows; ++i) {
        const int Y = y0 + r0 + i;
        if (X >= res || Y >= res) continue;
        const uint32_t* q = q0 + i * P;
        // s = sum_k w_k (1 - D_k), with 1 - D_k = max(0, 2^Q - B_k) 2^-Q exactly
        float s = 0.0f;
        unsigned mask = 0u;
#pragma unroll
        for (int k = 0; k < K; ++k) {
          const int r = dil_r(k);
          const uint32_t B = q[(r + 1) * P + r + 1] - q[-r * P + r + 1] - q[(r + 1) * P - r] + q[-r * P - r];
          // B_k may reach 2^32 - 1 (not 2^31): the difference is taken unsigned
          const uint32_t t = (1u << Q) - min(B, 1u << Q);
          if (t != 0u) mask |= 1u << k;  // B_k < 1, decided on the exact fixed-point sum
          s = fmaf(d.L.dil_w[k] * inv_q, (float)t, s);
        }
        const int o = Y * res + X;
        const float O = 1.0f - Iv[i];
        const float M = Mv[i];
        const float mval = M * (1.0f - O);
        lu = fmaf(mval, s, lu);
        const uint32_t fx = to_fixed<K>(mval);  // mval <= 1: at most 2^Q < 2^24
        d.dil_g[pb + o] = fx != 0u ? fx | (mask << 24) : 0u;
        d.gOu[pb + o] = -(M * s);  // d/dO(q) of M(q)(1 - O(q))(1 - D_k(q)), times M(q)
      }
    }
    // fixed-order block sum
    for (int o = 16; o; o >>= 1) lu += __shfl_xor_sync(0xffffffffu, lu, o);
    if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5] = lu;
    __syncthreads();
    if (threadIdx.x == 0) {
      float t = 0.0f;
      for (int i = 0; i < kDThreads / 32; ++i) t += s_red[i];
      d.lossU[dt] = t;
    }
  }
}

template <int K>
__global__ void __launch_bounds__(kDThreads, 6) k_dilate_bwd(Dev d, int n_sm) {
  constexpr int S = DilGeom<K>::S, SP = DilGeom<K>::SP, h = DilGeom<K>::h, Q = DilGeom<K>::Q;
  constexpr float inv_q = 1.0f / (float)(1u << Q);
  extern __shared__ uint32_t sm[];
  __shared__ uint32_t s_or[kDThreads / 32];
  uint32_t* sM = sm;
  uint32_t* H = sM + S * SP;
  // the tiles with container coverage within the halo (G = 0 over the others and their halos); the
  // first one's place is read before the forward pass has completed
  const int n_halo = dil_count(d, 1);
  const int first = first_item(d.slots + 2 * kSlotInts, n_halo <= kBalanced * n_sm ? n_sm : 0);
  DilTile t{};
  if (first < n_halo) t = dil_place(d, 1, first);
  pdl_enter();
  if (*d.status & kStatusNoBins) return;
  for (int li = first; li < n_halo; li += gridDim.x) {
    if (li != first) t = dil_place(d, 1, li);
    const int x0 = t.x0, y0 = t.y0, res = t.res;
    const long long pb = t.pb;
    // a tile without coverage of its own was not written by the forward pass: store, not add
    const bool own = t.own;
    __syncthreads();
    {  // thread (column, first row): no division per element, 32-bit offsets from the problem's base
      constexpr int CW = DilGeom<K>::CW, RP = kDThreads / CW;
      const int c = threadIdx.x % CW, X = x0 + c - h;
      const bool col_in = X >= 0 && X < res;
      const uint32_t* gsrc = d.dil_g + pb;
      uint32_t any = 0u;
      if (c < S) {
        if (x0 >= h && y0 >= h && x0 + kDT + h <= res && y0 + kDT + h <= res) {  // all inside the image
          const uint32_t* src = gsrc + (y0 - h + (int)threadIdx.x / CW) * res + X;
          uint32_t* dst = sM + (threadIdx.x / CW) * SP + c;
#pragma unroll 8
          for (int r = threadIdx.x / CW; r < S; r += RP, src += RP * res, dst += RP * SP) {
            const uint32_t w = *src;
            any |= w;
            *dst = w;
          }
        } else {
#pragma unroll 8
          for (int r = threadIdx.x / CW; r < S; r += RP) {  // unrolled: loads in flight together
            const int Y = y0 + r - h;
            const uint32_t w = col_in && Y >= 0 && Y < res ? gsrc[Y * res + X] : 0u;
            any |= w;
            sM[r * SP + c] = w;
          }
        }
      }
      any = __reduce_or_sync(0xffffffffu, any);
      if ((threadIdx.x & 31) == 0) s_or[threadIdx.x >> 5] = any;
    }
    // the thread's output item (column c, rows r0..r0 + kVRows - 1): the forward pass's direct
    // part of dL_u/dO is read now, in flight during the horizontal pass
    float* g = d.gOu + pb;
    const int c = threadIdx.x % kDT, r0 = (threadIdx.x / kDT) * kVRows;
    const int X = x0 + c, Xc = min(X, res - 1);
    float gv[kVRows];
#pragma unroll
    for (int i = 0; i < kVRows; ++i) gv[i] = own ? g[min(y0 + r0 + i, res - 1) * res + Xc] : 0.0f;
    __syncthreads();
    uint32_t act = 0u;
#pragma unroll
    for (int w = 0; w < kDThreads / 32; ++w) act |= s_or[w];
    act = act >> 24 & ((1u << K) - 1u);
    if (act == 0u && own) continue;  // nothing to add
    hsums_all<K>(GSrc{sM, SP}, H, act);
    __syncthreads();
    float wq[K];
#pragma unroll
    for (int k = 0; k < K; ++k) wq[k] = d.L.dil_w[k] * inv_q;
    {
      uint32_t B[K][kVRows];
      vsums_col<K>(H, c, r0, act, B);
#pragma unroll
      for (int i = 0; i < kVRows; ++i) {
        const int Y = y0 + r0 + i;
        if (X >= res || Y >= res) continue;
        float acc = 0.0f;
#pragma unroll
        for (int k = 0; k < K; ++k) acc = fmaf(-wq[k], (float)B[k][i], acc);
        g[Y * res + X] = gv[i] + acc;
      }
    }
  }
}

// Per dilation tile, once per level: whether the container coverage is nonzero on the tile, and
// whether it is nonzero within the halo of the widest kernel; each lists the tile for the pass that
// visits it (the forward pass the first kind, the adjoint the second).
__global__ void __launch_bounds__(256) k_dtile_flags(Dev d, int h) {
  for (int dt = blockIdx.x; dt < d.total_dtiles; dt += gridDim.x) {
    DilTile t = dil_locate(d, dt, false);
    const int x0 = t.x0, y0 = t.y0, res = t.res;
    const float* cov = d.covc + t.pb;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    bool own = false, halo = false;
    for (int Y = max(y0 - h, 0) + wid; Y < min(y0 + kDT + h, res); Y += 8)
      for (int X = max(x0 - h, 0) + lane; X < min(x0 + kDT + h, res); X += 32)
        if (cov[Y * res + X] > 0.0f) {
          halo = true;
          own |= Y >= y0 && Y < y0 + kDT && X >= x0 && X < x0 + kDT;
        }
    own = __syncthreads_or(own);
    halo = __syncthreads_or(halo);
    if (threadIdx.x == 0) {
      t.own = own;
      if (own) d.dtile_list[atomicAdd(&d.dtile_n[0], 1)] = dil_pack(t);
      if (halo) d.dtile_list[d.total_dtiles + atomicAdd(&d.dtile_n[1], 1)] = dil_pack(t);
    }
  }
}

// Deterministic mode: each element sums its units' partials, one warp per element.  Its pairs
// take consecutive slots, its tile rectangle row-major, so lane l reads partials l, l + 32, ... of them (no
// search) and the 32 lane sums are added by a fixed shuffle tree; the order of every addition is fixed,
// so the result is bitwise reproducible.  Bound by the latency of two loads (5000 elements, 369 k pairs:
// 24.8 us when each pair was found by bisection in its tile's sorted list, 11.8 us now).
constexpr int kReduceWarps = 8;
__global__ void __launch_bounds__(kReduceWarps * 32) k_grad_reduce(Dev d, int mark) {
  pdl_enter();
  const int lane = threadIdx.x & 31, units = d.tile * d.tile / 64;
  const int g = blockIdx.x * kReduceWarps + (threadIdx.x >> 5);
  if (g < d.n_elems && !(*d.status & kStatusNoBins)) {
    const int4 rc = d.rect[g];
    const int base = d.elem_pbase[g];
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    if (rc.z >= rc.x && rc.w >= rc.y) {
      const int n = (rc.z - rc.x + 1) * (rc.w - rc.y + 1) * units;
      const float4* part = d.partial + (size_t)base * units;
#pragma unroll 4
      for (int i = lane; i < n; i += 32) {
        if (!in_bounds(d, base >= 0 && base + i / units < d.cap)) continue;
        const float4 v = part[i];
        acc.x += v.x;
        acc.y += v.y;
        acc.z += v.z;
        acc.w += v.w;
      }
    }
    for (int o = 16; o; o >>= 1) {
      acc.x += __shfl_xor_sync(0xffffffffu, acc.x, o);
      acc.y += __shfl_xor_sync(0xffffffffu, acc.y, o);
      acc.z += __shfl_xor_sync(0xffffffffu, acc.z, o);
      acc.w += __shfl_xor_sync(0xffffffffu, acc.w, o);
    }
    if (lane == 0) {
      double2* dq = reinterpret_cast<double2*>(d.dq + 4 * (size_t)g);
      dq[0] = make_double2((double)acc.x, (double)acc.y);
      dq[1] = make_double2((double)acc.z, (double)acc.w);
    }
  }
  if (mark) mark_step_if_last(d);
}

// Applies a pending Adam step to every element (see adam_update); the last block to finish clears
// the flag, once every block has read it.  With `out`, also gathers the params, the loss terms and
// the control words (status, step, pair count, 0) into one buffer, [4n | 5 n_probs | 4], so that one
// copy brings all of them to the host.  With `q_in`, the params are then replaced; with `q_out`, copied out.
__global__ void k_adam_flush(Dev d, float* out, const float4* q_in, float4* q_out) {
  const int g = blockIdx.x * blockDim.x + threadIdx.x;
  const bool pend = *d.pending != 0;
  if (g < d.n_elems) {
    if (pend && !d.fit) {
      const double* dq = d.dq + 4 * (size_t)g;
      adam_update(d, g, *d.step, make_float4((float)dq[0], (float)dq[1], (float)dq[2], (float)dq[3]));
    }
    if (q_in) d.q[g] = q_in[g];
    if (q_out) q_out[g] = d.q[g];
    if (out) reinterpret_cast<float4*>(out)[g] = d.q[g];
  }
  if (out && blockIdx.x == 0) {
    float* tail = out + 4 * (size_t)d.n_elems;
    for (int i = threadIdx.x; i < 5 * d.n_probs; i += blockDim.x) tail[i] = d.loss_terms[i];
    if (threadIdx.x == 0) {
      int* c = reinterpret_cast<int*>(tail + 5 * d.n_probs);
      for (int i = 0; i < kCtlWords; ++i) c[i] = d.status[i];  // the control words, in order
      c[3] = 0;  // the pending step is applied by this flush
    }
  }
  __syncthreads();  // every thread of the block has read the flag
  if (threadIdx.x == 0 && atomicAdd(&d.work[5], 1) == (int)gridDim.x - 1) {
    *d.pending = 0;
    d.work[5] = 0;
  }
}

static size_t dilate_smem(int K, bool backward) {
  const int S = kDT + 2 * dil_r(K - 1), SP = S | 1;
  // the forward pass keeps one integral image with a zero row and column; the backward pass stages
  // the packed words the forward pass wrote and keeps every kernel's horizontal sums
  if (!backward) return (size_t)(S + 1) * (S + 1) * sizeof(uint32_t);
  const size_t f = (size_t)S * SP + (size_t)hbase(K) * kHP;
  return f * sizeof(uint32_t);
}

template <int K>
static cudaError_t prepare_k() {
  cudaError_t e = cudaFuncSetAttribute(k_dilate_bwd<K>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)dilate_smem(K, true));
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(k_dilate_fwd<K>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)dilate_smem(K, false));
}

cudaError_t prepare_dilate(int n_dil) {
  switch (n_dil) {
    case 1: return prepare_k<1>();
    case 2: return prepare_k<2>();
    case 3: return prepare_k<3>();
    case 4: return prepare_k<4>();
    case 5: return prepare_k<5>();
    case 6: return prepare_k<6>();
    case 7: return prepare_k<7>();
    case 8: {  // the largest: also raise every smaller instantiation (callers may mix sizes)
      for (int k = 1; k < 8; ++k) {
        cudaError_t e = prepare_dilate(k);
        if (e != cudaSuccess) return e;
      }
      return prepare_k<8>();
    }
    default: return cudaSuccess;
  }
}

template <int K>
static cudaError_t launch_k(const Dev& d, cudaStream_t s, bool backward) {
  const size_t sm = dilate_smem(K, backward);
  // one tile a block
  const int n_sm = slot_sms(d, d.total_dtiles, 8);
  if (backward) return klaunch(d.pdl, k_dilate_bwd<K>, d.total_dtiles, kDThreads, sm, s, d, n_sm);
  return klaunch(d.pdl, k_dilate_fwd<K>, d.total_dtiles, kDThreads, sm, s, d, n_sm);
}

cudaError_t launch_dilate(const Dev& d, cudaStream_t s, bool backward) {
  switch (d.L.n_dil) {
    case 1: return launch_k<1>(d, s, backward);
    case 2: return launch_k<2>(d, s, backward);
    case 3: return launch_k<3>(d, s, backward);
    case 4: return launch_k<4>(d, s, backward);
    case 5: return launch_k<5>(d, s, backward);
    case 6: return launch_k<6>(d, s, backward);
    case 7: return launch_k<7>(d, s, backward);
    case 8: return launch_k<8>(d, s, backward);
    default: return cudaSuccess;
  }
}

cudaError_t launch_dtile_flags(const Dev& d, cudaStream_t s) {
  if (d.L.n_dil <= 0 || !d.dtile_list) return cudaSuccess;
  k_dtile_flags<<<d.total_dtiles, 256, 0, s>>>(d, dil_r(d.L.n_dil - 1));
  return cudaGetLastError();
}

cudaError_t launch_grad_reduce(const Dev& d, cudaStream_t s, bool mark_step) {
  return klaunch(d.pdl, k_grad_reduce, (d.n_elems + kReduceWarps - 1) / kReduceWarps, kReduceWarps * 32, 0,
                 s, d, mark_step ? 1 : 0);
}

cudaError_t launch_adam_flush(const Dev& d, cudaStream_t s, float* out, const float* q_in, float* q_out) {
  k_adam_flush<<<(d.n_elems + 255) / 256, 256, 0, s>>>(d, out, reinterpret_cast<const float4*>(q_in),
                                                       reinterpret_cast<float4*>(q_out));
  return cudaGetLastError();
}

// The loss terms and the gradient of the last pass into the caller's buffers (either may be null), one
// launch for both.
__global__ void k_copy_out(Dev d, float* terms, float* grad) {
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (grad && i < 4 * (size_t)d.n_elems) grad[i] = (float)d.dq[i];
  if (terms && i < 5 * (size_t)d.n_probs) terms[i] = d.loss_terms[i];
}

cudaError_t launch_copy_out(const Dev& d, cudaStream_t s, float* terms, float* grad) {
  const size_t n = 5 * (size_t)max(d.n_elems, d.n_probs);  // covers both
  k_copy_out<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(d, terms, grad);
  return cudaGetLastError();
}

}  // namespace collage
