// Internal device-side layout of libcollage (not part of the C ABI).
//
// HBM layout, all problems of a handle concatenated:
//   per element g (SoA):   prob, vertex offset, closed flag, stroke half-width, bin radius,
//                          params q / Adam m, v (float4), world translation in pixels (hi, lo),
//                          tile rectangle, first pair slot, gradient dq
//   per flattened vertex:  local position (unit coords), per-iteration segment record relative to
//                          the element translation in pixels (float, within an ulp of the exact value)
//   per (tile, element) pair, capacity `cap`: per pixel of the tile the signed distance + closest
//                          segment saved by the forward pass, per 64 pixels a deterministic gradient
//                          partial; the work lists of the emission and the adjoint
//   per pixel (level):     container coverage, Ihat, prod(1 - tau c^pad), uniform-loss scratch
//   per tile:              its list of pairs (slot, class, element) and its length; per 64 pixels of
//                          it the loss partials
#pragma once
#include <cstdint>
#include <cstdio>
#include <cuda_runtime.h>

namespace collage {

constexpr int kMaxDil = 8;
constexpr int kTrigSteps = 4096;        // steps to a turn of the transform's table of sines
constexpr int kLossUnits = 2048;        // 64-px units of an image per part of its loss,
constexpr int kLossParts = 16;          //   in at most this many parts
constexpr int kCtlWords = 24;           // device control words (status first, see Dev)
constexpr int kChunkPx = 64;            // side, in pixels, of the emission's chunks of an element
constexpr int kHeavyChunk = 1024;       // segments x tiles above which a chunk is taken first
constexpr int kStatusOverflow = 1;      // device status bits
constexpr int kStatusBadParam = 2;
constexpr int kStatusInternal = 4;      // an internal bounds check failed (a bug)
constexpr int kStatusTileCap = 8;       // a tile's pair list outgrew its capacity (regrown, re-run)
constexpr int kStatusNoBins = kStatusOverflow | kStatusTileCap;  // the bins of the iteration are void
constexpr int kStatusVoid = kStatusNoBins | kStatusBadParam;      // the iteration is void

// Class of a (tile, element) pair.  A pair is near when some segment of the outline lies within
// the coverage margin (rho + pad + stroke half-width) of some pixel centre of the tile; otherwise
// the coverage and the padded coverage are the same saturated value (0 or 1) on every pixel of
// the tile and the pair carries no gradient.
constexpr unsigned kPairOut = 0;   // not near, outside the outline: c = c^pad = 0
constexpr unsigned kPairIn = 1;    // not near, inside: c = c^pad = 1
constexpr unsigned kPairNear = 2;  // per-pixel signed distances (the distance kernel)
constexpr int kSlotBits = 30;      // a tile list's entry: slot | class << kSlotBits, element
constexpr unsigned kSlotMask = (1u << kSlotBits) - 1u;

// What a composite launch leaves.
constexpr int kCompLoss = 1;  // loss partials, and the images where the adjoint reads them
constexpr int kCompAllI = 2;  // img_I of every pixel (the distribution term or the metrics follow)

struct LossParams {
  float alpha, beta, gamma, delta;
  int force_kind;               // 0: downward potential 1 - y; 1: |p - (fx, fy)|
  float fx, fy;
  float tau, w_in, w_out;
  int n_dil;
  float dil_w[kMaxDil];
  float pad_px, rho_px;
};

struct Dev {
  // ---- problem (fixed at create) ----
  int n_elems, n_probs;
  int max_segs;                 // the most segments of any element
  const int* elem_prob;
  const int* elem_voff;         // [n+1]
  const uint8_t* elem_closed;
  const float* elem_hw;         // unit coords
  float* elem_rbin;             // bin radius (largest |control point|), float
  float2* vloc;                 // flattened local vertices, unit coords (rewritten by
                                //   k_ctrl_step when the outlines are fitted)
  const int* prob_elem_base;    // [P+1]
  const double* ring_pts;       // container rings, unit coords (double)
  const float2* ring_f;         //   and as given
  const int* ring_off;          // [total rings + 1]
  const int* prob_ring_base;    // [P+1] into ring_off
  // ---- level ----
  const int* prob_res;          // [P]
  const int* prob_ntx;          // [P] tiles per side
  const int* prob_tile_base;    // [P+1]
  const long long* prob_pix_base;  // [P+1]
  const int* prob_dtile_base;   // [P+1] dilation tiles
  int total_tiles, total_dtiles;
  int max_tiles;                // tiles of the largest problem
  long long total_pix;
  int tile;                     // raster tile side
  int emit_threads;             // threads per block of the emission / distance kernel (128, 256)
  int chunk_tiles;              // side of the emission's chunks, in tiles (<= kChunkPx / tile)
  // ---- params / optimiser ----
  float4* q;
  float4* m;
  float4* v;
  const float4* q_in;           // [n] params the transform takes in place of q (the host-buffer
                                //   step's mapped input), or null
  const uchar4* trainable;      // may be null
  const float4* trig;           // [kTrigSteps / 4 + 1] sines of k (2 pi / kTrigSteps), in three floats each
  float lr, b1, b2, eps, s_min, s_max;
  // ---- per iteration ----
  float4* segA;                 // [V] segment k: start (px, relative to the translation), direction
  float2* segB;                 // [V] segment k: end point y, 1 / |direction|^2
  float* segS;                  // [V] segment k: dx/dy of its direction (0 if horizontal)
  float4* tpx;                  // [n] translation in px: (hi.x, hi.y, lo.x, lo.y)
  int4* rect;                   // [n] tile rectangle (tx0, ty0, tx1, ty1), empty if tx1 < tx0
  int* elem_pbase;              // [n] first pair slot of each element: its tile rectangle's pairs
                                //   take consecutive slots, row-major (the transform allocates them)
  int* pair_need;               // [1] pair slots allocated by this iteration's transform
  int* total_pairs;             // [1] pairs of the last binning (copied from pair_need)
  int cap;                      // pair capacity
  int* tile_n;                  // [total_tiles] pairs registered in each tile's list by the
                                //   emission (the composite zeroes it)
  int* tile_m;                  // [total_tiles] pairs of each tile (the composite's count, kept)
  uint2* tile_list;             // [total_tiles * tile_cap] each tile's pairs in emission order: (slot |
                                //   class << kSlotBits, element)
  unsigned* tile_sorted;        // [total_tiles * tile_cap] scratch of the composite: the first words of
                                //   a very long list's covering pairs, in element order
  int tile_cap;                 // pair-list capacity of a tile
  int* tile_max;                // [1] pairs of the fullest tile list of the iteration where one passed 3/4
                                //   of the capacity, else 0 (the emission's block 0 zeroes it)
  int4* near_list;              // [list_cap] the emission's work list: (element, chunk origin tile
                                //   column | row << 16, problem, 0), one per kChunkPx-square chunk of
                                //   every element's tile rectangle, appended by the transform: heavy
                                //   ones from the front, light ones from the back
  int list_cap;                 // entries near_list holds
  int* chunk_count;             // [2] heavy and light chunks appended by the transform (the
                                //   composite's block 0 zeroes them)
  int4* live_list;              // [cap * units per tile] units with some non-saturated pixel: (slot | unit <<
                                //   kSlotBits, element, tile column | row << 16, problem), the adjoint's
                                //   work list (order depends on atomics)
  float2* saved;                // [cap * tile*tile] (sd px, closest segment as int bits)
  float* covc;                  // [pix] container coverage
  float* img_I;                 // [pix] Ihat = prod(1 - c)
  float* img_Pt;                // [pix] +-prod(1 - tau c^pad), negative where A_tau > tau
  float* gOu;                   // [pix] dL_u/dO
  uint32_t* dil_g;              // [pix] the adjoint's staged word: round(M_C (1 - O) 2^Q) in bits
                                // 0..23, bit 24 + k set where B_k < 1 (Q of the kernel count)
  float4* lossA;                // per unit of 64 pixels of a tile (one of 8 x 8, four of 16 x 16), tile by
                                //   tile: (sum W(I-Ic)^2, sum relu(A-tau), sum O(1-y), 0)
  float* loss0;                 // per unit: the first of these where nothing covers it (level constant)
  float* lossU;                 // [total_dtiles] weighted uniform-loss partial
  int4* dtile_list;             // [2 total_dtiles] the places of the dilation tiles with container coverage
                                //   from 0, with coverage within the halo from total_dtiles, in no
                                //   particular order (or null: all tiles)
  int* dtile_n;                 // [2] lengths of the two lists
  double* dq;                   // [4n] gradient, summed in FP64: the adjoint's units add to it in whatever order
                                //   they end, which FP32 sums showed in their last bits
  float4* partial;              // [cap * units per tile] deterministic gradient partials, by slot
  float* loss_terms;            // [P*5]
  float2* loss_part;            // [P * kLossParts * 4] the four sums over each part of a problem's loss partials, (hi, lo)
  int* loss_done;               // [P] parts summed so far (the last one zeroes it)
  int* status;                  // [1]
  int* step;                    // [1] Adam step count (the last gradient kernel advances it)
  int* pending;                 // [1] 1: the Adam step `step` is computed (dq) but not yet applied
  int* sched_base;              // [1] Adam step count when the running schedule graph began
  int* work;                    // [8] per-iteration counters: [0] chunks taken by the emission's
                                //   blocks beyond the first (the composite's block 0 zeroes it), [1] entries of live_list and
                                //   [3] blocks of the last gradient kernel that have finished
                                //   (zeroed by the transform), [5] blocks of the Adam flush that
                                //   have finished (its last block zeroes it), [2, 4, 6, 7] spare
  int* slots;                   // [3 * kSlotInts] block counts of balanced_slot: the emission's (zeroed by the
                                //   composite), the distribution term's forward and adjoint ones (by the transform)
  unsigned long long* paths;    // [4] cumulative counts of the rarely taken kernel paths (since
                                //   create): [0] pixel rows of a near pair whose crossings
                                //   overflow the per-row list (winding over every segment),
                                //   [1] emission chunks of outlines with more segments than
                                //   are staged in shared memory,
                                //   [2] tiles listing more than 32 pairs (ranked in shared
                                //   or global memory), [3] container ring chunks after a ring's first
  LossParams L;
  int deterministic;
  int sms;                      // SMs of the device
  int few_chunks;               // 1: the level has at most eight chunks per SM, all taken in one wave of blocks
  int pdl;                      // launch the iteration's kernels with programmatic serialisation
  // ---- outline fitting (fit_controls): the points of each element are the parameters ----
  int fit;                      // 1: the adjoint accumulates dv and k_ctrl_step runs Adam on ctrl
  int spc;                      // segments per cubic
  const int* elem_coff;         // [n+1] CSR offsets of each element's points in ctrl
  const uint8_t* elem_cubic;    // [n] 1: closed cubic path (points are control points)
  float2* ctrl;                 // [C] points, element-local unit coordinates
  float2* ctrl_m;               // [C] Adam moments
  float2* ctrl_v;
  float2* dctrl;                // [C] dL/d(points) of the last backward pass
  float2* dv;                   // [V] dL/d(flattened vertex), element-local unit coordinates
};

// ---- the checked build (-DCOLLAGE_CHECKED, libcollage_checked.so) ----
// in_bounds(d, ok): a failed index check latches kStatusInternal (the next host call that reads
// the status word returns COLLAGE_ERR_STATE) and the caller skips the guarded access, so nothing
// is read or written past a bound and nothing traps; the checked build also prints the first
// failures' source lines.  In the regular build it is the constant true and compiles away.
#ifdef COLLAGE_CHECKED
static __device__ int g_bounds_reports = 0;
__device__ __forceinline__ bool in_bounds_at(const Dev& d, bool ok, int line, const char* file) {
  if (!ok) {
    atomicOr(d.status, kStatusInternal);
    if (atomicAdd(&g_bounds_reports, 1) < 8) printf("collage: bounds check failed at %s:%d\n", file, line);
  }
  return ok;
}
#define in_bounds(d, ok) in_bounds_at((d), (ok), __LINE__, __FILE__)
#else
__device__ __forceinline__ bool in_bounds(const Dev& d, bool ok) {
  (void)d;
  (void)ok;
  return true;
}
#endif

// Adam (bias-corrected, the update torch.optim.Adam performs; it stands in for the plain descent
// step of Eq. 4) of element g at step t >= 1 with gradient gr, then the clamp of s.
// An iteration's step is applied lazily: the last block of the kernel that completes the gradient marks
// it pending (mark_step_if_last), and the next iteration's transform kernel (which reads the params
// first anyway) applies it before forming the geometry; API calls that read or replace params flush it.
struct AdamScale {
  float step, root2;  // lr / (1 - b1^t), sqrt(1 - b2^t)
};
__device__ __forceinline__ AdamScale adam_scale(const Dev& d, float b1_t, float b2_t) {
  return {d.lr / (1.0f - b1_t), sqrtf(1.0f - b2_t)};
}
__device__ __forceinline__ void adam_entry(const Dev& d, AdamScale a, float g, float& q, float& m, float& v) {
  m = d.b1 * m + (1.0f - d.b1) * g;
  v = d.b2 * v + (1.0f - d.b2) * g * g;
  const float denom = sqrtf(v) / a.root2 + d.eps;
  q -= a.step * m / denom;
}
__device__ __forceinline__ void adam_update(const Dev& d, int g, int t, float4 gr) {
  float4 q = d.q[g], m = d.m[g], v = d.v[g];
  const uchar4 tr = d.trainable ? d.trainable[g] : make_uchar4(1, 1, 1, 1);
  const AdamScale a = adam_scale(d, powf(d.b1, (float)t), powf(d.b2, (float)t));
  if (tr.x) adam_entry(d, a, gr.x, q.x, m.x, v.x);
  if (tr.y) adam_entry(d, a, gr.y, q.y, m.y, v.y);
  if (tr.z) adam_entry(d, a, gr.z, q.z, m.z, v.z);
  if (tr.w) adam_entry(d, a, gr.w, q.w, m.w, v.w);
  q.w = fminf(fmaxf(q.w, d.s_min), d.s_max);
  d.q[g] = q;
  d.m[g] = m;
  d.v[g] = v;
}

// Potential of the force term at the pixel centre (px, py), unit coordinates.
__device__ __forceinline__ float force_potential(const LossParams& L, float px, float py) {
  if (L.force_kind == 1) return hypotf(px - L.fx, py - L.fy);
  return 1.0f - py;
}

// ---- programmatic dependent launch ----
// With Dev::pdl set, the kernels of an iteration are launched with programmatic stream
// serialisation: a kernel may be scheduled while its predecessor on the stream still runs.  Every
// thread of such a kernel calls pdl_enter() before it ends: griddepcontrol.wait returns once the
// predecessor grid has completed and its memory operations are visible, then launch_dependents lets
// the successor be scheduled (the wait comes first in every thread, so completion is transitive along
// the chain: when a kernel starts, all but its predecessor have completed).  Launched without the
// attribute, both instructions are no-ops.
//
// What a kernel K_n may touch before its own wait:
//  1. memory that no kernel of an iteration writes: the problem, the level's tables, the container
//     raster and the dilation tiles' lists.  They change only in work that the host separates from
//     iterations (create, a level switch, replaced outlines), and a launch that may follow such work
//     directly does not read them early (`follows` of the transform);
//  2. what K_{n-2} or an earlier kernel wrote and K_{n-1} does not write, by accesses that L2 serves:
//     atomics (the counts of balanced_slot) or __ldcg loads (the adjoint).  Those kernels have completed
//     and their writes lie in L2, but only the wait is documented to make a grid's writes visible to
//     ordinary loads, which may hit a line that this SM's L1 kept from an earlier iteration;
//  3. nothing else: no store before the wait except to what only K_n itself writes and reads in this
//     iteration (the loss terms and their parts).
__device__ __forceinline__ void pdl_enter() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// ---- which block takes which work item ----
// Blocks that are launched while the predecessor drains go to whichever SM has room: one SM takes eight
// consecutive blocks of the emission and another none (1000 elements at 1024^2: the 602 long outlines, first
// in the list, lay on 86 of 152 SMs), and an SM that is free early takes up to 18 of the distribution term's
// one-tile blocks, a mean of 6.7.  Where the items are few for the SMs (the callers' limits), each block takes
// its item by its rank among the blocks on its own SM instead: the r-th block of an SM takes the next of items
// [r n_sm, (r + 1) n_sm), so that each SM gets an even share of the front of the list, and the grid's idle
// rest lies on the SMs with the most blocks (resident at once or not: a later block ranks behind).  A block whose range is spent takes the last free item; as there
// are as many items as blocks, each item is taken exactly once whatever the placement.  Runs before the wait
// on the predecessor (`c` has been zero since the predecessor's predecessor or earlier), so that its two
// atomics are hidden; one thread of each block calls it once.  Per iteration: 1000 elements at 1024^2 86.9 ->
// 81.1 us, at 128^2 to 512^2 64.7, 65.6, 70.8 -> 62.6, 61.6, 64.7; 100 outlines at 1000^2 66.0 -> 62.1; 120
// elements at 200^2 48.6 -> 46.4.  (Dealing the items over the block indices by a multiplier left up to
// eight long outlines on some SMs and none on others: half the gain.)
constexpr int kSlotSms = 256, kSlotRanks = 32, kSlotInts = kSlotSms + kSlotRanks;
__device__ __forceinline__ int balanced_slot(int* c, int n_sm) {
  const int G = (int)gridDim.x, n = (G + n_sm - 1) / n_sm;
  unsigned sm;
  asm volatile("mov.u32 %0, %%smid;" : "=r"(sm));
  auto take = [&](int r) {
    const int i = r * n_sm + atomicAdd(&c[kSlotSms + r], 1);
    return i < min((r + 1) * n_sm, G) ? i : -1;
  };
  const int rank = atomicAdd(&c[sm % kSlotSms], 1);
  int i = rank < n ? take(rank) : -1;
  for (int r = n - 1; i < 0 && r >= 0; --r) i = take(r);
  return i < 0 ? G : i;
}
// The block's item: by balanced_slot, or by its index where n_sm is 0 (the same in every thread).
__device__ __forceinline__ int first_item(int* c, int n_sm) {
  __shared__ int s_first;
  if (n_sm == 0) return (int)blockIdx.x;
  if (threadIdx.x == 0) s_first = balanced_slot(c, n_sm);
  __syncthreads();
  return s_first;
}
// The n_sm of a grid of `grid` blocks: 0 beyond per_sm per SM (at most kSlotRanks).
inline int slot_sms(const Dev& d, long long grid, int per_sm) {
  return grid <= (long long)d.sms * per_sm ? d.sms : 0;
}

template <typename... KArgs, typename... Args>
inline cudaError_t klaunch(bool pdl, void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem,
                           cudaStream_t s, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

// The last block of the kernel that completes an iteration's gradient marks the iteration's Adam
// step pending (applied by the next transform) and advances the step count, unless the iteration
// overflowed or met non-finite params.  Every block calls this once, after its last write to the
// gradient; the counter work[3] is zeroed by the transform of each iteration.
__device__ __forceinline__ void mark_step_if_last(const Dev& d) {
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();  // this block's gradient writes are visible before it is counted
    if (atomicAdd(&d.work[3], 1) == (int)gridDim.x - 1 && !(atomicAdd(d.status, 0) & kStatusVoid)) {
      __threadfence();
      *d.step += 1;
      *d.pending = 1;
    }
  }
}

// ---- launchers (each enqueues on `s`, returns the launch error) ----
// follows: the previous launch on `s` is another iteration's, so the outlines were written long before
// and are read while it ends (never the first launch after a call that may replace them)
cudaError_t launch_transform(const Dev& d, cudaStream_t s, bool zero_grad, bool follows);
cudaError_t launch_container(const Dev& d, cudaStream_t s);
// part 1: pair emission, classification and per-pixel signed distances (per element chunk);
// part 2: per-tile composite and loss partials (flags: kComp*)
cudaError_t launch_raster_fwd(const Dev& d, cudaStream_t s, int pair_grid, int tile_grid,
                              float* out_bw, float* out_tau, int part, int flags = 0);
cudaError_t prepare_dilate(int n_dil);  // sets dynamic shared memory limits (not capturable)
cudaError_t launch_dilate(const Dev& d, cudaStream_t s, bool backward);
cudaError_t launch_dtile_flags(const Dev& d, cudaStream_t s);  // once per level, after the container
// the adjoint and the loss assembly; resident: unit_grid is a persistent one, not a block per unit; mark_step:
// the kernel's last block marks the iteration's Adam step (step mode)
cudaError_t launch_raster_bwd(const Dev& d, cudaStream_t s, int unit_grid, bool resident, bool mark_step);
cudaError_t launch_grad_reduce(const Dev& d, cudaStream_t s, bool mark_step);
// applies a pending Adam step to all elements and clears the flag (before params are read); then, where
// given, replaces the params by q_in, copies them to q_out (both 16-byte aligned, [4n]) and gathers them
// with the loss terms and the control words into out
cudaError_t launch_adam_flush(const Dev& d, cudaStream_t s, float* out = nullptr, const float* q_in = nullptr,
                              float* q_out = nullptr);
// outline fitting, one block per element: mode 0 maps dv to dctrl (and clears dv); mode 1 also
// takes an Adam step on ctrl at step *d.step and flattens again (vertices and bin radii); mode 2
// only flattens
cudaError_t launch_ctrl_step(const Dev& d, cudaStream_t s, int mode);
// skeleton-based initialisation: distance transform, medial axis, greedy placement into d.q (after
// prepare_mat_init, once per handle: the placement's shared-memory limits)
cudaError_t prepare_mat_init();
cudaError_t launch_mat_init(const Dev& d, cudaStream_t s, int max_res, unsigned* g, unsigned* d2,
                            unsigned* cand, int* n_cand, float* clear, int* placed, int* axis_out,
                            float* width_out);
// the captured level schedule: records the step count at the start of a run; sets a level's loop
// condition (1 while fewer than `target` iterations of the run are done and nothing latched)
cudaError_t launch_sched_begin(const Dev& d, cudaStream_t s);
cudaError_t launch_sched_cond(const Dev& d, cudaStream_t s, cudaGraphConditionalHandle cond, int target);
cudaError_t launch_copy_out(const Dev& d, cudaStream_t s, float* terms, float* grad);
// Resident blocks per SM of the raster kernels, the pairs one adjoint block and the tiles one
// composite block take at once (the forward distance kernel takes one pair per block).
struct RasterOcc {
  int fwd_per_sm, bwd_per_sm, tile_per_sm, bwd_pairs_per_block, tiles_per_block;
};
void raster_occupancy(int tile, int emit_threads, RasterOcc* o);
// quality metrics after a render pass: counts [4 * n_probs] and squared-distance sums [n_probs]
cudaError_t launch_metrics(const Dev& d, cudaStream_t s, uint8_t* obj, unsigned short* gcol,
                           unsigned long long* cnt, unsigned long long* sums, int max_res);

}  // namespace collage
