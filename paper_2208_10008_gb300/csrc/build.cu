// BVH construction on the device (Sec. II.B-C of arXiv 2208.10008).
//
// Pipeline, all asynchronous on one stream.  Every kernel after the first is
// launched with programmatic dependent launch and waits for its predecessor
// (griddepcontrol.wait) before it reads anything that kernel wrote, so the
// launches overlap their set-up with the previous kernel's tail.
//   memset        control block
//   k_prep        Eq. 3 box of every triangle -> build record; scene and
//                 centroid bounds
//   k_bin_root    30-bit Morton key of every box centre (kept in the record
//                 for the small subtrees); the root task; the root's bins
//   k_split       one persistent launch for the whole recursion of Fig. 2.
//                 Its first CTAs take the chunk items of big nodes (more than
//                 `big` triangles, cut into chunks of 256..2048 records, CTA
//                 per chunk): Eq. 2 at every bin plane from the node's merged
//                 bins, stable partition of the chunk into the other record
//                 buffer, and on the way the children's bins and per-chunk
//                 counts; the CTA finishing a node's last chunk writes the node
//                 and publishes its children's items.  Every CTA takes the
//                 subtrees (nodes of at most `big` triangles) from a second
//                 device queue, CTA per subtree, and builds each in shared
//                 memory: nodes of more than 32 triangles split by the whole
//                 CTA (the smaller child goes back to the queue), nodes of at
//                 most 32 finished by single warps in registers over the
//                 Morton order of their records.  No CTA waits for another
//                 except for work to appear (bounded waits).
//   k_small       (large scenes) the subtrees of the nodes of at most 64 or 128
//                 records that k_split then leaves, a warp each
//   k_post        4-wide traversal nodes (greedy by surface area), stored at the
//                 id of their binary root; triangles in leaf order
//
// Bins.  A bin holds 13 words: the record count, the union of the records'
// boxes and the bounds of their box centres, the floats as order-preserving
// unsigned codes (min slots store the complement) so that every merge is an
// atomicAdd or atomicMax and all-zero is the empty bin.  A node's bins give the
// exact boxes and centroid bounds of both children of any plane, so a child is
// binned while its parent is partitioned.
//
// Node identity: the binary node that splits its range at position s gets id
// s - 1.  Split positions of distinct internal nodes differ, so ids need no
// allocator and the tree is the same whatever order the work ran in.
#include <cuda_runtime.h>

#include <algorithm>
#include <cfloat>
#include <climits>
#include <type_traits>

#include "rt_internal.cuh"

namespace rt {
namespace {

constexpr int kBlock = 256;  // threads of every build CTA
constexpr int kWarps = kBlock / 32;
constexpr int kBinVals = 13;  // count, box lo xyz, box hi xyz, centre lo xyz, centre hi xyz
constexpr int kBinWords = 3 * kMaxBins * kBinVals;
constexpr int kCntStride = 3 * kMaxBins;
constexpr int kMaxRpt = 8;     // records per thread of a big node's chunk
constexpr int kRegRpt = 4;     // at most, where they stay in registers
constexpr int kStage = kBlock * kMaxRpt;  // records of a chunk in shared memory: all of them
constexpr int kLargeScene = 240000;  // records from which a build is bound by work and not by its longest chain
constexpr int kBigMin = 1024;  // big nodes have more triangles than this
constexpr unsigned kFull = 0xffffffffu;

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

__device__ __forceinline__ void set_status(BuildCtl* ctl, int code, int where) {
  if (atomicCAS(&ctl->status, 0, code) == 0) ctl->status_where = where;
}

__device__ __forceinline__ int ld_volatile(const int* p) { return *(const volatile int*)p; }

// Acquire load / release store / release add at GPU scope: the flag and
// counter protocol of the work queues without full memory fences.
__device__ __forceinline__ int ld_acquire(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release(int* p, int v) {
  asm volatile("st.release.gpu.b32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ int atom_add_acq_rel(int* p, int v) {
  int old;
  asm volatile("atom.acq_rel.gpu.add.s32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(v) : "memory");
  return old;
}
__device__ __forceinline__ void red_release_add(int* p, int v) {
  asm volatile("red.release.gpu.add.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// AABB centre, evaluated identically wherever a bin is needed.
__device__ __forceinline__ float centre(float lo, float hi) { return __fmul_rn(__fadd_rn(lo, hi), 0.5f); }

// Bin index of centroid coordinate c for slab [cmin, cmin + K/scale).
__device__ __forceinline__ int bin_of(float c, float cmin, float scale, int K) {
  int b = (int)__fmul_rn(__fsub_rn(c, cmin), scale);
  return min(max(b, 0), K - 1);
}

__device__ __forceinline__ float bin_scale(float cmin, float cmax, int K) {
  float ext = cmax - cmin;
  return ext > 0.f ? (float)K * (1.f - 1e-6f) / ext : 0.f;
}

__device__ __forceinline__ float area(float3 lo, float3 hi) {
  float dx = hi.x - lo.x, dy = hi.y - lo.y, dz = hi.z - lo.z;
  return 2.f * (dx * dy + dy * dz + dz * dx);
}

__device__ __forceinline__ float sel3(float x, float y, float z, int k) { return k == 0 ? x : (k == 1 ? y : z); }

struct CostP {
  float alpha, t_i, t_trav, sx, sy, sz;
  int dist_norm;
};

// Eq. 2 (Eq. 1 at alpha = 1): children L (nl triangles), R (nr) of node C.
// The two divisions by the node's area and squared diagonal are fast
// approximate reciprocals times products: the build's cost needs no correctly
// rounded quotient, only the same value for the same inputs.
__device__ __forceinline__ float eq2_cost(float3 llo, float3 lhi, int nl, float3 rlo, float3 rhi, int nr, float3 clo,
                                          float3 chi, const CostP& p) {
  const float sc = area(clo, chi);
  const float sah = sc > 0.f ? (area(llo, lhi) * (float)nl + area(rlo, rhi) * (float)nr) * __fdividef(1.f, sc) * p.t_i
                             : (float)(nl + nr) * p.t_i;
  const float ax = 0.5f * (llo.x + lhi.x) - p.sx, ay = 0.5f * (llo.y + lhi.y) - p.sy, az = 0.5f * (llo.z + lhi.z) - p.sz;
  const float bx = 0.5f * (rlo.x + rhi.x) - p.sx, by = 0.5f * (rlo.y + rhi.y) - p.sy, bz = 0.5f * (rlo.z + rhi.z) - p.sz;
  const float da2 = ax * ax + ay * ay + az * az, db2 = bx * bx + by * by + bz * bz;
  float d2 = 0.5f * (da2 + db2);
  if (p.dist_norm) {
    const float dx = chi.x - clo.x, dy = chi.y - clo.y, dz = chi.z - clo.z;
    const float diag2 = dx * dx + dy * dy + dz * dz;
    if (p.dist_norm == 2)  // each child's distance weighted by its triangles
      d2 = (diag2 > 0.f ? ((float)nl * da2 + (float)nr * db2) * __fdividef(1.f, diag2) : 0.f) * p.t_i;
    else
      d2 = (diag2 > 0.f ? d2 * __fdividef(1.f, diag2) : 0.f) * (float)(nl + nr) * p.t_i;
  }
  return p.alpha * sah + (1.f - p.alpha) * d2 + p.t_trav;
}

// Order-preserving unsigned code of a float: a < b <=> ucode(a) < ucode(b).
__device__ __forceinline__ unsigned ucode(float x) { return (unsigned)ford(x) ^ 0x80000000u; }
__device__ __forceinline__ float uval(unsigned u) { return iford((int)(u ^ 0x80000000u)); }

// ------------------------------------------------------------------ bins
// Union of a run of bins (or of records): count, box, centre bounds.
struct BinU {
  int n;
  float l0, l1, l2, h0, h1, h2;  // box
  float a0, a1, a2, b0, b1, b2;  // centre bounds
};

__device__ __forceinline__ BinU binu_empty() {
  return {0, FLT_MAX, FLT_MAX, FLT_MAX, -FLT_MAX, -FLT_MAX, -FLT_MAX,
          FLT_MAX, FLT_MAX, FLT_MAX, -FLT_MAX, -FLT_MAX, -FLT_MAX};
}
__device__ __forceinline__ BinU binu_join(const BinU& x, const BinU& y) {
  return {x.n + y.n,
          fminf(x.l0, y.l0), fminf(x.l1, y.l1), fminf(x.l2, y.l2),
          fmaxf(x.h0, y.h0), fmaxf(x.h1, y.h1), fmaxf(x.h2, y.h2),
          fminf(x.a0, y.a0), fminf(x.a1, y.a1), fminf(x.a2, y.a2),
          fmaxf(x.b0, y.b0), fmaxf(x.b1, y.b1), fmaxf(x.b2, y.b2)};
}
// Decode a 13-word bin entry.
__device__ __forceinline__ BinU binu_load(const unsigned* e) {
  const unsigned c = e[0];
  if (c == 0) return binu_empty();
  return {(int)c,          uval(~e[1]), uval(~e[2]), uval(~e[3]), uval(e[4]),  uval(e[5]), uval(e[6]),
          uval(~e[7]),     uval(~e[8]), uval(~e[9]), uval(e[10]), uval(e[11]), uval(e[12])};
}

// A record's 12 bin codes: box lo / hi and centre (twice: min and max slot).
struct RecCodes {
  unsigned v[12];
};
__device__ __forceinline__ RecCodes rec_codes(float4 lo, float4 hi, float cx, float cy, float cz) {
  RecCodes r;
  r.v[0] = ~ucode(lo.x);
  r.v[1] = ~ucode(lo.y);
  r.v[2] = ~ucode(lo.z);
  r.v[3] = ucode(hi.x);
  r.v[4] = ucode(hi.y);
  r.v[5] = ucode(hi.z);
  r.v[6] = ~ucode(cx);
  r.v[7] = ~ucode(cy);
  r.v[8] = ~ucode(cz);
  r.v[9] = ucode(cx);
  r.v[10] = ucode(cy);
  r.v[11] = ucode(cz);
  return r;
}

// Add the record of every lane with cell >= 0 to its bin on each axis: entry
// e[a] (count at bins + e[a] * kBinVals, then the 12 code maxima) and, if
// cnt is not null, cnt[e[a]].  The cell names the entries (equal cells,
// equal entries).  Lanes whose cells are equal and adjacent form a run: a
// segmented warp scan gives the run's last lane the run's count and code
// maxima, and that lane alone issues the shared-memory atomics, for all
// three axes.  Records in Morton or input order come in runs of one cell,
// so a warp costs one scan of 12 words instead of reductions per distinct
// bin and axis.  All 32 lanes of the warp must call.
__device__ __forceinline__ void bin_add_runs(int cell, const int* e, unsigned* bins, unsigned* cnt,
                                             const RecCodes& c) {
  const int lane = threadIdx.x & 31;
  __syncwarp();
  const int prev = __shfl_up_sync(kFull, cell, 1), next = __shfl_down_sync(kFull, cell, 1);
  const bool head = lane == 0 || prev != cell, tail = lane == 31 || next != cell;
  const unsigned heads = __ballot_sync(kFull, head);
  const int start = 31 - __clz(heads & (0xffffffffu >> (31 - lane)));  // first lane of the run
  unsigned v[12];
#pragma unroll
  for (int q = 0; q < 12; ++q) v[q] = c.v[q];
#pragma unroll 1
  for (int o = 1; o < 32; o <<= 1) {
    const int from = max(lane - o, start);  // (idempotent: nothing to select past the run's start)
#pragma unroll
    for (int q = 0; q < 12; ++q) v[q] = max(v[q], __shfl_sync(kFull, v[q], from));
  }
  if (tail && cell >= 0) {
    const unsigned m = (unsigned)(lane - start + 1);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      unsigned* b = bins + e[a] * kBinVals;
      atomicAdd(b, m);
#pragma unroll
      for (int q = 0; q < 12; ++q) atomicMax(b + 1 + q, v[q]);
      if (cnt) atomicAdd(cnt + e[a], m);
    }
  }
}

// A lane's run of records of one cell: the code maxima, the count, and per
// axis the word offset of its bin (from the bins) and of its count (<< 16,
// from the counts).
struct CellRun {
  unsigned v[12], n, off[3];
  int cell;  // -1: none
};

__device__ __forceinline__ void run_add(const CellRun& r, unsigned* bins, unsigned* cnt) {
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    unsigned* b = bins + (r.off[a] & 0xffffu);
    atomicAdd(b, r.n);
#pragma unroll
    for (int q = 0; q < 12; ++q) atomicMax(b + 1 + q, r.v[q]);
    atomicAdd(cnt + (r.off[a] >> 16), r.n);
  }
}

// Add the run that every lane holds, joined first with the adjacent lanes'
// runs of the same cell by a segmented warp scan (as many steps as the
// longest stretch of equal cells needs); the last lane of a stretch issues
// the atomics.  All 32 lanes of the warp must call.
__device__ __forceinline__ void run_add_warp(CellRun r, unsigned* bins, unsigned* cnt) {
  const int lane = threadIdx.x & 31;
  __syncwarp();
  const int prev = __shfl_up_sync(kFull, r.cell, 1), next = __shfl_down_sync(kFull, r.cell, 1);
  const bool head = lane == 0 || prev != r.cell, tail = lane == 31 || next != r.cell;
  const unsigned heads = __ballot_sync(kFull, head);
  const int start = 31 - __clz(heads & (0xffffffffu >> (31 - lane)));  // first lane of the stretch
  const int span = (int)__reduce_max_sync(kFull, (unsigned)(lane - start));
#pragma unroll 1
  for (int o = 1; o <= span; o <<= 1) {
    const int from = max(lane - o, start);
    const unsigned m = __shfl_sync(kFull, r.n, from);
    r.n += lane - o >= start ? m : 0u;
#pragma unroll
    for (int q = 0; q < 12; ++q) r.v[q] = max(r.v[q], __shfl_sync(kFull, r.v[q], from));  // (idempotent)
  }
  if (tail && r.cell >= 0) run_add(r, bins, cnt);
  __syncwarp();
}

// ------------------------------------------------------------------ Eq. 2 evaluation
struct Split {
  float cost;
  int cand;  // axis * (K - 1) + plane - 1 (INT_MAX: none)
  BinU L, R;
};

__device__ __forceinline__ void split_none(Split& s) {
  s.cost = INFINITY;
  s.cand = INT_MAX;
  s.L = binu_empty();
  s.R = binu_empty();
}

// Count and box of a run of bins: the part of a bin the cost needs.
struct BinB {
  int n;
  float l0, l1, l2, h0, h1, h2;
};
__device__ __forceinline__ BinB binb_empty() { return {0, FLT_MAX, FLT_MAX, FLT_MAX, -FLT_MAX, -FLT_MAX, -FLT_MAX}; }
__device__ __forceinline__ BinB binb_join(const BinB& x, const BinB& y) {
  return {x.n + y.n,          fminf(x.l0, y.l0), fminf(x.l1, y.l1), fminf(x.l2, y.l2),
          fmaxf(x.h0, y.h0),  fmaxf(x.h1, y.h1), fmaxf(x.h2, y.h2)};
}
// The bin at e, the empty one unless `in`: loaded and selected without a
// branch.  A lane that skips a load leaves its warp in two parts, and every
// warp-wide operation after that meets at a slow rendezvous.
__device__ __forceinline__ BinB binb_load(const unsigned* e, bool in) {
  const unsigned c = e[0], w1 = e[1], w2 = e[2], w3 = e[3], w4 = e[4], w5 = e[5], w6 = e[6];
  const bool f = in && c != 0;
  return {f ? (int)c : 0,         f ? uval(~w1) : FLT_MAX,  f ? uval(~w2) : FLT_MAX, f ? uval(~w3) : FLT_MAX,
          f ? uval(w4) : -FLT_MAX, f ? uval(w5) : -FLT_MAX, f ? uval(w6) : -FLT_MAX};
}
#define RT_BINB_SHFL(F, x, arg)                                                                            \
  BinB {                                                                                                   \
    F(kFull, (x).n, arg), F(kFull, (x).l0, arg), F(kFull, (x).l1, arg), F(kFull, (x).l2, arg),             \
        F(kFull, (x).h0, arg), F(kFull, (x).h1, arg), F(kFull, (x).h2, arg)                                 \
  }

// Eq. 2 at the K - 1 planes of na axes (a0 .. a0 + na - 1, na * K <= 32) by
// one warp.  Lanes are cut into segments of K, lane sl of segment g holding
// bin sl of axis a0 + g (`bins0` points at the bins of axis a0, the others
// follow); segmented warp scans (log2 K steps) of the bins' counts and boxes
// give every lane the union of the bins left of plane sl and right of it,
// and lane sl evaluates Eq. 2 there.  `best` (identical in every lane) is
// replaced if a plane has a lower cost, ties going to the lower candidate
// (lowest axis, then lowest plane); the winning children's centre bounds
// are then gathered by warp reductions over the bins' codes.  The union of
// a segment is the node box.
// kVals: words per bin (13, or 7 for bins of count and box only); kCentres:
// gather the children's centre bounds (13-word bins only; otherwise the
// caller derives the children's unions itself and only best.L.n is exact).
// eval_bins is the evaluation of bins held in registers (x: the lane's bin;
// in: the lane holds one), eval_seg the one of bins in shared memory.
template <bool kCentres>
__device__ __forceinline__ void eval_bins(const BinB& x, const unsigned* e, bool in, int g, int sl, int K, int n, int a0,
                                          const CostP& cp, Split& best) {
  const int a = a0 + (in ? g : 0);
  BinB pre = x, suf = x;
  const int l0 = threadIdx.x & 31, first = l0 - sl, last = min(first + K - 1, 31);
#pragma unroll 1
  for (int o = 1; o < K; o <<= 1) {
    // the boxes' unions are idempotent: a lane past its axis's end reads the
    // end's own union and only the counts are selected
    const int up = max(l0 - o, first), dn = min(l0 + o, last);
    BinB u = RT_BINB_SHFL(__shfl_sync, pre, up), d = RT_BINB_SHFL(__shfl_sync, suf, dn);
    u.n = sl >= o ? u.n : 0;
    d.n = 0;  // (the right side's count is n minus the left's)
    pre = binb_join(pre, u);
    suf = binb_join(suf, d);
  }
  const BinB L = RT_BINB_SHFL(__shfl_up_sync, pre, 1);  // lane sl: bins 0 .. sl-1 of its axis
  const BinB C = binb_join(L, suf);                     // the node (at sl >= 1, where a plane is)
  // Eq. 2 in every lane (a plane without records on both sides costs
  // infinity), then the lowest cost by two warp reductions: costs are >= +0
  // (alpha in [0, 1], t_i > 0, t_trav >= 0), so their bit patterns order as
  // their values, and the lowest candidate among equal costs wins
  const float c = eq2_cost(make_float3(L.l0, L.l1, L.l2), make_float3(L.h0, L.h1, L.h2), L.n,
                           make_float3(suf.l0, suf.l1, suf.l2), make_float3(suf.h0, suf.h1, suf.h2), n - L.n,
                           make_float3(C.l0, C.l1, C.l2), make_float3(C.h0, C.h1, C.h2), cp);
  const bool ok = in && sl >= 1 && L.n > 0 && L.n < n && c < INFINITY;
  const unsigned key = ok ? __float_as_uint(c + 0.f) : __float_as_uint(INFINITY);
  const unsigned kmin = __reduce_min_sync(kFull, key);
  const int cand = (int)__reduce_min_sync(kFull, ok && key == kmin ? (unsigned)(a * (K - 1) + sl - 1) : 0xffffffffu);
  const float cost = __uint_as_float(kmin);
  if (cand >= 0 && (cost < best.cost || (cost == best.cost && cand < best.cand))) {
    const int ax = cand / (K - 1), gw = ax - a0, pl = cand - ax * (K - 1) + 1;  // plane pl of axis ax
    const int w = gw * K + pl;
    const BinB Lb = RT_BINB_SHFL(__shfl_sync, L, w), Rb = RT_BINB_SHFL(__shfl_sync, suf, w);
    const bool mine = in && g == gw;
    unsigned lc[6] = {0u, 0u, 0u, 0u, 0u, 0u}, rc[6] = {0u, 0u, 0u, 0u, 0u, 0u};
    if (kCentres) {
#pragma unroll
      for (int q = 0; q < 6; ++q) {
        const unsigned w = e[7 + q], v = mine ? w : 0u;
        lc[q] = __reduce_max_sync(kFull, sl < pl ? v : 0u);
        rc[q] = __reduce_max_sync(kFull, sl >= pl ? v : 0u);
      }
    }
    best.cost = cost;
    best.cand = cand;
    best.L = {Lb.n, Lb.l0, Lb.l1, Lb.l2, Lb.h0, Lb.h1, Lb.h2,
              uval(~lc[0]), uval(~lc[1]), uval(~lc[2]), uval(lc[3]), uval(lc[4]), uval(lc[5])};
    best.R = {n - Lb.n, Rb.l0, Rb.l1, Rb.l2, Rb.h0, Rb.h1, Rb.h2,
              uval(~rc[0]), uval(~rc[1]), uval(~rc[2]), uval(rc[3]), uval(rc[4]), uval(rc[5])};
  }
}
template <int kVals, bool kCentres>
__device__ __forceinline__ void eval_seg(const unsigned* bins0, int K, int n, int a0, int na, const CostP& cp,
                                         Split& best) {
  const int lane = threadIdx.x & 31;
  const int g = lane / K, sl = lane - g * K;
  const bool in = g < na;
  const unsigned* e = bins0 + ((in ? g : 0) * K + sl) * kVals;
  __syncwarp();
  const BinB x = binb_load(e, in);
  eval_bins<kCentres>(x, e, in, g, sl, K, n, a0, cp, best);
}
__device__ __forceinline__ BinB binb_xor(const BinB& x, int o) { return RT_BINB_SHFL(__shfl_xor_sync, x, o); }
#undef RT_BINB_SHFL

__device__ __forceinline__ void eval_axis(const unsigned* bins, int K, int n, int a, const CostP& cp, Split& best) {
  eval_seg<kBinVals, true>(bins + a * K * kBinVals, K, n, a, 1, cp, best);
}
__device__ __forceinline__ void eval_axes(const unsigned* bins, int K, int n, int a0, int na, const CostP& cp,
                                          Split& best) {
  eval_seg<kBinVals, true>(bins + a0 * K * kBinVals, K, n, a0, na, cp, best);
}

// ------------------------------------------------------------------ arguments
struct BuildArgs {
  const float4* tri;  // input-order triangles
  const int* sel;     // nullable: input ids of the triangles in this build (a range build)
  float4* rec[2];     // [2T] records (lo.xyz, id) (hi.xyz, morton); a node's range lives
                      // in one buffer, its children go to the other
  Node2* node2;
  int2* link2;
  BuildCtl* ctl;
  Task* qa;  // subtree queue
  int* qa_ready;
  TopTask* ttask;  // big nodes
  int* tdone;
  unsigned* tbins;
  unsigned* tccnt;
  unsigned* tscnt;
  int2* titem;  // chunk items of big nodes
  int4* tplan;  // [cap_t][2]: what a big node reserved for each big child (task slots, count slots,
                // chunk items, count slots to clear), written by its chunk 0
  int* tready;
  WNode* wide;
  QNode* qwide;  // nullable: also write the 64-byte nodes
  WNode8* wide8; // nullable: write 8-wide traversal nodes (instead of the 4-wide ones)
  float4* tri_leaf;
  int32_t* order;
  int* epoch_dev;
  int n, K, max_leaf;  // n: records in this build
  int n_all;           // triangles in the scene (input ids are below it)
  int big, chunk, rpt, cap_t, cap_c, qa_cap, top_ctas;
  int wsm;             // nodes of up to this many records go to k_small (0: none do)
  int spin_limit;                    // polls without progress before a wait gives up
  int phantom_tasks, phantom_items;  // test hooks: pending work that never comes
  CostP cp;
};

__device__ __forceinline__ unsigned* tbins_at(const BuildArgs& A, int slot) {
  return A.tbins + (size_t)slot * kBinWords;
}
__device__ __forceinline__ unsigned* tccnt_at(const BuildArgs& A, int c) { return A.tccnt + (size_t)c * kCntStride; }
__device__ __forceinline__ unsigned* tscnt_at(const BuildArgs& A, int c) { return A.tscnt + (size_t)c * kCntStride; }

__device__ __forceinline__ TopTask load_top_cg(const TopTask* p) {
  const int4* q = reinterpret_cast<const int4*>(p);
  const int4 a = __ldcg(q), b = __ldcg(q + 1), c = __ldcg(q + 2), d = __ldcg(q + 3);
  TopTask t;
  t.begin = a.x;
  t.count = a.y;
  t.parent = a.z;
  t.side = a.w;
  t.clo[0] = __int_as_float(b.x);
  t.clo[1] = __int_as_float(b.y);
  t.clo[2] = __int_as_float(b.z);
  t.depth = b.w;
  t.chi[0] = __int_as_float(c.x);
  t.chi[1] = __int_as_float(c.y);
  t.chi[2] = __int_as_float(c.z);
  t.nchunk = c.w;
  t.chunk_first = d.x;
  t.child_slot = d.y;
  t.chunk_res = d.z;
  t.parity = d.w;
  return t;
}

// Hand a task to the subtree queue (one thread).  The slot's ready word
// takes this build's epoch, so stale slots from older builds never match.
__device__ void push_task(const BuildArgs& A, const Task& t, int epoch) {
  const int s = atomicAdd(&A.ctl->qa_tail, 1);
  if (s >= A.qa_cap) {
    set_status(A.ctl, kStQueueOverflow, 1);
    return;
  }
  atomicAdd(&A.ctl->qa_pending, 1);
  A.qa[s] = t;
  st_release(&A.qa_ready[s], epoch);
}

// Hand up to 3 tasks to the subtree queue at once (one thread): one slot
// reservation, one fence.
__device__ void push_tasks(const BuildArgs& A, const Task* t, int k, int epoch) {
  if (k <= 0) return;
  const int s = atomicAdd(&A.ctl->qa_tail, k);
  if (s + k > A.qa_cap) {
    set_status(A.ctl, kStQueueOverflow, 3);
    return;
  }
  atomicAdd(&A.ctl->qa_pending, k);
  for (int i = 0; i < k; ++i) A.qa[s + i] = t[i];
  for (int i = 0; i < k; ++i) st_release(&A.qa_ready[s + i], epoch);
}

// Hand a node of at most A.wsm records to k_small (one thread): its list
// grows down from the end of the task array (a tree node is in one of the
// two at most, so they never meet in a valid tree).
__device__ void push_small(const BuildArgs& A, const Task& t) {
  const int i = atomicAdd(&A.ctl->sq_count, 1);
  if (i >= A.qa_cap - ld_volatile(&A.ctl->qa_tail)) {
    set_status(A.ctl, kStQueueOverflow, 6);
    return;
  }
  A.qa[A.qa_cap - 1 - i] = t;
}

__device__ __forceinline__ Task make_task(int begin, int count, int parent, int side, int depth, const BinU& u,
                                          int parity) {
  Task t;
  t.begin = begin;
  t.count = count;
  t.parent = parent;
  t.side = side;
  t.clo[0] = u.a0;
  t.clo[1] = u.a1;
  t.clo[2] = u.a2;
  t.chi[0] = u.b0;
  t.chi[1] = u.b1;
  t.chi[2] = u.b2;
  t.depth = depth;
  t.pad = parity;
  return t;
}

// Reserve `amt` consecutive items of a counter bounded by `cap`: one atomic
// add; -1 if they do not fit (the items past cap are then never used).
__device__ __forceinline__ int reserve(int* ctr, int amt, int cap) {
  const int old = atomicAdd(ctr, amt);
  return old + amt <= cap ? old : -1;
}

// Write binary node `id` (both children's boxes, refs, counts) and link it
// to its parent.  One thread.
__device__ __forceinline__ void write_node(const BuildArgs& A, int id, int parent, int side, const BinU& L, int refl,
                                           int nl, const BinU& R, int refr, int nr, int epoch) {
  Node2 nd;
  nd.a_lo = make_float4(L.l0, L.l1, L.l2, __int_as_float(refl));
  nd.a_hi = make_float4(L.h0, L.h1, L.h2, __int_as_float(nl));
  nd.b_lo = make_float4(R.l0, R.l1, R.l2, __int_as_float(refr));
  nd.b_hi = make_float4(R.h0, R.h1, R.h2, __int_as_float(nr));
  A.node2[id] = nd;
  if (parent < 0)
    A.ctl->root_ref = id;
  else if (parent < A.n - 1)
    *(side == 0 ? &A.node2[parent].a_lo.w : &A.node2[parent].b_lo.w) = __int_as_float(id);
  else
    set_status(A.ctl, kStBadLink, 3);
  A.link2[id] = make_int2(parent, epoch);
}

// ------------------------------------------------------------------ range selection
// A build with a ray action range keeps the triangles whose box lies within
// the range of the source (Sec. II.B): no point of a path of total length
// <= range is farther from the source, at any reflection order.  The
// selection keeps input order (block counts, one scan, ordered writes), so
// the build is the same every time.  The range is widened by 1e-5 of itself
// so that rounding never drops a reachable triangle.
__device__ __forceinline__ bool tri_in_range(const float4* __restrict__ tri, int i, float3 s, float r2) {
  const float4 a = __ldg(tri + 3 * (size_t)i), b = __ldg(tri + 3 * (size_t)i + 1), c = __ldg(tri + 3 * (size_t)i + 2);
  const float dx = fmaxf(fmaxf(fminf(a.x, fminf(b.x, c.x)) - s.x, s.x - fmaxf(a.x, fmaxf(b.x, c.x))), 0.f);
  const float dy = fmaxf(fmaxf(fminf(a.y, fminf(b.y, c.y)) - s.y, s.y - fmaxf(a.y, fmaxf(b.y, c.y))), 0.f);
  const float dz = fmaxf(fmaxf(fminf(a.z, fminf(b.z, c.z)) - s.z, s.z - fmaxf(a.z, fmaxf(b.z, c.z))), 0.f);
  return dx * dx + dy * dy + dz * dz <= r2;
}

__global__ void __launch_bounds__(kBlock) k_sel_count(const float4* __restrict__ tri, int n, float3 s, float r2,
                                                      int* __restrict__ cnt) {
  const int i = blockIdx.x * kBlock + threadIdx.x;
  const int c = __syncthreads_count(i < n && tri_in_range(tri, i, s, r2));
  if (threadIdx.x == 0) cnt[blockIdx.x] = c;
}

// Exclusive scan of cnt[0 .. nb) in place by one CTA; the total goes to cnt[nb].
__global__ void __launch_bounds__(1024) k_sel_scan(int* __restrict__ cnt, int nb) {
  __shared__ int part[1024];
  const int t = threadIdx.x, per = (nb + 1023) / 1024, b0 = min(t * per, nb), b1 = min(b0 + per, nb);
  int sum = 0;
  for (int b = b0; b < b1; ++b) sum += cnt[b];
  part[t] = sum;
  __syncthreads();
  for (int o = 1; o < 1024; o <<= 1) {
    const int v = t >= o ? part[t - o] : 0;
    __syncthreads();
    part[t] += v;
    __syncthreads();
  }
  int run = part[t] - sum;
  for (int b = b0; b < b1; ++b) {
    const int v = cnt[b];
    cnt[b] = run;
    run += v;
  }
  if (t == 1023) cnt[nb] = part[1023];
}

__global__ void __launch_bounds__(kBlock) k_sel_write(const float4* __restrict__ tri, int n, float3 s, float r2,
                                                      const int* __restrict__ off, int* __restrict__ sel) {
  __shared__ int wc[kWarps];
  const int i = blockIdx.x * kBlock + threadIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool f = i < n && tri_in_range(tri, i, s, r2);
  const unsigned bal = __ballot_sync(kFull, f);
  if (lane == 0) wc[warp] = __popc(bal);
  __syncthreads();
  int base = off[blockIdx.x];
  for (int w = 0; w < warp; ++w) base += wc[w];
  if (f) sel[base + __popc(bal & ((1u << lane) - 1u))] = i;
}

// ------------------------------------------------------------------ prep
__global__ void __launch_bounds__(kBlock) k_prep(BuildArgs A) {
  pdl_wait();
  pdl_launch();
  __shared__ float red[kWarps][12];
  const int n = A.n;
  const int gt = blockIdx.x * kBlock + threadIdx.x, gs = gridDim.x * kBlock;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (gt == 0) {
    const int e = *A.epoch_dev + 1;
    *A.epoch_dev = e;
    A.ctl->epoch = e;
  }
  // the root's bins and 32-chunk group counts start empty
  const int nch = (n + A.chunk - 1) / A.chunk;
  for (int k = gt; k < kBinWords; k += gs) A.tbins[k] = 0u;
  for (int k = gt; k < (nch / 32 + 1) * kCntStride; k += gs) A.tscnt[k] = 0u;
  float v[12];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    v[k] = FLT_MAX;       // box lo
    v[3 + k] = -FLT_MAX;  // box hi
    v[6 + k] = FLT_MAX;   // centre lo
    v[9 + k] = -FLT_MAX;  // centre hi
  }
  for (int i = gt; i < n; i += gs) {
    const int t = A.sel ? __ldg(A.sel + i) : i;
    const float4 a = A.tri[3 * (size_t)t], b = A.tri[3 * (size_t)t + 1], c = A.tri[3 * (size_t)t + 2];
    float lx = fminf(a.x, fminf(b.x, c.x)), ly = fminf(a.y, fminf(b.y, c.y)), lz = fminf(a.z, fminf(b.z, c.z));
    float hx = fmaxf(a.x, fmaxf(b.x, c.x)), hy = fmaxf(a.y, fmaxf(b.y, c.y)), hz = fmaxf(a.z, fmaxf(b.z, c.z));
    // no ray meets a triangle whose three vertices have no number on an axis;
    // its box is a point there, or every union with it would be lost
    if (isnan(lx)) lx = hx = 0.f;
    if (isnan(ly)) ly = hy = 0.f;
    if (isnan(lz)) lz = hz = 0.f;
    A.rec[0][2 * (size_t)i] = make_float4(lx, ly, lz, __int_as_float(t));
    A.rec[0][2 * (size_t)i + 1] = make_float4(hx, hy, hz, 0.f);
    const float cx = centre(lx, hx), cy = centre(ly, hy), cz = centre(lz, hz);
    v[0] = fminf(v[0], lx);
    v[1] = fminf(v[1], ly);
    v[2] = fminf(v[2], lz);
    v[3] = fmaxf(v[3], hx);
    v[4] = fmaxf(v[4], hy);
    v[5] = fmaxf(v[5], hz);
    v[6] = fminf(v[6], cx);
    v[7] = fminf(v[7], cy);
    v[8] = fminf(v[8], cz);
    v[9] = fmaxf(v[9], cx);
    v[10] = fmaxf(v[10], cy);
    v[11] = fmaxf(v[11], cz);
  }
  __syncwarp();
#pragma unroll
  for (int k = 0; k < 12; ++k) {
    const bool mn = k < 3 || (k >= 6 && k < 9);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float y = __shfl_xor_sync(kFull, v[k], o);
      v[k] = mn ? fminf(v[k], y) : fmaxf(v[k], y);
    }
    if (lane == 0) red[warp][k] = v[k];
  }
  __syncthreads();
  if (threadIdx.x < 12) {
    const int k = threadIdx.x;
    const bool mn = k < 3 || (k >= 6 && k < 9);
    float x = red[0][k];
    for (int w = 1; w < kWarps; ++w) x = mn ? fminf(x, red[w][k]) : fmaxf(x, red[w][k]);
    if (n > 0) atomicMax(&A.ctl->sb[k], mn ? ~ucode(x) : ucode(x));
  }
}

// Spread the low 10 bits of v to every third bit.
__device__ __forceinline__ uint32_t spread10(uint32_t v) {
  v &= 0x3ffu;
  v = (v | (v << 16)) & 0x030000FFu;
  v = (v | (v << 8)) & 0x0300F00Fu;
  v = (v | (v << 4)) & 0x030C30C3u;
  v = (v | (v << 2)) & 0x09249249u;
  return v;
}

// ------------------------------------------------------------------ root
// Morton keys of all records; the root task (a top task, a subtree task, a
// leaf or nothing); the root's bins and per-chunk counts when it is a top task.
__global__ void __launch_bounds__(kBlock) k_bin_root(BuildArgs A) {
  pdl_wait();
  pdl_launch();
  __shared__ unsigned sbins[kBinWords];
  __shared__ unsigned scnt[kCntStride];
  const int n = A.n, K = A.K, K3 = 3 * K, CH = A.chunk;
  const int nch = (n + CH - 1) / CH;
  const bool top = n > A.big;
  const int gt = blockIdx.x * kBlock + threadIdx.x, gs = gridDim.x * kBlock;
  float cl[3], chh[3], msc[3], scl[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    cl[a] = uval(~__ldcg(&A.ctl->sb[6 + a]));
    chh[a] = uval(__ldcg(&A.ctl->sb[9 + a]));
    const float ext = chh[a] - cl[a];
    msc[a] = ext > 0.f ? 1023.99f / ext : 0.f;
    scl[a] = bin_scale(cl[a], chh[a], K);
  }
  if (gt == 0) {
    const int epoch = __ldcg(&A.ctl->epoch);
    BinU cu = binu_empty();
    cu.a0 = cl[0];
    cu.a1 = cl[1];
    cu.a2 = cl[2];
    cu.b0 = chh[0];
    cu.b1 = chh[1];
    cu.b2 = chh[2];
    if (n == 0) {
      A.ctl->root_ref = INT_MIN;
    } else if (n <= A.max_leaf) {
      A.ctl->root_ref = leaf_ref(0, n);
      A.ctl->n_leaves = 1;
      A.ctl->depth2 = 1;
      A.ctl->max_leaf_size = n;
    } else if (!top) {
      push_task(A, make_task(0, n, -1, 0, 1, cu, 0), epoch);
    } else {
      TopTask R;
      R.begin = 0;
      R.count = n;
      R.parent = -1;
      R.side = 0;
      for (int a = 0; a < 3; ++a) {
        R.clo[a] = cl[a];
        R.chi[a] = chh[a];
      }
      R.depth = 1;
      R.nchunk = nch;
      R.chunk_first = 0;   // count slots 0 .. nch-1: the root's chunks (written below)
      R.child_slot = 1;    // task slots 1, 2
      R.chunk_res = nch;   // count slots nch .. 2 nch + 1
      R.parity = 0;
      A.ttask[0] = R;
      A.ctl->t_slot_next = 3;
      A.ctl->t_cnt_next = 2 * nch + 2;
      A.ctl->ti_tail = nch;
      A.ctl->ti_pending = nch;
    }
    if (A.phantom_tasks) atomicAdd(&A.ctl->qa_pending, A.phantom_tasks);
    if (A.phantom_items) atomicAdd(&A.ctl->ti_pending, A.phantom_items);
  }
  if (top) {
    // the root's children start empty; the root's chunks become items
    const int epoch = __ldcg(&A.ctl->epoch);
    for (int k = gt; k < 2 * kBinWords; k += gs) tbins_at(A, 1)[k] = 0u;
    for (int k = gt; k < (nch + 2) * kCntStride; k += gs) {
      tccnt_at(A, nch)[k] = 0u;
      tscnt_at(A, nch)[k] = 0u;
    }
    if (gt < 3) A.tdone[gt] = 0;
    for (int c = gt; c < nch; c += gs) {
      A.titem[c] = make_int2(0, c);
      A.tready[c] = epoch;
    }
  }
  float4* rec = A.rec[0];
  for (int c = blockIdx.x; c < nch; c += gridDim.x) {
    if (top) {
      for (int w = threadIdx.x; w < K3 * kBinVals; w += kBlock) sbins[w] = 0u;
      for (int w = threadIdx.x; w < K3; w += kBlock) scnt[w] = 0u;
      __syncthreads();
    }
    for (int r = 0; r < A.rpt; ++r) {
      const int k = c * CH + r * kBlock + threadIdx.x;
      const bool valid = k < n;
      float4 lo = make_float4(0.f, 0.f, 0.f, 0.f), hi = lo;
      float cx = 0.f, cy = 0.f, cz = 0.f;
      if (valid) {
        lo = __ldcg(rec + 2 * (size_t)k);
        hi = __ldcg(rec + 2 * (size_t)k + 1);
        cx = centre(lo.x, hi.x);
        cy = centre(lo.y, hi.y);
        cz = centre(lo.z, hi.z);
        uint32_t q[3];
        const float cc[3] = {cx, cy, cz};
#pragma unroll
        for (int a = 0; a < 3; ++a) q[a] = (uint32_t)min(max((int)((cc[a] - cl[a]) * msc[a]), 0), 1023);
        const uint32_t key = (spread10(q[0]) << 2) | (spread10(q[1]) << 1) | spread10(q[2]);
        hi.w = __uint_as_float(key);
        rec[2 * (size_t)k + 1] = hi;
      }
      if (top) {
        const float cc[3] = {cx, cy, cz};
        const RecCodes rc = rec_codes(lo, hi, cx, cy, cz);
        int e[3], cell = 0;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          const int b = bin_of(cc[a], cl[a], scl[a], K);
          e[a] = a * K + b;
          cell = cell * kMaxBins + b;
        }
        bin_add_runs(valid ? cell : -1, e, sbins, scnt, rc);
      }
    }
    if (top) {
      __syncthreads();
      unsigned* gc = tccnt_at(A, c);
      unsigned* gg = tscnt_at(A, c >> 5);
      for (int w = threadIdx.x; w < K3; w += kBlock) {
        const unsigned v = scnt[w];
        gc[w] = v;
        if (v) atomicAdd(gg + w, v);
      }
      unsigned* gb = tbins_at(A, 0);
      for (int w = threadIdx.x; w < K3 * kBinVals; w += kBlock) {
        const unsigned v = sbins[w];
        if (v) {
          if (w % kBinVals == 0)
            atomicAdd(gb + w, v);
          else
            atomicMax(gb + w, v);
        }
      }
      __syncthreads();
    }
  }
}

// Tree facts gathered by a warp, added to the control block when it exits.
struct WarpStats {
  int n_int, n_leaf, big, deep;
};

// Account a written binary node (one thread per node).
__device__ __forceinline__ void note_node(WarpStats& ws, int nl, int nr, bool leafl, bool leafr, int depth) {
  ++ws.n_int;
  ws.n_leaf += (int)leafl + (int)leafr;
  if (leafl) ws.big = max(ws.big, nl);
  if (leafr) ws.big = max(ws.big, nr);
  ws.deep = max(ws.deep, (leafl || leafr) ? depth + 1 : depth);
}

// ------------------------------------------------------------------ big nodes
// Shared-memory place of record k of a chunk, in float4: four records and
// 16 bytes of padding per thread, so that 16-byte reads of consecutive
// records by consecutive lanes fall on distinct banks.
__device__ __forceinline__ int stage_at(int k) { return (k >> 2) * 9 + (k & 3) * 2; }

struct TopSmem {
  unsigned pbins[kBinWords];
  unsigned cbins[2][kBinWords];
  unsigned ccnt[2][2][kCntStride];
  Split ax[3];
  int wl[kWarps];
  int red[kWarps];
  int2 item;
  int last;
  int created[2], ibase[2];
  int4 plan[2];
  Task ptask[2];  // subtree-sized children the emit hands to the subtree queue
  int np;
};

// With the chunk's records.
struct StagedSmem {
  TopSmem top;
  alignas(16) float4 rec[kStage / 4 * 9];  // (stage_at)
  unsigned short order[kStage];            // its records, the left ones first
};

__device__ __forceinline__ int block_sum(int v, int* red) {
  __syncwarp();
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  int t = 0;
#pragma unroll
  for (int w = 0; w < kWarps; ++w) t += red[w];
  __syncthreads();
  return t;
}

// One thread takes the next chunk item and waits for it to be published
// (no warp-synchronous operation in this loop; the other threads wait at a
// barrier).  Returns (-1, 0) when no big node is left (or the build failed).
// The wait is bounded: spin_limit polls without new items set a timeout
// status.
__device__ int2 claim_item(const BuildArgs& A, int epoch) {
  const int s = atomicAdd(&A.ctl->ti_head, 1);
  int seen = -1;
  for (int it = 0;; ++it) {
    if (s < A.cap_c && ld_acquire(&A.tready[s]) == epoch) {
      return __ldcg(A.titem + s);
    }
    if ((it & 3) == 0) {
      if (ld_volatile(&A.ctl->ti_pending) == 0 || ld_volatile(&A.ctl->status) != 0) break;
      const int tail = ld_volatile(&A.ctl->ti_tail);
      if (tail != seen) {  // new items appeared: restart the no-progress budget
        seen = tail;
        it = 0;
      }
    }
    if (it > A.spin_limit) {
      set_status(A.ctl, kStQueueTimeout, 2);
      break;
    }
    __nanosleep(128);
  }
  return make_int2(-1, 0);
}

__device__ void top_emit(const BuildArgs& A, TopSmem& S, const TopTask& T, int slot, int epoch, int nl, int nr,
                         const BinU& cu0, const BinU& cu1, bool top0, bool top1, int nch0, int nch1, int cfirst0,
                         int cfirst1, WarpStats& ts);

// Chunk 0 of a big node, as soon as its split is known: one thread reserves
// what the node's big children will need (two task slots and the count slots
// for their own children, their chunk items) while the chunk is partitioned;
// then the CTA clears what their chunks will fill, so that the CTA finishing
// the node's last chunk only writes and publishes.  The clearing is ordered
// before that CTA's emit by chunk 0's release of its done count.
__device__ __forceinline__ void top_reserve(const BuildArgs& A, TopSmem& S, int slot, bool top0, bool top1, int nch0,
                                            int nch1) {
  int cs[2] = {-1, -1}, cr[2] = {-1, -1}, ib[2] = {-1, -1};
  // every reservation is issued before any result is used: one round trip
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    if (!(s ? top1 : top0)) continue;
    const int ncs = s ? nch1 : nch0;
    cs[s] = reserve(&A.ctl->t_slot_next, 2, A.cap_t);
    cr[s] = reserve(&A.ctl->t_cnt_next, ncs + 2, A.cap_c);
    ib[s] = reserve(&A.ctl->ti_tail, ncs, A.cap_c);
  }
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    const int ncs = s ? nch1 : nch0;
    const int4 pl =
        (cs[s] >= 0 && cr[s] >= 0 && ib[s] >= 0) ? make_int4(cs[s], cr[s], ib[s], ncs + 2) : make_int4(-1, -1, -1, 0);
    S.plan[s] = pl;
    A.tplan[2 * slot + s] = pl;
  }
}
// (after a barrier: the partition's)
__device__ __forceinline__ void top_clear(const BuildArgs& A, TopSmem& S) {
  const int tid = threadIdx.x;
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    const int4 pl = S.plan[s];
    if (pl.x < 0) continue;
    unsigned* zb = tbins_at(A, pl.x);
    for (int w = tid; w < 2 * kBinWords; w += kBlock) zb[w] = 0u;
    if (tid < 2) A.tdone[pl.x + tid] = 0;
    unsigned* zc = tccnt_at(A, pl.y);
    unsigned* zs = tscnt_at(A, pl.y);
    for (int w = tid; w < pl.w * kCntStride; w += kBlock) {
      zc[w] = 0u;
      zs[w] = 0u;
    }
  }
}

// Chunk j of big node T (one CTA): Eq. 2 at every bin plane from the node's
// merged bins (every chunk of the node picks the same plane), stable
// partition of the chunk into the other record buffer, and on the way the
// bins and per-chunk counts of the children that are big nodes too.  The CTA
// that finishes the node's last chunk writes the node and creates its
// children: big ones get their chunk items, the others go to the subtree
// queue.  No CTA ever waits for another.
template <bool kStaged>
__device__ void top_chunk(const BuildArgs& A, TopSmem& S, const TopTask& T, int slot, int j, int epoch,
                          WarpStats& ts) {
  StagedSmem& G = reinterpret_cast<StagedSmem&>(S);  // (where kStaged)
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int K = A.K, K3 = 3 * K, CH = A.chunk;
  const unsigned lt_mask = (1u << lane) - 1u;
  const int n = T.count;
  const int par = T.parity & 1;
  const float4* src = A.rec[par];
  float4* dst = A.rec[par ^ 1];
  const int r0 = j * CH;
  const int rn = min(CH, n - r0);
  float4 lo[kRegRpt], hi[kRegRpt];
  if (kStaged) {  // the chunk's records go to shared memory while the split is chosen
    const float4* p = src + 2 * ((size_t)T.begin + r0);
    const unsigned to = (unsigned)__cvta_generic_to_shared(&G.rec[0]);
    for (int i = tid; i < 2 * rn; i += kBlock)
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(to + 16 * (stage_at(i >> 1) + (i & 1))),
                   "l"(p + i)
                   : "memory");
  } else {
#pragma unroll
    for (int r = 0; r < kRegRpt; ++r) {
      const int k = r * kBlock + tid;
      lo[r] = hi[r] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (r < A.rpt && k < rn) {
        const float4* p = src + 2 * ((size_t)T.begin + r0 + k);
        lo[r] = __ldcg(p);
        hi[r] = __ldcg(p + 1);
      }
    }
  }
  {
    for (int w = tid; w < 2 * kBinWords; w += kBlock) (&S.cbins[0][0])[w] = 0u;
    for (int w = tid; w < 4 * kCntStride; w += kBlock) (&S.ccnt[0][0][0])[w] = 0u;
  }
  float cmin[3], scl[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    cmin[a] = T.clo[a];
    scl[a] = bin_scale(T.clo[a], T.chi[a], K);
  }
  __syncthreads();
  // Eq. 2 at every plane.  Up to 10 bins warp 0 evaluates all three axes in
  // one pass; otherwise warp a evaluates axis a (a < 3).  The others wait at
  // the barrier and read the choice from shared memory.  An axis without
  // extent has all records in bin 0 and yields no candidate.
  Split best;
  if (__any_sync(kFull, warp < (3 * K <= 32 ? 1 : 3))) {
    Split sp;
    split_none(sp);
    if (3 * K <= 32)
      eval_axes(S.pbins, K, n, 0, 3, A.cp, sp);
    else
      eval_axis(S.pbins, K, n, warp, A.cp, sp);
    if (lane == 0) S.ax[warp] = sp;
  }
  __syncthreads();
  if (3 * K <= 32) {
    best = S.ax[0];
  } else {
    best = S.ax[0];
#pragma unroll
    for (int a = 1; a < 3; ++a) {
      const float ca = S.ax[a].cost;
      const int ka = S.ax[a].cand;
      if (ka != INT_MAX && (ca < best.cost || (ca == best.cost && ka < best.cand))) best = S.ax[a];
    }
  }
  int axis, plane, nl;
  BinU cu0, cu1;
  if (best.cand != INT_MAX) {
    axis = best.cand / (K - 1);
    plane = 1 + best.cand % (K - 1);
    nl = best.L.n;
    cu0 = best.L;
    cu1 = best.R;
  } else {  // no usable plane: split the range in the middle, children take the node's bounds
    axis = -1;
    plane = 0;
    nl = n / 2;
    BinU node = binu_empty();
    for (int b = 0; b < K; ++b) node = binu_join(node, binu_load(S.pbins + b * kBinVals));
    node.a0 = T.clo[0];
    node.a1 = T.clo[1];
    node.a2 = T.clo[2];
    node.b0 = T.chi[0];
    node.b1 = T.chi[1];
    node.b2 = T.chi[2];
    cu0 = node;
    cu1 = node;
  }
  const int nr = n - nl;
  cu0.n = nl;
  cu1.n = nr;
  const bool top0 = nl > A.big, top1 = nr > A.big;
  const int nch0 = (nl + CH - 1) / CH, nch1 = (nr + CH - 1) / CH;
  const int cfirst0 = T.chunk_res, cfirst1 = T.chunk_res + nch0;
  // (in a small scene the clearing too comes first: a level waits for its
  // chunk 0, and the other chunks are few)
  if (j == 0 && tid == kBlock - 1) top_reserve(A, S, slot, top0, top1, nch0, nch1);
  if (!kStaged && j == 0) {
    __syncthreads();
    top_clear(A, S);
  }
  const float cmin0[3] = {cu0.a0, cu0.a1, cu0.a2}, cmin1[3] = {cu1.a0, cu1.a1, cu1.a2};
  const float scl0[3] = {bin_scale(cu0.a0, cu0.b0, K), bin_scale(cu0.a1, cu0.b1, K), bin_scale(cu0.a2, cu0.b2, K)};
  const float scl1[3] = {bin_scale(cu1.a0, cu1.b0, K), bin_scale(cu1.a1, cu1.b1, K), bin_scale(cu1.a2, cu1.b2, K)};
  // records of the node's earlier chunks that go left: 32-chunk group
  // totals, then the chunks of this chunk's own group
  int lbase;
  if (axis >= 0) {
    const int g = j >> 5;
    const int ng = g * plane, nc = (j - 32 * g) * plane;
    int part = 0;
    for (int it = tid; it < ng + nc; it += kBlock) {
      if (it < ng) {
        const int q = it / plane, b = it - q * plane;
        part += (int)__ldcg(tscnt_at(A, T.chunk_first + q) + axis * K + b);
      } else {
        const int i2 = it - ng, q = i2 / plane, b = i2 - q * plane;
        part += (int)__ldcg(tccnt_at(A, T.chunk_first + 32 * g + q) + axis * K + b);
      }
    }
    lbase = block_sum(part, S.red);
  } else {
    lbase = min(r0, nl);
  }
  const int rbase = r0 - lbase;
  const int dfirst0 = lbase / CH, dfirst1 = rbase / CH;
  const int dnext0 = (dfirst0 + 1) * CH, dnext1 = (dfirst1 + 1) * CH;  // first positions of the next child chunks
  const float pcmin = sel3(cmin[0], cmin[1], cmin[2], axis < 0 ? 0 : axis);
  const float pscl = sel3(scl[0], scl[1], scl[2], axis < 0 ? 0 : axis);
  // stable partition of the chunk; the records of children that are big nodes
  // too are binned for them on the way.  A thread takes up to 8 consecutive
  // records: runs of one cell (the records of a building, a wall) mostly lie
  // within a thread or its neighbours, so that one scan of 12 words by
  // shuffles, which bound this step, serves 256 records and not 32.
  if (kStaged) {
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    const float4* rec = G.rec;
    const int c = (rn + kBlock - 1) / kBlock, k0 = min(tid * c, rn), k1 = min(k0 + c, rn);
    unsigned fl = 0;  // bit i: record k0 + i goes left
#pragma unroll 1
    for (int k = k0; k < k1; ++k) {
      bool left;
      if (axis >= 0) {
        const float* q = reinterpret_cast<const float*>(rec + stage_at(k)) + axis;
        left = bin_of(centre(q[0], q[4]), pcmin, pscl, K) < plane;
      } else {
        left = r0 + k < nl;
      }
      fl |= (unsigned)left << (k - k0);
    }
    __syncwarp();
    int before = 0, wtot = 0;
#pragma unroll
    for (int r = 0; r < kStage / kBlock; ++r) {
      const unsigned bal = __ballot_sync(kFull, (fl >> r) & 1u);
      before += __popc(bal & lt_mask);
      wtot += __popc(bal);
    }
    if (lane == 0) S.wl[warp] = wtot;
    __syncthreads();
    int tl = 0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
      const int v = S.wl[w];
      before += w < warp ? v : 0;
      tl += v;
    }
    int lp = before, rp = k0 - before;  // positions of the thread's next left and right record in the chunk
    CellRun run;
    run.cell = -1;
    run.n = 0;
#pragma unroll
    for (int q = 0; q < 12; ++q) run.v[q] = 0u;
    run.off[0] = run.off[1] = run.off[2] = 0u;
    for (int r = 0; r < c; ++r) {  // (uniform)
      const int k = k0 + r;
      const bool valid = k < k1;
      const bool left = (fl >> r) & 1u;
      const int pos = left ? lp : rp;
      if (valid) G.order[left ? pos : tl + pos] = (unsigned short)k;
      lp += valid && left ? 1 : 0;
      rp += valid && !left ? 1 : 0;
      if (top0 || top1) {
        const bool act = valid && (left ? top0 : top1);
        const int kk = valid ? k : 0;
        const float4 lo = rec[stage_at(kk)], hi = rec[stage_at(kk) + 1];
        const float cx = centre(lo.x, hi.x), cy = centre(lo.y, hi.y), cz = centre(lo.z, hi.z);
        const RecCodes rc = rec_codes(lo, hi, cx, cy, cz);
        const int jj = left ? (lbase + pos >= dnext0 ? 1 : 0) : (rbase + pos >= dnext1 ? 1 : 0);
        int cell = (left ? 0 : 2) + jj;
        const unsigned cb = (unsigned)cell * kCntStride, bb = left ? 0u : (unsigned)kBinWords;
        unsigned off[3];
        const float cc[3] = {cx, cy, cz};
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          const int b = bin_of(cc[a], left ? cmin0[a] : cmin1[a], left ? scl0[a] : scl1[a], K);
          off[a] = (bb + (unsigned)((a * K + b) * kBinVals)) | (cb + (unsigned)(a * K + b)) << 16;
          cell = cell * kMaxBins + b;
        }
        const bool fresh = act && cell != run.cell, out = fresh && run.cell >= 0;
        if (__any_sync(kFull, out)) {
          if (out) run_add(run, &S.cbins[0][0], &S.ccnt[0][0][0]);
          __syncwarp();
        }
        run.n = fresh ? 1u : run.n + (act ? 1u : 0u);
        run.cell = fresh ? cell : run.cell;
#pragma unroll
        for (int a = 0; a < 3; ++a) run.off[a] = fresh ? off[a] : run.off[a];
#pragma unroll
        for (int q = 0; q < 12; ++q) run.v[q] = fresh ? rc.v[q] : max(run.v[q], act ? rc.v[q] : 0u);
      }
    }
    if (top0 || top1) run_add_warp(run, &S.cbins[0][0], &S.ccnt[0][0][0]);
    __syncthreads();
    // the records leave in the order of their places, 512 bytes a warp
    for (int i = tid; i < 2 * rn; i += kBlock) {
      const int p = i >> 1;
      const bool left = p < tl;
      const int dest = left ? lbase + p : rbase + p - tl;
      const float4 v = rec[stage_at(G.order[p]) + (i & 1)];
      if (dest < (left ? nl : nr))
        dst[2 * ((size_t)T.begin + (left ? 0 : nl) + dest) + (i & 1)] = v;
      else
        set_status(A.ctl, kStBadSplit, 3);
    }
  }
  int lrun = 0, rrun = 0;
#pragma unroll
  for (int r = 0; !kStaged && r < kRegRpt; ++r) {  // a round of 256 records, a record a thread
    if (r >= A.rpt || r * kBlock >= rn) break;
    const int k = r * kBlock + tid;
    const bool valid = k < rn;
    bool left = false;
    if (valid) {
      if (axis >= 0) {
        const float cc = axis == 0 ? centre(lo[r].x, hi[r].x)
                                   : (axis == 1 ? centre(lo[r].y, hi[r].y) : centre(lo[r].z, hi[r].z));
        left = bin_of(cc, sel3(cmin[0], cmin[1], cmin[2], axis), sel3(scl[0], scl[1], scl[2], axis), K) < plane;
      } else {
        left = r0 + k < nl;
      }
    }
    __syncwarp();
    const unsigned bal = __ballot_sync(kFull, left);
    if (lane == 0) S.wl[warp] = __popc(bal);
    __syncthreads();
    int woff = 0, rtot = 0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
      const int v = S.wl[w];
      woff += w < warp ? v : 0;
      rtot += v;
    }
    const int lbefore = woff + __popc(bal & lt_mask);
    const int dest = left ? lbase + lrun + lbefore : rbase + rrun + tid - lbefore;
    const int s = left ? 0 : 1;
    if (valid) {
      if (dest < (s ? nr : nl)) {
        const size_t gp = (size_t)T.begin + (s ? nl : 0) + dest;
        dst[2 * gp] = lo[r];
        dst[2 * gp + 1] = hi[r];
      } else {
        set_status(A.ctl, kStBadSplit, 3);
      }
    }
    if (top0 || top1) {
      const bool act = valid && (s ? top1 : top0);
      const int jj = (dest / CH - (s ? dfirst1 : dfirst0)) & 1;
      const float cx = centre(lo[r].x, hi[r].x), cy = centre(lo[r].y, hi[r].y), cz = centre(lo[r].z, hi[r].z);
      const float cc[3] = {cx, cy, cz};
      const RecCodes rc = rec_codes(lo[r], hi[r], cx, cy, cz);
      int e[3], cell = s * 2 + jj;
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const int b = s ? bin_of(cc[a], cmin1[a], scl1[a], K) : bin_of(cc[a], cmin0[a], scl0[a], K);
        e[a] = a * K + b;
        cell = cell * kMaxBins + b;
      }
      bin_add_runs(act ? cell : -1, e, &S.cbins[s][0], &S.ccnt[s][jj][0], rc);
    }
    lrun += rtot;
    rrun += min(kBlock, rn - r * kBlock) - rtot;
    __syncthreads();
  }
  if (kStaged && j == 0) top_clear(A, S);
  // the children's bins and chunk counts
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    if (!(s ? top1 : top0)) continue;
    unsigned* gb = tbins_at(A, T.child_slot + s);
    for (int w = tid; w < K3 * kBinVals; w += kBlock) {
      const unsigned v = S.cbins[s][w];
      if (v) {
        if (w % kBinVals == 0)
          atomicAdd(gb + w, v);
        else
          atomicMax(gb + w, v);
      }
    }
    const int cf = s ? cfirst1 : cfirst0, df = s ? dfirst1 : dfirst0, ncs = s ? nch1 : nch0;
    for (int q = tid; q < 2 * K3; q += kBlock) {
      const int jj = q / K3, e = q - jj * K3;
      const unsigned v = S.ccnt[s][jj][e];
      const int chunk = df + jj;
      if (v && chunk < ncs) {
        atomicAdd(tccnt_at(A, cf + chunk) + e, v);
        atomicAdd(tscnt_at(A, cf + (chunk >> 5)) + e, v);
      }
    }
  }
  // the last chunk of the node to finish writes it and creates its children:
  // the count is an acquire-release add (this CTA's writes, ordered before
  // thread 0 by the barrier, are released with it; the last chunk's thread 0
  // acquires every other chunk's, among them chunk 0's plan)
  __syncthreads();
  if (tid == 0) S.last = atom_add_acq_rel(&A.tdone[slot], 1) == T.nchunk - 1;
  __syncthreads();
  if (S.last) top_emit(A, S, T, slot, epoch, nl, nr, cu0, cu1, top0, top1, nch0, nch1, cfirst0, cfirst1, ts);
}

// Write the node split by the chunks just finished and create its children
// (the CTA that finished the node's last chunk), with what chunk 0 reserved
// for them; tree facts go to the CTA's own tally (thread 0).
__device__ void top_emit(const BuildArgs& A, TopSmem& S, const TopTask& T, int slot, int epoch, int nl, int nr,
                         const BinU& cu0, const BinU& cu1, bool top0, bool top1, int nch0, int nch1, int cfirst0,
                         int cfirst1, WarpStats& ts) {
  const int tid = threadIdx.x;
  const int par = T.parity & 1;
  if (tid == 0) {
    S.np = 0;
    const int id = T.begin + nl - 1;
    const int refl = nl <= A.max_leaf ? leaf_ref(T.begin, nl) : INT_MAX;
    const int refr = nr <= A.max_leaf ? leaf_ref(T.begin + nl, nr) : INT_MAX;
    write_node(A, id, T.parent, T.side, cu0, refl, nl, cu1, refr, nr, epoch);
    note_node(ts, nl, nr, refl != INT_MAX, refr != INT_MAX, T.depth);
    for (int s = 0; s < 2; ++s) {
      const int cn = s ? nr : nl, cb = T.begin + (s ? nl : 0);
      const BinU& cu = s ? cu1 : cu0;
      S.created[s] = 0;
      if (cn <= A.max_leaf) {
        if (par == 0) S.ptask[S.np++] = make_task(cb, cn, id, s, T.depth + 1, cu, 1);  // copy to buffer 0
        continue;
      }
      if (s ? top1 : top0) {
        const int4 pl = __ldcg(A.tplan + 2 * slot + s);
        if (pl.x >= 0) {
          TopTask X;
          X.begin = cb;
          X.count = cn;
          X.parent = id;
          X.side = s;
          X.clo[0] = cu.a0;
          X.clo[1] = cu.a1;
          X.clo[2] = cu.a2;
          X.chi[0] = cu.b0;
          X.chi[1] = cu.b1;
          X.chi[2] = cu.b2;
          X.depth = T.depth + 1;
          X.nchunk = s ? nch1 : nch0;
          X.chunk_first = s ? cfirst1 : cfirst0;
          X.child_slot = pl.x;
          X.chunk_res = pl.y;
          X.parity = par ^ 1;
          A.ttask[T.child_slot + s] = X;
          S.created[s] = 1;
          S.ibase[s] = pl.z;
          continue;
        }
      }
      S.ptask[S.np++] = make_task(cb, cn, id, s, T.depth + 1, cu, par ^ 1);  // pools full: a subtree task
    }
    if (S.created[0] || S.created[1])
      atomicAdd(&A.ctl->ti_pending, (S.created[0] ? nch0 : 0) + (S.created[1] ? nch1 : 0));
  }
  __syncthreads();
  // publish the children's chunk items: each release store also publishes
  // what every thread wrote before the barrier (the tasks, the pending
  // count); meanwhile a thread of warp 1 hands the subtree-sized children to
  // the subtree queue (one reservation, release stores), so that neither
  // publication waits for the other's fence
  if (tid == 32 && S.np > 0) {
    int k = 0;
    for (int i = 0; i < S.np; ++i) {
      if (A.wsm && S.ptask[i].count <= A.wsm && S.ptask[i].count > A.max_leaf)
        push_small(A, S.ptask[i]);
      else
        S.ptask[k++] = S.ptask[i];
    }
    push_tasks(A, S.ptask, k, epoch);
  }
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    if (!S.created[s]) continue;
    const int ncs = s ? nch1 : nch0;
    for (int q = tid; q < ncs; q += kBlock) {
      A.titem[S.ibase[s] + q] = make_int2(T.child_slot + s, q);
      st_release(&A.tready[S.ibase[s] + q], epoch);
    }
  }
}

// Chunk j of big node `slot`, after checking the node's fields.
template <bool kStaged>
__device__ void top_item(const BuildArgs& A, TopSmem& S, int slot, int j, int epoch, WarpStats& ts) {
  const int tid = threadIdx.x;
  TopTask T;
  bool ok = slot >= 0 && slot < A.cap_t;
  // the node's merged bins depend on the slot only: their loads go out with
  // the task's, into shared memory once both have arrived
  constexpr int kPer = (kBinWords + kBlock - 1) / kBlock;
  const int nw = 3 * A.K * kBinVals;
  unsigned bv[kPer];
  if (ok) {
    const unsigned* gb = tbins_at(A, slot);
#pragma unroll
    for (int q = 0; q < kPer; ++q) bv[q] = tid + q * kBlock < nw ? __ldcg(gb + tid + q * kBlock) : 0u;
    T = load_top_cg(A.ttask + slot);
#pragma unroll
    for (int q = 0; q < kPer; ++q)
      if (tid + q * kBlock < nw) S.pbins[tid + q * kBlock] = bv[q];
  }
  const int n = ok ? T.count : 0;
  ok = ok && T.begin >= 0 && n > A.big && T.begin <= A.n - n && j >= 0 && j < T.nchunk && T.chunk_first >= 0 &&
       T.chunk_first + T.nchunk <= A.cap_c && T.child_slot >= 0 && T.child_slot + 2 <= A.cap_t &&
       T.chunk_res >= 0 && T.chunk_res + T.nchunk + 2 <= A.cap_c;
  if (!ok) {
    if (tid == 0) set_status(A.ctl, kStBadSplit, 4);
  } else {
    top_chunk<kStaged>(A, S, T, slot, j, epoch, ts);
  }
}

template <bool kStaged>
__device__ void top_loop(const BuildArgs& A, TopSmem& S, int epoch) {
  WarpStats ts{0, 0, 0, 0};  // thread 0's tally of the nodes this CTA wrote
  for (;;) {
    if (threadIdx.x == 0) S.item = claim_item(A, epoch);
    __syncthreads();
    const int2 it = S.item;
    __syncthreads();
    if (it.x < 0) break;
    top_item<kStaged>(A, S, it.x, it.y, epoch, ts);
    __syncthreads();
    // release: the subtree tasks this item pushed are counted before the
    // item stops counting (the warps' exit test reads ti_pending first)
    if (threadIdx.x == 0) red_release_add(&A.ctl->ti_pending, -1);
  }
  if (threadIdx.x == 0) {
    if (ts.n_int) atomicAdd(&A.ctl->n_internal, ts.n_int);
    if (ts.n_leaf) atomicAdd(&A.ctl->n_leaves, ts.n_leaf);
    if (ts.big) atomicMax(&A.ctl->max_leaf_size, ts.big);
    if (ts.deep) atomicMax(&A.ctl->depth2, ts.deep);
  }
}

// ------------------------------------------------------------------ small subtrees
// A node of at most 32 triangles is finished by one warp in registers: lane
// j holds record j of the node's range in Morton order.  Every split of the
// subtree is the minimum of Eq. 2 over all splits of that order, evaluated
// from warp scans of the records' boxes; ranges never move, so there is no
// partition step, and all nodes of one level of the subtree are split
// together (scans that stop at each node's bounds).  Nothing in it branches
// by lane: where lanes part, every shuffle after that costs a rendezvous
// (with branches in the scans, the node writes and the load of a short
// node's records a node took 20k cycles of a busy SM, now 9k).
struct Box6 {
  float l0, l1, l2, h0, h1, h2;
};
__device__ __forceinline__ Box6 box_empty() { return {FLT_MAX, FLT_MAX, FLT_MAX, -FLT_MAX, -FLT_MAX, -FLT_MAX}; }
__device__ __forceinline__ Box6 box_join(const Box6& a, const Box6& b) {
  return {fminf(a.l0, b.l0), fminf(a.l1, b.l1), fminf(a.l2, b.l2),
          fmaxf(a.h0, b.h0), fmaxf(a.h1, b.h1), fmaxf(a.h2, b.h2)};
}
__device__ __forceinline__ Box6 box_sel(bool c, const Box6& a, const Box6& b) {
  return {c ? a.l0 : b.l0, c ? a.l1 : b.l1, c ? a.l2 : b.l2, c ? a.h0 : b.h0, c ? a.h1 : b.h1, c ? a.h2 : b.h2};
}
__device__ __forceinline__ Box6 box_shfl_down(const Box6& a, int o) {
  return {__shfl_down_sync(kFull, a.l0, o), __shfl_down_sync(kFull, a.l1, o), __shfl_down_sync(kFull, a.l2, o),
          __shfl_down_sync(kFull, a.h0, o), __shfl_down_sync(kFull, a.h1, o), __shfl_down_sync(kFull, a.h2, o)};
}
__device__ __forceinline__ Box6 box_shfl(const Box6& a, int src) {
  return {__shfl_sync(kFull, a.l0, src), __shfl_sync(kFull, a.l1, src), __shfl_sync(kFull, a.l2, src),
          __shfl_sync(kFull, a.h0, src), __shfl_sync(kFull, a.h1, src), __shfl_sync(kFull, a.h2, src)};
}


// Lane j: record j (box x) of the node of n records at gbase.  A lane is the
// split position of at most one node of the subtree, so it keeps that node
// (its own prefix and suffix unions are the children's boxes) and its
// children's references, which it and its right neighbour know one level
// later; all nodes are written together at the end.
__device__ __forceinline__ void micro_build(const BuildArgs& A, const Box6& x, int n, int gbase, int parent, int side,
                                            int depth, int epoch, WarpStats& ws) {
  const int lane = threadIdx.x & 31;
  // every lane follows the node its record belongs to: range [b, e), its
  // parent and depth; lanes past n sit in empty ranges of their own
  const bool valid = lane < n;
  int b = valid ? 0 : lane, e = valid ? n : lane + 1;
  int par = parent, dep = depth;
  // the node that this lane splits
  Box6 nl = box_empty(), nr = box_empty();
  int ob = 0, oe = 0, opar = 0, refl = 0, refr = 0;
  bool own = false, fresh = false, root = false;
#pragma unroll 1
  for (int level = 0; level < 32; ++level) {
    const bool active = valid && e - b > A.max_leaf;
    if (!__any_sync(kFull, active)) break;
    const int width = (int)__reduce_max_sync(kFull, active ? (unsigned)(e - b) : 0u);
    // unions of the records from the start of the lane's node up to the lane
    // (ip) and from the lane to the node's end (is): scans that stop at the
    // node's bounds, all nodes of the level at once
    Box6 ip = x, is = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      if (o >= width) break;
      // a lane past the node's bound reads the bound's own union instead
      // (unions are idempotent, so nothing has to be selected)
      ip = box_join(ip, box_shfl(ip, max(lane - o, b)));
      is = box_join(is, box_shfl(is, min(lane + o, e - 1)));
    }
    const Box6 sufn = box_shfl_down(is, 1);  // records after the lane, within the node
    const Box6 node = box_shfl(ip, e - 1);   // the whole node
    // candidate: the lane is the last left record
    const float c = eq2_cost(make_float3(ip.l0, ip.l1, ip.l2), make_float3(ip.h0, ip.h1, ip.h2), lane - b + 1,
                             make_float3(sufn.l0, sufn.l1, sufn.l2), make_float3(sufn.h0, sufn.h1, sufn.h2),
                             e - lane - 1, make_float3(node.l0, node.l1, node.l2),
                             make_float3(node.h0, node.h1, node.h2), A.cp);
    const bool ok = active && lane + 1 < e && c < INFINITY;
    // lowest cost of the node (found at its last lane), and the lowest
    // position that has it
    const float cost = ok ? c : INFINITY;
    float least = cost;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      if (o >= width) break;
      least = fminf(least, __shfl_sync(kFull, least, max(lane - o, b)));
    }
    least = __shfl_sync(kFull, least, e - 1);
    const unsigned at = __ballot_sync(kFull, ok && cost == least) & (0xffffffffu >> (32 - e)) & (0xffffffffu << b);
    const int q = !active ? lane : (at ? __ffs(at) - 1 : (b + e) / 2 - 1);  // no finite cost: middle
    // the references of the nodes of this level, for those split on the last
    const int ref = active ? gbase + q : leaf_ref(gbase + b, e - b), rref = __shfl_down_sync(kFull, ref, 1);
    refl = fresh ? ref : refl;
    refr = fresh ? rref : refr;
    fresh = active && lane == q;
    own = own || fresh;
    root = root || (fresh && level == 0);
    nl = box_sel(fresh, ip, nl);
    nr = box_sel(fresh, sufn, nr);
    ob = fresh ? b : ob;
    oe = fresh ? e : oe;
    opar = fresh ? par : opar;
    // follow the child holding this lane's record
    par = active ? gbase + q : par;
    dep += active ? 1 : 0;
    b = active && lane > q ? q + 1 : b;
    e = active && lane <= q ? q + 1 : e;
  }
  const int ref = leaf_ref(gbase + b, e - b), rref = __shfl_down_sync(kFull, ref, 1);
  refl = fresh ? ref : refl;
  refr = fresh ? rref : refr;
  // tree facts: every lane's last node is a leaf, one more leaf than nodes
  const int nn = __popc(__ballot_sync(kFull, own));
  ws.n_int += nn;
  ws.n_leaf += nn ? nn + 1 : 0;
  ws.big = max(ws.big, (int)__reduce_max_sync(kFull, valid ? (unsigned)(e - b) : 0u));
  ws.deep = max(ws.deep, (int)__reduce_max_sync(kFull, valid ? (unsigned)dep : 0u));
  if (own) {
    const int id = gbase + lane;
    Node2 nd;
    nd.a_lo = make_float4(nl.l0, nl.l1, nl.l2, __int_as_float(refl));
    nd.a_hi = make_float4(nl.h0, nl.h1, nl.h2, __int_as_float(lane + 1 - ob));
    nd.b_lo = make_float4(nr.l0, nr.l1, nr.l2, __int_as_float(refr));
    nd.b_hi = make_float4(nr.h0, nr.h1, nr.h2, __int_as_float(oe - lane - 1));
    A.node2[id] = nd;
    A.link2[id] = make_int2(opar, epoch);
    if (root) {
      if (parent < 0)
        A.ctl->root_ref = id;
      else if (parent < A.n - 1)
        *(side == 0 ? &A.node2[parent].a_lo.w : &A.node2[parent].b_lo.w) = __int_as_float(id);
      else
        set_status(A.ctl, kStBadLink, 4);
    }
  }
  __syncwarp();
}

// A node of 2 .. 32 records at src (shared memory, this warp's): order them
// by (Morton key, id), each lane counting the records before its own, write
// them to buffer 0 at gbegin in that order (the final order of their leaves)
// and build the subtree.
__device__ __forceinline__ void micro_sort_build(const BuildArgs& A, float4* src, int gbegin, int n, int parent,
                                                 int side, int depth, int epoch, WarpStats& ws) {
  const int lane = threadIdx.x & 31;
  const int k = min(lane, n - 1);
  float4 lo = src[2 * k], hi = src[2 * k + 1];
  const unsigned key = __float_as_uint(hi.w), id = __float_as_uint(lo.w);
  int rank = 0;
#pragma unroll 4
  for (int j = 0; j < n; ++j) {
    const unsigned kj = __float_as_uint(src[2 * j + 1].w), ij = __float_as_uint(src[2 * j].w);
    rank += (kj < key || (kj == key && ij < id)) ? 1 : 0;
  }
  __syncwarp();
  if (lane < n) {
    src[2 * rank] = lo;
    src[2 * rank + 1] = hi;
  }
  __syncwarp();
  lo = src[2 * k];
  hi = src[2 * k + 1];
  if (lane < n) {
    float4* p = A.rec[0] + 2 * ((size_t)gbegin + lane);
    p[0] = lo;
    p[1] = hi;
  }
  __syncwarp();
  const Box6 x = box_sel(lane < n, Box6{lo.x, lo.y, lo.z, hi.x, hi.y, hi.z}, box_empty());
  micro_build(A, x, n, gbegin, parent, side, depth, epoch, ws);
}

// ------------------------------------------------------------------ subtree queue
// One thread takes the next queue slot and waits for it to be filled (the
// other threads of the CTA wait at a barrier; nothing warp-synchronous runs
// in this loop).  Returns false when the queue is drained (no big node and
// no task pending) or the build failed.  The wait is bounded: spin_limit
// polls without progress set a timeout status.
__device__ bool claim_task(const BuildArgs& A, int epoch, Task& t) {
  const int s = atomicAdd(&A.ctl->qa_head, 1);
  int seen = -1;
  for (int it = 0;; ++it) {
    if (s < A.qa_cap && ld_acquire(&A.qa_ready[s]) == epoch) {
      const int4* q = reinterpret_cast<const int4*>(A.qa + s);
      const int4 a = __ldcg(q), b = __ldcg(q + 1), c = __ldcg(q + 2);
      t.begin = a.x;
      t.count = a.y;
      t.parent = a.z;
      t.side = a.w;
      t.clo[0] = __int_as_float(b.x);
      t.clo[1] = __int_as_float(b.y);
      t.clo[2] = __int_as_float(b.z);
      t.depth = b.w;
      t.chi[0] = __int_as_float(c.x);
      t.chi[1] = __int_as_float(c.y);
      t.chi[2] = __int_as_float(c.z);
      t.pad = c.w;
      return true;
    }
    if ((it & 3) == 0) {
      // done when no big node is left and then no subtree task either
      if (ld_acquire(&A.ctl->ti_pending) == 0 && ld_volatile(&A.ctl->qa_pending) == 0) return false;
      if (ld_volatile(&A.ctl->status) != 0) return false;
      const int prog = ld_volatile(&A.ctl->qa_tail) + ld_volatile(&A.ctl->ti_head);
      if (prog != seen) {  // work moved: restart the no-progress budget
        seen = prog;
        it = 0;
      }
    }
    if (it > A.spin_limit) {
      set_status(A.ctl, kStQueueTimeout, 1);
      return false;
    }
    __nanosleep(200);
  }
}

// ------------------------------------------------------------------ subtrees in shared memory
// A CTA takes a task of at most kSubMax records, loads its records into
// shared memory once and builds the subtree there.  Every node of more than
// 32 records is split by the whole CTA; the larger child stays with the CTA
// and the smaller one, if it has more than 32 records, goes back to the
// device queue (records to buffer 1) for an idle CTA, so a subtree spreads
// over the SMs as it branches.  Nodes of at most 32 records are collected
// and finished at the end by the warps in parallel, in registers.  Records
// leave shared memory only as leaves, in their final order, into buffer 0.
constexpr int kSubMax = 1024;            // records of a subtree built in shared memory
constexpr int kWarpMax = 128;            // largest node that a warp of k_small takes (4 records per lane)
constexpr int kMicroList = kSubMax / 2;  // nodes of at most 32 records (>= 2 each, disjoint)
constexpr int kNodeThread = kBlock - 32;  // writes a CTA split's node: the last warp's first lane, so that the
                                         // warps that evaluate Eq. 2 do not wait for its queue push
constexpr int kBoxVals = 7;              // a subtree bin: count, box lo (complemented codes), box hi
constexpr int kCtaBinWords = 3 * kMaxBins * kBoxVals + 4 * kBinVals;  // bins, then two sets of children's unions
static_assert(kSubMax <= kBlock * 4, "a CTA partition keeps at most 4 records per thread");
static_assert(kSubMax <= 1024 && kMicro < 64, "packed small-node fields");

// A node of the subtree: local range [b, b + n) of shared buffer `par`,
// parent id, side, depth, centroid bounds.
struct SubNode {
  int b, n, parent, side, depth, par;
  float clo[3], chi[3];
};

struct SubSmem {
  float4 rec[2][2 * kSubMax];
  unsigned bins[kCtaBinWords];
  int2 ml[kMicroList];  // nodes of at most 32: (parent, b | n << 10 | side << 16 | par << 17 | depth << 18)
  Task task;
  int red[kWarps];
  int2 pick[3];     // the split Eq. 2 chose on each group of axes: candidate, records on the left
  float pcost[3];
  int mord[32];  // the order in which the warps take the small nodes (largest first)
  float4 pbox[3][3];  // and the boxes of its children (left lo, hi; right lo, hi)
  int nm, mnext, got;
};

__device__ __forceinline__ SubNode sub_node(int b, int n, int parent, int side, int depth, int par, const BinU& u) {
  SubNode x;
  x.b = b;
  x.n = n;
  x.parent = parent;
  x.side = side;
  x.depth = depth;
  x.par = par;
  x.clo[0] = u.a0;
  x.clo[1] = u.a1;
  x.clo[2] = u.a2;
  x.chi[0] = u.b0;
  x.chi[1] = u.b1;
  x.chi[2] = u.b2;
  return x;
}

// Packed node of at most 32 records; depth is relative to the task (a
// subtree of kSubMax records is less than kSubMax deep).
__device__ __forceinline__ int2 micro_pack(int b, int n, int parent, int side, int depth, int par) {
  return make_int2(parent, b | (n << 10) | (side << 16) | (par << 17) | (depth << 18));
}

// Bin the run of records [k0, k1) of src on all three axes (count and box
// per bin).  Consecutive records of the Morton order mostly share a bin, so
// the run is accumulated in registers and each stretch of equal bins costs
// one flush of shared-memory atomics.
__device__ __forceinline__ void flush_box(unsigned* e, const unsigned* acc) {
  atomicAdd(e, acc[0]);
#pragma unroll
  for (int q = 1; q < kBoxVals; ++q) atomicMax(e + q, acc[q]);
}
template <bool kGlobal>
__device__ __forceinline__ float4 rec_load(const float4* p) {
  return kGlobal ? __ldcg(p) : *p;
}
template <bool kGlobal>
__device__ __forceinline__ void bin_run(unsigned* bins, const float4* src, int k0, int k1, int K, const float* cmin,
                                        const float* scl) {
  int key[3] = {-1, -1, -1};
  unsigned acc[3][kBoxVals];
  for (int k = k0; k < k1; ++k) {
    const float4 lo = rec_load<kGlobal>(src + 2 * k), hi = rec_load<kGlobal>(src + 2 * k + 1);
    const unsigned c6[6] = {~ucode(lo.x), ~ucode(lo.y), ~ucode(lo.z), ucode(hi.x), ucode(hi.y), ucode(hi.z)};
    const float cc[3] = {centre(lo.x, hi.x), centre(lo.y, hi.y), centre(lo.z, hi.z)};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const int kk = bin_of(cc[a], cmin[a], scl[a], K);
      if (kk != key[a]) {
        if (key[a] >= 0) flush_box(bins + (a * K + key[a]) * kBoxVals, acc[a]);
        key[a] = kk;
        acc[a][0] = 1u;
#pragma unroll
        for (int q = 0; q < 6; ++q) acc[a][1 + q] = c6[q];
      } else {
        acc[a][0] += 1u;
#pragma unroll
        for (int q = 0; q < 6; ++q) acc[a][1 + q] = max(acc[a][1 + q], c6[q]);
      }
    }
  }
#pragma unroll
  for (int a = 0; a < 3; ++a)
    if (key[a] >= 0) flush_box(bins + (a * K + key[a]) * kBoxVals, acc[a]);
}

// A warp's union of its lanes' 13 words (count, then the codes of a record).
__device__ __forceinline__ void acc13_warp(unsigned* v) {
  v[0] = __reduce_add_sync(kFull, v[0]);
#pragma unroll
  for (int q = 1; q < kBinVals; ++q) v[q] = __reduce_max_sync(kFull, v[q]);
}

// Copy a leaf's records from shared memory (or buffer 1) to buffer 0 (their
// final place).
template <bool kGlobal>
__device__ __forceinline__ void leaf_out(const BuildArgs& A, const float4* src, int gpos, int n, int t0, int nt) {
  for (int k = t0; k < 2 * n; k += nt) A.rec[0][2 * (size_t)gpos + k] = rec_load<kGlobal>(src + k);
}


// Split node X of the subtree with the whole CTA (split `it` of the task's
// chain): bins (count and box) in one shared array, each thread binning a
// run of records (thread (w, l) takes run l * 8 + w, so the lanes of a warp
// work far apart); Eq. 2 evaluated by one to three warps, the axes divided
// among them, their choices read by all from shared memory; stable partition
// by a block scan, which also gathers both children's unions (into one of two
// sets, alternating with `it`) and clears the bins and the other set for
// the next split.  One thread writes the node and routes the other children:
// the smaller one of more than 32 records goes to the device queue, those
// of at most 32 to the small-node list.  If the larger child has more than
// 32 records, every thread makes it X (true) and goes on without a barrier.
// Bound by the latency of its dependent steps: a split of 33 .. 64 records
// takes 7.0k cycles (11.9k when one warp evaluated all axes, with branches
// that left it in two parts), of which Eq. 2 2.7k (6.6k).
//
// kGlobal: the same split of a node too large for shared memory (more than
// kSubMax records: big = T / 4096 of a scene of more than 4M triangles, or a
// big node whose pools were full), its records in global buffer X.par, the
// children's in the other; both children that are not leaves become tasks
// except the larger one, which is X again whatever its size (true while it
// is still too large).
template <bool kGlobal>
__device__ __forceinline__ bool cta_split(const BuildArgs& A, SubSmem& S, SubNode& X, int it, int gbegin, int tdepth,
                                          int epoch, WarpStats& ws) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int K = A.K, n = X.n, p = X.par;
  const int nbw = 3 * K * kBoxVals;
  unsigned* cb = S.bins;  // zero on entry
  unsigned* cu = cb + nbw + (it & 1) * 2 * kBinVals;  // the children's unions, 2 x 13 words (zero on entry)
  unsigned* cu_next = cb + nbw + ((it + 1) & 1) * 2 * kBinVals;
  const float4* src = kGlobal ? A.rec[p] + 2 * ((size_t)gbegin + X.b) : S.rec[p] + 2 * X.b;
  float4* dst = kGlobal ? A.rec[p ^ 1] + 2 * ((size_t)gbegin + X.b) : S.rec[p ^ 1] + 2 * X.b;
  float cmin[3], scl[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    cmin[a] = X.clo[a];
    scl[a] = bin_scale(X.clo[a], X.chi[a], K);
  }
  // thread t owns records [t c, t c + c) for the partition; runs for the
  // bins use the spread order
  const int c = (n + kBlock - 1) / kBlock;
  {
    const int r = lane * kWarps + warp, k0 = min(r * c, n), k1 = min(k0 + c, n);
    bin_run<kGlobal>(cb, src, k0, k1, K, cmin, scl);
  }
  __syncthreads();
  // Eq. 2: as many axes per warp as 32 lanes hold, warp g the g-th group of
  // them (the others wait at the barrier); every thread then takes the lower
  // cost, the lower candidate among equal costs
  const int apw = min(3, 32 / K), ngr = (2 + apw) / apw;
  if (__any_sync(kFull, warp < ngr)) {
    const int a0 = warp * apw, m = min(3 - a0, apw);
    Split best;
    split_none(best);
    if (m >= 2 || __any_sync(kFull, sel3(scl[0], scl[1], scl[2], a0) > 0.f))
      eval_seg<kBoxVals, false>(cb + a0 * K * kBoxVals, K, n, a0, m, A.cp, best);
    if (lane == 0) {
      S.pcost[warp] = best.cost;
      S.pick[warp] = make_int2(best.cand, best.L.n);
      // both children's boxes: the unions of the bins' boxes on each side
      S.pbox[warp][0] = make_float4(best.L.l0, best.L.l1, best.L.l2, best.L.h0);
      S.pbox[warp][1] = make_float4(best.L.h1, best.L.h2, best.R.l0, best.R.l1);
      S.pbox[warp][2] = make_float4(best.R.l2, best.R.h0, best.R.h1, best.R.h2);
    }
  }
  __syncthreads();
  int win = 0;
  int2 pick = S.pick[0];
  float pcost = S.pcost[0];
  for (int g = 1; g < ngr; ++g) {
    const float c = S.pcost[g];
    const int2 q = S.pick[g];
    const bool lower = c < pcost || (c == pcost && q.x < pick.x);
    win = lower ? g : win;
    pick = lower ? q : pick;
    pcost = lower ? c : pcost;
  }
  int axis, plane, nl;
  if (pick.x != INT_MAX) {
    axis = pick.x / (K - 1);
    plane = 1 + pick.x % (K - 1);
    nl = pick.y;
  } else {
    axis = -1;
    plane = 0;
    nl = n / 2;
  }
  const float acmin = sel3(cmin[0], cmin[1], cmin[2], axis < 0 ? 0 : axis);
  const float ascl = sel3(scl[0], scl[1], scl[2], axis < 0 ? 0 : axis);
  const int k0 = min(tid * c, n);
  const int k1 = min(k0 + c, n);
  auto goes_left = [&](int k) {
    if (axis < 0) return k < nl;
    const float* q = reinterpret_cast<const float*>(src + 2 * k) + axis;
    const float cc = kGlobal ? centre(__ldcg(q), __ldcg(q + 4)) : centre(q[0], q[4]);
    return bin_of(cc, acmin, ascl, K) < plane;
  };
  int cnt = 0;
  // A node in shared memory gives a thread at most 4 records (1024 / 256): the
  // sides are kept as bits, so that the partition below does not bin each
  // record again (medium city: 16 bins 187.5 -> 184 us, 8 bins 181 -> 177).
  unsigned fl = 0;
#pragma unroll 1
  for (int k = k0; k < k1; ++k) {
    const bool l = goes_left(k);
    cnt += l;
    fl |= (unsigned)l << ((k - k0) & 31);
  }
  int inc = cnt;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int u = __shfl_up_sync(kFull, inc, o);
    if (lane >= o) inc += u;
  }
  if (lane == 31) S.red[warp] = inc;
  __syncthreads();
  int before = 0, total = 0;
#pragma unroll
  for (int w = 0; w < kWarps; ++w) {
    const int v = S.red[w];
    before += w < warp ? v : 0;
    total += v;
  }
  int lb = before + inc - cnt, rb = k0 - lb;
  // the bins are done with (Eq. 2 read them before the barriers above):
  // clear them, and the other unions, for the next split
  for (int w = tid; w < nbw; w += kBlock) cb[w] = 0u;
  if (tid < 2 * kBinVals) cu_next[tid] = 0u;
  // the larger child of more than 32 records stays; the other one of more
  // than 32 goes to the device queue, where an idle CTA takes it, so the
  // subtree spreads over the SMs as it branches: its records go straight to
  // buffer 1 here instead of to shared memory
  const int nr = n - nl;
  const int keep = nl >= nr ? 0 : 1;
  const int lim = kGlobal ? kSubMax : (A.wsm ? A.wsm : kMicro);  // the chain ends at nodes of this size
  bool ex[2];  // children that leave shared memory: the smaller one, to the queue, and k_small's nodes
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    const int cn = s ? nr : nl;
    ex[s] = cn > lim ? s != keep : A.wsm && cn > A.max_leaf;
  }
  float4* gx = A.rec[1] + 2 * ((size_t)gbegin + X.b);
  unsigned ua[kBinVals], ub[kBinVals];
#pragma unroll
  for (int q = 0; q < kBinVals; ++q) ua[q] = ub[q] = 0u;
#pragma unroll 1
  for (int k = k0; k < k1; ++k) {
    const float4 rl = rec_load<kGlobal>(src + 2 * k), rh = rec_load<kGlobal>(src + 2 * k + 1);
    const bool left = kGlobal ? goes_left(k) : ((fl >> (k - k0)) & 1u) != 0;
    const int d = left ? lb++ : nl + rb++;
    if (d < n) {
      if (kGlobal) {
        __stcg(dst + 2 * d, rl);
        __stcg(dst + 2 * d + 1, rh);
      } else if (left ? ex[0] : ex[1]) {
        __stcg(gx + 2 * d, rl);
        __stcg(gx + 2 * d + 1, rh);
      } else {
        dst[2 * d] = rl;
        dst[2 * d + 1] = rh;
      }
    }
    const RecCodes rc = rec_codes(rl, rh, centre(rl.x, rh.x), centre(rl.y, rh.y), centre(rl.z, rh.z));
    const unsigned ml = left ? 0xffffffffu : 0u;  // the codes of the other side count as empty (0)
    ua[0] += left ? 1u : 0u;
    ub[0] += left ? 0u : 1u;
#pragma unroll
    for (int q = 0; q < 12; ++q) {
      ua[1 + q] = max(ua[1 + q], rc.v[q] & ml);
      ub[1 + q] = max(ub[1 + q], rc.v[q] & ~ml);
    }
  }
  // the children's unions: with a plane, count and box are known (Eq. 2's
  // scans) and only the centre bounds (words 7..12) are gathered; without
  // one, all 13 words
  if (axis >= 0) {
#pragma unroll
    for (int q = 7; q < kBinVals; ++q) {
      ua[q] = __reduce_max_sync(kFull, ua[q]);
      ub[q] = __reduce_max_sync(kFull, ub[q]);
    }
    if (lane == 0) {
#pragma unroll
      for (int q = 7; q < kBinVals; ++q) {
        atomicMax(cu + q, ua[q]);
        atomicMax(cu + kBinVals + q, ub[q]);
      }
    }
  } else {
    acc13_warp(ua);
    acc13_warp(ub);
    if (lane == 0) {
      atomicAdd(cu, ua[0]);
      atomicAdd(cu + kBinVals, ub[0]);
#pragma unroll
      for (int q = 1; q < kBinVals; ++q) {
        atomicMax(cu + q, ua[q]);
        atomicMax(cu + kBinVals + q, ub[q]);
      }
    }
  }
  __syncthreads();
  BinU L, R;
  if (axis >= 0) {
    const float4 b0 = S.pbox[win][0], b1 = S.pbox[win][1], b2 = S.pbox[win][2];
    L = {nl, b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, uval(~cu[7]), uval(~cu[8]), uval(~cu[9]), uval(cu[10]),
         uval(cu[11]), uval(cu[12])};
    R = {n - nl, b1.z, b1.w, b2.x, b2.y, b2.z, b2.w, uval(~cu[kBinVals + 7]), uval(~cu[kBinVals + 8]),
         uval(~cu[kBinVals + 9]), uval(cu[kBinVals + 10]), uval(cu[kBinVals + 11]), uval(cu[kBinVals + 12])};
  } else {
    L = binu_load(cu);
    R = binu_load(cu + kBinVals);
  }
  const bool leafl = nl <= A.max_leaf, leafr = nr <= A.max_leaf;
  if (!kGlobal || p == 0) {  // (a leaf of a global split from buffer 1 is in buffer 0 already)
    if (leafl) leaf_out<kGlobal>(A, dst, gbegin + X.b, nl, tid, kBlock);
    if (leafr) leaf_out<kGlobal>(A, dst + 2 * nl, gbegin + X.b + nl, nr, tid, kBlock);
  }
  const int id = gbegin + X.b + nl - 1;
  if (tid == kNodeThread) {
    if (total != nl) set_status(A.ctl, kStBadSplit, 6);
    write_node(A, id, X.parent, X.side, L, leafl ? leaf_ref(gbegin + X.b, nl) : INT_MAX, nl, R,
               leafr ? leaf_ref(gbegin + X.b + nl, nr) : INT_MAX, nr, epoch);
    note_node(ws, nl, nr, leafl, leafr, X.depth);
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      const int cn = s ? nr : nl, b = X.b + (s ? nl : 0);
      if (cn <= A.max_leaf) continue;
      const bool small = A.wsm && cn <= A.wsm;
      if (kGlobal) {
        const Task c = make_task(gbegin + b, cn, id, s, X.depth + 1, s ? R : L, p ^ 1);
        if (s == keep) continue;
        if (small)
          push_small(A, c);
        else
          push_task(A, c, epoch);
      } else if (ex[s] && small) {
        push_small(A, make_task(gbegin + b, cn, id, s, X.depth + 1, s ? R : L, 1));
      } else if (ex[s]) {
        // the records written to buffer 1 by every thread are ordered before
        // this thread by the barrier; push_task's release store publishes them
        push_task(A, make_task(gbegin + b, cn, id, s, X.depth + 1, s ? R : L, 1), epoch);
      } else if (cn <= kMicro) {
        if (S.nm < kMicroList)
          S.ml[S.nm++] = micro_pack(b, cn, id, s, X.depth + 1 - tdepth, p ^ 1);
        else
          set_status(A.ctl, kStQueueOverflow, 4);
      }
    }
  }
  // every thread takes the kept child from the unions it read (no barrier:
  // the node thread's write and release fence overlap the next split's
  // binning, which reads only the kept child's records)
  if (!kGlobal && (keep ? nr : nl) <= lim) return false;
  X = sub_node(X.b + (keep ? nl : 0), keep ? nr : nl, id, keep, X.depth + 1, p ^ 1, keep ? R : L);
  return !kGlobal || X.n > kSubMax;
}

// The warps finish the collected nodes of at most 32 records, one node per
// warp at a time (no node is added any more).
__device__ __forceinline__ void micro_phase(const BuildArgs& A, SubSmem& S, int gbegin, int tdepth, int epoch,
                                            WarpStats& ws) {
  const int lane = threadIdx.x & 31;
  const int nm = S.nm;
  // more nodes than warps (up to 32): warp 0 orders them largest first, so
  // that the last round of builds holds the quickest ones
  const bool order = nm > kWarps && nm <= 32;
  if (order) {
    if (__any_sync(kFull, threadIdx.x < 32)) {
      unsigned key = lane < nm ? ((unsigned)(63 - ((S.ml[lane].y >> 10) & 63)) << 8) | (unsigned)lane : 0xffffffffu;
#pragma unroll 1
      for (int k = 2; k <= 32; k <<= 1) {
#pragma unroll 1
        for (int jj = k >> 1; jj > 0; jj >>= 1) {
          const unsigned ok = __shfl_xor_sync(kFull, key, jj);
          const bool up = (lane & k) == 0, lower = (lane & jj) == 0;
          if ((lower == up) ? (ok < key) : (ok > key)) key = ok;
        }
      }
      S.mord[lane] = (int)(key & 255u);
    }
    __syncthreads();
  }
  for (;;) {
    int i = 0;
    if (lane == 0) i = atomicAdd(&S.mnext, 1);
    i = __shfl_sync(kFull, i, 0);
    if (i >= nm) break;
    const int2 m = S.ml[order ? S.mord[i] : i];
    const int f = m.y;
    const int b = f & 1023, n = __shfl_sync(kFull, (f >> 10) & 63, 0), side = (f >> 16) & 1, par = (f >> 17) & 1,
              dep = f >> 18;
    micro_sort_build(A, S.rec[par] + 2 * b, gbegin + b, n, m.x, side, tdepth + dep, epoch, ws);
  }
}

// Task t as a node of its own range, its records in buffer par.
__device__ __forceinline__ SubNode task_node(const Task& t, int par) {
  SubNode X;
  X.b = 0;
  X.n = t.count;
  X.parent = t.parent;
  X.side = t.side;
  X.depth = t.depth;
  X.par = par;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    X.clo[a] = t.clo[a];
    X.chi[a] = t.chi[a];
  }
  return X;
}

// Build the subtree of task t (max_leaf < t.count <= kSubMax) in shared
// memory with the whole CTA.
__device__ void sub_tree(const BuildArgs& A, SubSmem& S, const Task& t, int epoch, WarpStats& ws) {
  const int tid = threadIdx.x;
  const int n = t.count;
  const float4* g = A.rec[t.pad & 1] + 2 * (size_t)t.begin;
  for (int k = tid; k < 2 * n; k += kBlock) S.rec[0][k] = __ldcg(g + k);
  // the first split's bins and unions start at zero
  for (int w = tid; w < kCtaBinWords; w += kBlock) S.bins[w] = 0u;
  __syncthreads();
  if (tid == kNodeThread) {
    S.nm = 0;
    S.mnext = 0;
    if (n <= kMicro) S.ml[S.nm++] = micro_pack(0, n, t.parent, t.side, 0, 0);
  }
  if (n > kMicro) {  // the chain of larger children, split by the whole CTA
    SubNode X = task_node(t, 0);
    for (int it = 0; cta_split<false>(A, S, X, it, t.begin, t.depth, epoch, ws); ++it) {
    }
  }
  __syncthreads();  // the node thread's last additions to the small-node list
  micro_phase(A, S, t.begin, t.depth, epoch, ws);
  __syncthreads();
}

// The subtree role of every CTA: take a task from the queue, build its
// subtree (tasks of more than kSubMax records are first split in global
// memory, down to a part that fits), repeat until the queue is drained.
__device__ void sub_loop(const BuildArgs& A, SubSmem& S, int epoch) {
  const int tid = threadIdx.x, lane = tid & 31;
  WarpStats ws{0, 0, 0, 0};
  for (;;) {
    if (tid == 0) S.got = claim_task(A, epoch, S.task);
    __syncthreads();
    const bool got = S.got;
    Task t = S.task;
    __syncthreads();
    if (!got) break;
    const int par = t.pad & 1;
    if (t.begin < 0 || t.count < 1 || t.begin > A.n - t.count) {
      if (tid == 0) set_status(A.ctl, kStBadSplit, 5);
    } else if (t.count <= A.max_leaf) {
      // a leaf made by a top level whose records sit in buffer 1
      if (par)
        for (int k = tid; k < 2 * t.count; k += kBlock)
          A.rec[0][2 * (size_t)t.begin + k] = __ldcg(A.rec[1] + 2 * (size_t)t.begin + k);
    } else {
      if (t.count > kSubMax) {
        // split in global memory, down to a part that fits
        for (int w = tid; w < kCtaBinWords; w += kBlock) S.bins[w] = 0u;
        __syncthreads();
        SubNode X = task_node(t, par);
        for (int it = 0; cta_split<true>(A, S, X, it, t.begin, t.depth, epoch, ws); ++it) {
        }
        t.begin += X.b;
        t.count = X.n;
        t.parent = X.parent;
        t.side = X.side;
        t.depth = X.depth;
        t.pad = X.par;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          t.clo[a] = X.clo[a];
          t.chi[a] = X.chi[a];
        }
        __syncthreads();
      }
      sub_tree(A, S, t, epoch, ws);
    }
    __syncthreads();
    // the pushes of this task counted first, so this never reads zero early
    if (tid == 0) atomicSub(&A.ctl->qa_pending, 1);
  }
  if (lane == 0) {
    if (ws.n_int) atomicAdd(&A.ctl->n_internal, ws.n_int);
    if (ws.n_leaf) atomicAdd(&A.ctl->n_leaves, ws.n_leaf);
    if (ws.big) atomicMax(&A.ctl->max_leaf_size, ws.big);
    if (ws.deep) atomicMax(&A.ctl->depth2, ws.deep);
  }
}

// Joins the box (lo, hi) to x where a == b, as predicated instructions: a
// branch here would cost a reconvergence per record.
__device__ __forceinline__ void binb_join_if(BinB& x, unsigned a, unsigned b, float4 lo, float4 hi) {
  asm("{\n\t.reg .pred p;\n\tsetp.eq.u32 p, %7, %8;\n\t@p add.s32 %0, %0, 1;\n\t@p min.f32 %1, %1, %9;\n\t"
      "@p min.f32 %2, %2, %10;\n\t@p min.f32 %3, %3, %11;\n\t@p max.f32 %4, %4, %12;\n\t"
      "@p max.f32 %5, %5, %13;\n\t@p max.f32 %6, %6, %14;\n\t}"
      : "+r"(x.n), "+f"(x.l0), "+f"(x.l1), "+f"(x.l2), "+f"(x.h0), "+f"(x.h1), "+f"(x.h2)
      : "r"(a), "r"(b), "f"(lo.x), "f"(lo.y), "f"(lo.z), "f"(hi.x), "f"(hi.y), "f"(hi.z));
}

// Split a node of 33 .. kWarpMax records (src, shared memory) with one warp.
// Lane s holds bin s: every lane reads every record (broadcasts) and joins
// those of its own bin in registers, as many axes at a time as 32 lanes hold
// (at most 16 bins in all: the half-warps take every other record each), so
// there is nothing to clear, no atomic and no bin in memory.  The records
// return to src in the order of the stable partition.  The same bins, costs
// and order as cta_split's, so the same tree.  Returns the records on the
// left; both children's boxes in L and R.
__device__ __forceinline__ int warp_split(const BuildArgs& A, unsigned* idx, float4* src, int n, BinU& L, BinU& R) {
  constexpr int kPer = kWarpMax / 32;
  const int lane = threadIdx.x & 31;
  const int K = A.K;
  unsigned ext[6] = {0u, 0u, 0u, 0u, 0u, 0u};  // centre bounds: ~code of the least, code of the largest
#pragma unroll
  for (int r = 0; r < kPer; ++r) {
    const int k = r * 32 + lane;
    if (k < n) {
      const float4 lo = src[2 * k], hi = src[2 * k + 1];
      const unsigned u0 = ucode(centre(lo.x, hi.x)), u1 = ucode(centre(lo.y, hi.y)), u2 = ucode(centre(lo.z, hi.z));
      ext[0] = max(ext[0], ~u0);
      ext[1] = max(ext[1], ~u1);
      ext[2] = max(ext[2], ~u2);
      ext[3] = max(ext[3], u0);
      ext[4] = max(ext[4], u1);
      ext[5] = max(ext[5], u2);
    }
  }
  __syncwarp();
  float cmin[3], scl[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    cmin[a] = uval(~__reduce_max_sync(kFull, ext[a]));
    scl[a] = bin_scale(cmin[a], uval(__reduce_max_sync(kFull, ext[3 + a])), K);
  }
#pragma unroll
  for (int r = 0; r < kPer; ++r) {
    const int k = r * 32 + lane;
    if (k < n) {
      const float4 lo = src[2 * k], hi = src[2 * k + 1];
      idx[k] = (unsigned)bin_of(centre(lo.x, hi.x), cmin[0], scl[0], K) |
               (unsigned)bin_of(centre(lo.y, hi.y), cmin[1], scl[1], K) << 8 |
               (unsigned)bin_of(centre(lo.z, hi.z), cmin[2], scl[2], K) << 16;
    }
  }
  __syncwarp();
  Split best;
  split_none(best);
  for (int a0 = 0; a0 < 3;) {
    const int m = min(3 - a0, 32 / K);
    if (m >= 2 || __any_sync(kFull, sel3(scl[0], scl[1], scl[2], a0) > 0.f)) {
      const bool half = m * K <= 16;
      const int ll = half ? lane & 15 : lane;
      const int g = ll / K, sl = ll - g * K;
      bool in = g < m;
      const int shift = 8 * (a0 + (in ? g : 0));
      const unsigned want = in ? (unsigned)sl : 0xffffffffu;
      const int step = half ? 2 : 1;
      BinB x = binb_empty();
#pragma unroll 4
      for (int k = half ? lane >> 4 : 0; k < n; k += step) {
        const unsigned w = idx[k];
        const float4 lo = src[2 * k], hi = src[2 * k + 1];
        binb_join_if(x, (w >> shift) & 255u, want, lo, hi);
      }
      __syncwarp();
      if (half) {
        x = binb_join(x, binb_xor(x, 16));
        in = in && lane < 16;
        if (!in) x = binb_empty();
      }
      eval_bins<false>(x, nullptr, in, in ? g : 32, sl, K, n, a0, A.cp, best);
    }
    a0 += m;
  }
  int axis = -1, plane = 0, nl = n / 2;
  if (best.cand != INT_MAX) {
    axis = best.cand / (K - 1);
    plane = 1 + best.cand % (K - 1);
    nl = best.L.n;
  }
  float4 lo[kPer], hi[kPer];
  int dest[kPer];
  int lrun = 0;
#pragma unroll
  for (int r = 0; r < kPer; ++r) {
    const int k = r * 32 + lane;
    bool left = false;
    if (k < n) {
      lo[r] = src[2 * k];
      hi[r] = src[2 * k + 1];
      left = axis >= 0 ? (int)((idx[k] >> (8 * axis)) & 255u) < plane : k < nl;
    }
    __syncwarp();
    const unsigned b = __ballot_sync(kFull, left);
    const int before = lrun + __popc(b & ((1u << lane) - 1u));  // records on the left before k
    dest[r] = left ? before : nl + k - before;
    lrun += __popc(b);
  }
  if (lane == 0 && lrun != nl) set_status(A.ctl, kStBadSplit, 7);
#pragma unroll
  for (int r = 0; r < kPer; ++r) {
    if (r * 32 + lane < n && dest[r] < n) {
      src[2 * dest[r]] = lo[r];
      src[2 * dest[r] + 1] = hi[r];
    }
  }
  L = best.L;
  R = best.R;
  if (__any_sync(kFull, axis < 0)) {  // no usable plane: the halves' boxes from their records
    unsigned u[12];  // codes of the left's box (lo complemented), then the right's
#pragma unroll
    for (int q = 0; q < 12; ++q) u[q] = 0u;
#pragma unroll
    for (int r = 0; r < kPer; ++r) {
      if (r * 32 + lane < n) {
        const unsigned c[6] = {~ucode(lo[r].x), ~ucode(lo[r].y), ~ucode(lo[r].z),
                               ucode(hi[r].x), ucode(hi[r].y), ucode(hi[r].z)};
        const bool left = dest[r] < nl;
#pragma unroll
        for (int q = 0; q < 6; ++q) {
          u[q] = max(u[q], left ? c[q] : 0u);
          u[6 + q] = max(u[6 + q], left ? 0u : c[q]);
        }
      }
    }
    __syncwarp();
#pragma unroll
    for (int q = 0; q < 12; ++q) u[q] = __reduce_max_sync(kFull, u[q]);
    L.l0 = uval(~u[0]), L.l1 = uval(~u[1]), L.l2 = uval(~u[2]);
    L.h0 = uval(u[3]), L.h1 = uval(u[4]), L.h2 = uval(u[5]);
    R.l0 = uval(~u[6]), R.l1 = uval(~u[7]), R.l2 = uval(~u[8]);
    R.h0 = uval(u[9]), R.h1 = uval(u[10]), R.h2 = uval(u[11]);
  }
  __syncwarp();  // src is written before any lane reads it again
  return nl;
}

// The subtrees of a large scene's nodes of at most kWarpMax records, a warp
// each from its node to its leaves: the records in shared memory, the larger
// child kept, the other on the warp's stack.  A CTA split of so few records
// waits at its barriers most of the time (7k cycles of 8 warps for 33-64
// records); here every warp of the SM has a node of its own and the issue of
// instructions bounds it (13.2M-triangle metro: 778k nodes of at most 32
// records and 767k splits in 5.3 ms, 14.9 ms inside the split kernel).  24
// warps per SM (80 registers, 184 bytes of spill stores and 260 of loads).
struct SmallSmem {
  float4 rec[kWarps][2 * kWarpMax];
  unsigned idx[kWarps][kWarpMax];
  int4 stack[kWarps][kWarpMax / 2];  // (first record, records | side << 16, parent, depth): disjoint, >= 2 records
};

__global__ void __launch_bounds__(kBlock, 3) k_small(BuildArgs A) {
  pdl_wait();
  pdl_launch();
  __shared__ SmallSmem S;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int epoch = __ldcg(&A.ctl->epoch);
  const int count = __shfl_sync(kFull, __ldcg(&A.ctl->sq_count), 0);
  float4* rec = S.rec[warp];
  int4* stack = S.stack[warp];
  WarpStats ws{0, 0, 0, 0};
  for (;;) {
    int i = 0;
    if (lane == 0) i = atomicAdd(&A.ctl->sq_head, 1);
    i = __shfl_sync(kFull, i, 0);
    if (i >= count) break;
    const int4* q = reinterpret_cast<const int4*>(A.qa + (A.qa_cap - 1 - i));
    const int4 t0 = __ldcg(q), t1 = __ldcg(q + 1), t2 = __ldcg(q + 2);
    const int begin = t0.x;
    int n = __shfl_sync(kFull, t0.y, 0), b = 0, parent = t0.z, side = t0.w, depth = t1.w, sp = 0;
    if (begin < 0 || n < 2 || n > kWarpMax || begin > A.n - n) {
      if (lane == 0) set_status(A.ctl, kStBadSplit, 8);
      continue;
    }
    const float4* g = A.rec[t2.w & 1] + 2 * (size_t)begin;
    for (int k = lane; k < 2 * n; k += 32) rec[k] = __ldcg(g + k);
    __syncwarp();
    for (;;) {
      while (n > kMicro) {
        float4* src = rec + 2 * b;
        BinU L, R;
        const int nl = __shfl_sync(kFull, warp_split(A, S.idx[warp], src, n, L, R), 0), nr = n - nl;
        const bool leafl = nl <= A.max_leaf, leafr = nr <= A.max_leaf;
        const int id = begin + b + nl - 1;
        const int keep = nl >= nr ? 0 : 1;
        if (leafl) leaf_out<false>(A, src, begin + b, nl, lane, 32);
        if (leafr) leaf_out<false>(A, src + 2 * nl, begin + b + nl, nr, lane, 32);
        if (lane == 0) {
          write_node(A, id, parent, side, L, leafl ? leaf_ref(begin + b, nl) : INT_MAX, nl, R,
                     leafr ? leaf_ref(begin + b + nl, nr) : INT_MAX, nr, epoch);
          note_node(ws, nl, nr, leafl, leafr, depth);
          if (!(keep ? leafl : leafr))  // the smaller child
            stack[sp] = keep ? make_int4(b, nl, id, depth + 1) : make_int4(b + nl, nr | (1 << 16), id, depth + 1);
        }
        __syncwarp();
        sp += (keep ? leafl : leafr) ? 0 : 1;
        parent = id;
        side = keep;
        ++depth;
        b += keep ? nl : 0;
        n = keep ? nr : nl;
      }
      if (n > A.max_leaf) micro_sort_build(A, rec + 2 * b, begin + b, n, parent, side, depth, epoch, ws);
      if (sp == 0) break;
      const int4 e = stack[--sp];
      b = e.x;
      n = __shfl_sync(kFull, e.y & 0xffff, 0);
      side = e.y >> 16;
      parent = e.z;
      depth = e.w;
    }
    __syncwarp();
  }
  if (lane == 0) {
    if (ws.n_int) atomicAdd(&A.ctl->n_internal, ws.n_int);
    if (ws.n_leaf) atomicAdd(&A.ctl->n_leaves, ws.n_leaf);
    if (ws.big) atomicMax(&A.ctl->max_leaf_size, ws.big);
    if (ws.deep) atomicMax(&A.ctl->depth2, ws.deep);
  }
}

template <bool kStaged>
union SplitSmem {
  std::conditional_t<kStaged, StagedSmem, TopSmem> top;
  SubSmem sub;
};

// The split phase: the first top_ctas CTAs work the chunk items of big nodes
// (CTA per item) and then join the others, which take the subtree queue
// (CTA per subtree).  Both run at once, so subtrees proceed while the big
// nodes of other branches are still being split; in large scenes every CTA
// takes chunks first.
//
// kStaged (large scenes): the big nodes' chunks go through shared memory, up
// to 8 consecutive records a thread, instead of registers, a record a thread
// and round.  The shuffles of the children's binning bound a chunk, 60 for 32
// records (an SM does one every two cycles); staged, 65 serve 256.  Builds of
// 600k triangles 1.09 -> 0.81 ms at alpha 1 and 1.63 -> 1.39 at 0.7, 4M 5.35 ->
// 4.55 and 8.71 -> 7.46; but 20k 0.203 -> 0.210, 199k 0.717 -> 0.765 at 0.7,
// where a level's latency counts and a chunk has few records.
template <bool kStaged>
__global__ void __launch_bounds__(kBlock, 2) k_split(BuildArgs A) {
  pdl_wait();
  pdl_launch();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  SplitSmem<kStaged>& S = *reinterpret_cast<SplitSmem<kStaged>*>(smem_raw);
  const int epoch = __ldcg(&A.ctl->epoch);
  if ((int)blockIdx.x < A.top_ctas) {
    top_loop<kStaged>(A, reinterpret_cast<TopSmem&>(S), epoch);
    __syncthreads();
  }
  sub_loop(A, S.sub, epoch);
}

// ------------------------------------------------------------------ traversal nodes + leaf order
__device__ __forceinline__ void child_of(const Node2& n, int s, int* ref, float3* lo, float3* hi) {
  const float4 l = s == 0 ? n.a_lo : n.b_lo, h = s == 0 ? n.a_hi : n.b_hi;
  *ref = __float_as_int(l.w);
  *lo = make_float3(l.x, l.y, l.z);
  *hi = make_float3(h.x, h.y, h.z);
}

__device__ __forceinline__ Node2 load_node_cg(const Node2* p) {
  const float4* q = reinterpret_cast<const float4*>(p);
  Node2 n;
  n.a_lo = __ldcg(q);
  n.a_hi = __ldcg(q + 1);
  n.b_lo = __ldcg(q + 2);
  n.b_hi = __ldcg(q + 3);
  return n;
}

// A child reference is usable if it is a leaf or a node written by this build.
__device__ __forceinline__ bool ref_ok(const BuildArgs& A, int ref, int epoch) {
  if (ref == INT_MIN) return false;
  if (ref < 0) return true;
  return ref < A.n - 1 && __ldcg(&A.link2[ref]).y == epoch;
}

// The 4-wide node rooted at binary node x: open the internal child of
// largest surface area until there are 4 children (the first of equal areas
// wins; the opened node's children take its slot and the next free one).
// The 64-byte form of wide node w: per axis the grid origin is the union
// box's lower corner and the step 2^e the smallest with 255 steps covering
// its extent; each lower plane takes the largest byte whose decoded value is
// not above it, each upper plane the smallest not below it (checked with
// qplane itself, so the decoded box contains the exact one); when 255 steps
// fall short after rounding, e grows.  An infinite plane is coded as the
// largest float's (lower ones) or decodes to infinity (upper ones, at the
// largest step), beyond every finite ray either way.
__device__ QNode quantize_node(const WNode& w) {
  const float lo[3][4] = {{w.lox.x, w.lox.y, w.lox.z, w.lox.w}, {w.loy.x, w.loy.y, w.loy.z, w.loy.w},
                          {w.loz.x, w.loz.y, w.loz.z, w.loz.w}};
  const float hi[3][4] = {{w.hix.x, w.hix.y, w.hix.z, w.hix.w}, {w.hiy.x, w.hiy.y, w.hiy.z, w.hiy.w},
                          {w.hiz.x, w.hiz.y, w.hiz.z, w.hiz.w}};
  const int ch[4] = {w.child.x, w.child.y, w.child.z, w.child.w};
  QNode q;
  float org[3];
  unsigned wlo[3], whi[3];
  int exps = 0;
  for (int a = 0; a < 3; ++a) {
    float ulo = INFINITY, uhi = -INFINITY;
    for (int i = 0; i < 4; ++i)
      if (ch[i] != INT_MIN) {
        ulo = fminf(ulo, lo[a][i]);
        uhi = fmaxf(uhi, hi[a][i]);
      }
    if (!(ulo <= uhi)) {  // no child
      ulo = 0.f;
      uhi = 0.f;
    }
    ulo = fminf(fmaxf(ulo, -FLT_MAX), FLT_MAX);
    int e = -126;
    const float ext = uhi - ulo;
    if (ext > FLT_MAX) {
      e = 127;
    } else if (ext > 0.f) {
      int k;
      frexpf(ext * (1.f / 255.f), &k);  // ext / 255 < 2^k
      e = max(-126, min(127, k));
    }
    unsigned bl = 0, bh = 0;
    for (int attempt = 0; attempt < 8; ++attempt) {
      const float s = qscale(e);
      bool ok = true;
      bl = bh = 0;
      for (int i = 0; i < 4; ++i) {
        unsigned ql = 255, qh = 0;  // empty slot: an empty decoded box
        if (ch[i] != INT_MIN) {
          int l = (int)floorf((lo[a][i] - ulo) / s), h = (int)ceilf((hi[a][i] - ulo) / s);
          l = max(0, min(255, l));
          h = max(0, min(255, h));
          while (l > 0 && qplane((unsigned)l, s, ulo) > lo[a][i]) --l;
          while (h < 255 && qplane((unsigned)h, s, ulo) < hi[a][i]) ++h;
          ok = ok && qplane((unsigned)l, s, ulo) <= lo[a][i] && qplane((unsigned)h, s, ulo) >= hi[a][i];
          ql = (unsigned)l;
          qh = (unsigned)h;
        }
        bl |= ql << (8 * i);
        bh |= qh << (8 * i);
      }
      if (ok || e >= 127) break;
      ++e;
    }
    org[a] = ulo;
    wlo[a] = bl;
    whi[a] = bh;
    exps |= (e + 128) << (8 * a);
  }
  q.ox = org[0];
  q.oy = org[1];
  q.oz = org[2];
  q.exps = exps;
  q.lox = wlo[0];
  q.hix = whi[0];
  q.loy = wlo[1];
  q.hiy = whi[1];
  q.loz = wlo[2];
  q.hiz = whi[2];
  q.parent = w.meta.x;
  q.pad = 0;
  q.child = w.child;
  return q;
}

// The W-wide node rooted at binary node x: open the internal child of
// largest surface area until there are W children (the first of equal areas
// wins; the opened node's children take its slot and the next free one).
// Slots past m are empty.
template <int W>
__device__ int collapse(const BuildArgs& A, int x, int epoch, int* ref, float3* lo, float3* hi) {
  const Node2 nd = load_node_cg(A.node2 + x);
  child_of(nd, 0, &ref[0], &lo[0], &hi[0]);
  child_of(nd, 1, &ref[1], &lo[1], &hi[1]);
  int m = 2;
  for (int q = 0; q < 2; ++q)
    if (!ref_ok(A, ref[q], epoch)) {
      set_status(A.ctl, kStBadLink, 1);
      ref[q] = INT_MIN;
    }
  while (m < W) {
    int pick = -1;
    float best = -1.f;
    for (int q = 0; q < m; ++q)
      if (ref[q] >= 0) {
        const float ar = area(lo[q], hi[q]);
        if (ar > best) {
          best = ar;
          pick = q;
        }
      }
    if (pick < 0) break;
    const Node2 g = load_node_cg(A.node2 + ref[pick]);
    child_of(g, 1, &ref[m], &lo[m], &hi[m]);
    child_of(g, 0, &ref[pick], &lo[pick], &hi[pick]);
    for (int q : {pick, m})
      if (!ref_ok(A, ref[q], epoch)) {
        set_status(A.ctl, kStBadLink, 2);
        ref[q] = INT_MIN;
      }
    ++m;
  }
  for (int q = m; q < W; ++q) ref[q] = INT_MIN;
  for (int q = 0; q < W; ++q)
    if (ref[q] == INT_MIN) {
      lo[q] = make_float3(INFINITY, INFINITY, INFINITY);
      hi[q] = make_float3(-INFINITY, -INFINITY, -INFINITY);
    }
  return m;
}

__device__ void make_wide(const BuildArgs& A, int x, int epoch) {
  int ref[4];
  float3 lo[4], hi[4];
  collapse<4>(A, x, epoch, ref, lo, hi);
  WNode w;
  w.lox = make_float4(lo[0].x, lo[1].x, lo[2].x, lo[3].x);
  w.hix = make_float4(hi[0].x, hi[1].x, hi[2].x, hi[3].x);
  w.loy = make_float4(lo[0].y, lo[1].y, lo[2].y, lo[3].y);
  w.hiy = make_float4(hi[0].y, hi[1].y, hi[2].y, hi[3].y);
  w.loz = make_float4(lo[0].z, lo[1].z, lo[2].z, lo[3].z);
  w.hiz = make_float4(hi[0].z, hi[1].z, hi[2].z, hi[3].z);
  w.child = make_int4(ref[0], ref[1], ref[2], ref[3]);
  w.meta = make_int4(__ldcg(&A.link2[x]).x, 0, 0, 0);
  A.wide[x] = w;
  if (A.qwide) A.qwide[x] = quantize_node(w);
}

__device__ void make_wide8(const BuildArgs& A, int x, int epoch) {
  int ref[8];
  float3 lo[8], hi[8];
  collapse<8>(A, x, epoch, ref, lo, hi);
  WNode8 w;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int b = 4 * h;
    w.lox[h] = make_float4(lo[b].x, lo[b + 1].x, lo[b + 2].x, lo[b + 3].x);
    w.hix[h] = make_float4(hi[b].x, hi[b + 1].x, hi[b + 2].x, hi[b + 3].x);
    w.loy[h] = make_float4(lo[b].y, lo[b + 1].y, lo[b + 2].y, lo[b + 3].y);
    w.hiy[h] = make_float4(hi[b].y, hi[b + 1].y, hi[b + 2].y, hi[b + 3].y);
    w.loz[h] = make_float4(lo[b].z, lo[b + 1].z, lo[b + 2].z, lo[b + 3].z);
    w.hiz[h] = make_float4(hi[b].z, hi[b + 1].z, hi[b + 2].z, hi[b + 3].z);
    w.child[h] = make_int4(ref[b], ref[b + 1], ref[b + 2], ref[b + 3]);
  }
  w.meta[0] = make_int4(__ldcg(&A.link2[x]).x, 0, 0, 0);
  w.meta[1] = make_int4(0, 0, 0, 0);
  A.wide8[x] = w;
}

__global__ void __launch_bounds__(kBlock) k_post(BuildArgs A) {
  pdl_wait();
  pdl_launch();
  const int n = A.n;
  const int epoch = __ldcg(&A.ctl->epoch);
  const int gt = blockIdx.x * kBlock + threadIdx.x, gs = gridDim.x * kBlock;
  if (gt == 0) {
    const int r = __ldcg(&A.ctl->root_ref);
    if (r >= 0) {
      A.ctl->wide_root = r;
    } else {  // the whole scene is one leaf (or empty): a wrapper node in slot 0
      WNode w;
      const float inf = INFINITY;
      w.lox = w.loy = w.loz = make_float4(inf, inf, inf, inf);
      w.hix = w.hiy = w.hiz = make_float4(-inf, -inf, -inf, -inf);
      w.child = make_int4(INT_MIN, INT_MIN, INT_MIN, INT_MIN);
      if (r != INT_MIN && leaf_count(r) > 0) {
        w.lox.x = uval(~__ldcg(&A.ctl->sb[0]));
        w.loy.x = uval(~__ldcg(&A.ctl->sb[1]));
        w.loz.x = uval(~__ldcg(&A.ctl->sb[2]));
        w.hix.x = uval(__ldcg(&A.ctl->sb[3]));
        w.hiy.x = uval(__ldcg(&A.ctl->sb[4]));
        w.hiz.x = uval(__ldcg(&A.ctl->sb[5]));
        w.child.x = r;
      }
      w.meta = make_int4(-1, 0, 0, 0);
      if (A.wide8) {
        WNode8 w8;
        w8.lox[0] = w.lox;
        w8.hix[0] = w.hix;
        w8.loy[0] = w.loy;
        w8.hiy[0] = w.hiy;
        w8.loz[0] = w.loz;
        w8.hiz[0] = w.hiz;
        w8.lox[1] = w8.loy[1] = w8.loz[1] = make_float4(inf, inf, inf, inf);
        w8.hix[1] = w8.hiy[1] = w8.hiz[1] = make_float4(-inf, -inf, -inf, -inf);
        w8.child[0] = w.child;
        w8.child[1] = make_int4(INT_MIN, INT_MIN, INT_MIN, INT_MIN);
        w8.meta[0] = w.meta;
        w8.meta[1] = make_int4(0, 0, 0, 0);
        A.wide8[0] = w8;
      } else {
        A.wide[0] = w;
        if (A.qwide) A.qwide[0] = quantize_node(w);
      }
      A.ctl->wide_root = 0;
    }
  }
  for (int i = gt; i < n; i += gs) {
    const int p = __float_as_int(__ldcg(A.rec[0] + 2 * (size_t)i).w);
    if (p < 0 || p >= A.n_all) {
      set_status(A.ctl, kStBadSplit, 20);
      continue;
    }
    A.order[i] = p;
    A.tri_leaf[3 * (size_t)i] = A.tri[3 * (size_t)p];
    A.tri_leaf[3 * (size_t)i + 1] = A.tri[3 * (size_t)p + 1];
    A.tri_leaf[3 * (size_t)i + 2] = A.tri[3 * (size_t)p + 2];
    if (i < n - 1 && __ldcg(&A.link2[i]).y == epoch) {
      if (A.wide8)
        make_wide8(A, i, epoch);
      else
        make_wide(A, i, epoch);
    }
  }
}

size_t split_smem(bool staged) { return staged ? sizeof(SplitSmem<true>) : sizeof(SplitSmem<false>); }

int sm_count() {
  static int n = 0;
  if (!n) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    if (n <= 0) n = 1;
  }
  return n;
}

// Launch with programmatic stream serialization when `pdl` is set: the
// kernel may start while its predecessor drains and waits for it in-kernel.
template <typename... P, typename... Q>
cudaError_t launch(void (*k)(P...), int grid, size_t smem, cudaStream_t st, bool pdl, Q... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3(kBlock);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = pdl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, k, args...);
}

}  // namespace

BuildGeom build_geometry(int64_t n, int nsm) {
  BuildGeom g{};
  const int64_t T = n < 1 ? 1 : n;
  g.big = (int)std::max<int64_t>(kBigMin, (T + 4095) / 4096);
  int64_t rpt = (T + (int64_t)nsm * 512 - 1) / ((int64_t)nsm * 512);
  // (8 from a million records: 1.2M 1.53 -> 1.37 ms at alpha 1, 2.52 -> 2.44 at
  // 0.7, 13.2M 30.8 -> 27.1; 400k 0.640 -> 0.660 and 1.05 -> 1.10; 16 gains
  // nothing more)
  rpt = std::min<int64_t>(std::max<int64_t>(rpt, 1), T >= 1000000 ? kMaxRpt : kRegRpt);
  g.rpt = (int)rpt;
  g.chunk = kBlock * g.rpt;
  // Pools of one build (a full pool sends further big nodes to the subtree queue,
  // slower but correct).  Big nodes of one depth are disjoint, so there are at
  // most T / big of them per depth; 16 depths' worth covers the uneven trees
  // of alpha < 1.  Chunk counts: a big node reserves its chunks + 2 for its
  // children; per depth that is at most T / chunk + 3 T / big, where
  // T' / chunk(T') <= max(2 nsm, T / 1024) + 1 for every T' <= T.
  const int64_t nb = (T + g.big - 1) / g.big;
  const int64_t nc = std::max<int64_t>(2 * (int64_t)nsm, (T + 1023) / 1024) + 1;
  g.cap_t = (int)(16 * nb + 256);
  g.cap_c = (int)(16 * nc + 3 * (int64_t)g.cap_t + 64);
  // pushes: at most one per binary node of more than max_leaf triangles plus
  // one per leaf cut from a big node
  g.qa_cap = (int)(2 * T + 16);
  return g;
}

cudaError_t launch_build(rt_scene_s* s, const rt_build_params& p, cudaStream_t st) {
  int n = (int)s->n_tri;
  const int* sel = nullptr;
  cudaError_t e;
  if (p.range > 0.f && p.range < 3.0e38f) {
    // the triangles within the ray action range, in input order; the build
    // is sized for their count, which the host reads back (one small copy)
    const int nb = (n + kBlock - 1) / kBlock;
    if (n > 0) {
      const float3 src = make_float3(p.source[0], p.source[1], p.source[2]);
      const float rr = p.range * 1.00001f;
      k_sel_count<<<nb, kBlock, 0, st>>>(s->tri_in, n, src, rr * rr, s->sel_cnt);
      k_sel_scan<<<1, 1024, 0, st>>>(s->sel_cnt, nb);
      k_sel_write<<<nb, kBlock, 0, st>>>(s->tri_in, n, src, rr * rr, s->sel_cnt, s->sel);
      count_launches(3);
      if ((e = cudaGetLastError())) return e;
      if ((e = cudaMemcpyAsync(s->sel_host, s->sel_cnt + nb, sizeof(int), cudaMemcpyDeviceToHost, st))) return e;
      if ((e = cudaStreamSynchronize(st))) return e;
      n = *s->sel_host;
    }
    sel = s->sel;
  }
  s->n_built = n;
  const int nsm = sm_count();
  const BuildGeom g = build_geometry(n, nsm);
  if (g.cap_t > s->geom.cap_t || g.cap_c > s->geom.cap_c || g.qa_cap > s->geom.qa_cap) return cudaErrorInvalidValue;
  BuildArgs A;
  A.tri = s->tri_in;
  A.sel = sel;
  A.rec[0] = s->rec[0];
  A.rec[1] = s->rec[1];
  A.node2 = s->node2;
  A.link2 = s->link2;
  A.ctl = s->ctl;
  A.qa = s->qa;
  A.qa_ready = s->qa_ready;
  A.ttask = s->top_task;
  A.tdone = s->top_done;
  A.tbins = s->top_bins;
  A.tccnt = s->top_ccnt;
  A.tscnt = s->top_scnt;
  A.titem = s->top_item;
  A.tplan = s->top_plan;
  A.tready = s->top_ready;
  A.wide = s->wide;
  A.qwide = p.quantize ? s->qwide : nullptr;
  A.wide8 = p.width == 8 ? s->wide8 : nullptr;
  A.tri_leaf = s->tri_leaf;
  A.order = s->idx[0];
  A.epoch_dev = s->epoch;
  A.n = n;
  A.n_all = (int)s->n_tri;
  A.K = p.bins;
  A.max_leaf = p.max_leaf;
  // k_small pays where the subtrees fill the device and the split kernel is
  // bound by what they cost, not by the longest of them.  Builds without it,
  // with 64 and with 128 records a node, alpha 1: 60k triangles 0.241 /
  // 0.255 / 0.289 ms, 279k 0.647 / 0.557 / 0.548, 600k 1.36 / 1.14 / 1.09, 4M
  // 7.70 / 5.93 / 5.33; alpha 0.7: 199k 0.716 / 0.737 / 0.750, 279k 0.912 /
  // 0.838 / 0.871, 600k 1.81 / 1.67 / 1.63, 4M 11.4 / 9.46 / 8.70.
  const bool large = n >= kLargeScene;
  A.wsm = !large ? 0 : (n < 500000 ? kWarpMax / 2 : kWarpMax);
  A.big = g.big;
  A.chunk = g.chunk;
  A.rpt = g.rpt;
  A.cap_t = s->geom.cap_t;
  A.cap_c = s->geom.cap_c;
  A.qa_cap = s->geom.qa_cap;
  static bool attr = false;
  static int split_per_sm = 2;  // resident split CTAs per SM (at most 2)
  if (!attr) {
    int occ = 2;
    for (bool staged : {false, true}) {
      void (*k)(BuildArgs) = staged ? k_split<true> : k_split<false>;
      const size_t sm = split_smem(staged);
      if ((e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm))) return e;
      int o = 0;
      if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, k, kBlock, sm))) return e;
      occ = std::min(occ, o);
    }
    split_per_sm = std::max(1, std::min(2, occ));
    attr = true;
  }
  // the big-node chunks go to the first nsm CTAs, which then join the rest on
  // the subtree queue, so that subtrees proceed while other branches' big
  // nodes are split; in large scenes every CTA takes chunks first (475k
  // triangles 1.55 -> 1.50 ms)
  A.top_ctas = n > g.big ? (large ? split_per_sm * nsm : nsm) : 0;
  const DebugHooks dh = debug_hooks();
  A.spin_limit = dh.spin_limit > 0 ? dh.spin_limit : kSpinLimit;
  A.phantom_tasks = dh.phantom_tasks;
  A.phantom_items = dh.phantom_items;
  if (A.phantom_items && !A.top_ctas) A.top_ctas = nsm;  // someone must wait for the phantom items
  A.cp = CostP{p.alpha, p.t_i, p.t_trav, p.source[0], p.source[1], p.source[2], p.dist_norm};
  if ((e = cudaMemsetAsync(s->ctl, 0, sizeof(BuildCtl), st))) return e;
  const int nch = (n + g.chunk - 1) / g.chunk;
  int gp = (n + kBlock - 1) / kBlock;
  gp = std::max(1, std::min(gp, nsm * 8));
  if ((e = launch(k_prep, gp, 0, st, false, A))) return e;
  if ((e = launch(k_bin_root, std::max(1, std::min(nch, nsm * 4)), 0, st, true, A))) return e;
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  if (s->split_ev[0] && (e = cudaStreamIsCapturing(st, &cs))) return e;
  const unsigned evflags = cs == cudaStreamCaptureStatusNone ? cudaEventRecordDefault : cudaEventRecordExternal;
  if (s->split_ev[0] && (e = cudaEventRecordWithFlags(s->split_ev[0], st, evflags))) return e;
  if ((e = launch(large ? k_split<true> : k_split<false>, split_per_sm * nsm, split_smem(large), st, true, A)))
    return e;
  if (A.wsm) {
    if ((e = launch(k_small, 3 * nsm, 0, st, true, A))) return e;
    count_launches(1);
  }
  if (s->split_ev[1] && (e = cudaEventRecordWithFlags(s->split_ev[1], st, evflags))) return e;
  if ((e = launch(k_post, gp, 0, st, true, A))) return e;
  count_launches(4);
  return cudaSuccess;
}

}  // namespace rt
