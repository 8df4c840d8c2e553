// Per-node top-k with 256-byte indexer rows (128 bf16 or 64 fp32) and up to four indexer heads, for lists beyond the short ones.
//
// Scoring (both forms; fp32 storage below): a warp scores sixteen entries at a time for eight nodes and all heads by tensor-core products (16
// entries x 32 query rows), its rows straight from global memory into the fragments: an inner product does not care for the
// order of its terms, so lane tq of a row's four takes the 16-byte pieces tq, tq + 4, ... and the queries are read the same
// way.  An indexer row is read once per sequence (one CTA per node read it once per node, in rounds of 96 rows through
// shared memory), and no warp waits for another.
//
//   topk_seq_kernel   lists of up to kSeqMax entries, trees of up to eight nodes: one cluster of eight CTAs per SEQUENCE.  The
//                     entries are split over the CTAs; a warp leaves its scores in the lists of the nodes' owners (CTA r owns
//                     node r) through distributed shared memory, and after one cluster barrier every node's whole list
//                     lies in its owner's shared memory.
//   score_rows_kernel + topk_list_kernel   longer lists or larger trees: the scores over all SMs into the workspace, then a
//                     cluster of eight CTAs per node with the list in shared memory.
//
// fp32 storage (cluster form only): a lane scores one entry for all nodes and heads, its row in registers, the queries
// broadcast from shared memory; exact fp32 products in eight interleaved partial sums per inner product.
//
// The selection finds the k largest by ONE histogram over equal intervals of [min, max] (the scores of a list share their high
// bits, so radix digits of the bit pattern take four passes with colliding bins): the interval of the k-th largest holds few
// candidates, which are ranked against each other exactly (ties to the lower index).  Degenerate lists (more than CAP
// candidates in that interval: ties, outliers; a score that is infinite or NaN) take four radix passes instead: the interval code
// compares floats, under which a NaN has no place, the radix digits are a total order of the bit patterns.
// Same result as topk_kernel: the exact k largest scores, ties to the lower index, ascending output.
#include "select_common.cuh"

namespace tsv {

namespace ssel {

constexpr int CS = 8;                  // CTAs per cluster = nodes scored together
constexpr int kSeqMax = 4096;          // longest list of the cluster form
constexpr int DI = 128, HMAX = 4;      // indexer width (bf16), heads (query row 4 n + h, absent ones zero)
constexpr int ROWB = 256;              // bytes of an indexer row
constexpr int QP = 320;                // pitch of a staged query row: conflict-free 16-byte fragment loads
constexpr int CAP = 256;               // candidates ranked against each other

__device__ __forceinline__ void mma_bf16_16816(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t map_to_rank(uint32_t saddr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(rank));
  return r;
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

// dynamic shared memory of the cluster form: queries | a step's scores per warp | score list of the owned node | bit per candidate
struct Layout {
  uint32_t loc, sc, bits, total;
  __host__ __device__ Layout(int nw, int cap) {
    loc = 32 * QP;
    sc = loc + (uint32_t)nw * 512;
    bits = sc + (uint32_t)cap * 4;
    total = bits + ((uint32_t)cap + 31) / 32 * 4;
  }
};

// Sixteen entries against the queries of eight nodes.
struct Scorer {
  const char* ikb;
  RowAddr rows;
  int g, tq, end;
  float iwr[4][2];                                       // head weights of this lane's columns 8 j + 2 tq, + 1
  // rows g and g + 8 of the sixteen entries from e on: lane tq's pieces of 16 bytes, four of a row
  template <bool PAGED>
  __device__ __forceinline__ void fetch(int e, uint4 (&lo)[4], uint4 (&hi)[4]) const {
    const int r0 = min(e + g, end - 1), r1 = min(e + g + 8, end - 1);
    const uint4* p0 = reinterpret_cast<const uint4*>(ikb + (size_t)(PAGED ? rows.rel(r0) : (int64_t)r0) * (DI * 2));
    const uint4* p1 = reinterpret_cast<const uint4*>(ikb + (size_t)(PAGED ? rows.rel(r1) : (int64_t)r1) * (DI * 2));
#pragma unroll
    for (int q = 0; q < 4; ++q) { lo[q] = __ldg(p0 + 4 * q); hi[q] = __ldg(p1 + 4 * q); }
  }
  __device__ __forceinline__ void weights(const float* iw, int n0, int D, int HI) {      // iw: [D][HI] of the sequence
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        const int n = n0 + 2 * j + (tq >> 1), h = ((2 * tq) & 3) + x;
        iwr[j][x] = n < D && h < HI ? __ldg(iw + n * HI + h) : 0.f;
      }
  }
  // scores into buf (this warp's, [8 nodes][16 entries]); qs: the staged queries
  __device__ __forceinline__ void score(const uint4 (&lo)[4], const uint4 (&hi)[4], const unsigned char* qs, float* buf) const {
    float acc[4][4];
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int x = 0; x < 4; ++x) acc[j][x] = 0.f;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {                      // column g of tile j = query row 8 j + g
        const uint4 bv = *reinterpret_cast<const uint4*>(qs + (8 * j + g) * QP + q * 64 + tq * 16);
        mma_bf16_16816(acc[j], lo[q].x, hi[q].x, lo[q].y, hi[q].y, bv.x, bv.y);
        mma_bf16_16816(acc[j], lo[q].z, hi[q].z, lo[q].w, hi[q].w, bv.z, bv.w);
      }
    }
    __syncwarp();                                        // (the step before has left the buffer)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float l = fmaf(iwr[j][1], fmaxf(acc[j][1], 0.f), iwr[j][0] * fmaxf(acc[j][0], 0.f));
      float h = fmaf(iwr[j][1], fmaxf(acc[j][3], 0.f), iwr[j][0] * fmaxf(acc[j][2], 0.f));
      l += __shfl_xor_sync(0xffffffffu, l, 1);
      h += __shfl_xor_sync(0xffffffffu, h, 1);
      if (!(tq & 1)) { float* o = buf + (2 * j + (tq >> 1)) * 16 + g; o[0] = l; o[8] = h; }
    }
    __syncwarp();
  }
};
// queries of nodes n0 .. n0 + 7 of sequence b into shared memory: row 4 (n - n0) + h; absent heads and node slots zero
__device__ __forceinline__ void stage_queries(unsigned char* qs, const void* iq_, int b, int n0, int D, int HI) {
  const uint4* iq = reinterpret_cast<const uint4*>(reinterpret_cast<const char*>(iq_) + (size_t)b * D * HI * ROWB);
  for (int idx = threadIdx.x; idx < 32 * 16; idx += blockDim.x) {
    const int row = idx >> 4, c16 = idx & 15, n = n0 + (row >> 2), h = row & 3;
    *reinterpret_cast<uint4*>(qs + row * QP + c16 * 16) = n < D && h < HI ? __ldg(iq + (n * HI + h) * (ROWB / 16) + c16) : make_uint4(0u, 0u, 0u, 0u);
  }
}
// Lane j = node j: the strict ancestors of node n that close a CSA block (from their positions), root first.  One warp.
__device__ __forceinline__ void path_of(PathEntries& pe, const TreeMeta& tm, const tsv_shape& s, int n, bool live) {
  const int t = threadIdx.x & 31;
  const bool valid = !tm.status && t < tm.nn;
  const uint32_t strict = live ? tm.anc[n] & ~(1u << n) : 0u;
  const uint32_t cm = __ballot_sync(0xffffffffu, valid && node_closes(tm.L, tm.depth[t], s.m_csa)) & strict;
  if ((cm >> t) & 1u) { const int o = __popc(cm & ((1u << t) - 1u)); pe.newc[o] = t; pe.newc_blk[o] = (tm.L + tm.depth[t]) / s.m_csa; }
  if (t == 0) pe.n_newc = __popc(cm);
}
// Scores of the in-tree entries on node n's path (the state build's results): warp w takes entries w, w + nw, ... and hands the
// score of entry i to put(i, score) in lane 0.  A lane holds 8 bytes of every head's query, which it may fetch long before.
template <typename T>
struct ExtraScorer {
  static constexpr int DI = ROWB / (int)sizeof(T), PER = 8 / (int)sizeof(T);
  uint2 q[4];
  float iw[4];
  static __device__ __forceinline__ void unpack(const uint2& v, float* o) {
    if (sizeof(T) == 2) {
      o[0] = __uint_as_float(v.x << 16); o[1] = __uint_as_float(v.x & 0xFFFF0000u);
      o[2] = __uint_as_float(v.y << 16); o[3] = __uint_as_float(v.y & 0xFFFF0000u);
    } else { o[0] = __uint_as_float(v.x); o[1] = __uint_as_float(v.y); }
  }
  __device__ __forceinline__ void fetch(const tsv_shape& s, const tsv_nodes& nd, int b, int n) {
    const int lane = threadIdx.x & 31;
    const size_t r0 = ((size_t)b * s.D + n) * s.HI;
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      q[h] = h < s.HI ? __ldg(reinterpret_cast<const uint2*>(reinterpret_cast<const char*>(nd.iq) + (r0 + h) * ROWB) + lane) : make_uint2(0u, 0u);
      iw[h] = h < s.HI ? __ldg(nd.iw + r0 + h) : 0.f;
    }
  }
  template <typename Put>
  __device__ __forceinline__ void score(const PathEntries& pe, const tsv_shape& s, const tsv_scratch& sc, int b, Put put) const {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int i = w; i < pe.n_newc; i += nw) {
      const uint2 kv = __ldcg(reinterpret_cast<const uint2*>(reinterpret_cast<const char*>(sc.new_csa_ik) + ((size_t)b * s.D + pe.newc[i]) * ROWB) + lane);
      float k4[PER], p[4];
      unpack(kv, k4);
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        float q4[PER];
        unpack(q[h], q4);
        p[h] = 0.f;
#pragma unroll
        for (int x = 0; x < PER; ++x) p[h] = fmaf(q4[x], k4[x], p[h]);
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int h = 0; h < 4; ++h) p[h] += __shfl_xor_sync(0xffffffffu, p[h], o);
      float tot = 0.f;
#pragma unroll
      for (int h = 0; h < 4; ++h) tot = fmaf(iw[h], fmaxf(p[h], 0.f), tot);
      if (lane == 0) put(i, tot);
    }
  }
};
// Everything is selected (or nothing: padding, a flagged sequence): the index list, where somebody reads it.
__device__ __forceinline__ void select_all(int n_cand, int n_csa, const PathEntries& pe, int k, int32_t* sel, int32_t* usr, int32_t* selcnt) {
  for (int i = threadIdx.x; i < k; i += blockDim.x) {
    const int v = i < n_cand ? (i < n_csa ? i : pe.newc_blk[i - n_csa]) : -1;
    sel[i] = v; if (usr) usr[i] = v;
  }
  if (threadIdx.x == 0) *selcnt = n_cand;
}

template <int NT, int NB>
struct SelectSmem {
  int hist[NB];                                          // zero at the start of the selection, like cnt
  float red[2][NT / 32];
  int wsum[2][NT / 32];
  int bin, rem, cnt;
  float cand_s[CAP];
  int cand_i[CAP];
};

// Selection of one node by the whole CTA, in two parts.  list: shared memory, the scores of the n_csa committed entries first, then
// those of the in-tree ones.  First part: the range and the histogram of the committed entries, which need nothing of the state build
// (the in-tree entries are added to it as they are scored; the intervals at either end take what lies beyond).
// (All passes over the list fetch several scores before they use one: one shared-memory latency for them all, where a pass that
// writes in between would take one for each.)
template <int NT, typename F>
__device__ __forceinline__ void each_score(const float* list, int n, F f) {
  constexpr int U = 8;
  for (int i0 = threadIdx.x; i0 < n; i0 += U * NT) {
    float v[U];
#pragma unroll
    for (int u = 0; u < U; ++u) v[u] = i0 + u * NT < n ? list[i0 + u * NT] : 0.f;
#pragma unroll
    for (int u = 0; u < U; ++u) if (i0 + u * NT < n) f(i0 + u * NT, v[u]);
  }
}
struct ScoreBins {
  float lo, scale;
  bool regular;                                          // (else: all equal, not finite, a NaN among them, or too narrow)
  // interval of a score: monotone in the score (a rounded subtraction and product are), so intervals order as scores do
  template <int NB> __device__ __forceinline__ int of(float v) const { return min(NB - 1, max(0, (int)((v - lo) * scale))); }
};
// Minimum that a NaN on either side makes NaN.  A list's range is NaN then, its scale 0, and the list not regular.
__device__ __forceinline__ float min_or_nan(float a, float b) {
  float r;
  asm("min.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}
template <int NT, int NB>
__device__ __forceinline__ ScoreBins count_committed(SelectSmem<NT, NB>& sm, const float* list, int n_csa) {
  constexpr int NW = NT / 32;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  float lo = INFINITY, hi = -INFINITY;
  each_score<NT>(list, n_csa, [&](int, float v) { lo = min_or_nan(lo, v); hi = fmaxf(hi, v); });
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) { lo = min_or_nan(lo, __shfl_xor_sync(0xffffffffu, lo, o)); hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o)); }
  if (lane == 0) { sm.red[0][w] = lo; sm.red[1][w] = hi; }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < NW; ++i) { lo = min_or_nan(lo, sm.red[0][i]); hi = fmaxf(hi, sm.red[1][i]); }
  ScoreBins bins;
  bins.lo = lo;
  bins.scale = hi > lo ? (float)NB / (hi - lo) : 0.f;
  bins.regular = bins.scale > 0.f && bins.scale < 1e30f;
  if (bins.regular) each_score<NT>(list, n_csa, [&](int, float v) { atomicAdd(&sm.hist[bins.of<NB>(v)], 1); });
  return bins;
}

// Second part (after a barrier; the histogram is complete).  bits: zero.  lists: write the index list; selmask: a bit per candidate
// for the tile plan, or null.
template <int NT, int NB>
__device__ __forceinline__ void select_node(SelectSmem<NT, NB>& sm, const ScoreBins& bins, const float* list, uint32_t* bits, int n_cand, int n_csa,
                                            const PathEntries& pe, int k, bool lists, int32_t* sel, int32_t* usr, int32_t* selcnt, uint32_t* selmask) {
  constexpr int NW = NT / 32;
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  auto bin_of = [&](float v) { return bins.of<NB>(v); };
  int m = CAP + 1, bstar = 0, rem = k;
  if (bins.regular) {
    // thread t holds intervals NB - 1 - t PER .. down: exclusive sum from the top
    constexpr int PER = NB / NT;
    int h[PER], tot = 0;
#pragma unroll
    for (int j = 0; j < PER; ++j) { h[j] = sm.hist[NB - 1 - (t * PER + j)]; tot += h[j]; }
    int incl = tot;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const int y = __shfl_up_sync(0xffffffffu, incl, o); if (lane >= o) incl += y; }
    if (lane == 31) sm.wsum[0][w] = incl;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < NW; ++i) if (i < w) incl += sm.wsum[0][i];
    int cum = incl - tot;
    if (cum < k && incl >= k) {                          // exactly one thread
#pragma unroll
      for (int j = 0; j < PER; ++j) {
        if (cum + h[j] >= k) { sm.bin = NB - 1 - (t * PER + j); sm.rem = k - cum; break; }
        cum += h[j];
      }
    }
    __syncthreads();
    bstar = sm.bin; rem = sm.rem;
    each_score<NT>(list, n_cand, [&](int i, float v) {
      if (bin_of(v) == bstar) { const int pos = atomicAdd(&sm.cnt, 1); if (pos < CAP) { sm.cand_s[pos] = v; sm.cand_i[pos] = i; } }
    });
    __syncthreads();
    m = sm.cnt;
    if (m <= CAP) {
      for (int x = t; x < m; x += NT) {
        const float v = sm.cand_s[x];
        const int ix = sm.cand_i[x];
        int r = 0;
        for (int y = 0; y < m; ++y) { const float u = sm.cand_s[y]; r += (u > v || (u == v && sm.cand_i[y] < ix)) ? 1 : 0; }
        if (r < rem) atomicOr(&bits[ix >> 5], 1u << (ix & 31));
      }
      __syncthreads();
    }
  }
  uint32_t thr = 0;
  const bool radix = m > CAP;
  if (radix) {                                           // four passes of 8 bits over the order-preserving keys
    uint32_t mask = 0;
    rem = k;
#pragma unroll 1
    for (int pass = 0; pass < 4; ++pass) {
      const int shift = 24 - 8 * pass;
      __syncthreads();
      for (int i = t; i < 256; i += NT) sm.hist[i] = 0;
      __syncthreads();
      for (int i = t; i < n_cand; i += NT) { const uint32_t key = order_key(list[i]); if ((key & mask) == thr) atomicAdd(&sm.hist[(key >> shift) & 255u], 1); }
      __syncthreads();
      // every warp finds the interval of the rem-th largest for itself: lane l owns bins 255 - 8 l .. 248 - 8 l
      int h[8], tot = 0;
#pragma unroll
      for (int j = 0; j < 8; ++j) { h[j] = sm.hist[255 - (lane * 8 + j)]; tot += h[j]; }
      int incl = tot;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) { const int y = __shfl_up_sync(0xffffffffu, incl, o); if (lane >= o) incl += y; }
      const bool own = incl - tot < rem && incl >= rem;  // exactly one lane
      int cum = incl - tot, bin = 255 - lane * 8;
      if (own) {
#pragma unroll
        for (int j = 0; j < 8; ++j) { if (cum + h[j] >= rem) { bin = 255 - (lane * 8 + j); break; } cum += h[j]; }
      }
      const int src = __ffs(__ballot_sync(0xffffffffu, own)) - 1;
      thr |= (uint32_t)__shfl_sync(0xffffffffu, bin, src) << shift;
      rem -= __shfl_sync(0xffffffffu, cum, src);
      mask |= 0xFFu << shift;
    }
  }
  // Warp w owns the candidates [w * part, (w + 1) * part), rows of 32.  above: certainly taken; edge (radix only): equal to the
  // threshold, of which the first rem in index order are taken.
  const int part = ((n_cand + NW - 1) / NW + 31) & ~31, beg = min(n_cand, w * part), end = min(n_cand, beg + part);
  constexpr int U = 4;                                   // rows of 32 candidates taken together
  auto classify = [&](int i0, bool (&above)[U], bool (&edge)[U]) {
    float v[U];
    uint32_t word[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i = i0 + 32 * u + lane;
      v[u] = i < end ? list[i] : 0.f;
      word[u] = i0 + 32 * u < end ? bits[(i0 >> 5) + u] : 0u;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (radix) { const uint32_t key = order_key(v[u]); above[u] = key > thr; edge[u] = key == thr; }
      else { const int bn = bin_of(v[u]); above[u] = bn > bstar || (bn == bstar && ((word[u] >> lane) & 1u)); edge[u] = false; }
      if (i0 + 32 * u + lane >= end) above[u] = edge[u] = false;
    }
  };
  int pos = 0, eq_base = 0;
  if (lists || radix) {
    int ca = 0, ce = 0;
    for (int i0 = beg; i0 < end; i0 += 32 * U) {
      bool above[U], edge[U];
      classify(i0, above, edge);
#pragma unroll
      for (int u = 0; u < U; ++u) { ca += __popc(__ballot_sync(0xffffffffu, above[u])); ce += __popc(__ballot_sync(0xffffffffu, edge[u])); }
    }
    __syncthreads();
    if (lane == 0) { sm.wsum[0][w] = ca; sm.wsum[1][w] = ce; }
    __syncthreads();
    for (int i = 0; i < w; ++i) { pos += sm.wsum[0][i]; eq_base += sm.wsum[1][i]; }
    if (radix) pos += min(rem, eq_base);
  }
  const uint32_t lt = (1u << lane) - 1u;
  for (int i0 = beg; i0 < end; i0 += 32 * U) {
    bool above[U], edge[U];
    classify(i0, above, edge);
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int r0 = i0 + 32 * u, i = r0 + lane;
      if (r0 >= end) break;                              // (uniform in the warp)
      bool take = above[u];
      if (radix) {
        const uint32_t eqm = __ballot_sync(0xffffffffu, edge[u]);
        take = take || (edge[u] && eq_base + __popc(eqm & lt) < rem);
        eq_base += __popc(eqm);
      }
      const uint32_t tkm = __ballot_sync(0xffffffffu, take);
      if (selmask && lane == 0) selmask[r0 >> 5] = tkm;
      if (lists) {
        if (take) {
          const int p = pos + __popc(tkm & lt), val = i < n_csa ? i : pe.newc_blk[i - n_csa];
          sel[p] = val; if (usr) usr[p] = val;
        }
        pos += __popc(tkm);
      }
    }
  }
  if (lists && t == 0) *selcnt = k;
}

}  // namespace ssel

// `cap`: floats of the score list (covers the padded shares of the eight CTAs and the in-tree entries).
template <bool PAGED, typename T>
__global__ void __launch_bounds__(128, 4) topk_seq_kernel(const tsv_shape s, const TvaPlan pl, const tsv_cache c, const tsv_nodes nd,
                                                         const tsv_scratch sc, int32_t* __restrict__ topk_user, char* __restrict__ ws,
                                                         int32_t* __restrict__ status, const int cap) {
  using namespace ssel;
  constexpr int NT = 128, NB = 1024, NW = NT / 32;
  constexpr bool BF = sizeof(T) == 2;
  extern __shared__ __align__(128) unsigned char dsm[];
  __shared__ TreeMeta tm;
  __shared__ TreeStage tstage;
  __shared__ PathEntries pe;
  __shared__ SelectSmem<NT, NB> sm;
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");   // the tile plan may start its selection-independent part
  const int rank = blockIdx.x, b = blockIdx.y, D = s.D, k = s.topk, HI = s.HI;
  const bool lists = !pl.tc || topk_user;               // somebody reads the index lists (the tile plan reads mask rows only)
  // (all that depends on the sequence alone is requested together: one memory latency)
  const TreeFetch tf = fetch_tree(s, c.L + b, nd.parent + (size_t)b * D, nd.n_nodes + b, c.csa_cap + b, c.hca_cap + b);
  const int L0 = c.L[b];
  const int64_t row0 = PAGED ? 0 : c.csa_row0[b];
  // some node may have more than k candidates (and the rows exist: a sequence of bad length or capacity is flagged below)
  const bool any_rank = L0 >= 0 && (int64_t)L0 + D <= s.max_L && (L0 + D) / s.m_csa <= c.csa_cap[b] && L0 / s.m_csa + D > k;
  if (!any_rank && !lists && rank != 0) return;          // (alike in the whole cluster but for CTA 0, which validates the sequence)
  const Layout lay(NW, cap);
  const uint32_t smem_s = (uint32_t)__cvta_generic_to_shared(dsm);
  float* loc = reinterpret_cast<float*>(dsm + lay.loc) + w * 128;
  float* list = reinterpret_cast<float*>(dsm + lay.sc);
  uint32_t* bits = reinterpret_cast<uint32_t*>(dsm + lay.bits);
  if (any_rank) cluster_arrive();                        // (every CTA runs before a peer writes to it; awaited before the first write)
  // this CTA's entries (a multiple of sixteen but for the end of the list)
  const int n_ent = any_rank ? L0 / s.m_csa : 0;
  const int share = ((n_ent + CS - 1) / CS + 15) & ~15, e0 = min(n_ent, rank * share), e1 = min(n_ent, e0 + share);
  Scorer sco;
  sco.g = lane >> 2; sco.tq = lane & 3; sco.end = e1;
  uint4 alo[4], ahi[4];
  const int first = e0 + 16 * w;
  if (any_rank) {
    if (PAGED) sco.rows = csa_rows_of(c, s, b); else { sco.rows.pt = nullptr; sco.rows.per_page = 1; sco.rows.row0 = row0; }
    sco.ikb = reinterpret_cast<const char*>(c.csa_ik) + (size_t)sco.rows.row0 * ROWB + (BF ? sco.tq * 16 : 0);
    if (BF && first < e1) sco.template fetch<PAGED>(first, alo, ahi);
    stage_queries(dsm, nd.iq, b, 0, D, HI);
    if (BF) sco.weights(nd.iw + (size_t)b * D * HI, 0, D, HI);
    else if (t < 32) reinterpret_cast<float*>(dsm + lay.loc)[t] = (t >> 2) < D && (t & 3) < HI ? __ldg(nd.iw + ((size_t)b * D + (t >> 2)) * HI + (t & 3)) : 0.f;
    for (int i = t; i < (cap + 31) / 32; i += NT) bits[i] = 0u;
    for (int i = t; i < NB; i += NT) sm.hist[i] = 0;
    if (t == 0) sm.cnt = 0;
  }
  derive_tree_meta(tm, tstage, s, tf, true, true);
  if (t == 0 && rank == 0 && tm.status) atomicOr(status + b, tm.status);
  const int n = rank;                                    // the node this CTA owns
  const bool live = !tm.status && n < tm.nn;
  const int n_csa = tm.n_csa;
  if (t < 32) path_of(pe, tm, s, n, live);
  __syncthreads();                                       // (the path entries: a warp without entries to score reads them at once)
  const int n_cand = live ? n_csa + pe.n_newc : 0;
  const bool ranks = any_rank && n_cand > k;             // (a node that ranks is of a sequence that may)
  ExtraScorer<T> ex;
  ScoreBins bins = {0.f, 0.f, false};
  // (a sequence flagged for its tree is scored too -- its rows exist -- and then dropped)
  if (any_rank) {
    cluster_wait();                                      // the peers run
    if constexpr (BF) {
    for (int e = first; e < e1; e += 16 * NW) {
      uint4 nlo[4], nhi[4];
      const bool more = e + 16 * NW < e1;
      if (more) sco.template fetch<PAGED>(e + 16 * NW, nlo, nhi);
      sco.score(alo, ahi, dsm, loc);
      // lane l: four entries of node l / 4 (up to three past the end of the list: overwritten below or never read)
      const float4 v = *reinterpret_cast<const float4*>(loc + 4 * lane);
      if ((lane >> 2) < D && e + 4 * (lane & 3) < e1)
        asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(map_to_rank(smem_s + lay.sc + (uint32_t)(e + 4 * (lane & 3)) * 4, lane >> 2)),
                     "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
      if (more) {
#pragma unroll
        for (int q = 0; q < 4; ++q) { alo[q] = nlo[q]; ahi[q] = nhi[q]; }
      }
    }
    } else {
      const float* iws = reinterpret_cast<const float*>(dsm + lay.loc);
      for (int e = e0 + 32 * w + lane; e < e1; e += 32 * NW) {
        const float4* row = reinterpret_cast<const float4*>(sco.ikb + (size_t)(PAGED ? sco.rows.rel(e) : (int64_t)e) * ROWB);
        float4 r[16];
#pragma unroll
        for (int x = 0; x < 16; ++x) r[x] = __ldg(row + x);
#pragma unroll 1
        for (int n = 0; n < D; ++n) {
          float tot = 0.f;
#pragma unroll 1
          for (int h = 0; h < HI; ++h) {
            const float4* q = reinterpret_cast<const float4*>(dsm + (4 * n + h) * QP);
            float p[8];
#pragma unroll
            for (int x = 0; x < 8; ++x) {               // partial sum x: pieces x and x + 8 of the row
              const float4 a = q[x], c2 = q[x + 8];
              p[x] = fmaf(a.w, r[x].w, fmaf(a.z, r[x].z, fmaf(a.y, r[x].y, a.x * r[x].x)));
              p[x] = fmaf(c2.w, r[x + 8].w, fmaf(c2.z, r[x + 8].z, fmaf(c2.y, r[x + 8].y, fmaf(c2.x, r[x + 8].x, p[x]))));
            }
            const float d = ((p[0] + p[1]) + (p[2] + p[3])) + ((p[4] + p[5]) + (p[6] + p[7]));
            tot = fmaf(iws[4 * n + h], fmaxf(d, 0.f), tot);
          }
          asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(map_to_rank(smem_s + lay.sc + (uint32_t)e * 4, n)), "f"(tot) : "memory");
        }
      }
    }
    __syncwarp();
    cluster_arrive();                                    // this CTA's scores are on their way
    if (ranks) ex.fetch(s, nd, b, n);
    cluster_wait();                                      // every peer's scores of this node are in the list; nobody touches a peer's memory from here on
    // (the histogram before the wait: it runs under the state build's tail like all of the above.  Counted after it, with the
    // queries of the in-tree entries fetched then too, one sequence of 4 k tokens took 40.9 us a pass, not 38.9; 64 grown ones no
    // more than the runs differ)
    if (ranks) bins = count_committed(sm, list, n_csa);
    // the state build's results: the first thing of that kernel this CTA reads
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (ranks)
      ex.score(pe, s, sc, b, [&](int i, float v) {
        list[n_csa + i] = v;
        if (v != v) atomicAdd(&sm.cnt, CAP + 1);         // (a NaN: the selection finds its interval overfull and takes the radix passes)
        if (bins.regular) atomicAdd(&sm.hist[bins.of<NB>(v)], 1);
      });
  } else if (rank == 0 && b == 0) {
    asm volatile("griddepcontrol.wait;" ::: "memory");   // (so that this kernel's completion implies the state build's)
  }
  __syncthreads();
  if (n >= D) return;
  int32_t* sel = reinterpret_cast<int32_t*>(ws + pl.off_sel) + ((size_t)b * D + n) * k;
  int32_t* selcnt = reinterpret_cast<int32_t*>(ws + pl.off_selcnt) + (size_t)b * D + n;
  int32_t* usr = topk_user ? topk_user + ((size_t)b * D + n) * k : nullptr;
  if (!ranks) {
    if (lists) select_all(n_cand, n_csa, pe, k, sel, usr, selcnt);
    return;
  }
  uint32_t* selmask = pl.tc ? reinterpret_cast<uint32_t*>(ws + pl.off_selmask) + ((size_t)b * D + n) * pl.mask_ld : nullptr;   // (for the tile plan)
  select_node(sm, bins, list, bits, n_cand, n_csa, pe, k, lists, sel, usr, selcnt, selmask);
}

// ------------------------------------------------------------------------------------------------ long lists
// Scores of all nodes of a sequence into the workspace.  grid (entry blocks, B, groups of eight nodes), four warps, kRowSteps steps
// of sixteen entries each; reads the caller's data and the committed caches only, so it runs under the state build's tail.
constexpr int kRowSteps = 4;
template <bool PAGED>
__global__ void __launch_bounds__(128) score_rows_kernel(const tsv_shape s, const TvaPlan pl, const tsv_cache c, const tsv_nodes nd, char* __restrict__ ws) {
  using namespace ssel;
  __shared__ __align__(16) unsigned char qs[32 * QP];
  __shared__ __align__(16) float bufs[4][128];
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");   // the selection waits for this kernel before it reads a score
  const int t = threadIdx.x, lane = t & 31, w = t >> 5, b = blockIdx.y, n0 = 8 * blockIdx.z, D = s.D, HI = s.HI;
  const int L0 = c.L[b];
  // (the rows exist: a sequence of bad length or capacity is flagged by the selection)
  const bool any_rank = L0 >= 0 && (int64_t)L0 + D <= s.max_L && (L0 + D) / s.m_csa <= c.csa_cap[b] && L0 / s.m_csa + D > s.topk;
  const int n_ent = any_rank ? L0 / s.m_csa : 0;
  const int first = (blockIdx.x * kRowSteps * 4 + w) * 16;
  if ((int)(blockIdx.x * kRowSteps * 64) >= n_ent) {
    if (blockIdx.x == 0 && b == 0 && blockIdx.z == 0) asm volatile("griddepcontrol.wait;" ::: "memory");   // (this kernel's completion implies the state build's)
    return;
  }
  Scorer sco;
  sco.g = lane >> 2; sco.tq = lane & 3; sco.end = n_ent;
  if (PAGED) sco.rows = csa_rows_of(c, s, b); else { sco.rows.pt = nullptr; sco.rows.per_page = 1; sco.rows.row0 = c.csa_row0[b]; }
  sco.ikb = reinterpret_cast<const char*>(c.csa_ik) + (size_t)sco.rows.row0 * (DI * 2) + sco.tq * 16;
  uint4 alo[4], ahi[4], nlo[4], nhi[4];
  sco.fetch<PAGED>(min(first, n_ent - 1), alo, ahi);
  stage_queries(qs, nd.iq, b, n0, D, HI);
  sco.weights(nd.iw + (size_t)b * D * HI, n0, D, HI);
  __syncthreads();
  float* scores = reinterpret_cast<float*>(ws + pl.off_scores) + (size_t)b * D * pl.score_ld;
  // No wait before the scores are written where the kernel before is this call's state build, whose dependents start when it has
  // waited for all earlier work (the call before on this workspace included): without it, and with the ranges kept below, four
  // sequences of 128 k tokens took 4 % less a pass.  In a call without the state build the kernel before may be any, such as a
  // selection that signals at its start and still reads scores and ranges.
  if (!pl.built) asm volatile("griddepcontrol.wait;" ::: "memory");
  float lo = INFINITY, hi = -INFINITY;                   // of node n0 + lane / 4, over this warp's entries (a NaN stays in lo)
#pragma unroll
  for (int st = 0; st < kRowSteps; ++st) {
    const int e = first + st * 64;
    if (e >= n_ent) break;
    if (st + 1 < kRowSteps) sco.fetch<PAGED>(min(e + 64, n_ent - 1), nlo, nhi);
    sco.score(alo, ahi, qs, bufs[w]);
    const float4 v = *reinterpret_cast<const float4*>(bufs[w] + 4 * lane);
    const int n = n0 + (lane >> 2), i = e + 4 * (lane & 3);            // (rows of the score array are padded to whole float4)
    if (n < D && i < n_ent) {                            // (entries past the last one are copies of it)
      *reinterpret_cast<float4*>(scores + (size_t)n * pl.score_ld + i) = v;
      lo = min_or_nan(min_or_nan(lo, v.x), min_or_nan(min_or_nan(v.y, v.z), v.w));
      hi = fmaxf(fmaxf(hi, v.x), fmaxf(fmaxf(v.y, v.z), v.w));
    }
    if (st + 1 < kRowSteps) {
#pragma unroll
      for (int q = 0; q < 4; ++q) { alo[q] = nlo[q]; ahi[q] = nhi[q]; }
    }
  }
  // The range of the scores for the selection, which bins them: two passes over the list and a cluster barrier less there (where there is
  // no room for the ranges, it makes those).
#pragma unroll
  for (int o = 1; o < 4; o <<= 1) { lo = min_or_nan(lo, __shfl_xor_sync(0xffffffffu, lo, o)); hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o)); }
  if (pl.ext_ld && (lane & 3) == 0 && n0 + (lane >> 2) < D)
    reinterpret_cast<float2*>(ws + pl.off_ext)[((size_t)b * D + n0 + (lane >> 2)) * pl.ext_ld + blockIdx.x * 4 + w] = make_float2(lo, hi);
  if (blockIdx.x == 0 && b == 0 && blockIdx.z == 0) asm volatile("griddepcontrol.wait;" ::: "memory");   // (this kernel's completion implies the state build's)
}

// Selection of one node from the score array by a cluster of eight CTAs: grid (8 D, B).  A CTA keeps its share of the list in
// shared memory; what the CTAs need of one another (extrema, histogram, the candidates of one interval) each leaves in its own
// shared memory and pulls from the others' after a cluster barrier.  (One CTA per node took 20 us over 32768 candidates.)
constexpr int kListThreads = 512, kListBins = 1024;
struct ListSmem {
  int hist[2][kListBins];                                // [0] the intervals; both: the digits of the radix passes
  float2 ext;
  int cnt[2];                                            // candidates; (entries certainly taken, entries equal to the threshold)
  int eqs;
  float cand_s[ssel::CAP];
  int cand_i[ssel::CAP];
  float all_s[ssel::CAP];
  int all_i[ssel::CAP];
  float red[2][kListThreads / 32];
  int wsum[2][kListThreads / 32];
  int bin, rem;
};
__global__ void __launch_bounds__(kListThreads, 2) topk_list_kernel(const tsv_shape s, const TvaPlan pl, const tsv_cache c, const tsv_nodes nd,
                                                                 const tsv_scratch sc, int32_t* __restrict__ topk_user, char* __restrict__ ws,
                                                                 int32_t* __restrict__ status) {
  using namespace ssel;
  constexpr int NT = kListThreads, NW = NT / 32, NB = kListBins;
  extern __shared__ __align__(128) unsigned char dsm[];
  __shared__ TreeMeta tm;
  __shared__ TreeStage tstage;
  __shared__ PathEntries pe;
  __shared__ float extra[TSV_MAX_D];
  __shared__ __align__(16) ListSmem sm;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");   // the tile plan may start its selection-independent part
  const int t = threadIdx.x, lane = t & 31, w = t >> 5, rank = blockIdx.x % CS, n = blockIdx.x / CS, b = blockIdx.y, D = s.D, k = s.topk;
  const bool lists = !pl.tc || topk_user;
  coop_tree_meta(tm, tstage, s, c.L + b, nd.parent + (size_t)b * D, nd.n_nodes + b, c.csa_cap + b, c.hca_cap + b);
  if (t == 0 && n == 0 && rank == 0 && tm.status) atomicOr(status + b, tm.status);
  const bool live = !tm.status && n < tm.nn;
  const int n_csa = tm.n_csa;
  if (t < 32) path_of(pe, tm, s, n, live);
  for (int i = t; i < NB; i += NT) { sm.hist[0][i] = 0; sm.hist[1][i] = 0; }
  if (t == 0) { sm.cnt[0] = sm.cnt[1] = 0; sm.eqs = 0; }
  __syncthreads();
  int32_t* sel = reinterpret_cast<int32_t*>(ws + pl.off_sel) + ((size_t)b * D + n) * k;
  int32_t* selcnt = reinterpret_cast<int32_t*>(ws + pl.off_selcnt) + (size_t)b * D + n;
  int32_t* usr = topk_user ? topk_user + ((size_t)b * D + n) * k : nullptr;
  const int n_cand = live ? n_csa + pe.n_newc : 0;
  // (every exit is taken by the whole cluster alike)
  asm volatile("griddepcontrol.wait;" ::: "memory");   // the scores, and (the scoring kernel waited) the entries closed inside the tree
  if (n_cand <= k) {
    if (lists && rank == 0) select_all(n_cand, n_csa, pe, k, sel, usr, selcnt);
    return;
  }
  // this CTA's candidates [c0, c1), a multiple of 32 but for the end of the list
  const int per = ((n_cand + CS - 1) / CS + 31) & ~31, c0 = min(n_cand, rank * per), c1 = min(n_cand, c0 + per), len = c1 - c0;
  float* list = reinterpret_cast<float*>(dsm);
  uint32_t* bits = reinterpret_cast<uint32_t*>(list + (((pl.score_ld + TSV_MAX_D + CS - 1) / CS + 63) & ~31));
  for (int i = t; i < (len + 31) / 32; i += NT) bits[i] = 0u;
  const float4* src = reinterpret_cast<const float4*>(reinterpret_cast<const float*>(ws + pl.off_scores) + ((size_t)b * D + n) * pl.score_ld + c0);
  float lo = INFINITY, hi = -INFINITY;                 // the range of the committed entries' scores
  const float2* ext = reinterpret_cast<const float2*>(ws + pl.off_ext) + ((size_t)b * D + n) * pl.ext_ld;
  for (int i = t; i < (pl.ext_ld ? (n_csa + 255) / 256 * 4 : 0); i += NT) { const float2 x = __ldcg(ext + i); lo = min_or_nan(lo, x.x); hi = fmaxf(hi, x.y); }
  const int n4 = (min(c1, n_csa) - c0 + 3) >> 2;       // (negative: none)
  for (int i = t; i < n4; i += NT) reinterpret_cast<float4*>(list)[i] = __ldcg(src + i);
  if (c1 > n_csa) {
    ExtraScorer<bf16> ex;
    ex.fetch(s, nd, b, n);
    ex.score(pe, s, sc, b, [&](int i, float v) {
      extra[i] = v;
      if (v != v && n_csa + i >= c0 && n_csa + i < c1) atomicAdd(&sm.cnt[0], CAP + 1);      // (a NaN: the interval is found overfull, the radix passes follow)
    });
    __syncthreads();
    for (int i = max(n_csa, c0) + t; i < c1; i += NT) list[i - c0] = extra[i - n_csa];
  }
  __syncthreads();
  if (!pl.ext_ld)                                        // (the range of this CTA's share, the in-tree entries with it)
    for (int i = t; i < len; i += NT) { const float v = list[i]; lo = min_or_nan(lo, v); hi = fmaxf(hi, v); }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) { lo = min_or_nan(lo, __shfl_xor_sync(0xffffffffu, lo, o)); hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o)); }
  if (lane == 0) { sm.red[0][w] = lo; sm.red[1][w] = hi; }
  __syncthreads();
  lo = sm.red[0][lane % NW]; hi = sm.red[1][lane % NW];
#pragma unroll
  for (int o = NW / 2; o > 0; o >>= 1) { lo = min_or_nan(lo, __shfl_xor_sync(0xffffffffu, lo, o)); hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o)); }
  auto peer = [&](const void* p, int r) { return map_to_rank((uint32_t)__cvta_generic_to_shared(p), r); };
  auto peer_i = [&](const int* p, int r) { int v; asm volatile("ld.shared::cluster.s32 %0, [%1];" : "=r"(v) : "r"(peer(p, r))); return v; };
  auto peer_f = [&](const float* p, int r) { float v; asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(peer(p, r))); return v; };
  auto meet = [&]() { __syncthreads(); cluster_arrive(); cluster_wait(); };
  if (!pl.ext_ld) {                                      // the ranges of all CTAs' shares
    if (t == 0) sm.ext = make_float2(lo, hi);
    meet();
    lo = peer_f(&sm.ext.x, lane & 7); hi = peer_f(&sm.ext.y, lane & 7);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) { lo = min_or_nan(lo, __shfl_xor_sync(0xffffffffu, lo, o)); hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o)); }
  }
  const float scale = hi > lo ? (float)NB / (hi - lo) : 0.f;
  const bool regular = scale > 0.f && scale < 1e30f;     // (else: all equal, not finite, a NaN among them, or too narrow)
  auto bin_of = [&](float v) { return min(NB - 1, max(0, (int)((v - lo) * scale))); };      // (in-tree entries may lie beyond the range)
  // the interval (of nb in h, over the whole cluster) of the rem-th largest: its number, and what of rem is left in it
  auto locate = [&](const int* h, int nb, int rem, int& bin, int& left) {
    int v[2] = {0, 0};
    const int hi2 = nb - 2 - 2 * t;                      // thread t: intervals nb - 1 - 2 t and nb - 2 - 2 t
    if (hi2 >= 0) {
      int x[CS], y[CS];
#pragma unroll
      for (int r = 0; r < CS; ++r) asm volatile("ld.shared::cluster.v2.s32 {%0, %1}, [%2];" : "=r"(x[r]), "=r"(y[r]) : "r"(peer(h + hi2, r)));
#pragma unroll
      for (int r = 0; r < CS; ++r) { v[0] += y[r]; v[1] += x[r]; }
    }
    int incl = v[0] + v[1];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const int y = __shfl_up_sync(0xffffffffu, incl, o); if (lane >= o) incl += y; }
    if (lane == 31) sm.wsum[0][w] = incl;
    __syncthreads();
#pragma unroll 1
    for (int i = 0; i < w; ++i) incl += sm.wsum[0][i];
    const int excl = incl - v[0] - v[1];
    if (excl < rem && incl >= rem) {                     // exactly one thread
      const bool first = excl + v[0] >= rem;
      sm.bin = hi2 + (first ? 1 : 0); sm.rem = rem - excl - (first ? 0 : v[0]);
    }
    __syncthreads();
    bin = sm.bin; left = sm.rem;
  };
  int m = CAP + 1, bstar = 0, rem = k;
  if (regular) {
    for (int i = t; i < len; i += NT) atomicAdd(&sm.hist[0][bin_of(list[i])], 1);
    meet();
    locate(sm.hist[0], NB, k, bstar, rem);
    for (int i = t; i < len; i += NT) {
      const float v = list[i];
      if (bin_of(v) == bstar) { const int pos = atomicAdd(&sm.cnt[0], 1); if (pos < CAP) { sm.cand_s[pos] = v; sm.cand_i[pos] = c0 + i; } }
    }
    meet();
    int base[CS + 1];
    base[0] = 0;
#pragma unroll
    for (int r = 0; r < CS; ++r) base[r + 1] = base[r] + peer_i(&sm.cnt[0], r);
    m = base[CS];
    if (m <= CAP) {
      for (int x = t; x < m; x += NT) {
        int r = 0, at = x;
#pragma unroll
        for (int q = 1; q < CS; ++q) if (x >= base[q]) { r = q; at = x - base[q]; }
        sm.all_s[x] = peer_f(&sm.cand_s[at], r); sm.all_i[x] = peer_i(&sm.cand_i[at], r);
      }
      __syncthreads();
      const int own = sm.cnt[0];
      for (int x = t; x < own; x += NT) {
        const float v = sm.cand_s[x];
        const int ix = sm.cand_i[x];
        int r = 0;
        for (int y = 0; y < m; ++y) { const float u = sm.all_s[y]; r += (u > v || (u == v && sm.all_i[y] < ix)) ? 1 : 0; }
        if (r < rem) atomicOr(&bits[(ix - c0) >> 5], 1u << (ix & 31));
      }
      __syncthreads();
    }
  }
  uint32_t thr = 0;
  const bool radix = m > CAP;                            // (alike in the cluster)
  if (radix) {                                           // four passes of 8 bits over the order-preserving keys
    uint32_t mask = 0;
    rem = k;
    meet();                                              // (everyone has pulled the intervals)
    for (int i = t; i < 256; i += NT) { sm.hist[0][i] = 0; sm.hist[1][i] = 0; }
    __syncthreads();
#pragma unroll 1
    for (int pass = 0; pass < 4; ++pass) {
      const int shift = 24 - 8 * pass, buf = pass & 1;
      for (int i = t; i < len; i += NT) { const uint32_t key = order_key(list[i]); if ((key & mask) == thr) atomicAdd(&sm.hist[buf][(key >> shift) & 255u], 1); }
      meet();
      for (int i = t; i < 256; i += NT) sm.hist[buf ^ 1][i] = 0;       // (pulled by everyone before this barrier)
      int bin;
      locate(sm.hist[buf], 256, rem, bin, rem);
      thr |= (uint32_t)bin << shift;
      mask |= 0xFFu << shift;
    }
  }
  // Warp w owns the candidates [w * part, (w + 1) * part) of the share, rows of 32.  above: certainly taken; edge (radix only): equal
  // to the threshold, of which the first rem in index order are taken.
  const int part = ((len + NW - 1) / NW + 31) & ~31, beg = min(len, w * part), end = min(len, beg + part);
  auto classify = [&](int i, bool& above, bool& edge) {
    above = edge = false;
    if (i >= end) return;
    const float v = list[i];
    if (radix) { const uint32_t key = order_key(v); above = key > thr; edge = key == thr; }
    else { const int bn = bin_of(v); above = bn > bstar || (bn == bstar && ((bits[i >> 5] >> (i & 31)) & 1u)); }
  };
  int pos = 0, eq_base = 0;
  if (lists || radix) {
    int ca = 0, ce = 0;
    for (int i0 = beg; i0 < end; i0 += 32) {
      bool above, edge;
      classify(i0 + lane, above, edge);
      ca += __popc(__ballot_sync(0xffffffffu, above)); ce += __popc(__ballot_sync(0xffffffffu, edge));
    }
    __syncthreads();
    if (lane == 0) { sm.wsum[0][w] = ca; sm.wsum[1][w] = ce; }
    __syncthreads();
    if (t == 0) { int a = 0, e = 0; for (int i = 0; i < NW; ++i) { a += sm.wsum[0][i]; e += sm.wsum[1][i]; } sm.cnt[1] = a; sm.eqs = e; }
    meet();
    for (int r = 0; r < rank; ++r) { pos += peer_i(&sm.cnt[1], r); eq_base += peer_i(&sm.eqs, r); }
    for (int i = 0; i < w; ++i) { pos += sm.wsum[0][i]; eq_base += sm.wsum[1][i]; }
    if (radix) pos += min(rem, eq_base);
  }
  uint32_t* selmask = pl.tc ? reinterpret_cast<uint32_t*>(ws + pl.off_selmask) + ((size_t)b * D + n) * pl.mask_ld : nullptr;   // (for the tile plan)
  const uint32_t lt = (1u << lane) - 1u;
  for (int i0 = beg; i0 < end; i0 += 32) {
    const int i = i0 + lane;
    bool take, edge;
    classify(i, take, edge);
    if (radix) {
      const uint32_t eqm = __ballot_sync(0xffffffffu, edge);
      take = take || (edge && eq_base + __popc(eqm & lt) < rem);
      eq_base += __popc(eqm);
    }
    const uint32_t tkm = __ballot_sync(0xffffffffu, take);
    if (selmask && lane == 0) selmask[(c0 + i0) >> 5] = tkm;
    if (lists) {
      if (take) {
        const int p = pos + __popc(tkm & lt), val = c0 + i < n_csa ? c0 + i : pe.newc_blk[c0 + i - n_csa];
        sel[p] = val; if (usr) usr[p] = val;
      }
      pos += __popc(tkm);
    }
  }
  if (lists && rank == 0 && t == 0) *selcnt = k;
  cluster_arrive();                                      // no CTA leaves while a peer may still read its memory
  cluster_wait();
}

// ------------------------------------------------------------------------------------------------ dispatch
static int seq_cap(const tsv_shape& s) {                 // padded shares of eight CTAs, the in-tree entries
  const int ent = (int)(s.max_L / s.m_csa), share = ((ent + ssel::CS - 1) / ssel::CS + 15) & ~15;
  return (share * ssel::CS + TSV_MAX_D + 127) & ~127;
}
static size_t list_bytes(const TvaPlan& p) {             // a share of the list, a bit per candidate of it
  const size_t fl = (((size_t)p.score_ld + TSV_MAX_D + ssel::CS - 1) / ssel::CS + 63) & ~(size_t)31;
  return fl * 4 + (fl + 31) / 32 * 4;
}
// The cluster form: its CTAs are small and all resident up to some 70 sequences; beyond kSeqMax entries a node's list is the work of
// too few threads.
static bool seq_form(const tsv_shape& s) { return s.D <= ssel::CS && s.max_L / s.m_csa <= ssel::kSeqMax; }

// 256-byte indexer rows, at most four heads.  fp32: the cluster form's lists.  bf16: lists that fit the cluster's shared memory as scores and are too long for
// topk_fused_kernel (which is the shorter chain while a list is three keys a thread).
bool topk_seq_applies(const tsv_shape& s, const TvaPlan& p) {
  if (p.need_scores && s.dtype == TSV_FP32) return s.di * 4 == ssel::ROWB && s.HI <= ssel::HMAX && seq_form(s);
  return p.need_scores && s.dtype == TSV_BF16 && s.di == ssel::DI && s.HI <= ssel::HMAX && !topk_fused_applies(s, p) &&
         (seq_form(s) || list_bytes(p) <= 200 * 1024);
}

int launch_topk_seq(const tsv_shape& s, const TvaPlan& p, const tsv_cache& c, const tsv_nodes& nd, const tsv_scratch& sc,
                    int32_t* topk_idx, char* ws, int32_t* status, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;          // may start under the tail of the kernel before (it waits inside)
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = ssel::CS; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cudaError_t e;
  if (seq_form(s)) {
    const int cap = seq_cap(s);
    const int bytes = (int)ssel::Layout(4, cap).total;
    cfg.numAttrs = 2;
    cfg.gridDim = dim3(ssel::CS, s.B, 1); cfg.blockDim = dim3(128, 1, 1); cfg.dynamicSmemBytes = bytes;
    TSV_PREP((topk_seq_kernel<true, bf16>)); TSV_PREP((topk_seq_kernel<false, bf16>)); TSV_PREP((topk_seq_kernel<true, float>)); TSV_PREP((topk_seq_kernel<false, float>));
    auto go = [&](auto kern) {
      if (bytes > 32 * 1024 && !ensure_smem((const void*)kern, bytes)) return cudaErrorInvalidValue;
      return cudaLaunchKernelEx(&cfg, kern, s, p, c, nd, sc, topk_idx, ws, status, cap);
    };
    if (s.dtype == TSV_BF16) e = c.page_table ? go(topk_seq_kernel<true, bf16>) : go(topk_seq_kernel<false, bf16>);
    else e = c.page_table ? go(topk_seq_kernel<true, float>) : go(topk_seq_kernel<false, float>);
    count_launch();
  } else {
    const int bytes = (int)list_bytes(p);
    if (bytes > 24 * 1024 && !ensure_smem((const void*)topk_list_kernel, bytes)) return TSV_ERR_CUDA;
    cfg.numAttrs = 1;
    const int ent = (int)(s.max_L / s.m_csa), per = kRowSteps * 64;
    cfg.gridDim = dim3((ent + per - 1) / per, s.B, (s.D + 7) / 8); cfg.blockDim = dim3(128, 1, 1);
    TSV_PREP(score_rows_kernel<true>); TSV_PREP(score_rows_kernel<false>); TSV_PREP(topk_list_kernel);
    e = c.page_table ? cudaLaunchKernelEx(&cfg, score_rows_kernel<true>, s, p, c, nd, ws) : cudaLaunchKernelEx(&cfg, score_rows_kernel<false>, s, p, c, nd, ws);
    count_launch();
    if (e != cudaSuccess) { cudaGetLastError(); return TSV_ERR_CUDA; }
    cfg.gridDim = dim3(ssel::CS * s.D, s.B, 1); cfg.blockDim = dim3(kListThreads, 1, 1); cfg.dynamicSmemBytes = bytes; cfg.numAttrs = 2;
    e = cudaLaunchKernelEx(&cfg, topk_list_kernel, s, p, c, nd, sc, topk_idx, ws, status);
    count_launch();
  }
  return e == cudaSuccess && cudaGetLastError() == cudaSuccess ? TSV_OK : TSV_ERR_CUDA;
}

}  // namespace tsv
