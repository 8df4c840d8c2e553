// tree_verify_attn on the 5th-generation tensor cores (tcgen05 + TMEM), bf16 storage, d = 512: the tile plan and the
// merge of multi-chunk tiles.  (The attention kernel itself is in tva_tc_pair.cu.)
//
// Rows are grouped in plan tiles of 256 query rows = 256/H consecutive tree nodes x H heads; all of them attend over the
// SAME staged key rows (key == value, MQA), so S = Q K^T and O = P K are dense contractions.  Which node sees which key is
// a per-key bitmask applied to the S fragment after it is read back from tensor memory.
//
//   tc_plan_kernel   per (sequence, plan tile): the keys visible to at least one node of the tile, as four runs {HCA
//                    entries, window ring, packed misc rows, CSA entries} padded to 32 rows, with a node mask per key.
//                    Contiguous-run tiles (every node selects all CSA candidates, or the CSA slab is at most 2 x topk
//                    rows): the runs as 32-row TMA boxes.  Gathered tiles (selection far from dense, or a paged pool
//                    whose pages do not hold whole boxes): the CSA run holds only the entries some node of the tile
//                    selected, and every key is named by array << 30 | row for four-row TMA gathers.
//                    Each tile CTA leaves its record (tile_record) at the tile's scheduling position (its rank by
//                    estimated length of its work items, longest first); an extra CTA per sequence packs the small scattered rows.
//   tc_combine_pair_kernel  merges the chunks of the paired kernel's multi-chunk tiles (fixed order).
#include <type_traits>

#include "tc_common.cuh"

namespace tsv {


// ------------------------------------------------------------------------------------------------ plan
constexpr int kRankTilesMax = 2048;                    // beyond that many tiles they keep their natural order
// Estimated length of a tile's work items: the keys it stages, from its committed length and node count alone (for tiles on the
// contiguous-run path it is exact up to the entries closed inside the tree; only the order of the tiles depends on it).
__device__ __forceinline__ int tile_keys_estimate(const tsv_shape& s, int L, int nn, int tile, int npt) {
  if (L < 0 || (int64_t)L + s.D > s.max_L || nn < 1 || nn > s.D || tile * npt >= nn) return 0;
  auto r32 = [](int x) { return (x + kBoxRows - 1) / kBoxRows * kBoxRows; };
  const int n_csa = L / s.m_csa, n_hca = L / s.m_hca, nh_in = n_hca <= kHcaMiscMax ? n_hca : 0, win = min(L, s.window);
  const int nk = n_csa <= 2 * s.topk ? r32(n_csa) + (n_hca > kHcaMiscMax ? r32(n_hca) : 0) + r32(win) + r32(nh_in + nn)
                                     : min(n_csa, npt * s.topk) + n_hca + win + 3 * nn;
  // The order is by the length of the work items (chunks), longest first: the pairs take them in that order, and an item of 600-768
  // keys (a whole tile) taken last would leave one pair working alone (64 sequences of 1-4 k tokens: the slowest pair ended at
  // 132 k cycles against a mean of 107 k when the order was by the tile's keys).
  return nk <= tc::NCX ? nk : min(nk, tc::NC);
}

// GENERAL: gathered tiles may occur (see gathered_tiles_possible); the instantiation without them keeps the short
// latency chain of the contiguous-run plan.
template <bool GENERAL, int PARTS>
__device__ __forceinline__ void tc_plan_tile(const tsv_shape& s, const TvaPlan& pl, const tsv_cache& c, const tsv_nodes& nd,
                                             const tsv_scratch& sc, char* __restrict__ ws, uint32_t* words, int* est, int* ahead_sm) {
  __shared__ TreeMeta tm;
  __shared__ TreeStage tstage;
  __shared__ int n_cand[8], win_lo[8];
  __shared__ int dense;
  // PARTS CTAs per tile (part 0 does everything but its share of a long list's compaction), then the packing CTA
  const int tile = blockIdx.x / PARTS, part = PARTS > 1 ? blockIdx.x % PARTS : 0, b = blockIdx.y, D = s.D, H = s.H;
  const bool packer = tile >= pl.tc_nt;
  const int npt = tc::PR / H, n0 = tile * npt;
  const size_t tix = (size_t)b * pl.tc_nt + tile;
  uint32_t* krow = reinterpret_cast<uint32_t*>(ws + pl.off_krow) + tix * pl.tc_maxk;    // gathered tiles: array << 30 | row per key
  uint8_t* kmask = reinterpret_cast<uint8_t*>(ws + pl.off_kmask) + tix * pl.tc_maxk;
  // the cache row offsets are fetched together with the tree scalars (one memory latency for all)
  __shared__ uint8_t cdone[TSV_MAX_D], hdone[TSV_MAX_D];
  __shared__ int64_t row0_sm[2];
  // (the length and node count of "its" tile's sequence, for the ranking of the tiles: requested now, used after the tree's loads)
  const int ntile = s.B * pl.tc_nt;
  const bool ranked_order = ntile <= kRankTilesMax && !packer && part == 0;
  int eL = -1, enn = 0;
  if (ranked_order && (int)threadIdx.x < ntile) { eL = c.L[threadIdx.x / pl.tc_nt]; enn = nd.n_nodes[threadIdx.x / pl.tc_nt]; }
  if (threadIdx.x == 40) row0_sm[0] = c.page_table ? 0 : c.csa_row0[b];
  if (threadIdx.x == 41) row0_sm[1] = c.page_table ? 0 : c.hca_row0[b];
  coop_tree_meta(tm, tstage, s, c.L + b, nd.parent + (size_t)b * D, nd.n_nodes + b, c.csa_cap + b, c.hca_cap + b);
  if (ranked_order) {                                  // estimated key counts of all tiles
    if ((int)threadIdx.x < ntile) est[threadIdx.x] = tile_keys_estimate(s, eL, enn, threadIdx.x % pl.tc_nt, npt);
#pragma unroll 1
    for (int i = threadIdx.x + blockDim.x; i < ntile; i += blockDim.x)
      est[i] = tile_keys_estimate(s, c.L[i / pl.tc_nt], nd.n_nodes[i / pl.tc_nt], i % pl.tc_nt, npt);
  }
  // thread 0 leaves the tile's record at that position as soon as it knows the key count
  auto leave_record = [&](int nk, int md) {
    reinterpret_cast<int4*>(ws + pl.off_order)[ntile <= kRankTilesMax ? *ahead_sm : (int)tix] = tc::tile_record(pl, b, tile, md, nk);
  };
  // The kernel is launched as a programmatic dependent of the selection kernel (itself one of the state build) and runs
  // under those kernels' tails as far as it reads only the caller's inputs and the committed caches: the done flags are
  // worked out from the positions, and a tile no node of which ranks is planned completely.  It waits for the two kernels
  // (griddepcontrol.wait, below) before it reads what they write: the entries closed inside the tree (packing CTA), the
  // ranking nodes' mask rows.
  if (threadIdx.x < D) {
    const bool valid = !tm.status && (int)threadIdx.x < tm.nn;
    cdone[threadIdx.x] = valid && node_closes(tm.L, tm.depth[threadIdx.x], s.m_csa);
    hdone[threadIdx.x] = valid && node_closes(tm.L, tm.depth[threadIdx.x], s.m_hca);
  }
  __syncthreads();
  // The tile's scheduling position: how many tiles come before it by estimated key count (complete after the next barrier).
  if (ranked_order) {
    const int mine = est[tix];
    int ahead = 0;
#pragma unroll 1
    for (int j = threadIdx.x; j < ntile; j += blockDim.x) { const int e = est[j]; ahead += (e > mine) || (e == mine && j < (int)tix); }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ahead += __shfl_xor_sync(0xffffffffu, ahead, o);
    if ((threadIdx.x & 31) == 0 && ahead) atomicAdd(ahead_sm, ahead);
  }
  // rows of the sequence's CSA and HCA entries: slabs, or through the page table of a paged pool
  RowAddr csa_row, hca_row;
  csa_row.pt = hca_row.pt = c.page_table ? c.page_table + (size_t)b * c.max_pages : nullptr;
  csa_row.per_page = c.page_table ? c.page_tokens / s.m_csa : 1; hca_row.per_page = c.page_table ? c.page_tokens / s.m_hca : 1;
  csa_row.row0 = row0_sm[0]; hca_row.row0 = row0_sm[1];
  // runs of consecutive rows exist in a paged pool only where a page holds whole 32-row boxes of the layer
  const bool csa_runs = !c.page_table || (csa_row.per_page % kBoxRows == 0 && c.page_tokens % kBoxRows == 0), hca_runs = !c.page_table || hca_row.per_page % kBoxRows == 0;
  if (packer) {
    // The extra CTA of the sequence (the last in grid x): rows that are small and scattered (few HCA entries, tree nodes,
    // entries closed inside the tree) are packed into one contiguous per-sequence buffer so that TMA boxes can fetch
    // them.  Kept off the tile CTAs: the copy is a chain of its own (addresses, loads, stores).  Within a cycle launched by one
    // call the state build has put the entries closed inside the tree here already: no wait for them then, and no copy.
    if (tm.status) return;
    const size_t rowb = (size_t)s.d * 2;
    const int nh_in = tm.n_hca <= kHcaMiscMax ? tm.n_hca : 0;
    int ncd = 0, nhd = 0;
#pragma unroll 1
    for (int j = 0; j < tm.nn; ++j) { ncd += cdone[j] != 0; nhd += hdone[j] != 0; }
    const int n_misc = nh_in + tm.nn + ncd + nhd;
    uint4* dst = reinterpret_cast<uint4*>(ws + pl.off_misc + (size_t)b * pl.tc_misc_rows * rowb);
    const int rows_out = (n_misc + kBoxRows - 1) / kBoxRows * kBoxRows;
    // The source of every packed row is worked out once (thread r: row r), then the copy runs flat over (row, 16-byte
    // piece) items, eight of a thread in flight.  Rows [0, first) and the zero padding behind n_misc are the caller's
    // data; the rows between are the state build's and copied after the wait.  (Compact code on purpose: the kernel runs
    // once per layer with cold instruction caches.)
    __shared__ const uint4* srcs[kHcaMiscMax + 3 * TSV_MAX_D];
    constexpr int CPR = tc::DH * 2 / 16;               // 16-byte pieces per row
#pragma unroll 1
    for (int r = threadIdx.x; r < rows_out; r += blockDim.x) {
      const char* src = nullptr;
      if (r < nh_in) src = (const char*)c.hca_kv + (size_t)hca_row(r) * rowb;
      else if (r < nh_in + tm.nn) src = (const char*)nd.kv + ((size_t)b * D + (r - nh_in)) * rowb;
      else if (r < n_misc && !pl.tc_packed) {
        int ord = r - nh_in - tm.nn;
        const bool isc = ord < ncd;
        if (!isc) ord -= ncd;
        const uint8_t* dn = isc ? cdone : hdone;
        int a = 0;
#pragma unroll 1
        for (int j = 0; j < tm.nn; ++j) if (dn[j]) { if (ord == 0) { a = j; break; } --ord; }
        src = (const char*)(isc ? sc.new_csa_kv : sc.new_hca_kv) + ((size_t)b * D + a) * rowb;
      }
      srcs[r] = reinterpret_cast<const uint4*>(src);
    }
    __syncthreads();
    const int first = nh_in + tm.nn;
#pragma unroll 1
    for (int phase = 0; phase < 2; ++phase) {
      if (phase) {
        if (n_misc == first || pl.tc_packed) break;
        asm volatile("griddepcontrol.wait;" ::: "memory");   // the entries closed inside the tree
      }
      const int lo = phase ? first * CPR : 0, hi = phase ? n_misc * CPR : rows_out * CPR;
#pragma unroll 1
      for (int i0 = lo + threadIdx.x; i0 < hi; i0 += 8 * blockDim.x) {
        uint4 v[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const int i = i0 + k * blockDim.x, r = i / CPR;
          const bool in = i < hi && (phase || r < first || r >= n_misc);
          const uint4* src = in ? srcs[r] : nullptr;
          v[k] = src ? __ldg(src + (i - r * CPR)) : make_uint4(0, 0, 0, 0);
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const int i = i0 + k * blockDim.x, r = i / CPR;
          if (i < hi && (phase || r < first || r >= n_misc)) dst[i] = v[k];
        }
      }
    }
    return;
  }
  if (threadIdx.x < 32) {                              // lane nl: candidates and window start of node n0 + nl
    const int lane = threadIdx.x, n = n0 + lane;
    const uint32_t cmaskbits = __ballot_sync(0xffffffffu, lane < D && cdone[lane]);   // nodes that close a CSA block
    const bool real = lane < npt && n < tm.nn;
    const int nc = tm.n_csa + (real ? __popc(tm.anc[n] & ((1u << n) - 1u) & cmaskbits) : 0);   // + blocks closed at strict ancestors
    if (lane < npt) {
      n_cand[lane] = nc;
      win_lo[lane] = max(0, tm.L + tm.depth[real ? n : 0] - s.window + 1);
    }
    const uint32_t over = __ballot_sync(0xffffffffu, real && nc > s.topk);
    if (lane == 0) dense = over == 0;
  }
  __syncthreads();
  if (tm.status || n0 >= tm.nn) { if (threadIdx.x == 0 && part == 0) leave_record(0, 1); return; }
  const int nvalid = min(npt, tm.nn - n0);
  const uint32_t validbits = (1u << nvalid) - 1u;
  const int n_csa = tm.n_csa;
  // Four runs of keys, each padded to whole boxes: HCA entries (when too many for the packed rows), the window ring, the packed
  // rows, and last the committed CSA entries, the only run that depends on the selection: everything else is written before the
  // CTA waits for it.
  //   contiguous-run tiles: every run as TMA boxes; ranked nodes still take this path while the CSA run is at most twice the
  //     selection size: all committed entries are staged and the unselected ones are masked per node
  //   gathered tiles (a longer CSA run, or a paged pool whose pages do not hold whole boxes): the CSA run holds only the entries
  //     some node of the tile selected, and every key is named by its row (array << 30 | row) for four-row TMA gathers
  const bool runs_ok = !GENERAL || ((dense || n_csa <= 2 * s.topk) && csa_runs && (hca_runs || tm.n_hca <= kHcaMiscMax));
  if (PARTS > 1 && part && (dense || runs_ok)) return;   // (the parts share the compaction of a ranked gathered tile only)
  uint32_t rankbits = 0;                               // nodes that rank (the others take every committed entry)
#pragma unroll 1
  for (int nl = 0; nl < nvalid; ++nl) if (n_cand[nl] > s.topk) rankbits |= 1u << nl;
  // The selection kernel left, for every node that ranks, a bit per candidate.
  const uint32_t* mrow = reinterpret_cast<const uint32_t*>(ws + pl.off_selmask) + ((size_t)b * D + n0) * pl.mask_ld;
  const int nwords = (n_csa + 31) >> 5, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
  // word wi of node n0 + nl: entries [32 wi, 32 wi + 32), those that do not exist cleared
  auto node_word = [&](int nl, int wi) -> uint32_t {
    const int left = n_csa - 32 * wi;
    return (((rankbits >> nl) & 1u) ? __ldcg(mrow + (size_t)nl * pl.mask_ld + wi) : 0xffffffffu) & (left >= 32 ? 0xffffffffu : (1u << left) - 1u);
  };
  // the packed per-sequence rows (written by the sequence's extra CTA): few HCA entries, tree nodes, entries closed in the tree
  const int nh_in = tm.n_hca <= kHcaMiscMax ? tm.n_hca : 0;
  int ncd = 0, nhd = 0;
#pragma unroll 1
  for (int j = 0; j < tm.nn; ++j) { ncd += cdone[j] != 0; nhd += hdone[j] != 0; }
  const int n_misc = nh_in + tm.nn + ncd + nhd;
  // the window: the ring in slot order, or (paged pool) the positions from the 32-aligned start of the box that holds the oldest
  // window position up to L - 1 (the positions before the window are masked like every position a node cannot see)
  const int win_a = c.page_table ? (max(0, tm.L - s.window) & ~(kBoxRows - 1)) : 0;
  auto r32 = [](int x) { return (x + kBoxRows - 1) / kBoxRows * kBoxRows; };
  const int c1 = tm.n_hca > kHcaMiscMax ? tm.n_hca : 0, c2 = c.page_table ? tm.L - win_a : min(tm.L, s.window), c3 = n_misc;
  const int k2 = r32(c1), k3 = k2 + r32(c2), k4 = k3 + r32(c3);        // first keys of the window, the packed rows, the CSA run
  // row of key i of run g (g = 0: the whole CSA slab)
  auto run_row = [&](int g, int i) -> int64_t {
    return g == 0 ? csa_row(i) : g == 1 ? hca_row(i) : g == 3 ? (int64_t)b * pl.tc_misc_rows + i
                  : c.page_table ? tok_row_of(c, s, b, win_a + i) : (int64_t)b * s.window + i;
  };
  auto run_of = [&](int k) { return k >= k4 ? 0 : k >= k3 ? 3 : k >= k2 ? 2 : 1; };
  auto run_first = [&](int g) { return g == 0 ? k4 : g == 3 ? k3 : g == 2 ? k2 : 0; };
  const int newc0 = nh_in + tm.nn;                     // first packed row of the CSA entries closed inside the tree
  // node a that closed the ord-th CSA (HCA) block of the tree
  auto closer = [&](const uint8_t* dn, int ord) {
    int a = 0;
#pragma unroll 1
    for (int j = 0; j < tm.nn; ++j) if (dn[j]) { if (ord == 0) { a = j; break; } --ord; }
    return a;
  };
  if (part == 0) {
    const int kb = dense || runs_ok ? k4 + r32(n_csa) : k4;
    if (runs_ok) {
      int2* box = reinterpret_cast<int2*>(ws + pl.off_box) + tix * (size_t)(pl.tc_maxk / kBoxRows);
#pragma unroll 1
      for (int bi = threadIdx.x; bi < kb / kBoxRows; bi += blockDim.x) {
        const int k = bi * kBoxRows, g = run_of(k);
        // (a box of a cache run never crosses a page: it starts on a multiple of 32 entries and per_page is one too)
        box[bi] = make_int2(g, (int)run_row(g, k - run_first(g)));
      }
    }
    // One pass over all keys: a thread finds the run of its key by comparison, so the runs' (short, latency-bound) mask
    // computations overlap instead of following each other.
#pragma unroll 1
    for (int k = threadIdx.x; k < (dense ? kb : k4); k += blockDim.x) {
      const int g = run_of(k), i = k - run_first(g), cg = g == 0 ? n_csa : g == 1 ? c1 : g == 2 ? c2 : c3;
      uint32_t m = 0;
      if (i < cg) {
        if (g < 2 || (g == 3 && i < nh_in)) m = validbits;
        else if (g == 2) {
          const int pos = c.page_table ? win_a + i : tm.L - 1 - ((tm.L - 1 - i) % s.window);
#pragma unroll 1
          for (int nl = 0; nl < nvalid; ++nl) if (pos >= win_lo[nl]) m |= 1u << nl;
        } else {
          // a tree node (visible to itself and its descendants) or an entry closed at one (to its strict descendants; a CSA
          // entry to those that selected it: ranked tiles write these masks after the wait)
          const bool own = i < newc0, isc = !own && i < newc0 + ncd;
          const int a = own ? i - nh_in : isc ? closer(cdone, i - newc0) : closer(hdone, i - newc0 - ncd);
#pragma unroll 1
          for (int nl = 0; nl < nvalid; ++nl) if (((tm.anc[n0 + nl] >> a) & 1u) && (own || a != n0 + nl)) m |= 1u << nl;
        }
      }
      if (dense || !(g == 3 && i >= newc0 && i < newc0 + ncd)) kmask[k] = (uint8_t)m;
      // gathered tiles: the key's row; the padding of a run repeats the run's first row (masked)
      if (!runs_ok) krow[k] = ((uint32_t)g << 30) | (uint32_t)(cg ? run_row(g, i < cg ? i : 0) : 0);
    }
    if ((dense || runs_ok) && threadIdx.x == 0) leave_record(kb, runs_ok ? 1 : 2);
  }
  if (dense) return;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");    // the selection's mask rows
  // In-tree entries: candidate n_csa + o of a node is the block closed at the o-th of its strict ancestors that closed one.
  // Thread i: the i-th closed entry of the tree, its mask over the tile's nodes.
  if (part == 0 && (int)threadIdx.x >= (int)blockDim.x - 32 && lane < ncd) {
    const int a = closer(cdone, lane);
    uint32_t closed = 0, m = 0;
#pragma unroll 1
    for (int j = 0; j < tm.nn; ++j) closed |= (uint32_t)(cdone[j] != 0) << j;
#pragma unroll 1
    for (int nl = 0; nl < nvalid; ++nl) {
      const uint32_t up = tm.anc[n0 + nl] & ((1u << (n0 + nl)) - 1u);      // strict ancestors
      if (!((up >> a) & 1u)) continue;
      const int cand = n_csa + __popc(up & closed & ((1u << a) - 1u));
      if (!((rankbits >> nl) & 1u) || ((__ldcg(mrow + (size_t)nl * pl.mask_ld + (cand >> 5)) >> (cand & 31)) & 1u)) m |= 1u << nl;
    }
    kmask[k3 + newc0 + lane] = (uint8_t)m;
  }
  if (runs_ok) {
    // the committed CSA run, a word of 32 entries per warp and step (its padding is zero): lane nl fetches node nl's word
#pragma unroll 2
    for (int wi = warp; wi < nwords; wi += nwarp) {
      const uint32_t v = lane < nvalid ? node_word(lane, wi) : 0u;
      uint32_t m = 0;
#pragma unroll
      for (int nl = 0; nl < 8; ++nl) m |= ((__shfl_sync(0xffffffffu, v, nl) >> lane) & 1u) << nl;
      kmask[k4 + 32 * wi + lane] = (uint8_t)m;
    }
    return;
  }
  if (!GENERAL) return;
  // Gathered: ordered compaction of the entries some node selected.  A thread counts those of a word of 32 entries, one block scan
  // gives each word its place, then a warp writes a word's entries (lane = entry: consecutive places, coalesced stores).  Over
  // long lists (PARTS > 1) several CTAs do the count each for itself and share the writing, which is bound by the issue slots of
  // one SM (32768 entries: 22 us by one CTA).
  __shared__ int wsum_c[33];
  const int wld = (pl.cand_cap + 31) >> 5;             // words: [wld] place of the word's first entry, then [wld] per node
  int* place = reinterpret_cast<int*>(words);
  int n_uni = 0;
#pragma unroll 1
  for (int w0 = 0; w0 < nwords; w0 += blockDim.x) {
    const int wi = w0 + threadIdx.x;
    uint32_t u = 0u;
    if (wi < nwords) {
      uint32_t v[8];
#pragma unroll
      for (int nl = 0; nl < 8; ++nl) v[nl] = nl < nvalid ? node_word(nl, wi) : 0u;
#pragma unroll
      for (int nl = 0; nl < 8; ++nl) if (nl < nvalid) { u |= v[nl]; words[(1 + nl) * wld + wi] = v[nl]; }
    }
    int total;
    const int at = block_excl_scan(__popc(u), wsum_c, total);
    if (wi < nwords) place[wi] = n_uni + at;
    n_uni += total;
  }
  if (part == 0 && threadIdx.x == 0) leave_record(k4 + r32(n_uni), 2);
  __syncthreads();
#pragma unroll 1
  for (int wi = warp * PARTS + part; wi < nwords; wi += nwarp * PARTS) {
    uint32_t m = 0;
#pragma unroll
    for (int nl = 0; nl < 8; ++nl) if (nl < nvalid) m |= ((words[(1 + nl) * wld + wi] >> lane) & 1u) << nl;
    const uint32_t u = __ballot_sync(0xffffffffu, m != 0);
    if (m) {
      const int p = k4 + place[wi] + __popc(u & ((1u << lane) - 1u));
      krow[p] = (uint32_t)csa_row(32 * wi + lane);
      kmask[p] = (uint8_t)m;
    }
  }
  if (part == 0 && threadIdx.x < kBoxRows) {            // the run's padding (masked)
    const int p = k4 + n_uni + threadIdx.x;
    if (p < k4 + r32(n_uni)) { krow[p] = (uint32_t)csa_row(0); kmask[p] = 0; }
  }
}

// Plan of every (sequence, 256-row tile).  Each tile CTA leaves one 16-byte record (tile_record) at the tile's
// scheduling position: its rank among all tiles by estimated key count, most first, which every CTA works out for itself
// from the lengths and node counts of all sequences (the paired attention kernel takes the tiles in that order, long
// ones first and short ones in the tail, and learns all it needs about its tile from one load).  A tile no node of which
// ranks is planned from the caller's inputs alone: its CTA never waits for the kernels before this one.
// NT threads per CTA: 256, or 1024 for gathered tiles over long candidate lists (the union of a tile's selections over tens
// of thousands of entries is the work of ONE CTA, alone on its SM).
constexpr int kPlanParts = 8;                          // CTAs per tile over long candidate lists
template <bool GENERAL, int NT>
__global__ void __launch_bounds__(NT) tc_plan_kernel(const tsv_shape s, const TvaPlan pl, const tsv_cache c, const tsv_nodes nd,
                                                                         const tsv_scratch sc, char* __restrict__ ws) {
  extern __shared__ uint32_t words_sm[];               // gathered tiles: per word of 32 entries its place and the nodes' selections
  __shared__ int est_sm[kRankTilesMax];
  __shared__ int ahead_sm;
  constexpr int PARTS = NT > 256 ? kPlanParts : 1;
  const int tile = blockIdx.x / PARTS;
  const bool tile_cta = tile < pl.tc_nt && blockIdx.x % PARTS == 0;
  const size_t tix = (size_t)blockIdx.y * pl.tc_nt + tile;
  if (threadIdx.x == 0) ahead_sm = 0;
  if (threadIdx.x < 2 && blockIdx.x == 0 && blockIdx.y == 0) reinterpret_cast<int32_t*>(ws + pl.off_sched)[threadIdx.x] = 0;   // the attention kernel's item counters
  if (threadIdx.x < 2 && tile_cta)                      // finished-chunk counters of the tile's two 128-row halves
    reinterpret_cast<int32_t*>(ws + pl.off_tcnt)[tix * 2 + threadIdx.x] = 0;
  tc_plan_tile<GENERAL, PARTS>(s, pl, c, nd, sc, ws, words_sm, est_sm, &ahead_sm);
  // Signalled here, and by a tile that waits for the selection before that wait: the attention kernel's CTAs take their places as the
  // CTAs of the small kernels leave (64 grown sequences 842 -> 830 us per pass of eight layers against after the wait).  At the start
  // of the CTA it is worse (865 -> 901 us): then all pairs begin at the same instant, and their first instructions queue behind
  // everyone's first operands.
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  // one CTA waits for the selection in any case, so that the completion of this kernel implies that one's
  if (blockIdx.x == 0 && blockIdx.y == 0) asm volatile("griddepcontrol.wait;" ::: "memory");
}

// ------------------------------------------------------------------------------------------------ merge
// Merge of the paired kernel's multi-chunk tiles (launched with its general instantiation): every chunk left its NORMALISED partial output with
// the row's (reference max, sum); the row's output is the average of the partial outputs weighted by sum * 2^(max - row max), the
// chunks accumulated in order.
// 1-d grid (scheduling position of the tile, its two 128-row halves, groups of 8 * rpw rows): a warp merges rpw rows, one after the
// other or (bf16, rpw = 2) together, a lane owns 16 columns as 16-byte pieces of the row (coalesced).  Bound by latency and by the
// L2 and HBM traffic (67 MB read and 34 MB written at 64 sequences of 1-4 k tokens, 15 us): a row's (max, sum) and its first four
// chunks, or those of two rows and their first two chunks, are requested together (after the maxima had been reduced they cost a
// third latency), and a CTA lives for several rows (rpw: 1, 2 or 4).
// The CTAs take the places of the attention kernel's as those run out of items, and a tile is merged as soon as all warps of its
// chunks have said that their rows are stored (it is looked for in the order in which the tiles are worked on), the rest when
// that kernel has ended: at those 64 sequences a pass of eight layers takes 798 instead of 830 us.  Tiles cut to fill the device
// all end with that kernel, and looking earlier loses 0.4 us a layer: there the merge waits for it at once.
// ANY32: some tiles' partial outputs may be fp32 (else all are bf16, and the kernel keeps its registers low).  ROWS: rows merged together.
constexpr int kMergePolls = 256;       // times a warp looks for its tile's chunks (0.3 us each) before it waits for the whole attention kernel
template <bool ANY32, int ROWS>
__global__ void __launch_bounds__(256) tc_combine_pair_kernel(const tsv_shape s, const TvaPlan pl, void* __restrict__ out_, const char* __restrict__ ws, const int rpw) {
  using namespace tc;
  constexpr uint32_t FULL = 0xffffffffu;
  const int lg = 31 - __clz(BM / 8 / rpw), pos = blockIdx.x >> (lg + 1), half = (blockIdx.x >> lg) & 1, group = blockIdx.x & ((1 << lg) - 1);
  // Launched as a programmatic dependent of the attention kernel, when all CTAs of that have started: the tile plan is complete.
  const int4 rec = __ldcg(reinterpret_cast<const int4*>(ws + pl.off_order) + pos);
  // (What other kernels wrote is read past the L1.)  One CTA waits for that kernel in any case, so that the completion of this one
  // implies that one's.
  const bool early = pl.tc_split == 1;
  if (blockIdx.x == 0 || !early) asm volatile("griddepcontrol.wait;" ::: "memory");
  const int b = rec.x, rt = rec_tile(rec) * 2 + half, nch = rec_chunks(rec);
  const size_t rix = (size_t)b * 2 * pl.tc_nt + rt;
  if (rec.z <= 0 || nch <= 1) return;                            // (one chunk: the paired kernel wrote the output itself)
  const bool f32 = ANY32 && rec_f32(rec);                        // (where no tile is split, one with more than one chunk was too long for one: bf16)
  const int rows_seq = s.D * s.H, row0 = rt * BM, lane = threadIdx.x & 31;
  const int first = group * 8 * rpw + (threadIdx.x >> 5), last = min(min(BM, rows_seq - row0), (group + 1) * 8 * rpw);
  if (first >= last) return;
  if (early) {
    const int32_t* cnt = reinterpret_cast<const int32_t*>(ws + pl.off_tcnt) + rix;
    int done = 0;
    for (int i = 0; i < kMergePolls; ++i) {                      // (every lane reads it: one request a warp)
      asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(done) : "l"(cnt) : "memory");
      if (done >= 8 * nch) break;
      __nanosleep(200);
    }
    if (done < 8 * nch) asm volatile("griddepcontrol.wait;" ::: "memory");
  }
  const float2* pml = reinterpret_cast<const float2*>(ws + pl.off_tpml) + rix * pl.tc_chmax * BM;
  // vec: 16-byte pieces of a lane's 16 columns; R: rows merged together (their requests are in flight together)
  auto merge = [&](auto vec, auto rows) {
    constexpr int V = decltype(vec)::value, R = decltype(rows)::value, U = R > 1 ? 2 : 4;      // U: chunks requested together
    // (a chunk's bf16 tile lies at the start of the chunk's slot of BM x DH floats)
    const uint4* po = reinterpret_cast<const uint4*>(ws + pl.off_tpo) + rix * pl.tc_chmax * BM * (DH / 4) + lane;
#pragma unroll 1
    for (int row = first; row < last; row += 8 * R) {
      float2 x[R];
      uint4 v[U][R][V];
      auto fetch_ml = [&](int c0) {
#pragma unroll
        for (int r = 0; r < R; ++r) x[r] = c0 + lane < nch && row + 8 * r < last ? __ldcg(pml + (size_t)(c0 + lane) * BM + row + 8 * r) : make_float2(-INFINITY, 0.f);
      };
      auto fetch = [&](int c0) {
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
          for (int r = 0; r < R; ++r)
            if (c0 + u < nch && row + 8 * r < last) {
#pragma unroll
              for (int q = 0; q < V; ++q) v[u][r][q] = __ldcg(po + (size_t)(row + 8 * r) * (DH / (V == 4 ? 4 : 8)) + (size_t)(c0 + u) * BM * (DH / 4) + 32 * q);
            }
      };
      fetch_ml(0);
      fetch(0);
      float m[R], wt[R], l[R], acc[R][16];
#pragma unroll
      for (int r = 0; r < R; ++r) {
        m[r] = x[r].y > 0.f ? x[r].x : -INFINITY;
#pragma unroll 1
        for (int ch = lane + 32; ch < nch && row + 8 * r < last; ch += 32) { const float2 y = __ldcg(pml + (size_t)ch * BM + row + 8 * r); if (y.y > 0.f) m[r] = fmaxf(m[r], y.x); }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) m[r] = fmaxf(m[r], __shfl_xor_sync(FULL, m[r], o));
        wt[r] = x[r].y > 0.f ? x[r].y * exp2f(x[r].x - m[r]) : 0.f;      // lane c: weight of chunk c (of the 32 chunks at hand)
        l[r] = 0.f;
#pragma unroll
        for (int k = 0; k < 16; ++k) acc[r][k] = 0.f;
      }
#pragma unroll 1
      for (int c0 = 0; c0 < nch; c0 += U) {
        if (c0) {
          fetch(c0);
          if ((c0 & 31) == 0) {                                  // (lists of more than 32 chunks)
            fetch_ml(c0);
#pragma unroll
            for (int r = 0; r < R; ++r) wt[r] = x[r].y > 0.f ? x[r].y * exp2f(x[r].x - m[r]) : 0.f;
          }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
#pragma unroll
          for (int r = 0; r < R; ++r) {
            const float w = __shfl_sync(FULL, wt[r], (c0 + u) & 31);
            if (c0 + u >= nch) continue;
            l[r] += w;
#pragma unroll
            for (int q = 0; q < V; ++q) {
              const uint32_t wd[4] = {v[u][r][q].x, v[u][r][q].y, v[u][r][q].z, v[u][r][q].w};
#pragma unroll
              for (int k = 0; k < 4; ++k) {
                if (V == 4) acc[r][4 * q + k] = fmaf(__uint_as_float(wd[k]), w, acc[r][4 * q + k]);
                else {
                  acc[r][8 * q + 2 * k] = fmaf(__uint_as_float(wd[k] << 16), w, acc[r][8 * q + 2 * k]);
                  acc[r][8 * q + 2 * k + 1] = fmaf(__uint_as_float(wd[k] & 0xFFFF0000u), w, acc[r][8 * q + 2 * k + 1]);
                }
              }
            }
          }
        }
      }
#pragma unroll
      for (int r = 0; r < R; ++r) {
        if (row + 8 * r >= last) break;
        const float inv = l[r] > 0.f ? 1.f / l[r] : 0.f;
        uint32_t o[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const __nv_bfloat162 h2 = __floats2bfloat162_rn(acc[r][2 * k] * inv, acc[r][2 * k + 1] * inv);
          o[k] = *reinterpret_cast<const uint32_t*>(&h2);
        }
        bf16* orow = reinterpret_cast<bf16*>(out_) + ((size_t)b * rows_seq + row0 + row + 8 * r) * DH;
        if (V == 4) {
#pragma unroll
          for (int q = 0; q < 4; ++q) reinterpret_cast<uint2*>(orow)[lane + 32 * q] = make_uint2(o[2 * q], o[2 * q + 1]);
        } else {
#pragma unroll
          for (int q = 0; q < 2; ++q) reinterpret_cast<uint4*>(orow)[lane + 32 * q] = make_uint4(o[4 * q], o[4 * q + 1], o[4 * q + 2], o[4 * q + 3]);
        }
      }
    }
  };
  if (ANY32 && f32) merge(std::integral_constant<int, 4>(), std::integral_constant<int, 1>());
  else merge(std::integral_constant<int, 2>(), std::integral_constant<int, ROWS>());
}

bool tva_tc_eligible(const tsv_shape& s) {
  return s.dtype == TSV_BF16 && s.d == tc::DH && s.H >= 32 && s.H <= 128 && (128 % s.H) == 0 && !(s.flags & TSV_FLAG_FORCE_SIMT);
}

void tva_tc_plan_sizes(const tsv_shape& s, TvaPlan& p) {
  const int npt = tc::PR / s.H;
  p.tc_nt = (s.D * s.H + tc::PR - 1) / tc::PR;
  const int64_t ksel = p.cand_cap < s.topk ? p.cand_cap : s.topk;
  int64_t uni = (int64_t)npt * ksel;
  if (uni > p.cand_cap) uni = p.cand_cap;
  int64_t mk = uni + s.max_L / s.m_hca + s.window + 3 * (int64_t)s.D + 8;
  const int64_t br = kBoxRows;
  p.tc_misc_rows = (int32_t)((kHcaMiscMax + 3 * s.D + br - 1) / br * br);
  // (+ one box: in a paged pool the window run starts on a 32-aligned position and may be a box longer than the window)
  // (a tile takes the whole committed CSA run only while that is at most twice the selection size)
  const int64_t run_csa = p.cand_cap < 2 * (int64_t)s.topk ? p.cand_cap : 2 * (int64_t)s.topk;
  const int64_t runs = (run_csa + br - 1) / br * br + (s.max_L / s.m_hca + br - 1) / br * br + (s.window + br - 1) / br * br + br + p.tc_misc_rows;
  if (runs > mk) mk = runs;
  // gathered tiles: the union of the nodes' selections, HCA entries, window and packed rows as four runs padded to boxes
  const int64_t gath = (uni + br - 1) / br * br + (s.max_L / s.m_hca + br - 1) / br * br + (s.window + br - 1) / br * br + br + p.tc_misc_rows;
  if (gath > mk) mk = gath;
  p.tc_maxk = (int32_t)((mk + 127) / 128 * 128);
  p.tc_chmax = (p.tc_maxk + tc::NC - 1) / tc::NC;
}

// (only where gathered tiles may occur)
static size_t plan_smem_bytes(const tsv_shape& s, const TvaPlan& p, bool gathered) {
  return gathered ? (((size_t)p.cand_cap + 31) / 32) * 4 * (1 + (size_t)(tc::PR / s.H)) : 0;
}
// Can the plan kernel produce a gathered tile for these capacities?  (A committed CSA run longer than twice the
// selection size, or a paged pool whose pages do not hold whole 32-row boxes of a layer.)
static bool gathered_tiles_possible(const tsv_shape& s, const TvaPlan& p, const tsv_cache& c) {
  if (p.need_scores && p.cand_cap > 2 * (int64_t)s.topk) return true;
  if (c.page_table) {
    const int epp = c.page_tokens / s.m_csa, hpp = c.page_tokens / s.m_hca;
    if (epp % kBoxRows || c.page_tokens % kBoxRows) return true;
    if (hpp % kBoxRows && s.max_L / s.m_hca > kHcaMiscMax) return true;
  }
  return false;
}

// Host-side work of the tensor-core path that can fail, before anything of the call is enqueued.
int prepare_tva_tc(const tsv_shape& s, const TvaPlan& p, const tsv_cache& c, const tsv_nodes& nd, void* out, char* ws, TvaTcPrep& prep) {
  const size_t plan_sm = plan_smem_bytes(s, p, gathered_tiles_possible(s, p, c));
  if (plan_sm > 32 * 1024 && !(ensure_smem((const void*)tc_plan_kernel<true, 1024>, (int)plan_sm) && ensure_smem((const void*)tc_plan_kernel<true, 256>, (int)plan_sm) &&
                               ensure_smem((const void*)tc_plan_kernel<false, 256>, (int)plan_sm)))
    return TSV_ERR_CUDA;
  TSV_PREP((tc_plan_kernel<true, 1024>));
  TSV_PREP((tc_plan_kernel<true, 256>));
  TSV_PREP((tc_plan_kernel<false, 256>));
  TSV_PREP((tc_combine_pair_kernel<true, 1>));
  TSV_PREP((tc_combine_pair_kernel<false, 1>));
  TSV_PREP((tc_combine_pair_kernel<false, 2>));
  return prepare_tva_tc_pair(s, p, c, nd, out, ws, prep);
}

int launch_tva_tc(const tsv_shape& s, const TvaPlan& p_in, const TvaTcPrep& prep, const tsv_cache& c, const tsv_nodes& nd, const tsv_scratch& sc,
                  void* out, char* ws, int32_t* status, cudaStream_t st, bool with_plan) {
  TvaPlan p = p_in;
  const bool gathered = gathered_tiles_possible(s, p, c);
  // general: some tile may have more than two chunks of the longest kind, or be gathered; then every multi-chunk tile leaves
  // partial outputs for the merge kernel: bf16, or fp32 where the tile would fit one chunk and is cut because tiles are few
  const bool general = (p.tc_maxk + tc::NCX - 1) / tc::NCX > 2 || gathered;
  p.tc_f32 = !general;                                 // (no more than two long chunks a tile: merged without rounding in the attention kernel)
  // 19-37 general tiles are neither cut nor shared further: mostly of several chunks, they have items enough, and shares fetch the keys
  // again (not cut and cut, us a pass: 16 sequences of 512-8192 tokens 69.7 and 73.0, 18 of them 75.6 and 80.7, 12 of 16-64 k 180.5 and
  // 189.4, 10 of 8-32 k 110.0 and 112.0; the other way where lists are short: 12 of 1-4 k 56.4 and 55.7, 14 paged of 256-4096 59.5 and 57.1).
  if (general && p.tc_split < 4) p.tc_split = 1;
  p.tc_general = general;
  const dim3 pgrid(p.tc_nt + 1, s.B);                                                                              // x: tiles + the packing CTA
  if (with_plan) {
    cudaLaunchConfig_t cfg = {};
    const bool wide = gathered && p.cand_cap > 8192;    // long candidate lists: the CTA's passes over all entries want many threads
    cfg.gridDim = wide ? dim3(p.tc_nt * kPlanParts + 1, s.B) : pgrid; cfg.blockDim = dim3(wide ? 1024 : 256, 1, 1); cfg.dynamicSmemBytes = plan_smem_bytes(s, p, gathered); cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;        // may start under the selection kernel's tail (it waits inside)
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    if (wide) cudaLaunchKernelEx(&cfg, tc_plan_kernel<true, 1024>, s, p, c, nd, sc, ws);
    else if (gathered) cudaLaunchKernelEx(&cfg, tc_plan_kernel<true, 256>, s, p, c, nd, sc, ws);
    else cudaLaunchKernelEx(&cfg, tc_plan_kernel<false, 256>, s, p, c, nd, sc, ws);
  }
  count_launch();
  const int r = launch_tva_tc_pair(s, p, prep, general, nd.q, out, ws, status, st);
  if (r != TSV_OK) return r;
  if (general && p.tc_chmax > 1) {
    cudaLaunchConfig_t cfg = {};
    // Rows a warp takes: one while that leaves SMs idle otherwise; two, merged together, up to 74 tiles (what is left to merge when the
    // attention ends is one row's latency then: 32 paged sequences 257 -> 242 us a pass, four rows one after the other before); four
    // beyond (there the merge runs under the attention's tail, and the registers of two rows at once take a third of the warps:
    // 64 grown sequences take 2-3 % more with two rows).
    const int64_t groups = (int64_t)2 * p.tc_nt * s.B * (tc::BM / 8);
    const int rpw = groups <= 4 * 148 ? 1 : groups <= 16 * 148 ? 2 : 4;
    cfg.gridDim = dim3(2 * p.tc_nt * s.B * (tc::BM / 8 / rpw)); cfg.blockDim = dim3(256, 1, 1); cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    if (p.tc_split > 1) cudaLaunchKernelEx(&cfg, tc_combine_pair_kernel<true, 1>, s, p, out, (const char*)ws, rpw);
    else if (rpw == 2) cudaLaunchKernelEx(&cfg, tc_combine_pair_kernel<false, 2>, s, p, out, (const char*)ws, rpw);
    else cudaLaunchKernelEx(&cfg, tc_combine_pair_kernel<false, 1>, s, p, out, (const char*)ws, rpw);
    count_launch();
  }
  return cudaGetLastError() == cudaSuccess ? TSV_OK : TSV_ERR_CUDA;
}

}  // namespace tsv
