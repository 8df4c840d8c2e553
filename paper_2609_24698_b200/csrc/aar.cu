// accept_and_refresh: greedy acceptance walk, then commit of the accepted path into the
// persistent per-sequence state of every layer.
//   aar_kernel  up to eight layers: one CTA per (sequence, layer), the layers of a sequence as a cluster.  Every
//               CTA validates all layers and walks the tree itself (one warp, one memory latency); after a cluster barrier
//               (all have read the lengths) each commits its layer.  One launch and two memory latencies, where two kernels
//               took two launches and a chain of loads per accepted node.
//   more layers: aar_walk (one warp per sequence) validates and walks, then aar_commit (one CTA per sequence, layer) reads
//               its verdict, so that all layers of a sequence commit or none does.
#include "kernels.h"

namespace tsv {

// One warp: lane l checks layer l's length and capacities (the same checks as build_tree_meta), lane n checks node n's parent;
// the greedy walk runs on ballots: lane c holds node c's parent and draft token.  found: flags found here; flags: those and
// what the cycle raised before.  path: [D], written by lane 0.
struct Walk { int found, flags, len, bonus; };
__device__ __forceinline__ Walk walk_sequence(const tsv_shape& s, const AarLayers& ls, int b, const int32_t* parent, const int32_t* n_nodes,
                                              const int32_t* draft, const int32_t* target, const int32_t* status, bool do_walk, int32_t* path) {
  const int D = s.D, lane = threadIdx.x & 31;
  int st = 0;
  int nn = n_nodes[b];
  const int earlier = do_walk ? status[b] : 0;
  const int par0 = lane < D ? parent[(size_t)b * D + lane] : -1;
  const int dr = do_walk && lane < D ? draft[(size_t)b * D + lane] : 0, tg = do_walk && lane < D ? target[(size_t)b * D + lane] : 0;
  if (nn < 1 || nn > D) { st |= TSV_ST_NODES; nn = 0; }
  for (int l = lane; l < ls.n; l += 32) {
    int L = ls.l[l].c.L[b];
    if (L < 0 || (int64_t)L + D > s.max_L) { st |= TSV_ST_LENGTH; L = 0; }
    if ((L + D) / s.m_csa > ls.l[l].c.csa_cap[b]) st |= TSV_ST_CSA_CAP;
    if ((L + D) / s.m_hca > ls.l[l].c.hca_cap[b]) st |= TSV_ST_HCA_CAP;
  }
  const int par = lane < nn ? par0 : -1;
  if (lane < nn && (lane == 0 ? par != -1 : (par < 0 || par >= lane))) st |= TSV_ST_PARENT;
  st = __reduce_or_sync(0xffffffffu, st);
  Walk r;
  r.found = st; r.flags = st | earlier; r.len = 0; r.bonus = -1;
  if (!do_walk || r.flags) return r;
  int cur = 0;
  if (lane == 0) path[0] = 0;
  r.len = 1;
  for (;;) {
    const int want = __shfl_sync(0xffffffffu, tg, cur);
    const uint32_t match = __ballot_sync(0xffffffffu, lane > cur && lane < nn && par == cur && dr == want);
    if (!match) break;
    const int nxt = __ffs(match) - 1;                  // the first matching child in node order
    if (lane == 0) path[r.len] = nxt;
    ++r.len;
    cur = nxt;
  }
  r.bonus = __shfl_sync(0xffffffffu, tg, cur);
  return r;
}

__global__ void __launch_bounds__(32) aar_walk_kernel(const tsv_shape s, const AarLayers ls, const int32_t* __restrict__ parent,
                                                      const int32_t* __restrict__ n_nodes, const int32_t* __restrict__ draft,
                                                      const int32_t* __restrict__ target, int32_t* __restrict__ accept_len,
                                                      int32_t* __restrict__ accept_path, int32_t* __restrict__ bonus,
                                                      int32_t* __restrict__ status, const int do_walk) {
  const int b = blockIdx.x, D = s.D, lane = threadIdx.x;
  const Walk r = walk_sequence(s, ls, b, parent, n_nodes, draft, target, status, do_walk, accept_path + (size_t)b * D);
  if (lane == 0 && r.found) atomicOr(status + b, r.found);
  if (!do_walk) return;
  if (lane == 0) {
    for (int i = r.len; i < D; ++i) accept_path[(size_t)b * D + i] = -1;
    accept_len[b] = r.len;
    bonus[b] = r.bonus;
  }
}

__device__ __forceinline__ void copy_row16(void* dst, const void* src, int bytes, int tid, int nthr) {
  const uint4* s4 = reinterpret_cast<const uint4*>(src);
  uint4* d4 = reinterpret_cast<uint4*>(dst);
  for (int i = tid; i < bytes / 16; i += nthr) d4[i] = s4[i];
}

// Commit of the accepted path (al nodes, path: [al]) of sequence b, whose length was L, into one layer.  A warp per copied row:
// all of them are in flight together.  (Which entries close is a function of the positions.)
__device__ __forceinline__ void commit_layer(const tsv_shape& s, const AarLayer& ly, int b, int L, int al, const int32_t* path) {
  __shared__ float coef_a[TSV_MAX_D], coef_b[TSV_MAX_D];
  const int D = s.D, es = s.dtype == TSV_BF16 ? 2 : 4;
  const int rowb = s.d * es, ikb = s.di * es;
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
  const size_t last = (size_t)b * D + path[al - 1];
  // Open-block states of the last accepted node.  A block that this node closed leaves an empty state, whose stored numbers
  // nobody reads (emptiness is known from the position count): that copy is skipped.
  const bool csa_open = (L + al) % s.m_csa != 0, hca_open = (L + al) % s.m_hca != 0;
  const bool hdef = hca_deferred(s, L);
  // copies: 4 i + {0: token row, 1: CSA entry, 2: its indexer key, 3: HCA entry} of accepted node i, then the three states
  for (int k = warp; k < 4 * al + 3; k += nw) {
    void* dst;
    const void* src;
    int bytes;
    if (k < 4 * al) {
      const int i = k >> 2, what = k & 3, pos = L + i;
      const size_t nidx = (size_t)b * D + path[i];
      if (what == 0) { dst = (char*)ly.c.win_kv + (size_t)tok_row_of(ly.c, s, b, pos) * rowb; src = (const char*)ly.node_kv + nidx * rowb; bytes = rowb; }
      else if (what == 3) {
        if ((pos + 1) % s.m_hca) continue;
        dst = (char*)ly.c.hca_kv + (size_t)hca_rows_of(ly.c, s, b)(pos / s.m_hca) * rowb; src = (const char*)ly.sc.new_hca_kv + nidx * rowb; bytes = rowb;
      } else {
        if ((pos + 1) % s.m_csa) continue;
        const size_t row = (size_t)csa_rows_of(ly.c, s, b)(pos / s.m_csa);
        if (what == 1) { dst = (char*)ly.c.csa_kv + row * rowb; src = (const char*)ly.sc.new_csa_kv + nidx * rowb; bytes = rowb; }
        else { dst = (char*)ly.c.csa_ik + row * ikb; src = (const char*)ly.sc.new_csa_ik + nidx * ikb; bytes = ikb; }
      }
    } else if (k == 4 * al) { if (!csa_open) continue; dst = ly.c.csa_acc_kv + (size_t)b * s.d; src = ly.sc.csa_acc_kv + last * s.d; bytes = s.d * 4; }
    else if (k == 4 * al + 1) { if (!csa_open) continue; dst = ly.c.csa_acc_ik + (size_t)b * s.di; src = ly.sc.csa_acc_ik + last * s.di; bytes = s.di * 4; }
    else { if (!hca_open || hdef) continue; dst = ly.c.hca_acc_kv + (size_t)b * s.d; src = ly.sc.hca_acc_kv + last * s.d; bytes = s.d * 4; }
    copy_row16(dst, src, bytes, lane, 32);
  }
  if (hdef) {
    // C128-deferred schedule: branch_state_build built no HCA states for this sequence (no block closes inside its tree);
    // the accepted tokens are folded into the persistent open block here, in path order, with the arithmetic of the state
    // build (scalar part by every thread alike, each thread its own vector elements), so the result has the same bits.
    float mx = ly.c.hca_mx[b], sw = ly.c.hca_s[b];
    for (int i = 0; i < al; ++i) {
      const float g = ly.node_g_hca[(size_t)b * D + path[i]];
      float ca = 0.f, cb = 1.f;
      if ((L + i) % s.m_hca == 0) { mx = g; sw = 1.f; }
      else {
        const float mx2 = fmaxf(mx, g);
        ca = expf(mx - mx2); cb = expf(g - mx2);
        sw = fmaf(sw, ca, cb);
        mx = mx2;
      }
      if (tid == 0) { coef_a[i] = ca; coef_b[i] = cb; }
    }
    __syncthreads();                    // (also: every thread has read the old scalars before thread 0 replaces them)
    for (int e = tid; e < s.d; e += nt) {
      float acc = ly.c.hca_acc_kv[(size_t)b * s.d + e];
      for (int i = 0; i < al; ++i) {
        const size_t nidx = (size_t)b * D + path[i];
        const float cv = s.dtype == TSV_BF16 ? to_f(reinterpret_cast<const bf16*>(ly.node_c_hca)[nidx * s.d + e])
                                             : reinterpret_cast<const float*>(ly.node_c_hca)[nidx * s.d + e];
        acc = (L + i) % s.m_hca == 0 ? cv : fmaf(coef_a[i], acc, coef_b[i] * cv);
      }
      ly.c.hca_acc_kv[(size_t)b * s.d + e] = acc;
    }
    if (tid == 0) { ly.c.hca_mx[b] = mx; ly.c.hca_s[b] = sw; }
  }
  if (tid == 0) {
    ly.c.csa_mx[b] = ly.sc.csa_mx[last]; ly.c.csa_s[b] = ly.sc.csa_s[last];
    if (!hdef) { ly.c.hca_mx[b] = ly.sc.hca_mx[last]; ly.c.hca_s[b] = ly.sc.hca_s[last]; }
    ly.c.L[b] = L + al;
  }
}

__global__ void __launch_bounds__(256) aar_commit_kernel(const tsv_shape s, const AarLayers ls, const int32_t* __restrict__ accept_len,
                                                         const int32_t* __restrict__ accept_path, const int32_t* __restrict__ status) {
  const int b = blockIdx.x;
  const AarLayer& ly = ls.l[blockIdx.y];
  const int al = accept_len[b];
  if (status[b] != 0 || al <= 0) return;
  const int L = ly.c.L[b];
  __syncthreads();                      // every thread holds L before anyone moves it
  commit_layer(s, ly, b, L, al, accept_path + (size_t)b * s.D);
}

constexpr int kAarFusedLayers = 8;      // layers of a portable cluster
__global__ void __launch_bounds__(256) aar_kernel(const tsv_shape s, const AarLayers ls, const int32_t* __restrict__ parent,
                                                  const int32_t* __restrict__ n_nodes, const int32_t* __restrict__ draft,
                                                  const int32_t* __restrict__ target, int32_t* __restrict__ accept_len,
                                                  int32_t* __restrict__ accept_path, int32_t* __restrict__ bonus, int32_t* __restrict__ status) {
  // launched as a programmatic dependent (its CTAs take their places as those of the kernel before leave); waits first
  asm volatile("griddepcontrol.wait;" ::: "memory");
  __shared__ int32_t path[TSV_MAX_D];
  __shared__ int verdict[2];
  const int layer = blockIdx.x, b = blockIdx.y, D = s.D, tid = threadIdx.x;
  const AarLayer& ly = ls.l[layer];
  const int L = ly.c.L[b];
  if (tid < 32) {
    const Walk r = walk_sequence(s, ls, b, parent, n_nodes, draft, target, status, true, path);
    __syncwarp();
    if (tid == 0) { verdict[0] = r.flags; verdict[1] = r.len; }
    if (layer == 0) {
      if (tid < D) accept_path[(size_t)b * D + tid] = tid < r.len ? path[tid] : -1;
      if (tid == 0) { accept_len[b] = r.len; bonus[b] = r.bonus; }
    }
  }
  __syncthreads();
  // every CTA of the sequence has read the lengths and the status before anyone moves them
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
  if (verdict[0]) {
    if (layer == 0 && tid == 0) atomicOr(status + b, verdict[0]);
    return;
  }
  commit_layer(s, ly, b, L, verdict[1], path);
}

int launch_aar(const tsv_shape& s, int n_layers, const tsv_cache* const* caches, const tsv_nodes* const* nodes,
               const tsv_scratch* const* scratch, const int32_t* parent, const int32_t* n_nodes,
               const int32_t* draft, const int32_t* target, int32_t* accept_len, int32_t* accept_path,
               int32_t* bonus, int32_t* status, cudaStream_t st) {
  AarLayers ls;
  auto layer = [&](int l) {
    AarLayer a;
    a.c = *caches[l]; a.node_kv = nodes[l]->kv; a.node_c_hca = nodes[l]->c_hca; a.node_g_hca = nodes[l]->g_hca; a.sc = *scratch[l];
    return a;
  };
  if (n_layers <= kAarFusedLayers) {
    ls.n = n_layers;
    for (int i = 0; i < n_layers; ++i) ls.l[i] = layer(i);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(n_layers, s.B, 1); cfg.blockDim = dim3(256, 1, 1); cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = n_layers; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr; cfg.numAttrs = 2;
    TSV_PREP(aar_kernel);
    const cudaError_t e = cudaLaunchKernelEx(&cfg, aar_kernel, s, ls, parent, n_nodes, draft, target, accept_len, accept_path, bonus, status);
    count_launch();
    return e == cudaSuccess && cudaGetLastError() == cudaSuccess ? TSV_OK : TSV_ERR_CUDA;
  }
  for (int l0 = 0; l0 < n_layers; l0 += kAarLayersPerLaunch) {
    ls.n = n_layers - l0 < kAarLayersPerLaunch ? n_layers - l0 : kAarLayersPerLaunch;
    for (int i = 0; i < ls.n; ++i) ls.l[i] = layer(l0 + i);
    const int last = l0 + ls.n >= n_layers;
    TSV_PREP(aar_walk_kernel);
    aar_walk_kernel<<<s.B, 32, 0, st>>>(s, ls, parent, n_nodes, draft, target, accept_len, accept_path, bonus, status, last);
    count_launch();
  }
  for (int l0 = 0; l0 < n_layers; l0 += kAarLayersPerLaunch) {
    ls.n = n_layers - l0 < kAarLayersPerLaunch ? n_layers - l0 : kAarLayersPerLaunch;
    for (int i = 0; i < ls.n; ++i) ls.l[i] = layer(l0 + i);
    TSV_PREP(aar_commit_kernel);
    aar_commit_kernel<<<dim3(s.B, ls.n), 256, 0, st>>>(s, ls, accept_len, accept_path, status);
    count_launch();
  }
  return cudaGetLastError() == cudaSuccess ? TSV_OK : TSV_ERR_CUDA;
}

}  // namespace tsv
