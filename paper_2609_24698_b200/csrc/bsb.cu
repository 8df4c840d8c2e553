// branch_state_build: chain-private online compression along every root-to-node path.
//
// Grid (sequence, element slab).  The scalar part of every fold (max gate, sum of weights, the two
// blend coefficients, done flags) follows the tree: in every CTA one warp per compressed layer (CSA,
// HCA) holds a node per lane, loads gates and parents up front (independent loads, one memory
// latency) and folds level by level, the parent's result arriving by shuffle.  Each thread then owns
// four neighbouring elements: it loads them of every node's compression vector up front, folds along
// the tree with the inherited values kept in shared memory (indexed by parent), and stores states and
// closed entries.  No load depends on a store.
//
// Bound by latency (the tree's loads, the scalar folds, the vector folds, one after the other); the traffic is 9 MB at 64
// sequences.  Every CTA repeats the scalar part, so few CTAs with four elements per thread (8- and 16-byte accesses)
// beat many with one.  In a cycle launched by one call it also puts the closed entries where the attention reads them, which
// the tile plan otherwise copies after waiting for this kernel (both together, per layer: 1 sequence 27.0 -> 25.6 us, 64 grown
// ones 108 -> 105 us).
#include "kernels.h"

namespace tsv {

struct FoldCoef {
  float a, b, s;     // acc' = a * acc_parent + b * c ; s = sum of weights after the fold
  int32_t done;      // block closes at this node
  int32_t empty;     // the inherited block holds no token (inherited numbers are ignored)
};

// empty / done: position p opens / closes a block of blk tokens (they depend on the position alone: a caller that folds
// along a chain works them out ahead of it)
__device__ __forceinline__ void scalar_fold(FoldCoef& fc, float& mx_out, float& s_out, bool empty, bool done, float mxp, float sp, float g) {
  float mx2, a, b, s2;
  if (empty) { mx2 = g; a = 0.f; b = 1.f; s2 = 1.f; }
  else {
    mx2 = fmaxf(mxp, g);
    a = expf(mxp - mx2);
    b = expf(g - mx2);
    s2 = fmaf(sp, a, b);
  }
  fc.a = a; fc.b = b; fc.s = s2; fc.empty = empty;
  fc.done = done;
  mx_out = fc.done ? 0.f : mx2;
  s_out = fc.done ? 0.f : s2;
}

constexpr int kBsbThreads = 96;    // (rows of 512, 512 and 128 elements, four per thread: three CTAs per sequence exactly)
constexpr int VEC = 4;             // (rows are multiples of eight elements, the arrays 16-byte aligned)

template <typename T> struct alignas(sizeof(T) * VEC) Quad { T x[VEC]; };

// DEFER: the C128-deferred schedule is on (a separate instantiation, so that the timely schedule's code is untouched by it)
// misc: the packed buffer of the attention that follows (misc_rows rows per sequence), or NULL
template <typename T, int DMAX, bool DEFER>
__global__ void __launch_bounds__(kBsbThreads) bsb_kernel(const tsv_shape s, const tsv_cache c, const tsv_nodes nd,
                                                          const tsv_scratch sc, int32_t* __restrict__ status, const bool reset_status,
                                                          T* __restrict__ misc, const int misc_rows) {
  using VT = Quad<T>;
  using VF = Quad<float>;
  extern __shared__ __align__(16) char hist_raw[];
  VF* hist = reinterpret_cast<VF*>(hist_raw);          // [D][kBsbThreads] post-fold values of this thread's elements per node
  __shared__ TreeMeta tm;
  __shared__ TreeStage tstage;
  __shared__ FoldCoef fcs[TSV_MAX_D], fhs[TSV_MAX_D];
  __shared__ uint32_t closed[2];                       // nodes that close a CSA / HCA block
  const int b = blockIdx.x, D = s.D;
  // Launched as a programmatic dependent (its CTAs take their places as those of the kernel before leave); waits before it reads or
  // signals anything, so nothing of this call starts before what came earlier on the stream is complete.
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");   // the selection may start the part of it that does not read this kernel's results
  const int d = s.d, di = s.di;
  const int e = (blockIdx.y * kBsbThreads + threadIdx.x) * VEC;     // first element: [0,d) CSA kv | [d,d+di) CSA indexer key | [d+di,2d+di) HCA kv
  const bool live = e < 2 * d + di;
  const int which = e < d ? 0 : (e < d + di ? 1 : 2);
  const int el = which == 0 ? e : (which == 1 ? e - d : e - d - di);
  const int dim = which == 1 ? di : d;
  const T* cin = reinterpret_cast<const T*>(which == 0 ? nd.c_csa : (which == 1 ? nd.ikc : nd.c_hca));
  const float* pers = which == 0 ? c.csa_acc_kv : (which == 1 ? c.csa_acc_ik : c.hca_acc_kv);
  // C128-deferred schedule: the HCA slabs of a sequence in which no HCA block can close inside the tree have nothing to do
  // (they learn the length first, one load, and leave before fetching any vector)
  if (DEFER && (int)(blockIdx.y * kBsbThreads * VEC) >= d + di && hca_deferred(s, c.L[b])) return;
  // All loads are issued before the scalar chain is known, the chain's own (which it starts from) first.  Padding slots load too: the
  // memory is there.
  const int lane = threadIdx.x & 31, chain = threadIdx.x >> 5;      // chain 0: CSA, 1: HCA (warp 2 takes no part)
  const TreeFetch tf = fetch_tree(s, c.L + b, nd.parent + (size_t)b * D, nd.n_nodes + b, c.csa_cap + b, c.hca_cap + b);
  float gate = 0.f, pmx = 0.f, psum = 0.f;
  if (chain < 2 && lane < D) gate = (chain == 0 ? nd.g_csa : nd.g_hca)[(size_t)b * D + lane];
  if (chain < 2 && lane == 0) { pmx = (chain == 0 ? c.csa_mx : c.hca_mx)[b]; psum = (chain == 0 ? c.csa_s : c.hca_s)[b]; }
  VT cvr[DMAX];                                        // kept as loaded: a conversion here would wait for the data
  const VT* cinv = reinterpret_cast<const VT*>(cin + (size_t)b * D * dim + el);
#pragma unroll
  for (int n = 0; n < DMAX; ++n) { cvr[n] = VT{}; if (live && n < D) cvr[n] = cinv[n * (dim / VEC)]; }
  VF pv = {};
  if (live) pv = *reinterpret_cast<const VF*>(pers + (size_t)b * dim + el);
  derive_tree_meta(tm, tstage, s, tf, true, true);

  // The scalar chains: warp 0 folds the CSA block states, warp 1 the HCA ones, lane n owning node n.  A node's fold needs
  // its parent's result, so the warp walks the tree level by level (nodes of one depth fold together, the parent's
  // running max and sum arrive by shuffle): as many steps as the tree is deep, not as it has nodes.
  const bool hdef = DEFER && hca_deferred(s, tm.L) && !tm.status;     // (tm.L is 0 for a flagged length: such a sequence commits nothing)
  if (chain < 2) {
    const bool writer = blockIdx.y == 0;
    if (writer && threadIdx.x == 0) {
      // (a selection CTA that runs early may have or-ed in what it found: the same bits)
      if (reset_status) status[b] = tm.status; else if (tm.status) atomicOr(status + b, tm.status);
    }
    const int nn = tm.status ? 0 : tm.nn, n = lane;
    const bool valid = n < nn;
    const int depth = valid ? tm.depth[n] : -1, par = valid && n ? tm.parent[n] : 0;
    const int maxd = __reduce_max_sync(0xffffffffu, depth);
    FoldCoef fc;
    fc.a = fc.b = fc.s = 0.f; fc.done = 0; fc.empty = 0;
    float mx = 0.f, sm = 0.f;                          // this node's running max and sum after its fold
    const bool skip = chain == 1 && hdef;              // deferred schedule: no HCA branch states
    const int blk = chain == 0 ? s.m_csa : s.m_hca, p = tm.L + max(depth, 0);
    const bool opens = (p % blk) == 0, closes = ((p + 1) % blk) == 0;
    if (!skip) {
      for (int level = 0; level <= maxd; ++level) {    // uniform trip count
        const float mp = __shfl_sync(0xffffffffu, mx, par), sp = __shfl_sync(0xffffffffu, sm, par);
        if (depth == level)
          scalar_fold(fc, mx, sm, opens, closes, n ? mp : pmx, n ? sp : psum, gate);
      }
    }
    const uint32_t cl = __ballot_sync(0xffffffffu, fc.done != 0);
    if (lane == 0) closed[chain] = cl;
    if (n < D) {
      (chain == 0 ? fcs : fhs)[n] = fc;
      if (writer) {
        if (chain == 0) { sc.csa_mx[(size_t)b * D + n] = mx; sc.csa_s[(size_t)b * D + n] = sm; sc.csa_done[(size_t)b * D + n] = (uint8_t)fc.done; }
        else {
          if (!hdef) { sc.hca_mx[(size_t)b * D + n] = mx; sc.hca_s[(size_t)b * D + n] = sm; }
          sc.hca_done[(size_t)b * D + n] = (uint8_t)fc.done;
        }
      }
    }
  }
  __syncthreads();
  if (!live || (which == 2 && hdef)) return;
  const int nn = tm.status ? 0 : tm.nn;
  float* sacc = which == 0 ? sc.csa_acc_kv : (which == 1 ? sc.csa_acc_ik : sc.hca_acc_kv);
  T* newe = reinterpret_cast<T*>(which == 0 ? sc.new_csa_kv : (which == 1 ? sc.new_csa_ik : sc.new_hca_kv));
  const FoldCoef* fc = which == 2 ? fhs : fcs;
  // packed buffer: [few HCA entries][tree nodes][closed CSA entries][closed HCA entries]
  const uint32_t mine = closed[which == 2];
  T* pack = nullptr;
  if (misc && which != 1)
    pack = misc + ((size_t)b * misc_rows + (tm.n_hca <= kHcaMiscMax ? tm.n_hca : 0) + nn + (which == 2 ? __popc(closed[0]) : 0)) * d + el;
#pragma unroll
  for (int n = 0; n < DMAX; ++n) {
    if (n < D) {
      const size_t o = ((size_t)b * D + n) * dim + el;
      VF acc = {}, ent = {};
      if (n < nn) {
        const FoldCoef f = fc[n];
        VF ap = pv;
        if (!f.empty && n) ap = hist[tm.parent[n] * kBsbThreads + threadIdx.x];
#pragma unroll
        for (int x = 0; x < VEC; ++x) {
          const float cvn = to_f(cvr[n].x[x]);
          acc.x[x] = f.empty ? cvn : fmaf(f.a, ap.x[x], f.b * cvn);
        }
        if (f.done) {
#pragma unroll
          for (int x = 0; x < VEC; ++x) { ent.x[x] = acc.x[x] / f.s; acc.x[x] = 0.f; }
        }
      }
      hist[n * kBsbThreads + threadIdx.x] = acc;
      VT en;
#pragma unroll
      for (int x = 0; x < VEC; ++x) en.x[x] = from_f<T>(ent.x[x]);
      *reinterpret_cast<VF*>(sacc + o) = acc;
      *reinterpret_cast<VT*>(newe + o) = en;
      if (pack && ((mine >> n) & 1u)) *reinterpret_cast<VT*>(pack + (size_t)__popc(mine & ((1u << n) - 1u)) * d) = en;
    }
  }
}

template <typename T, int DMAX, bool DEFER>
static int launch_bsb_as(const tsv_shape& s, const tsv_cache& c, const tsv_nodes& nd, const tsv_scratch& sc, int32_t* status, bool reset_status,
                         void* misc, int misc_rows, cudaStream_t st) {
  const auto kernel = bsb_kernel<T, DMAX, DEFER>;
  TSV_PREP(kernel);
  const int per_cta = kBsbThreads * VEC;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(s.B, (2 * s.d + s.di + per_cta - 1) / per_cta); cfg.blockDim = dim3(kBsbThreads, 1, 1);
  cfg.dynamicSmemBytes = (size_t)s.D * per_cta * sizeof(float); cfg.stream = st;
  if (DMAX > 8 && !ensure_smem((const void*)kernel, (int)cfg.dynamicSmemBytes)) return TSV_ERR_CUDA;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr; cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kernel, s, c, nd, sc, status, reset_status, reinterpret_cast<T*>(misc), misc_rows);
  count_launch();
  return cudaGetLastError() == cudaSuccess ? TSV_OK : TSV_ERR_CUDA;
}

int launch_bsb(const tsv_shape& s, const tsv_cache& c, const tsv_nodes& nd, const tsv_scratch& sc, int32_t* status, bool reset_status,
               void* misc, int misc_rows, cudaStream_t st) {
  const bool defer = (s.flags & TSV_FLAG_HCA_DEFERRED) != 0, bf = s.dtype == TSV_BF16, small = s.D <= 8;
#define TSV_BSB(T_, DM_)                                                                                              \
  return defer ? launch_bsb_as<T_, DM_, true>(s, c, nd, sc, status, reset_status, misc, misc_rows, st)                 \
               : launch_bsb_as<T_, DM_, false>(s, c, nd, sc, status, reset_status, misc, misc_rows, st)
  if (small) { if (bf) TSV_BSB(bf16, 8); TSV_BSB(float, 8); }
  if (bf) TSV_BSB(bf16, TSV_MAX_D);
  TSV_BSB(float, TSV_MAX_D);
#undef TSV_BSB
}

}  // namespace tsv
