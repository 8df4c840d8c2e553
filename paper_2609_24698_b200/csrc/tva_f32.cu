// tree_verify_attn for fp32 storage with 128-wide rows: one cluster of CTAs per (sequence, node, group of 16 heads).
//
// The node's key list, first the keys that nothing before this kernel decides (committed HCA entries | window | ancestors-or-self),
// then the others (selected CSA entries | in-tree HCA entries of the path), is split over the CTAs of the cluster, either part evenly;
// each works through its shares in tiles of 64 rows (16-byte asynchronous copies, the next tile's under the arithmetic of this
// one), and the CTAs merge their (max, sum, O) through distributed shared memory.
//
// Exact fp32 FMAs, so the bound is the shared-memory port or the FMA pipe, whichever the tiling feeds worse (the kernel for all other
// shapes reads three operands from shared memory per eight FMAs):
//   S = Q K^T: lane = (4 heads, an eighth of the row); its queries stay in registers for the whole list, a key's row is one
//              128-byte read for the four lane groups of a warp: 16 reads per 256 FMAs; the eighths meet by 14 shuffles.
//   O = P K:   warp = (8 heads, a quarter of the tile's keys), lane = 4 columns: three reads per 32 FMAs.
// The kernel is a programmatic dependent of the selection and waits for it between the two parts: of 16 sequences of 256-4096 tokens with
// 64 selected two thirds of the keys are done under the selection (42.0 us a pass without, 38.0 with).
#include "kernels.h"

namespace tsv {

namespace f32a {

constexpr int DH = 128, HG = 16, KT = 64, NT = 256, PP = 20;      // row width, heads per CTA, keys per tile, threads, pitch of P

__device__ __forceinline__ void cp16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ uint32_t map_to_rank(uint32_t saddr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(rank));
  return r;
}
__device__ __forceinline__ float4 ld_peer4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr));
  return v;
}
__device__ __forceinline__ float2 ld_peer2(uint32_t addr) {
  float2 v;
  asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(addr));
  return v;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

}  // namespace f32a

// EARLY: the keys known before the wait go first.  Else one part, the known keys at its start.
template <bool EARLY>
__global__ void __launch_bounds__(f32a::NT, 2) attn_f32_kernel(const tsv_shape s, const TvaPlan pl, const tsv_cache c, const tsv_nodes nd,
                                                               const tsv_scratch sc, float* __restrict__ out, char* __restrict__ ws) {
  using namespace f32a;
  extern __shared__ __align__(16) unsigned char dsm[];               // [2][KT][DH] rows; at the end [4][HG][DH] parts of O
  __shared__ TreeMeta tm;
  __shared__ TreeStage tstage;
  __shared__ __align__(16) float P[KT * PP];
  __shared__ __align__(16) float osum[HG * DH];
  __shared__ __align__(8) float2 ml[HG];
  __shared__ float alpha_sm[HG];
  __shared__ int32_t newc[TSV_MAX_D], newc_blk[TSV_MAX_D], newh[TSV_MAX_D], path[TSV_MAX_D];
  __shared__ int cnt[3];                                              // in-tree CSA entries, in-tree HCA entries, ancestors-or-self
  __shared__ const float* rows[2][KT];
  const int D = s.D, H = s.H, hgroups = (H + HG - 1) / HG;
  const int cs = gridDim.x, rank = blockIdx.x, n = blockIdx.y / hgroups, h0 = (blockIdx.y % hgroups) * HG, b = blockIdx.z;
  const int t = threadIdx.x, lane = t & 31, w = t >> 5, nh = min(HG, H - h0);
  const size_t row0 = ((size_t)b * D + n) * H + h0;                   // first query row of this CTA
  // this lane's queries: heads 4 (lane / 8) .., float4 pieces slice, slice + 8, ... of the row
  const int hq = 4 * (lane >> 3), slice = lane & 7;
  float4 q[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int x = 0; x < 4; ++x)
      q[i][x] = hq + i < nh ? __ldg(reinterpret_cast<const float4*>(reinterpret_cast<const float*>(nd.q) + (row0 + hq + i) * DH) + x * 8 + slice)
                            : make_float4(0.f, 0.f, 0.f, 0.f);
  coop_tree_meta(tm, tstage, s, c.L + b, nd.parent + (size_t)b * D, nd.n_nodes + b, c.csa_cap + b, c.hca_cap + b);
  const bool live = !tm.status && n < tm.nn;
  if (t < 32) {                                                       // lane j = node j: what of it node n sees
    const bool valid = !tm.status && t < tm.nn;
    const uint32_t self = live ? tm.anc[n] : 0u, strict = self & ~(1u << n), lt = (1u << t) - 1u;
    const uint32_t cm = __ballot_sync(0xffffffffu, valid && node_closes(tm.L, tm.depth[t], s.m_csa)) & strict;
    const uint32_t hm = __ballot_sync(0xffffffffu, valid && node_closes(tm.L, tm.depth[t], s.m_hca)) & strict;
    if ((cm >> t) & 1u) { const int o = __popc(cm & lt); newc[o] = t; newc_blk[o] = (tm.L + tm.depth[t]) / s.m_csa; }
    if ((hm >> t) & 1u) newh[__popc(hm & lt)] = t;
    if ((self >> t) & 1u) path[__popc(self & lt)] = t;
    if (t == 0) { cnt[0] = __popc(cm); cnt[1] = __popc(hm); cnt[2] = __popc(self); }
  }
  __syncthreads();
  if (!live) {                                                        // flagged sequence / padding node: zeros (the whole cluster alike)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (rank == 0)
      for (int i = t; i < nh * DH / 4; i += NT) reinterpret_cast<float4*>(out + row0 * DH)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    return;
  }
  // The keys in two parts, of each an equal share per CTA: those that neither the selection nor the state build decides
  // (committed HCA | window | ancestors-or-self), then those that they do (selected CSA | in-tree HCA).
  const int n_hca = tm.n_hca, n_newh = cnt[1], pos = tm.L + tm.depth[n], win_lo = max(0, pos - s.window + 1), n_win = max(0, tm.L - win_lo);
  const int32_t* sel = reinterpret_cast<const int32_t*>(ws + pl.off_sel) + ((size_t)b * D + n) * s.topk;
  const int lead = EARLY ? 0 : n_hca + n_win + cnt[2];
  int n_sel = 0;
  int k0 = 0, k1 = 0;                                                 // this CTA's share of the part at hand
  auto known_row = [&](int j) -> const float* {
    if (j < n_hca) return reinterpret_cast<const float*>(c.hca_kv) + (size_t)hca_rows_of(c, s, b)(j) * DH;
    j -= n_hca;
    if (j < n_win) return reinterpret_cast<const float*>(c.win_kv) + (size_t)tok_row_of(c, s, b, win_lo + j) * DH;
    return reinterpret_cast<const float*>(nd.kv) + ((size_t)b * D + path[j - n_win]) * DH;
  };
  auto chosen_row = [&](int j) -> const float* {
    if (j >= n_sel) return reinterpret_cast<const float*>(sc.new_hca_kv) + ((size_t)b * D + newh[j - n_sel]) * DH;
    const int idx = __ldcg(sel + j);
    if (idx < tm.n_csa) return reinterpret_cast<const float*>(c.csa_kv) + (size_t)csa_rows_of(c, s, b)(idx) * DH;
    int a = newc[0];
    for (int i = 0; i < cnt[0]; ++i) if (newc_blk[i] == idx) a = newc[i];
    return reinterpret_cast<const float*>(sc.new_csa_kv) + ((size_t)b * D + a) * DH;
  };
  const uint32_t ks = (uint32_t)__cvta_generic_to_shared(dsm);
  auto resolve = [&](int part, int tile) {
    const int j = k0 + tile * KT + t;
    if (t < KT && j < k1) {
      if (EARLY) rows[tile & 1][t] = part ? chosen_row(j) : known_row(j);
      else rows[tile & 1][t] = j < lead ? known_row(j) : chosen_row(j - lead);
    }
  };
  auto issue = [&](int tile) {                                        // after a barrier behind resolve(.., tile); one copy group per call
    const int nk = min(KT, k1 - (k0 + tile * KT));
    const uint32_t dst = ks + (uint32_t)(tile & 1) * (KT * DH * 4);
    for (int r = w; r < nk; r += NT / 32) cp16(dst + r * (DH * 4) + lane * 16, rows[tile & 1][r] + 4 * lane);
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  float m_run[2] = {-INFINITY, -INFINITY}, l_run[2] = {0.f, 0.f};     // heads 2 w, 2 w + 1 (alike in all lanes)
  float4 o[8];                                                        // heads 8 (w & 1) .., columns 4 lane ..
#pragma unroll
  for (int i = 0; i < 8; ++i) o[i] = make_float4(0.f, 0.f, 0.f, 0.f);
  const float scale = s.sm_scale;
  bool any = false;                                                   // a tile has been worked on
#pragma unroll 1
  for (int part = EARLY ? 0 : 1; part < 2; ++part) {
    int N = n_hca + n_win + cnt[2];
    if (part) {
      asm volatile("griddepcontrol.wait;" ::: "memory");               // the selection, and through it the state build
      n_sel = __ldcg(reinterpret_cast<const int32_t*>(ws + pl.off_selcnt) + (size_t)b * D + n);
      N = n_sel + n_newh + lead;
      __syncthreads();                                                  // (the buffers and row pointers of the part before)
    }
    const int per = (N + cs - 1) / cs;
    k0 = min(N, rank * per); k1 = min(N, k0 + per);
    const int ntile = (k1 - k0 + KT - 1) / KT;
    resolve(part, 0);
    resolve(part, 1);
    __syncthreads();
    issue(0);                                                           // (an empty share: an empty group)
#pragma unroll 1
    for (int tile = 0; tile < ntile; ++tile, any = true) {
      const int nk = min(KT, k1 - (k0 + tile * KT));
      if (tile) __syncthreads();                                        // the tile before has been read (its buffer is filled again)
      if (tile + 1 < ntile) issue(tile + 1); else asm volatile("cp.async.commit_group;" ::: "memory");
      asm volatile("cp.async.wait_group 1;" ::: "memory");
      __syncthreads();                                                  // the tile's rows are there; rows[tile & 1] has been read
      const float* K = reinterpret_cast<const float*>(dsm) + (size_t)(tile & 1) * (KT * DH);
      if (tile + 2 < ntile) resolve(part, tile + 2);
#pragma unroll 1
      for (int kb = 4 * w; kb < nk; kb += 32) {                         // (rows past nk of a group of four: stale, masked)
        float a[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) a[i] = 0.f;
#pragma unroll
        for (int x = 0; x < 4; ++x)
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const float4 kv = reinterpret_cast<const float4*>(K + (kb + k) * DH)[x * 8 + slice];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              a[4 * i + k] = fmaf(q[i][x].x, kv.x, a[4 * i + k]);
              a[4 * i + k] = fmaf(q[i][x].y, kv.y, a[4 * i + k]);
              a[4 * i + k] = fmaf(q[i][x].z, kv.z, a[4 * i + k]);
              a[4 * i + k] = fmaf(q[i][x].w, kv.w, a[4 * i + k]);
            }
          }
        // the eight slices: each exchange halves the values a lane is responsible for
#pragma unroll
        for (int half = 8, bit = 4; half >= 2; half >>= 1, bit >>= 1) {
          const bool up = lane & bit;
#pragma unroll
          for (int i = 0; i < half; ++i) {
            const float send = up ? a[i] : a[half + i], keep = up ? a[half + i] : a[i];
            a[i] = keep + __shfl_xor_sync(0xffffffffu, send, bit);
          }
        }
        const int h = hq + (slice >> 1), k = kb + 2 * (slice & 1);      // this lane: (head h, keys k, k + 1)
        P[k * PP + h] = k < nk ? a[0] * scale : -INFINITY;
        P[(k + 1) * PP + h] = k + 1 < nk ? a[1] * scale : -INFINITY;
      }
      __syncthreads();
#pragma unroll
      for (int x = 0; x < 2; ++x) {                                     // softmax of heads 2 w, 2 w + 1
        const int h = 2 * w + x;
        const float s0 = lane < nk ? P[lane * PP + h] : -INFINITY, s1 = lane + 32 < nk ? P[(lane + 32) * PP + h] : -INFINITY;
        float mx = fmaxf(s0, s1);
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, d));
        const float m_new = fmaxf(m_run[x], mx);                        // finite: every tile holds a key
        const float p0 = expf(s0 - m_new), p1 = expf(s1 - m_new);
        const float al = expf(m_run[x] - m_new);                        // 0 on the first tile
        l_run[x] = fmaf(l_run[x], al, warp_sum(p0 + p1));
        m_run[x] = m_new;
        if (lane < nk) P[lane * PP + h] = p0;
        if (lane + 32 < nk) P[(lane + 32) * PP + h] = p1;
        if (lane == 0) alpha_sm[h] = al;
      }
      __syncthreads();
      {
        const int hb = 8 * (w & 1), kq = w >> 1;
        if (any) {
#pragma unroll
          for (int i = 0; i < 8; ++i) { const float al = alpha_sm[hb + i]; o[i].x *= al; o[i].y *= al; o[i].z *= al; o[i].w *= al; }
        }
        const int beg = kq * (KT / 4), end = min(nk, beg + KT / 4);
#pragma unroll 4
        for (int k = beg; k < end; ++k) {
          const float4 kv = reinterpret_cast<const float4*>(K + k * DH)[lane];
          const float4 pa = *reinterpret_cast<const float4*>(P + k * PP + hb), pb = *reinterpret_cast<const float4*>(P + k * PP + hb + 4);
          const float pv[8] = {pa.x, pa.y, pa.z, pa.w, pb.x, pb.y, pb.z, pb.w};
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            o[i].x = fmaf(pv[i], kv.x, o[i].x); o[i].y = fmaf(pv[i], kv.y, o[i].y);
            o[i].z = fmaf(pv[i], kv.z, o[i].z); o[i].w = fmaf(pv[i], kv.w, o[i].w);
          }
        }
      }
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  {   // the quarters of the keys meet
    float4* part = reinterpret_cast<float4*>(dsm);
#pragma unroll
    for (int i = 0; i < 8; ++i) part[((w >> 1) * HG + 8 * (w & 1) + i) * (DH / 4) + lane] = o[i];
    if (lane < 2) ml[2 * w + lane] = make_float2(lane ? m_run[1] : m_run[0], lane ? l_run[1] : l_run[0]);
    __syncthreads();
#pragma unroll
    for (int x = 0; x < 2; ++x) {
      const int u = t + x * NT;
      float4 a = part[u];
#pragma unroll
      for (int k = 1; k < 4; ++k) { const float4 v = part[k * HG * (DH / 4) + u]; a.x += v.x; a.y += v.y; a.z += v.z; a.w += v.w; }
      reinterpret_cast<float4*>(osum)[u] = a;
    }
  }
  cluster_sync();
  // CTA r merges the r-th share of the output (16-byte units), in the order of the CTAs
  const uint32_t osum_s = (uint32_t)__cvta_generic_to_shared(osum), ml_s = (uint32_t)__cvta_generic_to_shared(ml);
  const int units = HG * DH / 4 / cs;
  for (int i = t; i < units; i += NT) {
    const int u = rank * units + i, h = u >> 5;
    float2 x[8];
    float4 v[8];
#pragma unroll
    for (int r = 0; r < 8; ++r) if (r < cs) { x[r] = ld_peer2(map_to_rank(ml_s + h * 8, r)); v[r] = ld_peer4(map_to_rank(osum_s + u * 16, r)); }
    float m = -INFINITY, l = 0.f;
#pragma unroll
    for (int r = 0; r < 8; ++r) if (r < cs) m = fmaxf(m, x[r].x);
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int r = 0; r < 8; ++r)
      if (r < cs) {
        const float wt = expf(x[r].x - m);                            // 0 for an empty share
        l = fmaf(x[r].y, wt, l);
        a.x = fmaf(v[r].x, wt, a.x); a.y = fmaf(v[r].y, wt, a.y); a.z = fmaf(v[r].z, wt, a.z); a.w = fmaf(v[r].w, wt, a.w);
      }
    if (h < nh) reinterpret_cast<float4*>(out + row0 * DH)[u] = make_float4(a.x / l, a.y / l, a.z / l, a.w / l);
  }
  cluster_sync();                                                     // no CTA leaves while a peer may still read its memory
}

bool tva_f32_applies(const tsv_shape& s) { return s.dtype == TSV_FP32 && s.d == f32a::DH; }

int launch_tva_f32(const tsv_shape& s, const TvaPlan& p, const tsv_cache& c, const tsv_nodes& nd, const tsv_scratch& sc,
                   void* out, char* ws, cudaStream_t st) {
  // The keys known before the wait go first where some node may rank, which takes the selection long enough to work under it; else they
  // are a part of the one list, whose shares leave one remainder of a tile instead of two (16 sequences of 2048 tokens with up to 1024
  // selected: 54.4 us a pass, 56.5 in two parts).
  const bool early = p.need_scores != 0;
  const int64_t known = early ? s.max_L / s.m_hca + s.window + s.D : 0, chosen = p.keys_max - known;
  // CTAs per node: as many as fit the device at once while a share still holds 32 keys.  One per SM where many of the keys precede the
  // wait: beside the selection's CTAs there is room for one, and the others would begin when the selection has ended (16 sequences of
  // 256-4096 tokens with 64 selected: 38.0 us, 40.0 with two per SM).  Two, as the registers admit, where two thirds follow it (512
  // selected: 74.9 us, 85.0 with one), or half if a node would have one CTA only (18 sequences with 256 selected: 50.2, 56.4).  Of
  // clusters of four and eight 296 CTAs are not resident at once (72 clusters of four: 61 us, 58 of two).
  const int64_t base = (int64_t)s.B * s.D * ((s.H + f32a::HG - 1) / f32a::HG);
  auto ctas = [&](int large, int small) {
    int cs = 8;
    while (cs > 1 && (base * cs > (cs > 2 ? large : small) || (cs - 1) * 32 >= p.keys_max)) cs >>= 1;
    return cs;
  };
  int cs = ctas(148, 148);
  if (chosen >= 2 * known || (cs == 1 && chosen >= known)) cs = ctas(256, 296);
  const int bytes = 2 * f32a::KT * f32a::DH * 4;
  if (!ensure_smem((const void*)attn_f32_kernel<true>, bytes) || !ensure_smem((const void*)attn_f32_kernel<false>, bytes)) return TSV_ERR_CUDA;
  TSV_PREP(attn_f32_kernel<true>); TSV_PREP(attn_f32_kernel<false>);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(cs, s.D * ((s.H + f32a::HG - 1) / f32a::HG), s.B); cfg.blockDim = dim3(f32a::NT, 1, 1); cfg.dynamicSmemBytes = bytes; cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = cs; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr; cfg.numAttrs = 2;
  const cudaError_t e = early ? cudaLaunchKernelEx(&cfg, attn_f32_kernel<true>, s, p, c, nd, sc, (float*)out, ws)
                              : cudaLaunchKernelEx(&cfg, attn_f32_kernel<false>, s, p, c, nd, sc, (float*)out, ws);
  count_launch();
  return e == cudaSuccess && cudaGetLastError() == cudaSuccess ? TSV_OK : TSV_ERR_CUDA;
}

}  // namespace tsv
