// tree_verify_attn, tensor-core kernel run by PAIRS of CTAs (thread-block cluster of 2, tcgen05 cta_group::2), for key
// lists made of contiguous runs (fetched as TMA boxes) and for key lists of scattered rows (fetched four rows at a
// time by TMA gather).
//
// A pair covers 256 query rows of one sequence (256/H consecutive tree nodes x H heads); each CTA owns
// 128 of them in its own tensor memory.  The two SMs execute every MMA together (M = 256): the B operand
// -- the staged key rows -- is split between the two shared memories, so each SM fetches only HALF of
// the K tile (S = Q K^T: half of the keys) and half of the V tile (O = P K: half of the columns of d).
// That halves the bytes each SM pulls from L2.
// The pairs are persistent (one per two SMs): they take (tile, chunk of keys) items from a counter until none is left.
//   warps 0, 3, 12-15  producers: TMA boxes or four-row gathers (cp.async.bulk.tensor, 128-byte swizzle) into 16 KiB slots, each
//                slot owned by one producer; the copies of BOTH CTAs complete on the mbarriers of the leader (rank 0) CTA
//   warp 1       MMA issuer (leader CTA only): tcgen05.mma.cta_group::2, slot release and accumulator
//                events by tcgen05.commit multicast to both CTAs
//   warp 2       hands out the items (leader's counter, both CTAs told)
//   warps 4-11   one-pass softmax on the CTA's own S rows (TMEM), P written back to TMEM, epilogue of O straight from
//                registers, or through swizzled shared-memory tiles and TMA stores; events to the leader's MMA warp by remote arrive
// Stage stream, TMEM column plan, running-max rule and chunking are those described at the kernel.
#include <cuda.h>
#include <stdio.h>
#include <cudaTypedefs.h>

#include <atomic>

#include "tc_common.cuh"

namespace tsv {

namespace pair {

using namespace tc;

// Warps: 0, 3, 12-15 producers; 1 MMA issuer; 2 hands out the items; 4-11 softmax and epilogue.  The service warpgroups give
// registers to the compute warpgroups: 128 x (120 + 136 + 136 + 120) of the 512 x 128 the CTA is launched with.
constexpr int TTHREADS = 512;
constexpr int NPROD = 6;                    // (12 slots: six producers with two each)
constexpr int REGS_SERVICE = 120, REGS_COMPUTE = 136;
static_assert(128 * (2 * REGS_SERVICE + 2 * REGS_COMPUTE) <= TTHREADS * 128, "register split beyond what the CTA is launched with");
constexpr int BOXB = kBoxRows * 128;       // bytes of one box: kBoxRows rows x 128 bytes
constexpr float RESCALE_GAP = 16.f;        // log2 units a later piece's row max may exceed the running reference
constexpr float REF_FLOOR = -3e38f;        // lowest reference: a row whose first visible scores are all -inf gives them the weight zero, not NaN

constexpr int NSX = 14;                    // 16 KiB slots of the staging area
constexpr int NQS = 8;                     // Q slices of an item (all of d, resident for every piece)
constexpr int NKS = NSX - NQS;             // K stages in flight
constexpr int NSV = 12;                    // Slots [0, 12) are one FIFO: an item's first six Q slices and its ring of six K stages take the next twelve
                                           // places, its V stages (once the S products are complete) the places from the same start on; so
                                           // the next item's operands land where the V stages are released first.  Slots 12, 13: the last
                                           // two Q slices, and, when O is read out, the staging of the output where it is staged (a 4 KiB tile per warp).
// The FIFO's places of an item, about in the order in which the S products want them: Q0 K0 Q1 K1 Q2 K2 K3 Q3 K4 Q4 K5 Q5 (of places
// p and p + 6, which are one producer's, one is a Q slice, the other a K stage).  Six stages of operands are requested before the item
// before is done with; with all of Q and four K stages in the FIFO, and the ring's other two stages waiting for the output's staging,
// the products waited for the fifth stage, requested when the first product was complete (640-key items 20.2 us, now 19.4).
__device__ __forceinline__ int q_place(int dk) { return dk < 3 ? 2 * dk : 2 * dk + 1; }         // dk < 6; slices 6 and 7 are in slots 12 and 13
__device__ __forceinline__ int k_place(int pos) { return pos < 3 ? 2 * pos + 1 : 2 * pos; }     // pos: stage modulo NKS

struct Ctl {                               // control block at the start of dynamic shared memory; no barrier is ever re-initialised
  uint64_t fullQ[NQS];                     // Q slice dk of the item has arrived
  uint64_t fullK[NKS], emptyK[NKS];        // ring of the K stages
  uint64_t fullV[NSV], emptyV[NSV];        // ring of the V stages (starts when the S products are complete)
  uint64_t acc_ev[7];                      // MMA -> other warps, one barrier per event, at most once per item:
                                           //   [pc] S of piece pc is complete   [3 + p] the item's part p of O is complete
  uint64_t cmp_ev[7];                      // compute warps -> MMA, likewise:
                                           //   [pc] P of piece pc is in TMEM   [3 + p] part p of O has been read out
  uint64_t stage_free;                     // the item's output tiles have left the staging slots (this CTA's; not used where GENERAL)
  uint64_t item_ev;                        // the next item has been handed out
  uint32_t tmem_base;
  int32_t merge_here;                      // set for the CTA that finished a multi-chunk tile last
  alignas(16) int4 item[2];                // the pair's current and next work: the tile's record with the item in its last word (sequence -1: no more)
  float xch[2][2][BM];                     // first-slab maxima of the rows, by the two warps that share them (two buffers in turn)
};
constexpr int CTLB = 3072;                 // control block bytes; the ring follows (needs a 1024-byte aligned base)
constexpr int SLOTP = 16384;               // ring slot: every stage of a CTA is at most 16 KiB
constexpr int SMEM_X = CTLB + NSX * SLOTP;
static_assert(sizeof(Ctl) <= CTLB, "control block overflow");
constexpr int NBAR = NQS + 2 * NKS + 2 * NSV + 7 + 7 + 2;      // barriers, at the start of the block
static_assert(offsetof(Ctl, tmem_base) == NBAR * 8 && NBAR <= 64, "the barriers are initialised by a thread each");

__device__ __forceinline__ void mbar_init(uint64_t* b, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(b)), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* b, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(b)), "r"(bytes) : "memory");
}
// shared::cluster address of the same variable in CTA `rank` of the cluster
__device__ __forceinline__ uint32_t map_to_rank(uint32_t saddr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(rank));
  return r;
}
// Arrival on a barrier of the pair for events in tensor memory only (tcgen05.wait and tcgen05.fence::before_thread_sync come
// before it, tcgen05.fence::after_thread_sync after the wait): relaxed, because a release at cluster scope would also
// order the thread's ordinary writes, which takes about 900 cycles and which nobody needs here.
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_addr) {
  asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
// TMA box copy into this CTA's shared memory; completion is counted on an mbarrier given by its cluster address
__device__ __forceinline__ void tma_box2(uint32_t dst, const CUtensorMap* map, int x, int y, uint32_t bar_cluster_addr) {
  asm volatile("cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
               ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar_cluster_addr) : "memory");
}
// the same box into L2 only
__device__ __forceinline__ void tma_box_l2(const CUtensorMap* map, int x, int y) {
  asm volatile("cp.async.bulk.prefetch.tensor.2d.L2.global.tile [%0, {%1, %2}];" ::"l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y) : "memory");
}
// four rows of a 2D tensor, given by their row indices, as four consecutive 128-byte lines of this CTA's shared memory
__device__ __forceinline__ void tma_gather4(uint32_t dst, const CUtensorMap* map, int x, const uint4& code, uint32_t bar_cluster_addr) {
  asm volatile("cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.tile::gather4.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5, %6}], [%7];"
               ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"((int)(code.x & 0x3FFFFFFFu)), "r"((int)(code.y & 0x3FFFFFFFu)),
                 "r"((int)(code.z & 0x3FFFFFFFu)), "r"((int)(code.w & 0x3FFFFFFFu)), "r"(bar_cluster_addr) : "memory");
}
__device__ __forceinline__ void mma2_ss(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
               ::"r"(d_tmem), "l"(a), "l"(b), "r"(idesc), "r"(acc) : "memory");
}
__device__ __forceinline__ void mma2_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::2.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
               ::"r"(d_tmem), "r"(a_tmem), "l"(b), "r"(idesc), "r"(acc) : "memory");
}
// arrives on the same barrier (same shared-memory offset) in both CTAs of the pair once all prior MMAs have completed
__device__ __forceinline__ void mma2_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
               ::"r"(smem_u32(bar)), "h"((uint16_t)3) : "memory");
}
__device__ __forceinline__ uint32_t make_idesc2(int N, int b_mn_major) {      // M = 256 over the pair
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)b_mn_major << 16) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(256 >> 4) << 24);
}
// 16 bytes into the shared memory of a CTA of the pair, counted on a barrier of the same CTA (both by cluster address)
__device__ __forceinline__ void st_async16(uint32_t cluster_addr, const int4& v, uint32_t bar_cluster_addr) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];"
               ::"r"(cluster_addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w), "r"(bar_cluster_addr) : "memory");
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// the two halves of the pair-wide barrier, for work that does not depend on the peer in between
__device__ __forceinline__ bool elect_one() {           // true in one lane of the (converged) warp
  uint32_t r;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.b32 %0, 1, 0, p;\n\t}" : "=r"(r));
  return r != 0;
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void compute_sync() { asm volatile("bar.sync 1, 256;" ::: "memory"); }

// Tensor maps of one call: every source array with boxes of 32, 64 and 128 rows (64 columns, 128-byte swizzle), so that
// a stage whose key rows are consecutive rows of one array is fetched by ONE large request.
struct alignas(64) MapSet {
  CUtensorMap q;          // 128-row boxes
  CUtensorMap out;        // 32-row boxes (stores; not used where GENERAL)
  CUtensorMap src[4][3];  // [csa, hca, window, packed misc][32, 64, 128 rows]
  CUtensorMap row[4];     // the same arrays with one-row boxes: gathers of four rows by index
};
constexpr int NMAPS = 18;

constexpr uint32_t OOB_BOX = 0x3FFFFF00u;   // map 0, a row beyond every tensor: the box is zero-filled

}  // namespace pair

// One item of work: a chunk of CL keys (pieces of 256 keys, the last may hold 128) of one 256-row tile.
namespace pair {
constexpr int NQ = 4, OW = tc::DH / NQ;      // the PV product is computed in NQ parts of OW columns of d
struct Item {
  int tix, b, tile, nk, chunk, nch, CL, cbeg, cend;      // (nch: kManyChunks for more than that)
  int npc;                 // S pieces
  int lds, p0, np;         // log2 of the items of a chunk; this one's parts of O: [p0, p0 + np)
  bool dbl;                // two O buffers: a part is computed while the one before is read out
  bool f32;                // partial outputs are fp32
  bool gather;             // the key list is a list of row codes (array << 30 | row), not of boxes
  __device__ __forceinline__ Item(int4 r, const TvaPlan& pl, bool general) {      // a tile's record, the item in its last word
    b = r.x; tile = rec_tile(r); tix = b * pl.tc_nt + tile;
    gather = general && rec_gather(r); f32 = general && rec_f32(r);
    lds = rec_lds(r);
    nk = r.z; chunk = r.w >> lds; nch = rec_chunks_or_many(r);
    np = NQ >> lds; p0 = (r.w & ((1 << lds) - 1)) * np;
    const int stride = rec_chunk_keys(r);
    cbeg = chunk * stride; cend = min(nk, cbeg + stride);
    CL = max(128, (cend - cbeg + 127) & ~127);           // (the tile's last chunk is as long as what is left)
    npc = (CL + 255) / 256;
    dbl = CL <= 512;
  }
  __device__ __forceinline__ uint32_t acc_used() const { return ((1u << npc) - 1u) | (((1u << np) - 1u) << 3); }
  __device__ __forceinline__ uint32_t cmp_used() const { return (1u << (npc - 1)) | (npc == 3 ? 2u : 0u) | (((1u << np) - 1u) << 3); }
};
}  // namespace pair

// PERSISTENT: one pair per two SMs walks its share of the items.  What a pair that served one item each lost on every item
// (start-up of the CTAs and barriers 4 k cycles, the gap between two CTAs on an SM 5 k, the first operands' latency
// 4-6 k, of 47 k for 512 keys) happens once: barriers and tensor memory live as long as the kernel, the next item's Q
// slices go into the V slots the last part of O has released, its first K stages follow, and its S products run under the
// read-out and the stores of the last part of O.
//
// Stages per item and CTA (rank r of the pair):
//   Q slices:  per 64-wide slice dk of d  [this CTA's 128 rows x 64 dims], fetched once, resident for all pieces
//   K stages:  piece after piece, per slice dk  [this CTA's half of the piece's keys x 64 dims]
//   V stages (after the last S product): per quarter of d, per 128 keys: [128 keys x this CTA's 64 of the quarter's 128 dims]
// TMEM columns (per CTA, its own 128 rows).  S piece 0 -> [0,256), pieces 1 and 2 -> [256,512) (fp32); P piece pc (bf16 pairs) ->
// [128 pc, 128 pc + 128); O, in four quarters of 128 columns: CL <= 512 alternately at [256,384) and [384,512), so that a quarter's
// products run while the one before is read out (halves of 256 columns left the tensor core idle for 2.4 k cycles of 31 k per
// 512-key item), else at [384,512).
//
// Every barrier phase is counted by its users: each role keeps, per barrier, the parity of its next use, and a slot's
// latest release is awaited before it is filled again, across items too.
//
// GENERAL: gathered tiles and tiles of more than two chunks may occur (shapes whose capacities rule both out run the
// instantiation without that code).
template <bool GENERAL>
__global__ void __launch_bounds__(pair::TTHREADS, 1)
tc_attn_pair_kernel(const __grid_constant__ pair::MapSet maps, const tsv_shape s,
                    const TvaPlan pl, const void* __restrict__ q, void* __restrict__ out_, char* __restrict__ ws, int32_t* __restrict__ status) {
  using namespace pair;
  extern __shared__ unsigned char smem_raw[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  uint32_t rank;                                                // the two CTAs of a pair are neighbours in x
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  Ctl& sm = *reinterpret_cast<Ctl*>(smem_raw);
  const uint32_t ring = smem_u32(smem_raw + CTLB);
  int fail = (smem_u32(smem_raw) & 1023u) ? 1 : 0;             // the swizzled tiles need a 1024-byte aligned base
  // Set-up, a warp for each part of it: one thread that initialised the sixty barriers before it allocated tensor memory took 1.7 us
  // from the CTA's start to the wait below, of the 25 us a layer of one short sequence takes.
  if (tid < NBAR) {
    mbar_init(&sm.fullQ[0] + tid, tid >= offsetof(Ctl, cmp_ev) / 8 && tid < offsetof(Ctl, cmp_ev) / 8 + 7 ? 16       // 8 compute warps of each CTA
                                  : tid == offsetof(Ctl, stage_free) / 8 ? 8 : 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 2) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&sm.tmem_base)) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  if (warp == 3 && lane < (GENERAL ? NMAPS : 14))   // the descriptors of the tensor maps in use are fetched while the plan is read
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&maps) + (uint64_t)lane * sizeof(CUtensorMap)) : "memory");
  __syncwarp();
  fence_before();
  cluster_arrive();                                              // this CTA's barriers exist and its tensor memory is allocated
  auto leave = [&]() {
    if (fail) for (int b = (int)(blockIdx.x >> 1); b < s.B; b += (int)(gridDim.x >> 1)) atomicOr(status + b, TSV_ST_INTERNAL);   // (an internal error: every sequence is flagged)
    fence_before();
    __syncthreads();
    cluster_sync_all();                                          // neither CTA leaves while the other may still signal it or read its memory
    fence_after();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, 512;" ::"r"(sm.tmem_base) : "memory");
  };
  // The queries of tile p by pair p into L2 (its first item is another tile: the longest ones go first, but all pairs' first phase
  // is bound by what arrives from HBM).  Here, and not by the tile plan's CTAs, which do not end before the copies they have asked
  // for: of 64 sequences the wait below ended 2.6 us sooner.  Before that wait: the queries are the caller's.
  if (warp == 2 && lane == 0) {
    const int p = blockIdx.x >> 1, b = p / pl.tc_nt, r0 = (p - b * pl.tc_nt) * PR + (int)rank * BM, rows = min(BM, s.D * s.H - r0);
    if (b < s.B && rows > 0)
      asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(reinterpret_cast<const char*>(q) + ((size_t)b * s.D * s.H + r0) * (DH * 2)), "r"(rows * DH * 2) : "memory");
  }
  // Launched as a programmatic dependent of the tile plan: the CTAs take their places and set up while that kernel's last
  // CTAs finish, and read nothing of its before it has completed.
  asm volatile("griddepcontrol.wait;" ::: "memory");
  // The merge kernel, where one follows, may take its places: it waits for this kernel before it does anything.  (Nothing else may
  // start before this kernel has ended: the next call's tile plan would overwrite what is read here.)
  if (GENERAL && pl.tc_chmax > 1) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  // Item 0 of pair p is item p / ntile of tile p % ntile, which every warp looks up itself; the others are handed out (warp 2).
  const int ntile = s.B * pl.tc_nt, P = gridDim.x >> 1, me = blockIdx.x >> 1, item0 = (uint32_t)me / (uint32_t)ntile;
  const int4 rec0 = __ldcg(reinterpret_cast<const int4*>(ws + pl.off_order) + (me - item0 * ntile));
  cluster_wait();                                                // barriers of both CTAs exist before anyone signals them
  fence_after();
  const uint32_t tm = sm.tmem_base;
  const int rows_seq = s.D * s.H;
  // Item n of this pair (sequence -1: no more).  The wait is made whatever failed before (a failure skips later
  // waits, never a step of the protocol, so that no warp is left alone at a barrier), and is longer than any other.
  const int own = rec0.z > 0 && item0 < rec_items(rec0) ? 1 : 0;
  auto next_item = [&](int n) {
    if (n < own) return make_int4(rec0.x, rec0.y, rec0.z, item0);
    bool ok = false;
    for (int i = 0; i < 8 && !ok; ++i) ok = mbar_wait(&sm.item_ev, (uint32_t)(n - own) & 1u);
    int4 r = sm.item[(n - own) & 1];
    if (!ok) { r.x = -1; fail = 1; }
    return r;
  };

  // (the register split dominates each side's code, which the compiler budgets by it)
  if (warp < 4 || warp >= 12) {
  asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(REGS_SERVICE));
  if (warp == 0 || warp == 3 || warp >= 12) {
    // ------------------------------------------------------------------ producers (both CTAs)
    // Every slot belongs to one producer, which issues all its copies and awaits all its releases in order (a parity wait
    // is only good for the phase after the last one seen).  Both CTAs' copies complete on the leader's barriers.
    // (Six warps because of the gathered tiles: a stage is 32 four-row requests there, and a warp takes about 70 cycles to
    // issue one; boxes would do with two.)
    // A producer steps from one of its own stages to the next: going over all stages of the item and picking out its own took it 1.1 us
    // from one copy to the next, longer than the slots were in use (512-key items 17.2 us, see k_ring).
    const int pw = warp == 0 ? 0 : warp == 3 ? 1 : warp - 10;
    uint32_t kcnt = 0, accb = 0;                                  // parities of the uses so far: ring positions of the K stages; events
    uint32_t vcnt = 0, vused = 0;                                 // of this producer's FIFO slots pw and pw + 6 (bits 0, 1): parity of the V stages so far, any
    int n_real = 0;                                               // items with keys so far
    auto v_wait = [&](int h) {                                    // the release of the latest V stage in FIFO slot pw + 6 h
      if (((vused >> h) & 1u) && !fail && !mbar_wait(&sm.emptyV[pw + NPROD * h], ((vcnt >> h) & 1u) ^ 1u)) fail = 1;
    };
    // the boxes of a chunk: lane i holds box i of up to NCX / kBoxRows
    auto load_box = [&](const Item& w) {
      uint32_t v = OOB_BOX;
      if (!w.gather && lane < NCX / kBoxRows && w.cbeg + lane * kBoxRows < w.cend) {
        const int2 bx = __ldg(reinterpret_cast<const int2*>(ws + pl.off_box) + (size_t)w.tix * (pl.tc_maxk / kBoxRows) + w.cbeg / kBoxRows + lane);
        v = ((uint32_t)bx.x << 30) | (uint32_t)bx.y;
      }
      return v;
    };
    int g0 = 0;                                                   // slot of the item's first place in the FIFO
#pragma unroll 1
    for (int it = 0;; ++it) {
      const int4 r = next_item(it);
      if (r.x < 0) break;
      const Item w(r, pl, GENERAL);
      const uint32_t box = load_box(w);
      const int CL = w.CL, row0 = w.tile * PR + (int)rank * BM;
      const int nvb = CL / 128;                                    // V stages per part
      const int NKST = 8 * w.npc, NVST = w.np * nvb;
      // This producer's places of the item are u and u + 6: slots pw + 6 h0 and pw + 6 (1 - h0).
      const int u = (pw + 2 * NPROD - g0) % NPROD, h0 = (g0 + u) % NSV >= NPROD ? 1 : 0;
      const int kpos = (u & 1) ? u >> 1 : 3 + (u >> 1);            // its ring position of the K stages
      const int khalf = (u & 1) ? h0 : h0 ^ 1, kphys = pw + NPROD * khalf;
      // bit i: boxes i and i + 1 name consecutive rows of one array (one request can fetch both)
      uint32_t cons = 0;
      auto consecutive = [&](int i0, int nb) { return ((~(cons >> i0)) & ((1u << (nb - 1)) - 1u)) == 0u; };
      // Gathered tiles: the keys' row codes stay in global memory (the tile plan left them there, four-aligned groups
      // never mix arrays); lane l fetches the codes of rows 4 l .. 4 l + 3 of a stage itself.  Keys past the end of the list
      // read row 0 of the first array (they are masked).
      const uint4* code_g = reinterpret_cast<const uint4*>(reinterpret_cast<const uint32_t*>(ws + pl.off_krow) + (size_t)w.tix * pl.tc_maxk + w.cbeg);
      auto codes_at = [&](int key) { return w.cbeg + key < w.cend ? __ldg(code_g + (key >> 2)) : make_uint4(0u, 0u, 0u, 0u); };
      uint4 kcode = make_uint4(0u, 0u, 0u, 0u);                                // this lane's codes of the current piece's K stages
      int kcode_pc = -1;
      auto issue_q = [&](int dk, int slot) {
        if (lane == 0) {
          if (slot < NSV) v_wait(slot >= NPROD);                   // (a V stage of the item before)
          else if (!GENERAL && n_real && !fail && !mbar_wait(&sm.stage_free, (uint32_t)(n_real - 1) & 1u)) fail = 1;
          if (rank == 0) mbar_expect_tx(&sm.fullQ[dk], 2 * SLOTP);
          tma_box2(ring + (uint32_t)slot * SLOTP, &maps.q, dk * 64, w.b * rows_seq + row0, map_to_rank(smem_u32(&sm.fullQ[dk]), 0));
          if (!GENERAL && n_real && dk < 2) tma_box_l2(&maps.q, (dk + 6) * 64, w.b * rows_seq + row0);     // (the slots of slices 6 and 7 are free last)
        }
        __syncwarp();
      };
      uint32_t kc = (kcnt >> kpos) & 1u;
      bool kuse = n_real > 0, kfirst = true;                           // the position has been used; the item's first use is still to come
      auto issue_k = [&](int gk) {
        const int pc = gk >> 3, dk = gk & 7;
        const uint32_t slot = ring + (uint32_t)kphys * SLOTP;
        const uint32_t fb_leader = map_to_rank(smem_u32(&sm.fullK[kpos]), 0);
        const int bytes = min(256, CL - pc * 256) * 64;                        // bytes THIS CTA copies in the stage
        if (w.gather && kcode_pc != pc) {                                      // this CTA's half of the piece's keys: bytes / 128 rows
          kcode_pc = pc;
          if (lane * 512 < bytes) kcode = codes_at(pc * 256 + (int)rank * (bytes >> 7) + 4 * lane);
        }
        if (lane == 0) {
          if (kfirst) v_wait(khalf);                               // (a V stage of the item before)
          if (kuse && !fail && !mbar_wait(&sm.emptyK[kpos], kc ^ 1u)) fail = 1;
          if (rank == 0) mbar_expect_tx(&sm.fullK[kpos], 2 * bytes);            // bytes of both CTAs
        }
        kfirst = false; kuse = true; kc ^= 1u;
        __syncwarp();
        // this CTA's half of the piece's keys: boxes [rank * nb, rank * nb + nb) of the piece
        const int nb = bytes / BOXB, i0 = pc * (256 / kBoxRows) + (int)rank * nb;
        if (w.gather) {
          if (lane * 512 < bytes) tma_gather4(slot + lane * 512, &maps.row[kcode.x >> 30], dk * 64, kcode, fb_leader);
        } else {
          const bool one = consecutive(i0, nb);                    // nb = 4 (128 rows) or 2 (64 rows)
          const uint32_t bx = __shfl_sync(0xffffffffu, box, one ? i0 : i0 + (lane & 3));
          // (the stage of this piece that takes its place has to wait for its product: its rows come from L2 then)
          const bool ahead = gk < 8 - NKS && n_real;
          if (one) {
            const CUtensorMap* map = &maps.src[bx >> 30][nb == 4 ? 2 : 1];
            if (lane == 0) {
              tma_box2(slot, map, dk * 64, (int)(bx & 0x3FFFFFFFu), fb_leader);
              if (ahead) tma_box_l2(map, (dk + NKS) * 64, (int)(bx & 0x3FFFFFFFu));
            }
          } else if (lane < nb) {
            tma_box2(slot + lane * BOXB, &maps.src[bx >> 30][0], dk * 64, (int)(bx & 0x3FFFFFFFu), fb_leader);
            if (ahead) tma_box_l2(&maps.src[bx >> 30][0], (dk + NKS) * 64, (int)(bx & 0x3FFFFFFFu));
          }
        }
        __syncwarp();
      };
      if (!(u & 1)) issue_q(u >> 1, pw + NPROD * h0);
      {
        const uint32_t box_up = __shfl_down_sync(0xffffffffu, box, 1);
        cons = __ballot_sync(0xffffffffu, lane < 31 && (box & 0x3FFFFFFFu) < (OOB_BOX & 0x3FFFFFFFu) && box_up == box + kBoxRows);
      }
      issue_k(kpos);
      if (u & 1) issue_q(3 + (u >> 1), pw + NPROD * (h0 ^ 1));
      if (u == 2 || u == 4) issue_q(5 + (u >> 1), NSV - 1 + (u >> 1));       // (slots 12 and 13: free since the S products of the item before, which this warp has awaited, or since its output left them)
#pragma unroll 1
      for (int gk = kpos + NKS; gk < NKST; gk += NKS) issue_k(gk);
      kcnt ^= w.npc == 1 ? 0x3Cu : w.npc == 2 ? 0x0Fu : 0u;        // (8, 16 or 24 stages over six positions)
      // V stages reuse the whole staging area: they start when the last S product is complete (the softmax of the last
      // piece is still to come, so the ring is full by the time the PV products start)
      if (lane == 0 && !fail && !mbar_wait(&sm.acc_ev[w.npc - 1], (accb >> (w.npc - 1)) & 1u)) fail = 1;
      __syncwarp();
      {
        int part = w.p0, kb = u, h = h0;
#pragma unroll 1
        for (int gv = u; gv < NVST; gv += NPROD) {
          while (kb >= nvb) { kb -= nvb; ++part; }
          const int sl = pw + NPROD * h;
          const uint32_t slot = ring + (uint32_t)sl * SLOTP;
          const uint32_t fb_leader = map_to_rank(smem_u32(&sm.fullV[sl]), 0);
          uint4 vcode = make_uint4(0u, 0u, 0u, 0u);                 // (fetched before the wait for the slot)
          if (w.gather) vcode = codes_at(kb * 128 + 4 * lane);
          if (lane == 0) {
            v_wait(h);
            if (rank == 0) mbar_expect_tx(&sm.fullV[sl], 2 * SLOTP);
          }
          __syncwarp();
          if (w.gather) tma_gather4(slot + lane * 512, &maps.row[vcode.x >> 30], (part * 2 + (int)rank) * 64, vcode, fb_leader);
          else {                    // key boxes 0..3
            const int i0 = kb * (128 / kBoxRows);
            const bool one = consecutive(i0, 4);
            const uint32_t bx = __shfl_sync(0xffffffffu, box, one ? i0 : i0 + (lane & 3));
            if (one) { if (lane == 0) tma_box2(slot, &maps.src[bx >> 30][2], (part * 2 + (int)rank) * 64, (int)(bx & 0x3FFFFFFFu), fb_leader); }
            else if (lane < 4) tma_box2(slot + lane * BOXB, &maps.src[bx >> 30][0], (part * 2 + (int)rank) * 64, (int)(bx & 0x3FFFFFFFu), fb_leader);
          }
          vcnt ^= 1u << h; vused |= 1u << h;
          h ^= 1; kb += NPROD;
        }
      }
      g0 = (g0 + NVST) % NSV;
      accb ^= w.acc_used();
      ++n_real;
    }
    // every release has arrived in this CTA before it may leave
    if (lane == 0) {
      if (n_real) for (int sl = 0; sl < NKS; ++sl) if (!fail && !mbar_wait(&sm.emptyK[sl], ((kcnt >> sl) & 1u) ^ 1u)) fail = 1;
      v_wait(0); v_wait(1);
    }
    __syncwarp();
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer (leader CTA only)
    // The whole warp walks the stages and one elected lane issues: with control flow and indices uniform over the warp the
    // descriptors are computed in uniform registers, where the instruction wants them.  (Inside a one-lane branch every
    // operand is moved there first, and the issuing thread was the pacemaker: 175 cycles per 256-wide product.)
    if (rank == 0) {
      const uint32_t idesc_k256 = make_idesc2(256, 0), idesc_k128 = make_idesc2(128, 0);
      uint32_t accb = 0, cmpb = 0, kpar = 0, vpar = 0;    // parities of the next use, per event / slot
      int g0 = 0;
      uint32_t pend = 0;                                  // read-out events of the item before that are still to be awaited
      uint32_t pend_par = 0;
      const bool one = elect_one();
      auto need_ev = [&](int e) { if (!fail && !mbar_wait(&sm.cmp_ev[e], (cmpb >> e) & 1u)) fail = 1; };
      // the columns [256, 512) of the item before have been read out
      auto need_pend = [&]() {
#pragma unroll
        for (int e = 3; e < 3 + NQ; ++e) if (((pend >> e) & 1u) && !fail && !mbar_wait(&sm.cmp_ev[e], (pend_par >> e) & 1u)) fail = 1;
        pend = 0;
      };
#pragma unroll 1
      for (int it = 0;; ++it) {
        int4 r = next_item(it);
        r = make_int4(__shfl_sync(0xffffffffu, r.x, 0), __shfl_sync(0xffffffffu, r.y, 0), __shfl_sync(0xffffffffu, r.z, 0), __shfl_sync(0xffffffffu, r.w, 0));
        if (r.x < 0) break;
        const Item w(r, pl, GENERAL);
        const int CL = w.CL, npc = w.npc, nvb = CL / 128;
        const uint32_t idesc_v = make_idesc2(OW, 1);
        // The issuing thread is the pacemaker of the tensor pipe: stages are walked with counters (no divisions), and the
        // descriptors of a stage are the slot-0 descriptor plus a multiple of the slot size (the address field counts
        // 16-byte units and cannot overflow within the ring).
        const uint64_t dk0 = make_desc(ring, 16, 1024), dv0 = make_desc(ring, 16384, 1024);
        // S, piece after piece (the softmax of a piece runs while the tensor core works on the next one): per piece the
        // eight slices of d, Q slice from its resident slot, K stage from the ring
        auto place = [&](int i) { const int p = g0 + i; return p >= NSV ? p - NSV : p; };
        int sl = 0;                                        // ring position of the next K stage
#pragma unroll 1
        for (int pc = 0; pc < npc; ++pc) {
          if (pc == 1) need_pend();                        // piece 1 overwrites the last part of O of the item before
          if (pc == 2) need_ev(1);                         // piece 2 reuses the S columns of piece 1
          const uint32_t scol = tm + (pc == 0 ? 0 : 256);
          const uint32_t idesc = CL - pc * 256 >= 256 ? idesc_k256 : idesc_k128;
#pragma unroll 1
          for (int dk = 0; dk < 8; ++dk) {
            if (pc == 0 && !fail && !mbar_wait(&sm.fullQ[dk], (uint32_t)it & 1u)) fail = 1;
            if (!fail && !mbar_wait(&sm.fullK[sl], (kpar >> sl) & 1u)) fail = 1;
            kpar ^= 1u << sl;
            fence_after();
            const int kphys = place(k_place(sl)), qphys = dk < NKS ? place(q_place(dk)) : NSV - NKS + dk;
            const uint64_t qd = dk0 + (uint64_t)(qphys * (SLOTP >> 4)), kd = dk0 + (uint64_t)(kphys * (SLOTP >> 4));
#pragma unroll
            for (int ks = 0; ks < 4; ++ks) if (one) mma2_ss(scol, qd + 2 * ks, kd + 2 * ks, idesc, (dk | ks) != 0);
            if (one) mma2_commit(&sm.emptyK[sl]);
            if (++sl == NKS) sl = 0;
          }
          if (one) mma2_commit(&sm.acc_ev[pc]);                     // S of the piece is complete
        }
        need_pend();
        sl = g0;                                           // slot of the next V stage
#pragma unroll 1
        for (int part = 0; part < w.np; ++part) {
          const uint32_t ocol = tm + (w.dbl ? 256 + (part & 1) * OW : 384);
          if (part == 0) need_ev(npc - 1);                 // all of P is in TMEM
          else if (!w.dbl || part >= 2) need_ev(3 + part - (w.dbl ? 2 : 1));      // the part before in these columns has been read out
#pragma unroll 1
          for (int kb = 0; kb < nvb; ++kb) {
            if (!fail && !mbar_wait(&sm.fullV[sl], (vpar >> sl) & 1u)) fail = 1;
            vpar ^= 1u << sl;
            fence_after();
            const uint64_t vd = dv0 + (uint64_t)(sl * (SLOTP >> 4));
            // per CTA: 128 keys x 64 dims = one [128 x 64] tile
#pragma unroll
            for (int ks = 0; ks < 8; ++ks) if (one) mma2_ts(ocol, tm + (kb >> 1) * 128 + (ks >> 2) * 64 + (kb & 1) * 32 + (ks & 3) * 8, vd + ks * (2048 >> 4), idesc_v, (kb | ks) != 0);
            if (one) mma2_commit(&sm.emptyV[sl]);
            if (++sl == NSV) sl = 0;
          }
          if (one) mma2_commit(&sm.acc_ev[3 + part]);
        }
        // P (overwritten by the next item's first piece) is free when the last part is complete
        if (!fail && !mbar_wait(&sm.acc_ev[2 + w.np], (accb >> (2 + w.np)) & 1u)) fail = 1;
        pend = ((1u << w.np) - (1u << max(0, w.np - (w.dbl ? 2 : 1)))) << 3; pend_par = cmpb;      // the last part or two
        accb ^= w.acc_used(); cmpb ^= w.cmp_used();
        g0 = sl;
      }
    }
    __syncwarp();
  } else {
    // ------------------------------------------------------------------ hands out the items
    // The plan kernel left a record per tile, longest work items first.  The items are the tiles' chunks (or shares of the columns of
    // chunks) in that order; pair p starts with the one every warp knows, all others are taken from a counter (items differ in length and in
    // where their rows come from, so a fixed deal leaves pairs idle: 177 k cycles for the slowest of 74 pairs against a mean
    // of 125 k on 64 sequences of 1-4 k tokens).  The leader's warp takes the next item when the current one's S is complete and
    // passes it on when all compute warps have stored its P: every warp of the pair has seen the current one then, and the
    // producers are about to need the next.
    const int4* order = reinterpret_cast<const int4*>(ws + pl.off_order);
    if (rank == 0) {
      int32_t* counter = reinterpret_cast<int32_t*>(ws + pl.off_sched);
      uint32_t cmpb = 0, accb = 0;
      int base = 0, w0 = -32;                           // window: tiles w0 .. w0 + 31, a lane each; base: items before it
      int4 rec = make_int4(-1, 0, 0, 0);
      int n = 0, incl = 0, tot = 0, given = 0;          // of the lane's tile: items handed out here, those of the lanes up to it, all lanes'; items given
      auto take = [&]() {                               // the next item of the device
        int q = 0x7fffffff;
        if (lane == 0 && !fail) q = atomicAdd(counter, 1);
        q = __shfl_sync(0xffffffffu, q, 0);
        while (q >= base + tot && w0 + 32 < ntile) {
          base += tot; w0 += 32;
          n = 0;
          if (w0 + lane < ntile) {
            rec = order[w0 + lane];
            if (rec.z > 0) { n = rec_items(rec); given = min(n, (P - (w0 + lane) + ntile - 1) / ntile); n -= given; }
          }
          incl = n;
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) { const int y = __shfl_up_sync(0xffffffffu, incl, o); if (lane >= o) incl += y; }
          tot = __shfl_sync(0xffffffffu, incl, 31);
        }
        int4 r = make_int4(-1, 0, 0, 0);
        if (q < base + tot) {
          const uint32_t has = __ballot_sync(0xffffffffu, q - base < incl);
          const int src = __ffs(has) - 1;
          r.x = __shfl_sync(0xffffffffu, rec.x, src); r.y = __shfl_sync(0xffffffffu, rec.y, src); r.z = __shfl_sync(0xffffffffu, rec.z, src);
          r.w = q - base - __shfl_sync(0xffffffffu, incl - n - given, src);
        }
        return r;
      };
      int4 r = own ? make_int4(rec0.x, rec0.y, rec0.z, item0) : take();
#pragma unroll 1
      for (int it = 0;; ++it) {
        if (it >= own) {
          if (lane < 2) st_async16(map_to_rank(smem_u32(&sm.item[(it - own) & 1]), lane), r, map_to_rank(smem_u32(&sm.item_ev), lane));
          if (lane == 0) mbar_expect_tx(&sm.item_ev, 16);
          __syncwarp();
        }
        if (r.x < 0) break;
        const Item w(r, pl, GENERAL);
        const int last = w.npc - 1;
        if (!fail && !mbar_wait(&sm.acc_ev[last], (accb >> last) & 1u)) fail = 1;
        const int4 next = take();
        if (!fail && !mbar_wait(&sm.cmp_ev[last], (cmpb >> last) & 1u)) fail = 1;
        accb ^= w.acc_used(); cmpb ^= w.cmp_used();
        fail = __any_sync(0xffffffffu, fail);
        r = next;
      }
      // the last pair to run out of items leaves the counters as it found them
      if (lane == 0 && atomicAdd(counter + 1, 1) == P - 1) { counter[0] = 0; counter[1] = 0; __threadfence(); }
    } else {
#pragma unroll 1
      for (int it = own;; ++it) {
        if (lane == 0) mbar_expect_tx(&sm.item_ev, 16);
        __syncwarp();
        if (next_item(it).x < 0) break;
      }
    }
    // tiles without keys (flagged sequences, padding): zeros, tile t by pair t mod P, each CTA its own rows
#pragma unroll 1
    for (int t0 = me; t0 < ntile; t0 += 32 * P) {
      int4 rz = make_int4(0, 0, 1, 0);
      if (t0 + lane * P < ntile) rz = order[t0 + lane * P];
      uint32_t zero = __ballot_sync(0xffffffffu, rz.z <= 0);
      while (zero) {
        const int src = __ffs(zero) - 1, b = __shfl_sync(0xffffffffu, rz.x, src), row0 = __shfl_sync(0xffffffffu, rec_tile(rz), src) * PR + (int)rank * BM;
        zero &= zero - 1;
        uint4* o4 = reinterpret_cast<uint4*>(reinterpret_cast<bf16*>(out_) + ((size_t)b * rows_seq + row0) * DH);
        const int n16 = min(BM, rows_seq - row0) * (DH / 8);
#pragma unroll 1
        for (int i = lane; i < n16; i += 32) o4[i] = make_uint4(0, 0, 0, 0);
      }
    }
  }
  leave();
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(REGS_COMPUTE));
    // ------------------------------------------------------------------ softmax + epilogue (8 warps)
    const int q4 = warp & 3, hh = (warp - 4) >> 2;
    const int row = q4 * 32 + lane;
    const uint32_t tlane = tm + ((uint32_t)(q4 * 32) << 16);
    const uint32_t mybit = 1u << ((int)rank * (BM / s.H) + row / s.H);      // node of this row within the pair's plan tile
    const float scale2 = s.sm_scale * 1.4426950408889634f;
    uint32_t accb = 0;                               // parity of the next use of each acc_ev
    // The merge kernel is told, per warp, that an item's rows are stored: half an item later, when the stores are
    // long complete (right after them the release waits a memory latency for them), and the pair's last item is signalled at the end.  Not where
    // tiles are cut to fill the device: all items end at about the same time there.
    int stored_rix = -1;
    auto signal_stored = [&]() {
      if (GENERAL && stored_rix >= 0) {
        __syncwarp();                                // (the other lanes' stores are before the release)
        if (lane == 0) asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(reinterpret_cast<int32_t*>(ws + pl.off_tcnt) + stored_rix) : "memory");
      }
      stored_rix = -1;
    };
#pragma unroll 1
    for (int it = 0;; ++it) {
    const int4 rec = next_item(it);
    if (rec.x < 0) break;
    const Item w(rec, pl, GENERAL);
    const int b = w.b, nch = w.nch, CL = w.CL, chunk = w.chunk, npc = w.npc;
    const int row0 = w.tile * PR + (int)rank * BM;   // first of this CTA's rows within the sequence
    const size_t rix = (size_t)b * 2 * pl.tc_nt + 2 * w.tile + rank;      // this CTA's 128-row tile (partials of multi-chunk tiles)
    const uint8_t* kmask_g = reinterpret_cast<const uint8_t*>(ws + pl.off_kmask) + (size_t)w.tix * pl.tc_maxk + w.cbeg;
    float m_run = -INFINITY;                         // reference max of the row (log2 units)
    float lp[4] = {0.f, 0.f, 0.f, 0.f};              // this thread's share of the row sum, four independent chains

    auto p_stored = [&](int pc) {                    // this warp's P of piece pc is in TMEM: tell the leader's MMA warp
      asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
      fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(map_to_rank(smem_u32(&sm.cmp_ev[pc]), 0));
    };
    // The softmax goes over a piece ONCE, in slabs of 32 keys, one after the other: a slab is read from tensor memory, checked against
    // the row's reference maximum, exponentiated and stored as P.
    //
    // Reference: the maximum over the visible keys of the first slab that has any (the two warps of a row, which share
    // its keys, exchange it once).  bf16 and fp32 have the range for weights above 1, so a later slab changes the reference
    // only where it exceeds it by more than RESCALE_GAP (then the warp rescales what it has stored, and the two warps settle
    // on one reference before the PV product: rare).
    //
    // Slabs: the warps with hh = 0 take slabs 0, 1, 4, 5 of a piece, those with hh = 1 slabs 2, 3, 6, 7.  P of piece pc lands in
    // columns [128 pc, 128 pc + 128), a warp's slabs side by side from 64 hh on: P of pieces 0 and 1 overlays S of piece 0, P of
    // piece 2 overlays S of piece 2, and with this split every column a warp writes held S of its OWN slabs, all read
    // before: no warp waits for another.  (A two-pass softmax with contiguous halves needed three barriers a piece and
    // read S twice.)
    constexpr uint32_t FULL = 0xffffffffu;
    uint32_t* xch = reinterpret_cast<uint32_t*>(sm.xch) + (it & 1) * 2 * BM;
    auto pair_sync = [&]() { asm volatile("bar.sync %0, 64;" ::"r"(2 + q4) : "memory"); };     // the two warps of these rows
    auto pair_or = [&](uint32_t x) {                 // the same, and whether x is set in any of their threads
      uint32_t y;
      asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %1, 0;\n\tbarrier.cta.red.or.pred q, %2, 64, p;\n\tselp.b32 %0, 1, 0, q;\n\t}" : "=r"(y) : "r"(x), "r"(2 + q4) : "memory");
      return y;
    };
    auto slab_of = [&](int i) { return (i & 1) + ((i & 2) << 1) + 2 * hh; };
    // slab i of this warp in the piece whose S begins at column scol: read, invisible keys as -inf; the maximum (unscaled)
    auto read_slab = [&](uint32_t scol, int i, uint32_t vis, uint32_t (&sv)[32]) {
      tmem_ld32(scol + slab_of(i) * 32, sv);
      if (vis != FULL) {
#pragma unroll
        for (int t = 0; t < 32; ++t) if (!((vis >> t) & 1u)) sv[t] = 0xff800000u;
      }
      float mc[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) mc[c] = __uint_as_float(sv[c]);
#pragma unroll
      for (int t = 4; t < 32; ++t) mc[t & 3] = fmaxf(mc[t & 3], __uint_as_float(sv[t]));
      return fmaxf(fmaxf(mc[0], mc[1]), fmaxf(mc[2], mc[3]));
    };
    // multiplies this thread's P columns [64 hh of every piece before pc, the first n slabs of piece pc] by f
    auto rescale_p = [&](int pc, int n, float f) {
      asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
#pragma unroll 1
      for (int v = 0; v < 4 * pc + n; ++v) {
        const uint32_t col = tlane + (v >> 2) * 128 + hh * 64 + (v & 3) * 16;
        uint32_t r[16];
        tmem_ld16(col, r);
#pragma unroll
        for (int t = 0; t < 16; ++t) {
          const float2 pv = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&r[t]));
          const __nv_bfloat162 h2 = __floats2bfloat162_rn(pv.x * f, pv.y * f);
          r[t] = *reinterpret_cast<const uint32_t*>(&h2);
        }
        tmem_st16(col, r);
      }
#pragma unroll
      for (int c = 0; c < 4; ++c) lp[c] *= f;
    };
    // A visible key has been found.  The branches that hold warp-collective instructions follow this, which is alike in all threads of
    // the two warps, and not the rows' references: finite queries and keys can have a product of -inf in one row alone.
    uint32_t seen = 0;
    int moved = 0;                                   // this warp changed its reference after the exchange
    // Node masks of this lane's keys of a piece, a byte per slab; fetched a piece ahead (fetched when needed they cost the chain a
    // memory latency, 1.3 k cycles per piece after the first).
    uint32_t km = 0;
    auto fetch_masks = [&](int pc) {
      km = 0;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int key = pc * 256 + slab_of(i) * 32 + lane;
        if (key < CL && w.cbeg + key < w.cend) km |= (uint32_t)__ldg(kmask_g + key) << (8 * i);
      }
    };
    fetch_masks(0);
#pragma unroll 1
    for (int pc = 0; pc < npc; ++pc) {
      const int ns = CL - pc * 256 >= 256 ? 4 : 2;   // slabs of this warp
      const uint32_t km_now = km;
      // visibility of a slab, a bit per key: the 32 rows of a warp belong to one node (H >= 32 on this path), so one ballot over the
      // keys' node masks gives the word
      auto visible = [&](int i) { return __ballot_sync(FULL, (km_now >> (8 * i)) & mybit); };
      if (pc + 1 < npc) fetch_masks(pc + 1);
      if (!fail && !mbar_wait(&sm.acc_ev[pc], (accb >> pc) & 1u)) fail = 1;
      fence_after();
      const uint32_t scol = tlane + (pc == 0 ? 0 : 256);
      // One slab after the other in a loop of one slab's code: what the two warps of a scheduler leave idle is the other's, and the
      // instructions of four slabs side by side did not stay in the instruction cache (kernel of 97 KB, a slab 900 cycles; 512 is what
      // the special-function unit needs for the two warps).
      if (!seen) {
        int i = 0;
        uint32_t vis = 0;
#pragma unroll 1
        for (; i < ns; ++i) if ((vis = visible(i)) != 0) break;
        uint32_t sv[32];
        const float mc = i < ns ? read_slab(scol, i, vis, sv) : -INFINITY;
        xch[hh * BM + row] = __float_as_uint(mc);
        seen = pair_or(i < ns);                      // (if not, nobody reads the words before they are written again)
        if (seen) m_run = fmaxf(fmaxf(mc, __uint_as_float(xch[(hh ^ 1) * BM + row])) * scale2, REF_FLOOR);
      }
#pragma unroll 1
      for (int i = 0; i < ns; ++i) {
        uint32_t pk[16];
        const uint32_t vis = visible(i);
        if (seen && vis) {
          uint32_t sv[32];
          const float mc = read_slab(scol, i, vis, sv) * scale2;
          if (__any_sync(FULL, mc > m_run + RESCALE_GAP)) {        // (warp-uniform: tensor-memory accesses are warp-collective)
            const float to = mc > m_run + RESCALE_GAP ? mc : m_run;
            rescale_p(pc, i, ex2(m_run - to));
            m_run = to;
            moved = 1;
          }
#pragma unroll
          for (int t = 0; t < 32; t += 2) {
            const float p0 = ex2(fmaf(__uint_as_float(sv[t]), scale2, -m_run)), p1 = ex2(fmaf(__uint_as_float(sv[t + 1]), scale2, -m_run));
            lp[(t >> 1) & 3] += p0 + p1;
            const __nv_bfloat162 h2 = __floats2bfloat162_rn(p0, p1);
            pk[t >> 1] = *reinterpret_cast<const uint32_t*>(&h2);
          }
        } else {
#pragma unroll
          for (int t = 0; t < 16; ++t) pk[t] = 0u;
        }
        tmem_st16(tlane + pc * 128 + hh * 64 + i * 16, pk);
      }
      // the MMA warp waits for the last piece only (and, with three pieces, for piece 1 before it overwrites that
      // piece's S columns); the wait for the stores of a later piece covers the earlier ones
      if (npc == 3 && pc == 1) p_stored(1);
    }
    // The row sums meet, in the words in which the maxima did (the two warps have read those when they are past the barrier below, and
    // write them again two items on); where a warp moved its reference, the two settle on the larger one first.
    float l_row = (lp[0] + lp[1]) + (lp[2] + lp[3]);
    {
      // (no reference moved, as nearly always: P is announced before the sums are exchanged)
      const uint32_t any_moved = pair_or(moved);
      auto exchange = [&](float v) {
        xch[hh * BM + row] = __float_as_uint(v);
        pair_sync();
        return __uint_as_float(xch[(hh ^ 1) * BM + row]);
      };
      if (any_moved) {                               // (alike in both warps)
        const float m_other = exchange(m_run), to = fmaxf(m_run, m_other), f = ex2(m_run - to);
        const int last = npc - 1;
        if (__any_sync(FULL, f != 1.f)) rescale_p(last, CL - last * 256 >= 256 ? 4 : 2, f);
        l_row *= f;
        m_run = to;
        pair_sync();                                 // (the words are written again)
      }
      p_stored(npc - 1);
      l_row += exchange(l_row);
    }
    signal_stored();                                 // (of the item before; after P, which the tensor core waits for)

    const float inv = l_row > 0.f ? 1.f / l_row : 0.f;
    constexpr int cw = OW / 2;                        // columns of the part this thread handles
    // The output leaves by one of two ways.  GENERAL: straight from registers, so that the next item's last two Q slices need not wait until
    // staging in their slots has been read (4 x 128 k 103.0 -> 99.7 us, 16 of 512-8192 tokens 3 %).  Else, where most pairs have an item or
    // two and the code is run through cold, staged for TMA stores, in half the instructions (one short stack takes 2 % more the other way).
    const bool full_tile = row0 + BM <= rows_seq;     // whole tile inside the sequence: rows may be stored as 32-row boxes
    const uint32_t stage = ring + (uint32_t)NSV * SLOTP + (uint32_t)(warp - 4) * 4096;   // this warp's tile of 32 rows x 64 columns (bf16)
    bool stored = false;
    // GENERAL: rows of the output, or of the chunk's slot of partial outputs: fp32, or bf16 at the start of the slot, which has room for
    // fp32; normalised, a merge kernel follows.  Read out so that four lanes share a row; they transpose their 4 x 4 words, and a
    // warp's store is whole 128-byte lines of eight rows.  (A row per lane, 32 bytes of a line each: 64 short sequences 423 -> 448 us.)
    const bool p32 = nch > 1 && w.f32;
    const int quad = lane >> 2, q = lane & 3, rowb = p32 ? DH * 4 : DH * 2;
    char* dst = nch == 1 ? reinterpret_cast<char*>(out_) + ((size_t)b * rows_seq + row0) * (DH * 2)
                         : ws + pl.off_tpo + (rix * pl.tc_chmax + chunk) * ((size_t)BM * DH * 4);
    const bool wide = (reinterpret_cast<uintptr_t>(dst) & 31) == 0;
    const int nrow = (nch > 1 ? BM : rows_seq - row0) - q4 * 32 - quad;       // rows 8 x of this lane with 8 x < nrow are written
    dst += (q4 * 32 + quad) * rowb;
    auto put32 = [&](char* p, const uint32_t (&v)[8]) {
      if (wide) asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]) : "memory");
      else {                                         // (the caller's output is aligned to 16 bytes)
        reinterpret_cast<uint4*>(p)[0] = make_uint4(v[0], v[1], v[2], v[3]);
        reinterpret_cast<uint4*>(p)[1] = make_uint4(v[4], v[5], v[6], v[7]);
      }
    };
    auto transpose4 = [&](uint32_t& v0, uint32_t& v1, uint32_t& v2, uint32_t& v3) {      // lane q's word i <-> lane i's word q
      const bool h2 = q & 2, h1 = q & 1;
      const uint32_t a = __shfl_xor_sync(FULL, h2 ? v0 : v2, 2), c = __shfl_xor_sync(FULL, h2 ? v1 : v3, 2);
      if (h2) { v0 = a; v1 = c; } else { v2 = a; v3 = c; }
      const uint32_t d = __shfl_xor_sync(FULL, h1 ? v0 : v1, 1), e = __shfl_xor_sync(FULL, h1 ? v2 : v3, 1);
      if (h1) { v0 = d; v2 = e; } else { v1 = d; v3 = e; }
    };
#pragma unroll 1
    for (int part = 0; part < w.np; ++part) {
      if (!fail && !mbar_wait(&sm.acc_ev[3 + part], (accb >> (3 + part)) & 1u)) fail = 1;
      fence_after();
      const uint32_t ocol = tlane + (w.dbl ? 256 + (part & 1) * OW : 384) + hh * cw;
      const int col = (w.p0 + part) * OW + hh * cw;
      uint32_t r[64];                                // GENERAL: [half of 16 rows][group of 8 columns][8 rows further][column]: row quad, columns 2 q, 2 q + 1
      if (GENERAL) {
        tmem_ld16x256b_x8_nowait(ocol, r);
        tmem_ld16x256b_x8_nowait(ocol + (16u << 16), r + 32);
      } else {
        tmem_ld32_nowait(ocol, r);
        tmem_ld32_nowait(ocol + 32, r + 32);
      }
      asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
      tmem_regs_ready(r);
      tmem_regs_ready(r + 32);
      fence_before();                                // in registers: the columns may be overwritten
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(map_to_rank(smem_u32(&sm.cmp_ev[3 + part]), 0));
      if (GENERAL) {
#pragma unroll
        for (int x = 0; x < 4; ++x) {                // rows 8 x + quad
          const float f = __shfl_sync(FULL, inv, 8 * x + quad);
          const uint32_t* rx = r + 32 * (x >> 1) + 2 * (x & 1);
          char* p = dst + 8 * x * rowb;
          uint32_t v[8];
          if (p32) {
#pragma unroll
            for (int j = 0; j < 2; ++j) {            // lane q: the columns of group 4 j + q
#pragma unroll
              for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int c = 0; c < 2; ++c) v[2 * i + c] = __float_as_uint(__uint_as_float(rx[4 * (4 * j + i) + c]) * f);
              transpose4(v[0], v[2], v[4], v[6]);
              transpose4(v[1], v[3], v[5], v[7]);
              if (8 * x < nrow) put32(p + (col + 8 * (4 * j + q)) * 4, v);
            }
          } else {                                   // lane q: the columns of groups 2 q and 2 q + 1
#pragma unroll
            for (int g = 0; g < 8; ++g) {
              const __nv_bfloat162 h2 = __floats2bfloat162_rn(__uint_as_float(rx[4 * g]) * f, __uint_as_float(rx[4 * g + 1]) * f);
              v[4 * (g & 1) + (g >> 1)] = *reinterpret_cast<const uint32_t*>(&h2);
            }
            transpose4(v[0], v[1], v[2], v[3]);
            transpose4(v[4], v[5], v[6], v[7]);
            if (8 * x < nrow) put32(p + (col + 16 * q) * 2, v);
          }
        }
      } else if (nch == 1) {
        // stage the 32 x 64 bf16 tile in the 128-byte swizzle pattern and store it with one TMA request
        if (stored) {                                // the store before has read the staging tile
          if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
          __syncwarp();
        }
        stored = true;
#pragma unroll
        for (int v = 0; v < 8; ++v) {
          uint32_t pk[4];
#pragma unroll
          for (int t = 0; t < 4; ++t) {
            const __nv_bfloat162 h2 = __floats2bfloat162_rn(__uint_as_float(r[8 * v + 2 * t]) * inv, __uint_as_float(r[8 * v + 2 * t + 1]) * inv);
            pk[t] = *reinterpret_cast<const uint32_t*>(&h2);
          }
          asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(stage + lane * 128 + ((v ^ (lane & 7)) << 4)), "r"(pk[0]), "r"(pk[1]), "r"(pk[2]),
                       "r"(pk[3]) : "memory");
        }
        if (full_tile) {
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          __syncwarp();
          if (lane == 0) {
            asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.tile.bulk_group [%0, {%1, %2}], [%3];"
                         ::"l"(reinterpret_cast<uint64_t>(&maps.out)), "r"(col), "r"(b * rows_seq + row0 + q4 * 32), "r"(stage) : "memory");
            asm volatile("cp.async.bulk.commit_group;" ::: "memory");
          }
        } else {                                     // the rows of this sequence only: plain stores, 64 columns of a row by eight lanes
          __syncwarp();
#pragma unroll 1
          for (int i = lane; i < 32 * 8; i += 32) {
            const int rr = i >> 3;
            uint4 v;
            asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(stage + rr * 128 + (((i ^ rr) & 7) << 4)) : "memory");
            if (row0 + q4 * 32 + rr < rows_seq)
              reinterpret_cast<uint4*>(reinterpret_cast<bf16*>(out_) + ((size_t)b * rows_seq + row0 + q4 * 32 + rr) * DH + col)[i & 7] = v;
          }
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");       // (the next item's queries are copied over the tile)
          __syncwarp();                              // (the tile is written again)
          stored = false;
        }
      } else {
        float* po = reinterpret_cast<float*>(ws + pl.off_tpo) + ((rix * pl.tc_chmax + chunk) * BM + row) * DH + col;
#pragma unroll
        for (int v = 0; v < 16; ++v)
          *reinterpret_cast<float4*>(po + v * 4) = make_float4(__uint_as_float(r[4 * v]), __uint_as_float(r[4 * v + 1]), __uint_as_float(r[4 * v + 2]), __uint_as_float(r[4 * v + 3]));
      }
      if (nch > 1 && w.p0 + part == 0 && hh == 0)
        reinterpret_cast<float2*>(ws + pl.off_tpml)[(rix * pl.tc_chmax + chunk) * BM + row] = make_float2(m_run, l_row);
    }
    if (!GENERAL && lane == 0) {                     // the staging slots are free for the next item's Q slices
      asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
      asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&sm.stage_free)) : "memory");
    }
    accb ^= w.acc_used();
    if (GENERAL && nch > 1 && pl.tc_split == 1) stored_rix = (int)rix;
    if (!GENERAL && nch > 1) {
      // Tiles of two chunks where nothing longer can occur: each chunk leaves its unnormalised part of O with (max, sum)
      // per row; the CTA that finishes a 128-row tile last merges the parts (fixed order, so the result does not depend
      // on who was last).  (In general a merge kernel follows: one CTA would take too long over many chunks.)
      __threadfence();
      compute_sync();
      if (warp == 4 && lane == 0) {
        int32_t* cnt = reinterpret_cast<int32_t*>(ws + pl.off_tcnt) + rix;
        const int done = atomicAdd(cnt, 1);
        sm.merge_here = done == (nch << w.lds) - 1;
      }
      compute_sync();
      if (sm.merge_here) {
        __threadfence();
        bf16* orow0 = reinterpret_cast<bf16*>(out_) + ((size_t)b * rows_seq + row0) * DH;
        const float* po = reinterpret_cast<const float*>(ws + pl.off_tpo) + rix * pl.tc_chmax * BM * DH;
        const float2* pml = reinterpret_cast<const float2*>(ws + pl.off_tpml) + rix * pl.tc_chmax * BM;
        // A warp takes 16 rows (wr, wr + 8, ...), a lane columns 4 (l + 32 k) .. + 3 of a row.  (Few registers on purpose: the path
        // is rare and must not cost the kernel around it any.)
        const int wr = warp - 4;
#pragma unroll 1
        for (int r = wr; r < BM && row0 + r < rows_seq; r += 8) {
          const float2 a0 = __ldcg(pml + r), a1 = __ldcg(pml + BM + r);
          const float m = fmaxf(a0.y > 0.f ? a0.x : -INFINITY, a1.y > 0.f ? a1.x : -INFINITY);
          const float w0 = a0.y > 0.f ? exp2f(a0.x - m) : 0.f, w1 = a1.y > 0.f ? exp2f(a1.x - m) : 0.f, l = a0.y * w0 + a1.y * w1;
          const float i0 = l > 0.f ? w0 / l : 0.f, i1 = l > 0.f ? w1 / l : 0.f;
          const float4* p0 = reinterpret_cast<const float4*>(po + (size_t)r * DH);
          const float4* p1 = reinterpret_cast<const float4*>(po + ((size_t)BM + r) * DH);
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const float4 x = __ldcg(p0 + lane + 32 * k), y = __ldcg(p1 + lane + 32 * k);
            const __nv_bfloat162 lo = __floats2bfloat162_rn(fmaf(x.x, i0, y.x * i1), fmaf(x.y, i0, y.y * i1));
            const __nv_bfloat162 hi = __floats2bfloat162_rn(fmaf(x.z, i0, y.z * i1), fmaf(x.w, i0, y.w * i1));
            uint2 o2;
            o2.x = *reinterpret_cast<const uint32_t*>(&lo); o2.y = *reinterpret_cast<const uint32_t*>(&hi);
            *reinterpret_cast<uint2*>(orow0 + (size_t)r * DH + 4 * (lane + 32 * k)) = o2;
          }
        }
      }
    }
    }
    if (!GENERAL && lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    signal_stored();
    leave();
  }
}

// ------------------------------------------------------------------------------------------------ host side
static PFN_cuTensorMapEncodeTiled encode_fn() {
  static PFN_cuTensorMapEncodeTiled fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess && q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled>(p);
  }
  return fn;
}

// rows x 512 bf16, row-major; boxes of 64 columns in the 128-byte swizzle
static bool make_map(CUtensorMap* m, const void* basep, int64_t rows, int box_rows) {
  PFN_cuTensorMapEncodeTiled fn = encode_fn();
  if (!fn || rows <= 0 || ((uintptr_t)basep & 15)) return false;
  const cuuint64_t gdim[2] = {(cuuint64_t)tc::DH, (cuuint64_t)rows};
  const cuuint64_t gstr[1] = {(cuuint64_t)tc::DH * 2};
  const cuuint32_t box[2] = {64u, (cuuint32_t)box_rows};
  const cuuint32_t estr[2] = {1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(basep), gdim, gstr, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool tva_tc_pair_usable(const tsv_cache& c) { return c.csa_rows > 0 && encode_fn() != nullptr; }


// Everything of the paired kernel's launch that can fail on the host, done before any kernel of the call is enqueued:
// the tensor maps and the kernel's shared-memory attribute.
int prepare_tva_tc_pair(const tsv_shape& s, const TvaPlan& p, const tsv_cache& c, const tsv_nodes& nd, void* out, char* ws, TvaTcPrep& prep) {
  // (a layer without HCA entries has no HCA array to map: its map is never used and stands in as a copy of the CSA one)
  const bool has_hca = c.hca_rows > 0 && c.hca_kv;
  const void* bases[4] = {c.csa_kv, has_hca ? c.hca_kv : c.csa_kv, c.win_kv, ws + p.off_misc};
  const int64_t rows[4] = {c.csa_rows, has_hca ? c.hca_rows : c.csa_rows, c.page_table ? c.tok_rows : (int64_t)s.B * s.window, (int64_t)s.B * p.tc_misc_rows};
  static_assert(sizeof(pair::MapSet) == sizeof(prep.maps), "TvaTcPrep holds a MapSet");
  pair::MapSet& ms = *reinterpret_cast<pair::MapSet*>(prep.maps);
  bool ok = make_map(&ms.q, nd.q, (int64_t)s.B * s.D * s.H, 128) && make_map(&ms.out, out, (int64_t)s.B * s.D * s.H, 32);
  for (int a = 0; a < 4 && ok; ++a) {
    for (int k = 0; k < 3 && ok; ++k) ok = make_map(&ms.src[a][k], bases[a], rows[a], 32 << k);
    ok = ok && make_map(&ms.row[a], bases[a], rows[a], 1);
  }
  if (!ok) {
    fprintf(stderr, "tsv: cuTensorMapEncodeTiled failed\n");
    return TSV_ERR_CUDA;
  }
  if (!ensure_smem((const void*)tc_attn_pair_kernel<true>, pair::SMEM_X) || !ensure_smem((const void*)tc_attn_pair_kernel<false>, pair::SMEM_X)) {
    fprintf(stderr, "tsv: cannot set %d bytes of dynamic shared memory\n", pair::SMEM_X);
    return TSV_ERR_CUDA;
  }
  TSV_PREP(tc_attn_pair_kernel<true>);
  TSV_PREP(tc_attn_pair_kernel<false>);
  return TSV_OK;
}

int launch_tva_tc_pair(const tsv_shape& s, const TvaPlan& p, const TvaTcPrep& prep, bool general, const void* q, void* out, char* ws, int32_t* status, cudaStream_t st) {
  const pair::MapSet& ms = *reinterpret_cast<const pair::MapSet*>(prep.maps);
  cudaLaunchConfig_t cfg = {};
  const int64_t most = (int64_t)p.tc_nt * s.B * (p.tc_split > 1 ? (p.tc_chmax > p.tc_split ? p.tc_chmax : p.tc_split) : p.tc_chmax);      // items, if every tile had the most
  cfg.blockDim = dim3(pair::TTHREADS, 1, 1);
  cfg.dynamicSmemBytes = pair::SMEM_X;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;          // may take its places under the plan kernel's tail (it waits inside)
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  // as many pairs as the device holds at once (asked for once; 74 on a B200), but no more than there can be items
  static std::atomic<int> resident{0};
  int pairs = resident.load(std::memory_order_relaxed);
  if (!pairs) {
    cfg.gridDim = dim3(2, 1, 1);
    if (cudaOccupancyMaxActiveClusters(&pairs, tc_attn_pair_kernel<true>, &cfg) != cudaSuccess || pairs < 1) { cudaGetLastError(); pairs = 64; }
    resident.store(pairs, std::memory_order_relaxed);
  }
  if (pairs > most) pairs = (int)most;
  cfg.gridDim = dim3(2 * pairs, 1, 1);
  const cudaError_t le = general ? cudaLaunchKernelEx(&cfg, tc_attn_pair_kernel<true>, ms, s, p, q, out, ws, status)
                                 : cudaLaunchKernelEx(&cfg, tc_attn_pair_kernel<false>, ms, s, p, q, out, ws, status);
  if (le != cudaSuccess) {
    int ncl = -1;
    cudaOccupancyMaxActiveClusters(&ncl, tc_attn_pair_kernel<true>, &cfg);
    fprintf(stderr, "tsv: cluster launch failed: %s (max active clusters %d, grid %d x %d x %d)\n", cudaGetErrorString(le), ncl,
            cfg.gridDim.x, cfg.gridDim.y, cfg.gridDim.z);
  }
  count_launch();
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) fprintf(stderr, "tsv: launch of the paired attention kernel failed: %s\n", cudaGetErrorString(e));
  return e == cudaSuccess ? TSV_OK : TSV_ERR_CUDA;
}

}  // namespace tsv
