// Shared pieces of the tensor-core (tcgen05) attention kernels: PTX wrappers, descriptors,
// the small shared-memory control block and the chunking rule.
#pragma once
#include "kernels.h"

namespace tsv {

namespace tc {

constexpr int DH = 512;             // head dim handled by this path
constexpr int BM = 128;             // rows per CTA
constexpr int PR = 256;             // rows per plan tile: two row tiles (one CTA pair) share one key list
constexpr int NC = 512;             // keys per chunk of a list that is cut into many
constexpr int NCMIN = 256;          // keys that are worth an SM pair of their own
constexpr uint32_t WAIT_LIMIT = 1u << 14;   // polls before a wait gives up (then no later wait of the thread is attempted)

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ uint64_t make_desc(uint32_t saddr, uint32_t lbo_bytes, uint32_t sbo_bytes) {
  // shared-memory matrix descriptor: 128-byte swizzle, descriptor version 1
  return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)(lbo_bytes >> 4) << 16) | ((uint64_t)(sbo_bytes >> 4) << 32) |
         (1ull << 46) | (2ull << 61);
}
__device__ __forceinline__ uint32_t make_idesc(int N, int b_mn_major) {
  // D fp32, A/B bf16, A K-major, M = 128
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)b_mn_major << 16) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
}
__device__ __forceinline__ void mma_ss(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
               ::"r"(d_tmem), "l"(a), "l"(b), "r"(idesc), "r"(acc) : "memory");
}
__device__ __forceinline__ void mma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Bounded wait on an mbarrier phase; false if the limit ran out.  Each try suspends the warp in hardware for up to
// SUSPEND_NS (it wakes as soon as the phase completes), so waiting warps do not compete for issue slots or for the
// shared-memory pipe with the warps that feed the tensor core.
constexpr uint32_t SUSPEND_NS = 4000;
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity) {
  const uint32_t a = smem_u32(bar);
  for (uint32_t it = 0; it < WAIT_LIMIT; ++it) {
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\tselp.b32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"(a), "r"(parity), "r"(SUSPEND_NS) : "memory");
    if (ok) return true;
  }
  return false;
}

__device__ __forceinline__ void cp16(uint32_t dst, const void* src, bool valid) {
  const int sz = valid ? 16 : 0;      // src-size 0: the 16 bytes are zero-filled
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(sz) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, %17, %18, %19, "
      "%20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]),
        "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]),
        "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]),
        "=r"(r[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_ld32_nowait(uint32_t taddr, uint32_t* r) {     // caller issues tcgen05.wait::ld before using r
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, %17, %18, %19, "
      "%20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]),
        "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]),
        "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]),
        "=r"(r[31])
      : "r"(taddr));
}
// 16 lanes x 64 columns: r[4 g + 2 h + c] is row 8 h + lane / 4, column 8 g + 2 (lane % 4) + c
__device__ __forceinline__ void tmem_ld16x256b_x8_nowait(uint32_t taddr, uint32_t* r) {     // likewise
  asm volatile(
      "tcgen05.ld.sync.aligned.16x256b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, %17, %18, %19, "
      "%20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]),
        "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]),
        "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]),
        "=r"(r[31])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]),
        "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
// Makes later uses of r depend on this point: placed after tcgen05.wait::ld so that the compiler cannot move a use of a
// loaded register above the wait.
__device__ __forceinline__ void tmem_regs_ready(uint32_t* r) {
  asm volatile("" : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]), "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]), "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]), "+r"(r[22]), "+r"(r[23]), "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]), "+r"(r[30]), "+r"(r[31]) :: "memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t* r) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
               ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
               "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]) : "memory");
}
__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

constexpr int NCX = 768;             // max keys per chunk of the TMA kernel: P (bf16) takes 384 TMEM columns, an O quarter 128
// Chunking of the TMA kernel: nch chunks of CL keys, CL a multiple of 128 and <= NCX.
// general = false (shapes whose capacities allow at most two chunks of NCX keys and no gathered tile): as few chunks as possible.
// general = true: a list that does not fit one chunk is cut into chunks of at most NC keys, whose quarters of O go through two
// buffers instead of one and which fill the SM pairs better (two chunks of up to NCX instead of three of NC cost 12 % of the
// attention kernel on 32 paged sequences of 256-4096 tokens, and gained nothing on 64 flat ones).
// split: items a tile may be cut into so that few tiles still use all pairs (1 where there are tiles enough).  general: a tile of more
// than NC keys into a chunk for every NCMIN keys or part of them (513 keys: 256, 256 and 1), up to split and to the slots of the
// workspace; one of up to NC keys stays whole.  Then, in both, by columns of the output: 1 << lds items of a chunk
// compute S and the softmax alike and each its own columns of O, which nobody has to merge.
// f32: the partial outputs of the tile are fp32 (a tile that is cut for the sake of parallelism alone is not rounded before
// the merge); f32_all: all multi-chunk tiles are.
__device__ __host__ __forceinline__ void chunking_x(int nk, bool general, int split, int chmax, bool f32_all, int& nch, int& CL, bool& f32, int& lds) {
  nch = (nk + NCX - 1) / NCX;
  if (general && nch > 1) nch = (nk + NC - 1) / NC;
  f32 = f32_all || nch <= 1;
  if (general && split > 1 && nk > NC) {
    int w = (nk + NCMIN - 1) / NCMIN;
    if (w > split) w = split;
    if (w > chmax) w = chmax;                            // (the workspace has slots for no more)
    if (w > nch) nch = w;
  }
  if (nch < 1) nch = 1;
  CL = (((nk + nch - 1) / nch) + 127) / 128 * 128;
  if (CL < 128) CL = 128;
  nch = (nk + CL - 1) / CL;
  if (nch < 1) nch = 1;
  lds = 4 * nch <= split ? 2 : 2 * nch <= split ? 1 : 0;
}
// The record of a tile, which the tile plan leaves and the kernels after it read: {sequence, what, keys, chunks}, what = mode (2 bits: 1
// boxes, 2 gathered) | fp32 partial outputs << 2 | chunk length / 128 << 4 | tile of the sequence << 7 | chunks, kManyChunks for that many
// and more, << 12 | log2 of the items of a chunk << 28.  In the record of a work item the last word is the item: its roles only ask for one
// chunk, two, or more.  (The chunking is three divisions: by every role of the attention kernel on its own they were 10 KB of its code.)
constexpr int kManyChunks = 0xFFFF;
__device__ __host__ __forceinline__ int4 tile_record(const TvaPlan& pl, int b, int tile, int mode, int nk) {
  int nch, CL, lds;
  bool f32;
  chunking_x(nk, pl.tc_general != 0, pl.tc_split, pl.tc_chmax, pl.tc_f32, nch, CL, f32, lds);
  return make_int4(b, mode | (f32 ? 4 : 0) | (CL / 128) << 4 | tile << 7 | (nch < kManyChunks ? nch : kManyChunks) << 12 | lds << 28, nk, nch);
}
static_assert(NCX / 128 < 8 && TSV_MAX_D * 128 / PR <= 32, "fields of a tile's record");
__device__ __host__ __forceinline__ bool rec_gather(const int4& r) { return (r.y & 3) == 2; }
__device__ __host__ __forceinline__ bool rec_f32(const int4& r) { return (r.y & 4) != 0; }
__device__ __host__ __forceinline__ int rec_chunk_keys(const int4& r) { return ((r.y >> 4) & 7) * 128; }
__device__ __host__ __forceinline__ int rec_tile(const int4& r) { return (r.y >> 7) & 31; }
__device__ __host__ __forceinline__ int rec_chunks_or_many(const int4& r) { return (r.y >> 12) & kManyChunks; }
__device__ __host__ __forceinline__ int rec_lds(const int4& r) { return r.y >> 28; }
// Of a tile's record.  (The packed count is read first, the word of its own only where that is saturated: with the word alone the merge
// kernel was slower, 64 sequences of 1-4 k tokens 755 us a pass, so 743.)
__device__ __host__ __forceinline__ int rec_chunks(const int4& r) { const int n = rec_chunks_or_many(r); return n < kManyChunks ? n : r.w; }
__device__ __host__ __forceinline__ int rec_items(const int4& r) { return rec_chunks(r) << rec_lds(r); }

}  // namespace tc

}  // namespace tsv
