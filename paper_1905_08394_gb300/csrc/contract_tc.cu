// K4 (tensor-core forms): one site absorption of the column sweep as a
// complex-as-real GEMM on the 5th-generation tensor cores (tcgen05), for a
// batch of lanes,
//   D[M x Nr] = A[M x Kr] * Bt[Nr x Kr]^T,   Kr = 2K, Nr = 2N,
// A = the running tensor G (interleaved re/im, the contracted legs (h_r, v)
// fastest), Bt = the real embedding of the site operand E:
//   Bt[2n  ][2k] =  Re E_kn   Bt[2n  ][2k+1] = -Im E_kn
//   Bt[2n+1][2k] =  Im E_kn   Bt[2n+1][2k+1] =  Re E_kn
// so that D's row is the interleaved complex output row (supplementary
// exact-overlap absorption step, transposed to columns).
//
// Forms: BF16 / FP16 (kind::f16, one MMA per k-step), BF16X2 / FP16X2 (hi/lo
// planes of A and Bt, three MMAs hi*hi + hi*lo + lo*hi accumulated in FP32),
// TF32 (kind::tf32, one MMA).
//
// Structure: persistent CTAs (one per SM) walk tiles (lane, M block, N block
// of up to 256 real columns).  Warp 0 issues TMA loads of A and Bt tiles
// (128-byte or 64-byte swizzle) into a ring of shared-memory stages, warp 1
// issues tcgen05.mma into one of two TMEM accumulators, the epilogue warps drain the
// other accumulator with tcgen05.ld, apply the step's power-of-two scale,
// split into the storage format and store permuted (the slowest untouched leg
// moves next to v'), and record the max |entry|.
//
// What bounds a short-K step is the epilogue's stores and its per-tile
// set-up, not the MMAs.  Rows are taken m_hi first (TcParams::mhi), so that a
// warp's stores cover whole 128-byte lines instead of one sector in each of 32
// lines (the L2 takes some 70 write requests per ns whatever their size);
// entries go out 32 bytes at a time; an item's set-up is loaded for 32 items
// at once; the index arithmetic has no 64-bit division.  16 lanes of a
// 32768 x 64 x 64 step (FP16X3, 537 MB read and written): 230 -> 95 us (5.6
// TB/s); of a 4096 x 64 x 512 step: 172 -> 61 us; the open-leg step 32768 x 128
// x 256 with P = 16, one item: 155 -> 38 us.
//
// CG = 2 (the default where the row tiles pair up and BN is a multiple of 32): a
// cluster of two CTAs on neighbouring SMs computes a 256-row tile with the 2-SM
// UMMA (tcgen05.mma.cta_group::2, M = 256).  Each CTA loads its own 128 rows of A
// and only half of the Bt tile; the even CTA issues the MMAs for both, and
// the TMA completions of both CTAs arrive on its barriers.  Per SM this
// halves the Bt bytes ingested per multiply-add, which is what bounds the
// single-CTA form (the MMA warp waits on operand arrival, not on the
// epilogue).  Every wait is bounded by a %globaltimer budget; on expiry the
// CTA raises the abort flag in both CTAs, sets the device timeout word,
// drains and releases TMEM before returning.
#include <cuda.h>
#include <cuda_runtime.h>

#include <cstring>
#include <mutex>

#include "common.h"
#include "format.cuh"
#include "share.cuh"

namespace peps {

namespace {

constexpr int BM = 128;
// Warps: a TMA producer, an MMA issuer and EPI epilogue warps; EPI = 4 (one per
// TMEM lane quadrant) or 8 (two per quadrant, each draining half of the
// tile's columns, for steps whose epilogue outlasts their MMAs).
// DR = 1 (a draining epilogue, eight warps): the accumulators take all of TMEM
// (256 columns of main and of correction sums), so a tile's MMAs wait for the
// epilogue of the one before.  A warp then reads its 128 columns into registers
// at once (the two sums added), releases TMEM, and scales, splits and stores
// from registers under the next tile's MMAs.  Its 128 held values need more
// registers than a thread gets at launch, so the producer's warpgroup (the
// producer, the MMA issuer and two idle warps) gives some up: 384 threads x 168
// = 128 x 72 + 256 x 216.
constexpr int first_epi(int dr) { return dr ? 4 : 2; }
constexpr int threads_of(int epi, int dr) { return 32 * (first_epi(dr) + epi); }

template <int FMT> struct FormTraits;
template <> struct FormTraits<FMT_BF16>   { static constexpr int NP = 1, ESZ = 2, KIND = 0, AB = 1; };
template <> struct FormTraits<FMT_FP16>   { static constexpr int NP = 1, ESZ = 2, KIND = 0, AB = 0; };
template <> struct FormTraits<FMT_BF16X2> { static constexpr int NP = 2, ESZ = 2, KIND = 0, AB = 1; };
template <> struct FormTraits<FMT_FP16X2> { static constexpr int NP = 2, ESZ = 2, KIND = 0, AB = 0; };
template <> struct FormTraits<FMT_TF32>   { static constexpr int NP = 1, ESZ = 4, KIND = 1, AB = 2; };

struct __align__(128) TcParams {   // the tensor maps need 128-byte alignment
  CUtensorMap mapA;        // {k, m, plane, lane}; m_hi-major steps: {k, m_hi, m_lo, b, plane/lane}
  CUtensorMap mapB[2];     // [plane] {k, n, operand variant}
  StepShape sh;
  const StepItem *items;
  const OpDesc *ops;
  Rec *recs;
  DeviceStatus *st;
  int n_items;
  int tiles_m, tiles_n;
  int BN;
  int stages;
  int tmem_cols;
  int ksplit;   // K segments accumulated in separate TMEM columns, summed in the
                // epilogue with round-to-nearest FP32 adds (long-K steps)
  int csep;     // 1: the split form's correction products (hi*lo, lo*hi) have
                // their own accumulator after the K segments
  int nacc;     // accumulators per buffer: ksplit + csep
  int nbuf;     // accumulator buffers (2: the epilogue of a tile overlaps the
                // next tile's MMAs)
  int mhi;      // 1: a tile's rows are ph consecutive m_hi x lh consecutive m_lo x
                // bh consecutive b (ph lh bh = BM, m_hi fastest), so that a
                // warp's stores (contiguous over m_hi) coalesce
  int lp_mul;   // m_hi-major: the A map's last coordinate is lane * lp_mul + plane
  int ph, lh, bh;  // m_hi-major: tile extent in m_hi, m_lo and b
  int wide;     // 1: the buffers are 32-byte aligned (256-bit stores)
  int gm;       // tile order: gm row groups at a time, n fastest within them
                // (1: n fastest over a whole row group)
  int64_t mlo;  // m_hi-major: Mr / P
  int64_t watchdog_ns;
  double2 *dot_partials;   // sh.dot: [item][tiles_per_item * CG * EPI]
  int blocked;  // 1: CTA pair c takes the consecutive tiles [c per, (c + 1) per);
                // 0: tiles c, c + pairs, ...
  // divisors of the tile and store index arithmetic
  Div d_tpi, d_tn;             // tiles per item, column tiles
  Div d_hper, d_lper, d_ph, d_lh;  // m_hi-major tiles: P / ph, (Mr / P) / lh, ph, lh
  Div d_Mr, d_Mlo, d_dv, d_dh; // output rows per batch slice, Mr / P, dim(v'), dim(h')
};

// ---------------------------------------------------------------------------
// PTX wrappers
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void *p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ uint64_t globaltimer() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
               "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_test(uint64_t *bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

__device__ __forceinline__ uint32_t cluster_ctarank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n"
               "barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Set the int at the same shared-memory offset in CTA `rank` of the cluster.
__device__ __forceinline__ void st_cluster_flag(volatile int *local, uint32_t rank, int v) {
  uint32_t remote;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote)
               : "r"(smem_u32((const void *)local)), "r"(rank));
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(remote), "r"(v) : "memory");
}

struct Watch {
  volatile int *abort;
  DeviceStatus *st;
  uint64_t deadline;
  int where;
  int cs;  // cluster size: an expired wait raises the abort flag in every CTA
};

// Bounded wait on an mbarrier phase.  Returns false on abort or timeout.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, Watch &w) {
  uint32_t spins = 0;
  while (!mbar_test(bar, parity)) {
    if ((++spins & 63) == 8) {   // on the eighth failed try, then on every 64th
      if (*w.abort) return false;
      if (globaltimer() > w.deadline) {
        *w.abort = 1;
        if (w.cs > 1)
          for (int r = 0; r < w.cs; ++r) st_cluster_flag(w.abort, (uint32_t)r, 1);
        atomicExch(&w.st->timeout, 1);
        atomicExch(&w.st->error_info, w.where);
        return false;
      }
    }
  }
  return true;
}

// What the producer and the epilogue need of the launch's items, one item per
// lane: the tiles of a CTA pair run through the items in increasing order, so a
// warp loads the next 32 items' entries at once and takes an item's from its
// lane by a shuffle.  Loaded one
// by one, the chain item -> bitstring -> operand -> record costs three
// dependent misses per item, which bounds launches of a tile or two per item.
struct ItemBlock {
  int base;          // first item held (item base + lane)
  int tau, a_lane;   // operand variant (B map coordinate), A map lane
};

__device__ __forceinline__ void tma_load_4d(void *dst, const CUtensorMap *map, uint64_t *bar,
                                            int c0, int c1, int c2, int c3) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(smem_u32(dst)),
      "l"((uint64_t)map), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(smem_u32(bar))
      : "memory");
}
// Shared::cluster address of the same shared-memory offset in CTA `rank`.
__device__ __forceinline__ uint32_t cluster_addr(const void *local, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_u32(local)), "r"(rank));
  return r;
}
// Arrive on an mbarrier given by its shared::cluster address (any CTA).
// Relaxed: the epilogue's arrival only has to follow its own completed TMEM
// reads (tcgen05.wait::ld, in program order); its global stores are for the
// next launch, so a release (which waits for them) would stall the epilogue.
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t bar_cluster_addr) {
  asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(
                   bar_cluster_addr)
               : "memory");
}
// Arrive with release semantics on an mbarrier given by its shared::cluster
// address: the stores to the cluster's shared memory before it are visible to
// a thread that sees the phase complete.
__device__ __forceinline__ void mbar_arrive_cluster_release(uint32_t bar_cluster_addr) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(
                   bar_cluster_addr)
               : "memory");
}
// Count `bytes` of transactions as complete on a local mbarrier (bytes that
// will never arrive: the pair's other CTA issued no load for that stage).
__device__ __forceinline__ void mbar_complete_tx(uint64_t *bar, uint32_t bytes) {
  asm volatile("mbarrier.complete_tx.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}
// TMA loads of a CTA pair: the data lands in this CTA's shared memory and the
// completion is counted on the mbarrier at `bar_cluster_addr` (the even CTA's).
__device__ __forceinline__ void tma_load_4d_cg2(void *dst, const CUtensorMap *map,
                                                uint32_t bar_cluster_addr, int c0, int c1, int c2,
                                                int c3) {
  asm volatile(
      "cp.async.bulk.tensor.4d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(smem_u32(dst)),
      "l"((uint64_t)map), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(bar_cluster_addr)
      : "memory");
}
__device__ __forceinline__ void tma_load_5d(void *dst, const CUtensorMap *map, uint64_t *bar,
                                            int c0, int c1, int c2, int c3, int c4) {
  asm volatile(
      "cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4, %5, %6}], [%7];" ::"r"(smem_u32(dst)),
      "l"((uint64_t)map), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4), "r"(smem_u32(bar))
      : "memory");
}
__device__ __forceinline__ void tma_load_5d_cg2(void *dst, const CUtensorMap *map,
                                                uint32_t bar_cluster_addr, int c0, int c1, int c2,
                                                int c3, int c4) {
  asm volatile(
      "cp.async.bulk.tensor.5d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4, %5, %6}], [%7];" ::"r"(smem_u32(dst)),
      "l"((uint64_t)map), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4), "r"(bar_cluster_addr)
      : "memory");
}
__device__ __forceinline__ void tma_load_3d_cg2(void *dst, const CUtensorMap *map,
                                                uint32_t bar_cluster_addr, int c0, int c1,
                                                int c2) {
  asm volatile(
      "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(smem_u32(dst)),
      "l"((uint64_t)map), "r"(c0), "r"(c1), "r"(c2), "r"(bar_cluster_addr)
      : "memory");
}
__device__ __forceinline__ void tma_load_3d(void *dst, const CUtensorMap *map, uint64_t *bar,
                                            int c0, int c1, int c2) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(smem_u32(dst)),
      "l"((uint64_t)map), "r"(c0), "r"(c1), "r"(c2), "r"(smem_u32(bar))
      : "memory");
}

// Tile `rem` of an item -> (row group mg, column tile nt).  Blocks of gm row
// groups are walked column by column, so that the tiles in flight at once
// (one per CTA pair) share the k-slabs of gm A row panels and of a few B
// column panels in L2; gm = 1 is the plain n-fastest order.
__device__ __forceinline__ void tile_of(int rem, int mgroups, int tiles_n, int gm, int &mg,
                                        int &nt) {
  if (gm <= 1) {
    mg = rem / tiles_n;
    nt = rem - mg * tiles_n;
    return;
  }
  const int blk = rem / (gm * tiles_n), within = rem - blk * gm * tiles_n;
  const int g0 = blk * gm, gsz = mgroups - g0 < gm ? mgroups - g0 : gm;
  nt = within / gsz;
  mg = g0 + (within - nt * gsz);
}

// Shared-memory matrix descriptor of a K-major swizzled tile (rows of
// `rowb` bytes, 8-row core groups `8 * rowb` bytes apart).
__device__ __forceinline__ uint64_t sdesc(uint32_t saddr, uint32_t rowb) {
  const uint64_t layout = rowb == 128 ? 2ull : 4ull;  // SWIZZLE_128B : SWIZZLE_64B
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)1 << 16;                               // leading offset (unused, K-major swizzled)
  d |= (uint64_t)(((8u * rowb) >> 4) & 0x3FFFu) << 32;  // stride offset between 8-row groups
  d |= (uint64_t)1 << 46;                               // descriptor version
  d |= layout << 61;
  return d;
}

template <int KIND, int CG>
__device__ __forceinline__ void mma(uint32_t dtmem, uint64_t a, uint64_t b, uint32_t idesc,
                                    uint32_t acc) {
  if (CG == 2) {
    if (KIND == 0)
      asm volatile(
          "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
          " tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(dtmem),
          "l"(a), "l"(b), "r"(idesc), "r"(acc));
    else
      asm volatile(
          "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
          " tcgen05.mma.cta_group::2.kind::tf32 [%0], %1, %2, %3, p;\n}\n" ::"r"(dtmem),
          "l"(a), "l"(b), "r"(idesc), "r"(acc));
    return;
  }
  if (KIND == 0) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(dtmem),
        "l"(a), "l"(b), "r"(idesc), "r"(acc));
  } else {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n}\n" ::"r"(dtmem),
        "l"(a), "l"(b), "r"(idesc), "r"(acc));
  }
}
__device__ __forceinline__ void mma_commit(uint64_t *bar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
          smem_u32(bar))
      : "memory");
}
// Commit of the pair's MMAs: arrives on the mbarrier at this offset in both CTAs.
__device__ __forceinline__ void mma_commit_cg2(uint64_t *bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64"
      " [%0], %1;" ::"r"(smem_u32(bar)),
      "h"((uint16_t)3)
      : "memory");
}
__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
// Issue a 32-lane x 16-column TMEM load (asynchronous: the registers are
// valid after tmem_wait()).
__device__ __forceinline__ void tmem_ld16_issue(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,"
      "%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
        "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}
// Wait for the outstanding TMEM loads; the registers of the last load are
// in/out operands so that no use of them can be scheduled before the wait.
__device__ __forceinline__ void tmem_wait(uint32_t (&r)[16]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]),
                 "+r"(r[6]), "+r"(r[7]), "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]),
                 "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])
               :
               : "memory");
}

// The same for two loads in flight.
__device__ __forceinline__ void tmem_wait2(uint32_t (&r)[16], uint32_t (&q)[16]) {
  tmem_wait(r);
  asm volatile("" : "+r"(q[0]), "+r"(q[1]), "+r"(q[2]), "+r"(q[3]), "+r"(q[4]), "+r"(q[5]),
               "+r"(q[6]), "+r"(q[7]), "+r"(q[8]), "+r"(q[9]), "+r"(q[10]), "+r"(q[11]),
               "+r"(q[12]), "+r"(q[13]), "+r"(q[14]), "+r"(q[15])
               :
               : "memory");
}

// ---------------------------------------------------------------------------
// Kernel
// ---------------------------------------------------------------------------
// CG: CTAs per MMA.  CG = 1: one CTA per 128-row tile.  CG = 2: a cluster of
// two CTAs per 256-row tile (2-SM UMMA), see the file comment.
template <int FMT, int ROWB, int CG, int EPI, int DR>
__global__ void __launch_bounds__(threads_of(EPI, DR), 1)
    k_contract_tc(const __grid_constant__ TcParams p) {
  using T = FormTraits<FMT>;
  constexpr int NP = T::NP;
  constexpr int KSTEPS = ROWB / 32;  // 32-byte MMA k-steps per stage
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char *smem =
      (unsigned char *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);

  const int BN = p.BN;              // real output columns per tile (MMA N)
  const int BNL = BN / CG;          // Bt rows held by this CTA
  const int S = p.stages;
  const uint32_t a_bytes = BM * ROWB;
  const uint32_t b_bytes = (uint32_t)BNL * ROWB;
  const uint32_t stage_bytes = NP * (a_bytes + b_bytes);  // this CTA's share
  uint64_t *bars = (uint64_t *)(smem + (size_t)S * stage_bytes);
  uint64_t *full = bars;
  uint64_t *empty = bars + S;
  uint64_t *tfull = bars + 2 * S;
  uint64_t *tempty = bars + 2 * S + 2;
  uint64_t *done = bars + 2 * S + 4;
  uint64_t *pdone = bars + 2 * S + 5;  // CG = 2: the odd producer has finished issuing
  uint32_t *tmem_slot = (uint32_t *)(bars + 2 * S + 6);
  volatile int *abort_flag = (volatile int *)(tmem_slot + 1);
  volatile uint32_t *odd_issued = tmem_slot + 2;  // CG = 2: stages the odd CTA issued

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = CG > 1 ? cluster_ctarank() : 0u;
  const bool leader = rank == 0;
  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(&tfull[a], 1);
      // the pair's epilogue warps (one elected lane each) release an accumulator
      mbar_init(&tempty[a], CG == 2 ? 2 * EPI : 32 * EPI);
    }
    mbar_init(done, 1);
    mbar_init(pdone, 1);
    *abort_flag = 0;
    *odd_issued = 0u;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    if (CG == 2) {
      asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                       smem_u32(tmem_slot)),
                   "r"(p.tmem_cols));
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;");
    } else {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                       smem_u32(tmem_slot)),
                   "r"(p.tmem_cols));
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
  }
  tc_fence_before();
  __syncthreads();
  if (CG > 1) cluster_sync();  // both CTAs' barriers exist before any remote signal
  tc_fence_after();
  pdl_trigger();
  const uint32_t tmem_base = *tmem_slot;

  const int cid = blockIdx.x / CG, ncl = gridDim.x / CG;
  const int mgroups = p.tiles_m / CG;               // CG == 2 only when tiles_m is even
  const int tiles_per_item = mgroups * p.tiles_n;  // tiles of the pair
  const int total = p.n_items * tiles_per_item;
  // this pair's tiles: a consecutive range (blocked) or every ncl-th
  const int per = p.blocked ? (total + ncl - 1) / ncl : 1;
  const int t_first = p.blocked ? cid * per : cid;
  const int t_end = p.blocked ? (t_first + per < total ? t_first + per : total) : total;
  const int t_step = p.blocked ? 1 : ncl;
  // a row of A holds 2K real entries of ESZ bytes; one stage covers ROWB bytes
  const int kb_count = (2 * p.sh.K * T::ESZ) / ROWB;
  Watch w{abort_flag, p.st, globaltimer() + (uint64_t)p.watchdog_ns, p.sh.q, CG};
  // the launch before has completed; the waits' budget counts from here
  auto start_watch = [&]() {
    pdl_wait();
    w.deadline = globaltimer() + (uint64_t)p.watchdog_ns;
  };
  // the even CTA's barriers, as cluster addresses
  const uint32_t full0 = CG == 2 ? cluster_addr(full, 0) : 0u;
  const uint32_t tempty0 = CG == 2 ? cluster_addr(tempty, 0) : 0u;

  if (warp < first_epi(DR)) {
  // DR: the warpgroups' register shares, 72 x 128 + 216 x 256 = 168 x 384
  if constexpr (DR != 0) asm volatile("setmaxnreg.dec.sync.aligned.u32 72;");
  if (warp == 0) {
    // ---------------- TMA producer (both CTAs) ----------------
    uint32_t it = 0;
    {
      ItemBlock ib{INT32_MIN, 0, 0};
      bool ok = true, first = true;
      for (int t = t_first; t < t_end; t += t_step) {
        const int item = (int)p.d_tpi.q(t);
        const int rem = t - item * tiles_per_item;
        int mg, nt;
        if (p.gm <= 1) {
          mg = (int)p.d_tn.q(rem);
          nt = rem - mg * p.tiles_n;
        } else {
          tile_of(rem, mgroups, p.tiles_n, p.gm, mg, nt);
        }
        const int mt = mg * CG + (int)rank;
        if (item >= ib.base + 32 || ib.base < 0) {
          ib.base = item;
          const int i = item + lane < p.n_items ? item + lane : item;
          const StepItem &si = p.items[i];
          ib.tau = block_variant(*si.bits, p.sh) + si.b_slot;
          ib.a_lane = si.a_lane;
          if (first) start_watch();
          first = false;
        }
        const int tau = __shfl_sync(0xffffffffu, ib.tau, item - ib.base);
        const int a_lane = __shfl_sync(0xffffffffu, ib.a_lane, item - ib.base);
        // m_hi-major: tile mt is rows m_hi = hb0 .. hb0+ph-1, m_lo = mlo_t ..
        // mlo_t+lh-1, b = b_t .. b_t+bh-1
        int b_t = 0, mlo_t = 0, hb0 = 0;
        if (p.mhi) {
          const uint32_t rest = p.d_hper.q(mt);
          hb0 = (int)(mt - rest * p.d_hper.d) * p.ph;
          b_t = (int)p.d_lper.q(rest);
          mlo_t = (int)(rest - b_t * p.d_lper.d) * p.lh;
          b_t *= p.bh;
        }
        if (lane == 0) {
          for (int kb = 0; kb < kb_count; ++kb, ++it) {
            const int s = it % S;
            const uint32_t ph = (it / S) & 1u;
            if (!mbar_wait(&empty[s], ph ^ 1u, w)) { ok = false; break; }
            unsigned char *st = smem + (size_t)s * stage_bytes;
            const int k0 = kb * (ROWB / T::ESZ);
            if (CG == 1) {
              mbar_expect_tx(&full[s], stage_bytes);
              for (int pl = 0; pl < NP; ++pl) {
                if (p.mhi)
                  tma_load_5d(st + pl * a_bytes, &p.mapA, &full[s], k0, hb0, mlo_t, b_t,
                              a_lane * p.lp_mul + pl);
                else
                  tma_load_4d(st + pl * a_bytes, &p.mapA, &full[s], k0, mt * BM, pl, a_lane);
                tma_load_3d(st + NP * a_bytes + pl * b_bytes, &p.mapB[pl], &full[s], k0,
                            nt * BN, tau);
              }
            } else {
              // the even CTA's full barrier counts both CTAs' bytes
              if (leader) mbar_expect_tx(&full[s], 2 * stage_bytes);
              for (int pl = 0; pl < NP; ++pl) {
                if (p.mhi)
                  tma_load_5d_cg2(st + pl * a_bytes, &p.mapA, full0 + (uint32_t)s * 8u, k0, hb0,
                                  mlo_t, b_t, a_lane * p.lp_mul + pl);
                else
                  tma_load_4d_cg2(st + pl * a_bytes, &p.mapA, full0 + (uint32_t)s * 8u, k0,
                                  mt * BM, pl, a_lane);
                tma_load_3d_cg2(st + NP * a_bytes + pl * b_bytes, &p.mapB[pl],
                                full0 + (uint32_t)s * 8u, k0, nt * BN + (int)rank * BNL, tau);
              }
            }
          }
        }
        ok = __shfl_sync(0xffffffffu, (int)ok, 0) != 0;
        if (!ok) break;
      }
    }
    if (lane == 0) {
      // Every issued stage must have landed before the pair may exit.  The
      // full barriers live in the even CTA and count the loads of both CTAs;
      // after an abort the two producers may have stopped at different
      // stages (at most S apart: a stage is issued only after the MMAs of
      // the stage S before it, which needed both CTAs' loads).  So the odd
      // producer reports how many stages it issued, and the even one settles
      // the difference: for a stage only the odd CTA issued it arrives with
      // the odd share's bytes, for a stage only it issued it counts the
      // missing odd share as complete; then it waits (bounded) on the full
      // barriers of the last S stages.  The odd CTA leaves only after the
      // teardown's cluster barrier, which the even CTA reaches after this.
      if (CG == 2 && !leader) {
        uint32_t slot;
        asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(slot)
                     : "r"(smem_u32((const void *)odd_issued)));
        asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(slot), "r"(it) : "memory");
        mbar_arrive_cluster_release(cluster_addr(pdone, 0));
      }
      if (leader) {
        Watch w2{abort_flag, p.st, globaltimer() + 100000000ull, p.sh.q, 1};
        volatile int zero = 0;
        w2.abort = &zero;
        uint32_t end = it;
        if (CG == 2 && mbar_wait(pdone, 0u, w2)) {
          asm volatile("fence.acq_rel.cluster;" ::: "memory");
          const uint32_t io = *odd_issued;
          const uint32_t half = stage_bytes;   // one CTA's share of a stage
          for (uint32_t j = it; j < io; ++j) mbar_expect_tx(&full[j % S], half);
          for (uint32_t j = io; j < it; ++j) mbar_complete_tx(&full[j % S], half);
          if (io > end) end = io;
        }
        for (uint32_t j = end > (uint32_t)S ? end - S : 0u; j < end; ++j)
          if (!mbar_wait(&full[j % S], (j / S) & 1u, w2)) break;
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer (the even CTA) ----------------
    if (lane == 0 && leader) {
      const uint32_t idesc = (1u << 4) | ((uint32_t)T::AB << 7) | ((uint32_t)T::AB << 10) |
                             ((uint32_t)(BN >> 3) << 17) | ((uint32_t)((BM * CG) >> 4) << 24);
      uint32_t it = 0, local = 0;
      start_watch();
      const int KSP = p.ksplit, NB = p.nbuf;
      for (int t = t_first; t < t_end; t += t_step, ++local) {
        const int acc = NB == 2 ? (int)(local & 1) : 0;
        const uint32_t aph = NB == 2 ? (local >> 1) & 1u : local & 1u;
        if (!mbar_wait(&tempty[acc], aph ^ 1u, w)) break;
        tc_fence_after();
        const uint32_t dbuf = tmem_base + (uint32_t)(acc * BN * p.nacc);
        const uint32_t dcorr = dbuf + (uint32_t)(KSP * BN);   // used when csep
        bool ok = true;
        int seg_prev = -1;
        for (int kb = 0; kb < kb_count; ++kb, ++it) {
          const int s = it % S;
          const uint32_t ph = (it / S) & 1u;
          if (!mbar_wait(&full[s], ph, w)) { ok = false; break; }
          tc_fence_after();
          const uint32_t sa = smem_u32(smem + (size_t)s * stage_bytes);
          const uint32_t sb = sa + NP * a_bytes;
          // K segment of this stage (each segment has its own accumulator)
          const int seg = (kb * KSP) / kb_count;
          const bool seg_start = seg != seg_prev;
          seg_prev = seg;
          const uint32_t dt = dbuf + (uint32_t)(seg * BN);
          const bool cs = NP == 2 && p.csep != 0;
          const uint32_t dc = cs ? dcorr : dt;
#pragma unroll
          for (int j = 0; j < KSTEPS; ++j) {
            const uint32_t first = (seg_start && j == 0) ? 0u : 1u;
            const uint64_t a0 = sdesc(sa + 32 * j, ROWB);
            const uint64_t b0 = sdesc(sb + 32 * j, ROWB);
            mma<T::KIND, CG>(dt, a0, b0, idesc, first);
            if (NP == 2) {
              const uint64_t a1 = sdesc(sa + a_bytes + 32 * j, ROWB);
              const uint64_t b1 = sdesc(sb + b_bytes + 32 * j, ROWB);
              const uint32_t cfirst = cs ? ((kb == 0 && j == 0) ? 0u : 1u) : 1u;
              mma<T::KIND, CG>(dc, a0, b1, idesc, cfirst);
              mma<T::KIND, CG>(dc, a1, b0, idesc, 1u);
            }
          }
          if (CG == 1) mma_commit(&empty[s]);
          else mma_commit_cg2(&empty[s]);  // frees the stage in both CTAs
        }
        if (!ok) break;
        if (CG == 1) mma_commit(&tfull[acc]);
        else mma_commit_cg2(&tfull[acc]);   // both CTAs' epilogues may drain
      }
      // all issued MMAs retire before TMEM is released
      if (CG == 1) mma_commit(done);
      else mma_commit_cg2(done);
      Watch w2{abort_flag, p.st, globaltimer() + 100000000ull, p.sh.q, 1};
      volatile int zero = 0;
      w2.abort = &zero;
      mbar_wait(done, 0u, w2);
    }
  }
  } else {
    // ---------------- epilogue (both CTAs) ----------------
    if constexpr (DR != 0) asm volatile("setmaxnreg.inc.sync.aligned.u32 216;");
    // Warp w drains TMEM lanes 32*(w%4) .. +31 (the rows it may access), all
    // columns of the tile, 16 at a time; the load of chunk c+1 is in flight
    // while chunk c is scaled, split and stored.
    const int quad = warp & 3;
    const int row = 32 * quad + lane;
    // EPI = 8: warps ew and ew + 4 share a quadrant and split its columns in
    // whole 16-column chunks (a 16-column tile stays with the first)
    const int ew = warp - first_epi(DR);
    const int c_mid = EPI == 8 ? (p.BN / 16 + 1) / 2 * 16 : p.BN;
    const int c_begin = ew < 4 ? 0 : c_mid;
    const int c_end = ew < 4 ? c_mid : p.BN;
    const bool idle = c_begin >= c_end;
    const int dv = p.sh.dv_out, dh = p.sh.dh_out;
    const uint32_t M = (uint32_t)p.sh.M;
    const int64_t P = p.sh.P;
    const int64_t Mr = p.sh.Mr > 0 ? p.sh.Mr : p.sh.M;
    const int64_t MrN = Mr * (int64_t)p.sh.N, Mrdh = Mr * (int64_t)dh;
    const bool vbm = p.sh.vb != 0;
    const bool dotm = p.sh.dot != 0;
    // Destination of complex column nc of a row:
    //   base + q(nc) * stride_q + r(nc) * stride_r  (q, r: nc / R, nc % R)
    //   vb = 0:          n = h' dv' + v', entry b Mr N + ((m_lo dh' + h') P + m_hi) dv' + v'
    //   vb = 1, nvs = 0: n = h' dv' + v', entry (b dv' + v') Mr dh' + (m_lo dh' + h') P + m_hi
    //   vb = 1, nvs = 1: n = v' dh' + h', the same entry
    // (R = 1: N = dh', the h' stride is stride_r over the whole N).  Runs of
    // consecutive nc with stride_r = 1 are contiguous: they are stored W
    // entries at a time (W = 8, 4, 2 dividing R), else one by one.
    const Div dR = vbm && p.sh.nvs != 0 ? p.d_dh : p.d_dv;
    const bool flat = dR.d == 1;
    const uint32_t R = flat ? (uint32_t)p.sh.N : dR.d;
    const int64_t stride_h = !vbm ? P * dv : P;
    const int64_t stride_q = flat ? 0 : (vbm && p.sh.nvs != 0 ? Mrdh : stride_h);
    const int64_t stride_r =
        flat ? (vbm && p.sh.nvs != 0 ? Mrdh : stride_h) : (!vbm ? 1 : (p.sh.nvs != 0 ? P : Mrdh));
    const int W = stride_r != 1 ? 1 : (R % 8 == 0 ? 8 : (R % 4 == 0 ? 4 : (R % 2 == 0 ? 2 : 1)));
    const int64_t wrap = stride_q - (int64_t)R * stride_r;   // added where nc crosses into a new q
    // m_hi-major tiles: this row's place in the tile, row = (bb lh + l) ph + h
    const uint32_t row_rl = p.d_ph.q(row);
    const uint32_t row_h = row - row_rl * p.d_ph.d, row_b = p.d_lh.q(row_rl),
                   row_l = row_rl - row_b * p.d_lh.d;
    uint32_t local = 0;
    // the warp's next 32 items, one per lane
    int ib_base = INT32_MIN, i_x = 0, i_exp = 0, i_rec = 0;
    unsigned long long i_D = 0;
    int cached_item = -1, out_rec = 0, out_exp = 0;
    void *D = nullptr;
    float sc = 1.f, vmax = 0.f;
    bool first = true;
    // the item's max |entry|, once per item and warp (non-negative floats
    // compare as their bits)
    auto flush_max = [&]() {
      const uint32_t mx = __reduce_max_sync(0xffffffffu, __float_as_uint(vmax));
      if (lane == 0) atomicMax(&p.recs[out_rec].maxbits, mx);
      vmax = 0.f;
    };
    for (int t = t_first; t < t_end; t += t_step, ++local) {
      const int item = (int)p.d_tpi.q(t);
      const int rem = t - item * tiles_per_item;
      int mg, nt;
      if (p.gm <= 1) {
        mg = (int)p.d_tn.q(rem);
        nt = rem - mg * p.tiles_n;
      } else {
        tile_of(rem, mgroups, p.tiles_n, p.gm, mg, nt);
      }
      const int mt = mg * CG + (int)rank;
      if (item != cached_item) {
        if (!dotm && cached_item >= 0) flush_max();
        cached_item = item;
        if (item >= ib_base + 32 || ib_base < 0) {
          ib_base = item;
          const int i = item + lane < p.n_items ? item + lane : item;
          const StepItem si = p.items[i];
          const OpDesc &op = p.ops[si.op_base + block_variant(*si.bits, p.sh)];
          if (first) start_watch();
          first = false;
          const bool unit_in = si.in_rec < 0;
          const float mu = unit_in ? 1.f : __uint_as_float(p.recs[si.in_rec].maxbits);
          const int s_in = unit_in ? 0 : p.recs[si.in_rec].exp;
          // a fused dot keeps the accumulator unscaled (nothing is stored)
          i_x = dotm ? 0 : step_scale_exp(mu, __uint_as_float(op.beta_t_bits), p.sh.target);
          i_exp = s_in + op.b_t + i_x + op.e_c;
          i_rec = si.out_rec;
          i_D = (unsigned long long)si.D;
        }
        const int src = item - ib_base;
        sc = pow2f(__shfl_sync(0xffffffffu, i_x, src));
        out_exp = __shfl_sync(0xffffffffu, i_exp, src);
        out_rec = __shfl_sync(0xffffffffu, i_rec, src);
        D = (void *)__shfl_sync(0xffffffffu, i_D, src);
      }
      const int acc = p.nbuf == 2 ? (int)(local & 1) : 0;
      const uint32_t aph = p.nbuf == 2 ? (local >> 1) & 1u : local & 1u;
      int ok = 1;
      if (lane == 0) ok = mbar_wait(&tfull[acc], aph, w) ? 1 : 0;
      ok = __shfl_sync(0xffffffffu, ok, 0);
      if (!ok) break;
      tc_fence_after();
      uint32_t b, m_hi, m_lo;
      bool live = true;
      if (p.mhi) {
        const uint32_t rest = p.d_hper.q(mt);
        m_hi = (mt - rest * p.d_hper.d) * (uint32_t)p.ph + row_h;
        b = p.d_lper.q(rest);
        m_lo = (rest - b * p.d_lper.d) * (uint32_t)p.lh + row_l;
        b = b * (uint32_t)p.bh + row_b;
      } else {
        const uint32_t m = (uint32_t)mt * BM + row;
        live = m < M;
        // row m = b * Mr + m_r (b: the batch of open legs, when there is one)
        b = p.d_Mr.q(m);
        const uint32_t mr = m - b * p.d_Mr.d;
        m_hi = p.d_Mlo.q(mr);
        m_lo = mr - m_hi * p.d_Mlo.d;
      }
      const int KSP = p.nacc;   // K segments, then the correction accumulator
      const uint32_t tbase =
          tmem_base + ((uint32_t)(32 * quad) << 16) + (uint32_t)(acc * BN * KSP);
      float dre = 0.f, dim = 0.f;   // fused dot: this row's partial sum
      // TMEM read: the accumulator goes back to the MMA issuer
      auto release = [&]() {
        tc_fence_before();
        if (CG == 1) {
          mbar_arrive(&tempty[acc]);
        } else {
          __syncwarp();
          if (lane == 0) mbar_arrive_cluster(tempty0 + (uint32_t)acc * 8u);
        }
      };
      // The columns in chunks of 16 (8 complex entries), the next chunk loaded
      // from TMEM while the current one is used.
      uint32_t ra[16], rb[16];
      if constexpr (DR != 0) {
        // this warp's 128 columns (BN = 256) into registers
        uint32_t v[8][16];
#pragma unroll
        for (int j = 0; j < 8; ++j) tmem_ld16_issue(tbase + (uint32_t)(c_begin + 16 * j), v[j]);
#pragma unroll
        for (int j = 0; j < 8; ++j) tmem_wait(v[j]);
        for (int sg = 1; sg < KSP; ++sg) {
          const uint32_t cb = tbase + (uint32_t)(sg * BN + c_begin);
          tmem_ld16_issue(cb, ra);
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            uint32_t (&cur)[16] = j & 1 ? rb : ra, (&next)[16] = j & 1 ? ra : rb;
            tmem_wait(cur);
            if (j < 7) tmem_ld16_issue(cb + (uint32_t)(16 * (j + 1)), next);
#pragma unroll
            for (int i = 0; i < 16; ++i)
              v[j][i] = __float_as_uint(__uint_as_float(v[j][i]) + __uint_as_float(cur[i]));
          }
        }
        release();
        if (dotm) {
          const int64_t dot_e = (int64_t)m_lo * p.sh.N + ((nt * BN + c_begin) >> 1);
          if (live) {
            Raw8 fcur, fnext;
            load8_raw<FMT>(D, dot_e, p.sh.plane, fcur);
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              if (j < 7) load8_raw<FMT>(D, dot_e + 8 * (j + 1), p.sh.plane, fnext);
              float2 f[8];
              unpack8<FMT>(fcur, f);
#pragma unroll
              for (int q = 0; q < 8; ++q) {
                const float vr = __uint_as_float(v[j][2 * q]), vi = __uint_as_float(v[j][2 * q + 1]);
                dre = fmaf(vr, f[q].x, fmaf(-vi, f[q].y, dre));
                dim = fmaf(vr, f[q].y, fmaf(vi, f[q].x, dim));
              }
              fcur = fnext;
            }
          }
        } else {
          // runs of 8 entries (the rule that takes this form)
          const int64_t base = !vbm ? (int64_t)b * MrN + ((int64_t)m_lo * dh * P + m_hi) * dv
                                    : (int64_t)b * dv * Mrdh + (int64_t)m_lo * dh * P + m_hi;
          const uint32_t nc0 = (uint32_t)(nt * BN + c_begin) >> 1;
          const uint32_t cq = flat ? 0u : dR.q(nc0);
          uint32_t cr = flat ? nc0 : nc0 - cq * R;
          int64_t dest = base + (int64_t)cq * stride_q + (int64_t)cr;
          if (live) {
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              float o[16];
#pragma unroll
              for (int i = 0; i < 16; ++i) o[i] = __uint_as_float(v[j][i]);
              Packed8<FMT> w;
              vmax = fmaxf(vmax, pack8<FMT>(o, sc, w));
              store_run8_wide<FMT>(D, dest, p.sh.plane, w);
              cr += 8;
              dest += 8;
              if (cr == R) {
                cr = 0;
                dest += wrap;
              }
            }
          }
        }
      } else {
      if (!idle) tmem_ld16_issue(tbase + (uint32_t)c_begin, ra);
      if (dotm) {
        // fused dot: the partner entries of row m (P = 1, row-major m N + n),
        // loaded one chunk ahead of their use
        const int64_t dot_e = (int64_t)m_lo * p.sh.N + ((nt * BN + c_begin) >> 1);
        Raw8 fcur, fnext;
        if (live && !idle) load8_raw<FMT>(D, dot_e, p.sh.plane, fcur);
        tmem_wait(ra);
        for (int c = c_begin; c < c_end; c += 16) {
          const bool more = c + 16 < c_end;
          float v[16];
#pragma unroll
          for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(ra[i]);
          if (more) tmem_ld16_issue(tbase + (uint32_t)(c + 16), ra);
          if (live && more) load8_raw<FMT>(D, dot_e + ((c + 16 - c_begin) >> 1), p.sh.plane, fnext);
          for (int sg = 1; sg < KSP; ++sg) {
            uint32_t rc[16];
            tmem_ld16_issue(tbase + (uint32_t)(sg * BN + c), rc);
            tmem_wait(rc);
#pragma unroll
            for (int i = 0; i < 16; ++i) v[i] += __uint_as_float(rc[i]);
          }
          if (live) {
            float2 f[8];
            unpack8<FMT>(fcur, f);
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              dre = fmaf(v[2 * j], f[j].x, fmaf(-v[2 * j + 1], f[j].y, dre));
              dim = fmaf(v[2 * j], f[j].y, fmaf(v[2 * j + 1], f[j].x, dim));
            }
            fcur = fnext;
          }
          if (more) tmem_wait(ra);
        }
      } else {
        const int64_t base = !vbm ? (int64_t)b * MrN + ((int64_t)m_lo * dh * P + m_hi) * dv
                                  : (int64_t)b * dv * Mrdh + (int64_t)m_lo * dh * P + m_hi;
        // the current column's place: dest = its entry, cr = r(nc)
        const uint32_t nc0 = (uint32_t)(nt * BN + c_begin) >> 1;
        const uint32_t cq = flat ? 0u : dR.q(nc0);
        uint32_t cr = flat ? nc0 : nc0 - cq * R;
        int64_t dest = base + (int64_t)cq * stride_q + (int64_t)cr * stride_r;
        // the next w columns (w divides R, or is 1)
        auto advance = [&](int w) {
          cr += w;
          dest += w * stride_r;
          if (cr == R) {
            cr = 0;
            dest += wrap;
          }
        };
        // the next 8 entries in runs of W
        auto store_any = [&](const Packed8<FMT> &w) {
          switch (W) {
            case 8:
              store_run<FMT, 8>(D, dest, p.sh.plane, w, 0);
              advance(8);
              break;
            case 4:
#pragma unroll
              for (int j = 0; j < 8; j += 4) {
                store_run<FMT, 4>(D, dest, p.sh.plane, w, j);
                advance(4);
              }
              break;
            case 2:
#pragma unroll
              for (int j = 0; j < 8; j += 2) {
                store_run<FMT, 2>(D, dest, p.sh.plane, w, j);
                advance(2);
              }
              break;
            default:
#pragma unroll
              for (int j = 0; j < 8; ++j) {
                store_run<FMT, 1>(D, dest, p.sh.plane, w, j);
                advance(1);
              }
          }
        };
        // 16 accumulator columns (8 complex entries) at a time: the other
        // accumulators added with FP32 round-to-nearest, scaled, rounded to the
        // storage format and stored, while the next chunk (of the first two
        // accumulators) is loaded.  One loop for the usual runs of 8, with no
        // choice between a chunk's load and its store, and one for the rest.
        auto chunks = [&](auto store) {
          const bool pair = KSP > 1;
          const uint32_t t2 = tbase + (uint32_t)BN;
          if (pair && !idle) tmem_ld16_issue(t2 + (uint32_t)c_begin, rb);
          tmem_wait2(ra, rb);
          for (int c = c_begin; c < c_end; c += 16) {
            const bool more = c + 16 < c_end;
            float o[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) o[i] = __uint_as_float(ra[i]);
            if (pair) {
#pragma unroll
              for (int i = 0; i < 16; ++i) o[i] += __uint_as_float(rb[i]);
            }
            if (more) {
              tmem_ld16_issue(tbase + (uint32_t)(c + 16), ra);
              if (pair) tmem_ld16_issue(t2 + (uint32_t)(c + 16), rb);
            }
            for (int sg = 2; sg < KSP; ++sg) {
              uint32_t rc[16];
              tmem_ld16_issue(tbase + (uint32_t)(sg * BN + c), rc);
              tmem_wait(rc);
#pragma unroll
              for (int i = 0; i < 16; ++i) o[i] += __uint_as_float(rc[i]);
            }
            if (live) {
              Packed8<FMT> w;
              vmax = fmaxf(vmax, pack8<FMT>(o, sc, w));
              store(w);
            }
            if (more) tmem_wait2(ra, rb);
          }
        };
        auto store8 = [&](const Packed8<FMT> &w) {
          store_run8_wide<FMT>(D, dest, p.sh.plane, w);
          advance(8);
        };
        if (W == 8 && p.wide) {
          if (NP == 1 && KSP == 1) {
            // single-plane forms: less arithmetic per chunk, so the chunk is
            // used where it was loaded, the two buffers in turn (16 lanes of
            // 32768 x 64 x 64 in BF16: 52.6 -> 47.7 us)
            auto emit = [&](const uint32_t (&r)[16]) {
              if (!live) return;
              float o[16];
#pragma unroll
              for (int i = 0; i < 16; ++i) o[i] = __uint_as_float(r[i]);
              Packed8<FMT> w;
              vmax = fmaxf(vmax, pack8<FMT>(o, sc, w));
              store8(w);
            };
            tmem_wait(ra);
            for (int c = c_begin; c < c_end; c += 32) {
              const bool two = c + 16 < c_end, more = c + 32 < c_end;
              if (two) tmem_ld16_issue(tbase + (uint32_t)(c + 16), rb);
              emit(ra);
              if (two) {
                tmem_wait(rb);
                if (more) tmem_ld16_issue(tbase + (uint32_t)(c + 32), ra);
                emit(rb);
                if (more) tmem_wait(ra);
              }
            }
          } else {
            chunks(store8);
          }
        } else {
          chunks(store_any);
        }
      }
      release();
      }
      if (dotm) {
        // the warp's 32 rows summed in FP64, one slot per (tile, CTA, warp)
        double r = (double)dre, i = (double)dim;
        for (int o = 16; o > 0; o >>= 1) {
          r += __shfl_xor_sync(0xffffffffu, r, o);
          i += __shfl_xor_sync(0xffffffffu, i, o);
        }
        if (lane == 0)
          p.dot_partials[((int64_t)item * tiles_per_item + rem) * (CG * EPI) + (int)rank * EPI +
                         ew] = make_double2(r, i);
      }
      if (mt == 0 && nt == 0 && ew == 0 && lane == 0) p.recs[out_rec].exp = out_exp;
    }
    if (!dotm && cached_item >= 0) flush_max();
  }

  // teardown: everyone done issuing; the last MMAs have retired (done
  // barrier) and the last loads have landed (full barriers) before the pair
  // releases TMEM and leaves.
  tc_fence_before();
  __syncthreads();
  if (CG > 1) cluster_sync();
  if (warp == 1) {
    tc_fence_after();
    if (CG == 2)
      asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base),
                   "r"(p.tmem_cols));
    else
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base),
                   "r"(p.tmem_cols));
  }
}

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *,
                                  const cuuint64_t *, const cuuint64_t *, const cuuint32_t *,
                                  const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void *f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &f, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = (EncodeTiledFn)f;
  });
  return fn;
}

int esz_of(int fmt) { return fmt == FMT_TF32 ? 4 : 2; }
int np_of(int fmt) { return (fmt == FMT_BF16X2 || fmt == FMT_FP16X2) ? 2 : 1; }

// Bytes of K per pipeline stage (the swizzle width): 128 where the row
// length allows and nothing else is asked, else 64.
int rowb_for(int Kr, int esz, int want = 0) {
  const int bytes = Kr * esz;
  if (want != 64 && bytes % 128 == 0) return 128;
  if (bytes % 64 == 0) return 64;
  return 0;
}

}  // namespace

int tc_Kr_pad(int K) { return 2 * K; }

bool tc_tuning_valid(int kchunk, int cluster, int epi) {
  return (kchunk == 0 || kchunk == 64 || kchunk == 128) && (cluster >= 0 && cluster <= 2) &&
         (epi == 0 || epi == 4 || epi == 8);
}
int tc_Nr_pad(int N) { return 2 * N; }

bool tc_supports(const StepShape &sh, int fmt) {
  if (!(fmt == FMT_BF16 || fmt == FMT_FP16 || fmt == FMT_BF16X2 || fmt == FMT_FP16X2 ||
        fmt == FMT_TF32))
    return false;
  const int Kr = 2 * sh.K, Nr = 2 * sh.N;
  if (rowb_for(Kr, esz_of(fmt)) == 0) return false;
  // fewer rows than a tile: the A box reaches past the tensor's M extent,
  // where TMA fills zeros, and the epilogue stores live rows only
  if (sh.M < 32) return false;
  if (!(Nr % 256 == 0 || (Nr % 16 == 0 && Nr <= 256))) return false;
  if (sh.M > 0x7fffffffLL) return false;
  return true;
}

// Accumulators and column width of a step's tiles, before what the launch
// (its items, its buffers' alignment) makes of them.
struct TileCols {
  int ksplit, csep;   // K segments, a correction accumulator (0 or 1)
  int BN;
};
static TileCols tile_cols(const StepShape &sh, int np, int kb_count) {
  const int Nr = 2 * sh.N;
  // K segments (long-K steps): at most one per k-chunk
  int KS = sh.ksplit > 1 ? sh.ksplit : 1;
  if (KS > kb_count) KS = kb_count;
  const int CS = (sh.csep && np == 2) ? 1 : 0;
  const int NA = KS + CS;
  // BN: the widest tile that divides Nr in whole 16-column chunks and whose NA
  // accumulators fit TMEM (twice where K is short, at most 16 k-chunks, which
  // needs the epilogue overlap of two buffers)
  const int cols_max = 512 / (kb_count <= 16 ? 2 * NA : NA);
  int BN = Nr < 256 ? Nr : 256;
  if (BN > cols_max) BN = cols_max / 16 * 16;
  while (BN > 16 && Nr % BN != 0) BN -= 16;
  return {KS, CS, BN};
}

// A fused dot keeps the width of tile_cols and takes eight epilogue warps unless
// four are asked for; every warp of every tile writes a slot, with columns of
// its own or not.
int64_t tc_dot_slots(const StepShape &sh, int fmt, int kchunk, int epi) {
  const int esz = esz_of(fmt), Kr = 2 * sh.K, rowb = rowb_for(Kr, esz, kchunk);
  if (!rowb) return 0;
  const int BN = tile_cols(sh, np_of(fmt), Kr * esz / rowb).BN;
  return ((sh.M + BM - 1) / BM) * (2 * sh.N / BN) * (epi == 4 ? 4 : 8);
}

struct TcLaunchData {
  TcParams prm;
  int rowb;
  int cg;   // CTAs per MMA: 1, or 2 for the 2-SM UMMA
  int epi;  // epilogue warps: 4, or 8 where the epilogue bounds the step
  int dr;   // 1: the draining epilogue
};

int tc_prepare(const StepShape &sh, int fmt, const void *a_base, int a_lanes,
               int64_t a_lane_stride, int64_t plane_stride_bytes, const void *const b_base[2],
               int n_var, int64_t b_var_stride, int n_items, int kchunk, int cluster, int epi,
               void **out_handle) {
  EncodeTiledFn enc = encode_fn();
  if (!enc) return -1;
  const int esz = esz_of(fmt), np = np_of(fmt);
  const int Kr = 2 * sh.K, Nr = 2 * sh.N;
  const int rowb = rowb_for(Kr, esz, kchunk);
  if (!rowb) return -2;
  auto *d = new TcLaunchData();
  std::memset(&d->prm, 0, sizeof(TcParams));
  d->rowb = rowb;
  const CUtensorMapDataType dt =
      esz == 4 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_UINT16;
  const CUtensorMapSwizzle sw =
      rowb == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B;
  // unused dimensions (one plane, one lane) get the packed stride
  const int64_t packed = (int64_t)Kr * esz * sh.M;
  // Rows are stored next to one another over m_hi (runs of dv' entries, or
  // of single entries where the step stores its open leg into the batch, vb),
  // but the input's consecutive rows are consecutive in m_lo, whose
  // destinations lie dh' P dv' entries apart.  So a tile takes ph consecutive
  // m_hi x lh consecutive m_lo x bh consecutive b (ph lh bh = BM), through a
  // 5-d map {k, m_hi, m_lo, b, plane/lane} (the plane and the lane share a
  // coordinate: lane * lp_mul + plane): a warp's stores then cover whole
  // 128-byte lines.  The box lands in shared memory as the usual 128 rows
  // (row = (bb lh + l) ph + h).  Nothing to gain where the rows' order is
  // already that (P = 1, or Mr = P) or nothing is stored (the fused dot).
  bool mhi = false;
  int64_t lp_mul = 1, lp_stride = 0, lp_ext = 1;
  int64_t ph = 1, lh = 1, bh = 1;
  if (!sh.dot && sh.P > 1 && sh.Mr > sh.P && sh.Mr % sh.P == 0 && sh.M % sh.Mr == 0) {
    const int64_t Mlo = sh.Mr / sh.P, B = sh.M / sh.Mr;
    const int64_t want = sh.vb ? BM : (sh.dv_out >= 64 ? 1 : 64 / sh.dv_out);
    while (2 * ph <= want && sh.P % (2 * ph) == 0 && 2 * ph <= BM) ph *= 2;
    while (2 * lh * ph <= BM && Mlo % (2 * lh) == 0) lh *= 2;
    while (2 * bh * lh * ph <= BM && B % (2 * bh) == 0) bh *= 2;
    mhi = ph > 1 && ph * lh * bh == BM && sh.nvs == 0;
  }
  if (mhi) {
    if (np > 1) {
      if (a_lanes == 1) {
        lp_stride = plane_stride_bytes;
        lp_ext = np;
      } else if (plane_stride_bytes > 0 && a_lane_stride % plane_stride_bytes == 0) {
        lp_mul = a_lane_stride / plane_stride_bytes;
        lp_stride = plane_stride_bytes;
        lp_ext = (int64_t)(a_lanes - 1) * lp_mul + np;
      } else {
        mhi = false;
      }
    } else {
      lp_stride = a_lanes > 1 ? a_lane_stride : packed;
      lp_ext = a_lanes;
    }
    if (lp_stride % 16 != 0) mhi = false;
  }
  if (mhi) {
    const int64_t Mlo = sh.Mr / sh.P, B = sh.M / sh.Mr;
    cuuint64_t dims[5] = {(cuuint64_t)Kr, (cuuint64_t)sh.P, (cuuint64_t)Mlo, (cuuint64_t)B,
                          (cuuint64_t)lp_ext};
    cuuint64_t strides[4] = {(cuuint64_t)(Mlo * Kr * esz), (cuuint64_t)Kr * esz,
                             (cuuint64_t)(sh.Mr * Kr * esz), (cuuint64_t)lp_stride};
    cuuint32_t box[5] = {(cuuint32_t)(rowb / esz), (cuuint32_t)ph, (cuuint32_t)lh, (cuuint32_t)bh, 1};
    cuuint32_t es[5] = {1, 1, 1, 1, 1};
    CUresult r = enc(&d->prm.mapA, dt, 5, const_cast<void *>(a_base), dims, strides, box, es,
                     CU_TENSOR_MAP_INTERLEAVE_NONE, sw, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
      delete d;
      return -3;
    }
    d->prm.mhi = 1;
    d->prm.lp_mul = (int)lp_mul;
    d->prm.ph = (int)ph;
    d->prm.lh = (int)lh;
    d->prm.bh = (int)bh;
    d->prm.mlo = Mlo;
  } else {
    cuuint64_t dims[4] = {(cuuint64_t)Kr, (cuuint64_t)sh.M, (cuuint64_t)np,
                          (cuuint64_t)a_lanes};
    const int64_t plane_st = np > 1 ? plane_stride_bytes : packed;
    const int64_t lane_st = a_lanes > 1 ? a_lane_stride : plane_st * np;
    cuuint64_t strides[3] = {(cuuint64_t)Kr * esz, (cuuint64_t)((plane_st + 15) / 16 * 16),
                             (cuuint64_t)((lane_st + 15) / 16 * 16)};
    cuuint32_t box[4] = {(cuuint32_t)(rowb / esz), (cuuint32_t)BM, 1, 1};
    cuuint32_t es[4] = {1, 1, 1, 1};
    CUresult r = enc(&d->prm.mapA, dt, 4, const_cast<void *>(a_base), dims, strides, box, es,
                     CU_TENSOR_MAP_INTERLEAVE_NONE, sw, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
      delete d;
      return -3;
    }
  }
  const int kb_count = (Kr * esz) / rowb;
  const TileCols tc = tile_cols(sh, np, kb_count);
  const int KS = tc.ksplit, CS = tc.csep, NA = KS + CS;
  int BN = tc.BN;
  // entries in contiguous runs of 8 (the epilogue's W = 8)
  const int run = sh.vb && sh.nvs ? sh.dh_out : (sh.dv_out == 1 && sh.P == 1 ? sh.N : sh.dv_out);
  const bool runs8 = !sh.dot && run % 8 == 0 && (sh.vb ? sh.nvs && sh.P == 1 : true);
  // The draining epilogue where main and correction accumulators fill TMEM on
  // 256-column tiles.  For a short K that is the alternative to 128-column
  // tiles with two buffers, which load every row of A twice as often: 16 lanes
  // of 65536 x 256 x 256 took 1408 us that way, at 9 TB/s from L2 into shared
  // memory; 1072 us drained, 993 with the interleaved order below as well (512
  // lanes of the fused 1024 x 1024 x 256 merge: 1912, 1756, 1632 us).  It needs tiles for every CTA pair; the fused dot's
  // tiles keep their width (it fixes the order of its partial sums).
  const bool wide32 = (uintptr_t)a_base % 32 == 0;
  const bool drain =
      CS == 1 && NA == 2 && rowb == 128 && Nr % 256 == 0 && epi != 4 && wide32 &&
      (sh.dot ? BN == 256
              : runs8 && (sh.M / 256) * (Nr / 256) * (int64_t)n_items >= (BN == 256 ? 38 : 152));
  if (drain) BN = 256;
  // A launch of fewer tiles than CTA pairs is as long as one tile: narrower
  // tiles (down to 64 columns, in whole 32s for the pairs) put more SMs on it.  One item of 256 x 1024 x
  // 1024: 38.9 -> 32.7 us, of 1024 x 128 x 512: 15.9 -> 12.4 us.
  const int64_t row_tiles = (sh.M + 2 * BM - 1) / (2 * BM);
  while (!drain && !sh.dot && BN >= 128 && BN % 64 == 0 && row_tiles * (Nr / BN) * n_items < 76)
    BN /= 2;
  const int tiles_m = (int)((sh.M + BM - 1) / BM);
  // The 2-SM UMMA when the 128-row tiles pair up and the columns are a multiple
  // of 32, as its M = 256 form is specified for (the one-CTA form: of 16).
  d->cg = (BN % 32 == 0 && tiles_m % 2 == 0 && cluster != 1) ? 2 : 1;
  // B: one map per plane over every operand variant {k, n, variant}; the
  // variants are equally spaced (a single variant gets the packed stride)
  const int64_t bpacked = (int64_t)Kr * esz * Nr;
  const int64_t vstride = n_var > 1 ? b_var_stride : bpacked;
  if (n_var < 1 || n_var > 64 || vstride < bpacked || vstride % 16 != 0) {
    delete d;
    return -6;
  }
  for (int pl = 0; pl < np; ++pl) {
    cuuint64_t dims[3] = {(cuuint64_t)Kr, (cuuint64_t)Nr, (cuuint64_t)n_var};
    cuuint64_t strides[2] = {(cuuint64_t)Kr * esz, (cuuint64_t)vstride};
    cuuint32_t box[3] = {(cuuint32_t)(rowb / esz), (cuuint32_t)(BN / d->cg), 1};
    cuuint32_t es[3] = {1, 1, 1};
    CUresult r = enc(&d->prm.mapB[pl], dt, 3, const_cast<void *>(b_base[pl]), dims, strides, box,
                     es, CU_TENSOR_MAP_INTERLEAVE_NONE, sw, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
      delete d;
      return -4;
    }
  }
  d->prm.sh = sh;
  d->prm.wide = wide32 ? 1 : 0;
  d->prm.BN = BN;
  d->prm.tiles_m = (int)((sh.M + BM - 1) / BM);
  d->prm.tiles_n = Nr / BN;
  // wide launches (the merges): 8 row groups at a time, so that concurrent
  // tiles reuse both operands' k-slabs from L2 instead of streaming one B
  // column panel per tile
  {
    const int mgroups = d->prm.tiles_m / d->cg;
    d->prm.gm = (d->prm.tiles_n >= 32 && mgroups >= 16) ? 8 : 1;
    // Outside the grouped order a pair walks consecutive tiles (an item's
    // set-up and operand once), or every ncl-th where the tiles are long and a
    // row panel has several of them: the pairs then work on the same k-slabs of
    // A and B at the same time, which L2 serves once, while consecutive tiles
    // re-read a panel of A after it has left.  Consecutive / interleaved: 32 lanes
    // of 512 x 1024 x 1024 339 / 226 us, 16 of 65536 x 256 x 256 1072 / 998 us,
    // 512 of 4096 x 64 x 256 908 / 846 us; but 512 of 2048 x 16 x 64 117 / 145 us,
    // 16 of 4096 x 64 x 512 60.2 / 61.8 us.
    const bool interleave = d->prm.tiles_n >= 2 && BN == 256 &&
                            (sh.K >= 128 || (sh.K >= 64 && d->prm.tiles_n == 2));
    d->prm.blocked = d->prm.gm == 1 && !interleave ? 1 : 0;
    d->prm.d_tpi = make_div((int64_t)mgroups * d->prm.tiles_n);
    d->prm.d_tn = make_div(d->prm.tiles_n);
  }
  {
    const int64_t Mr = sh.Mr > 0 ? sh.Mr : sh.M, P = sh.P > 0 ? sh.P : 1;
    d->prm.d_Mr = make_div(Mr);
    d->prm.d_Mlo = make_div(Mr / P);
    d->prm.d_dv = make_div(sh.dv_out);
    d->prm.d_dh = make_div(sh.dh_out);
    const int ph = d->prm.mhi ? d->prm.ph : 1, lh = d->prm.mhi ? d->prm.lh : 1;
    d->prm.d_ph = make_div(ph);
    d->prm.d_lh = make_div(lh);
    d->prm.d_hper = make_div(d->prm.mhi ? P / ph : 1);
    d->prm.d_lper = make_div(d->prm.mhi ? d->prm.mlo / lh : 1);
  }
  d->prm.ksplit = KS;
  d->prm.csep = CS;
  d->prm.nacc = NA;
  d->prm.nbuf = 2 * BN * NA <= 512 ? 2 : 1;
  int cols = 32;
  while (cols < d->prm.nbuf * BN * NA) cols *= 2;
  d->prm.tmem_cols = cols;
  const int stage_bytes = np * (BM + BN / d->cg) * rowb;  // this CTA's share
  // 227 KiB per CTA, less the 1 KiB alignment pad and the barriers
  const int budget = 227 * 1024 - 1024 - 256;
  int stages = budget / stage_bytes;
  if (stages > 8) stages = 8;
  d->prm.stages = stages;
  // Epilogue warps: eight where the epilogue bounds the tile (K <= 64 on
  // tiles of at least 64 columns, K <= 32 on 32) and where it is not hidden at
  // all (one accumulator buffer: the merges; the fused dot), four where the
  // MMAs do or where a second warp per quadrant finds no columns.  Measured,
  // eight / four warps: 16 lanes of 65536 x 16 x 256 446 / 460 us, of 4096 x 64 x
  // 512 58.6 / 59.3 us (BF16 36.1 / 38.1), one item of 256 x 1024 x 1024 49.5 / 59.0
  // us; 512 lanes of 1024 x 128 x 512 537 / 518 us, 16 of 32768 x 64 x 8 64.8 / 61.7
  // us.  (Drained against four warps: the fused 1024 x 1024 x 256 merge of 512
  // lanes 1632 / 1932 us, 16 lanes of 65536 x 256 x 256 993 / 1366 us.)
  const bool epi_bound = sh.dot || d->prm.nbuf == 1 || (sh.K <= 64 && BN >= 64) ||
                         (sh.K <= 32 && BN >= 32);
  d->epi = epi == 4 || epi == 8 ? epi : (epi_bound ? 8 : 4);
  d->dr = drain ? 1 : 0;
  if (drain) d->epi = 8;
  *out_handle = d;
  return stages >= 2 ? 0 : -5;
}

void tc_release(void *h) { delete (TcLaunchData *)h; }

// The kernel set up on the current device; *max_clusters: co-resident clusters
// at the largest shared-memory size (0: not known).
template <int FMT, int ROWB, int CG, int EPI, int DR>
static cudaError_t init_kernel(int *max_clusters) {
  static PerDevice state;
  return state.get(max_clusters, [](int *n) {
    auto kern = k_contract_tc<FMT, ROWB, CG, EPI, DR>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         227 * 1024);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t q = {};
    cudaLaunchAttribute qa[1];
    qa[0].id = cudaLaunchAttributeClusterDimension;
    qa[0].val.clusterDim.x = CG;
    qa[0].val.clusterDim.y = 1;
    qa[0].val.clusterDim.z = 1;
    q.gridDim = dim3(CG * 64);
    q.blockDim = dim3(threads_of(EPI, DR));
    q.dynamicSmemBytes = 227 * 1024;
    q.attrs = qa;
    q.numAttrs = 1;
    *n = 0;
    e = cudaOccupancyMaxActiveClusters(n, (void *)kern, &q);
    if (e != cudaSuccess || *n <= 0) {
      (void)cudaGetLastError();
      *n = 0;
    }
    return cudaSuccess;
  });
}

template <int FMT, int ROWB, int CG, int EPI, int DR>
static cudaError_t launch_one(const TcParams &prm, int units, size_t smem, cudaStream_t s) {
  auto kern = k_contract_tc<FMT, ROWB, CG, EPI, DR>;
  int max_clusters = 0;
  const cudaError_t e0 = init_kernel<FMT, ROWB, CG, EPI, DR>(&max_clusters);
  if (e0 != cudaSuccess) return e0;
  // units = SMs to use; one CTA per SM, clusters of CG
  int clusters = units / CG;
  if (max_clusters > 0 && clusters > max_clusters) clusters = max_clusters;
  if (clusters < 1) clusters = 1;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = CG;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  // Dependent launch (pdl_wait), but not for long launches in interleaved or
  // grouped order: started as SMs come free, the pairs that share k-slabs in L2
  // land on different dies (512 lanes of the 1024 x 1024 x 256 merge: 1616 us
  // placed in order, 1849 us so).
  const bool in_order = !prm.blocked && (int64_t)prm.n_items * (prm.tiles_m / CG) * prm.tiles_n >
                                            4 * (int64_t)clusters;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.gridDim = dim3(clusters * CG);
  cfg.blockDim = dim3(threads_of(EPI, DR));
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = in_order ? 1 : 2;
  return cudaLaunchKernelEx(&cfg, kern, prm);
}

// f.run<FMT, ROWB, CG, EPI, DR>() for the kernel that `d` launches
// (the draining form exists for the split formats and 128-byte stages only).
template <int FMT, class F>
static cudaError_t with_kernel(const TcLaunchData *d, F f) {
  if constexpr (FormTraits<FMT>::NP == 2) {
    if (d->dr) return d->cg == 2 ? f.template run<FMT, 128, 2, 8, 1>() : f.template run<FMT, 128, 1, 8, 1>();
  }
  if (d->dr) return cudaErrorInvalidValue;
  if (d->epi == 8) {
    if (d->rowb == 128)
      return d->cg == 2 ? f.template run<FMT, 128, 2, 8, 0>() : f.template run<FMT, 128, 1, 8, 0>();
    return d->cg == 2 ? f.template run<FMT, 64, 2, 8, 0>() : f.template run<FMT, 64, 1, 8, 0>();
  }
  if (d->rowb == 128)
    return d->cg == 2 ? f.template run<FMT, 128, 2, 4, 0>() : f.template run<FMT, 128, 1, 4, 0>();
  return d->cg == 2 ? f.template run<FMT, 64, 2, 4, 0>() : f.template run<FMT, 64, 1, 4, 0>();
}
template <class F>
static cudaError_t with_kernel_of(const TcLaunchData *d, F f) {
  switch (d->prm.sh.fmt) {
    case FMT_BF16: return with_kernel<FMT_BF16>(d, f);
    case FMT_FP16: return with_kernel<FMT_FP16>(d, f);
    case FMT_BF16X2: return with_kernel<FMT_BF16X2>(d, f);
    case FMT_FP16X2: return with_kernel<FMT_FP16X2>(d, f);
    case FMT_TF32: return with_kernel<FMT_TF32>(d, f);
  }
  return cudaErrorInvalidValue;
}
struct WarmKernel {
  template <int FMT, int ROWB, int CG, int EPI, int DR>
  cudaError_t run() const {
    int unused = 0;
    return init_kernel<FMT, ROWB, CG, EPI, DR>(&unused);
  }
};
struct LaunchKernel {
  const TcParams &prm;
  int units;
  size_t smem;
  cudaStream_t s;
  template <int FMT, int ROWB, int CG, int EPI, int DR>
  cudaError_t run() const { return launch_one<FMT, ROWB, CG, EPI, DR>(prm, units, smem, s); }
};

cudaError_t tc_warm(void *handle) {
  return with_kernel_of((const TcLaunchData *)handle, WarmKernel{});
}

int64_t tc_dot_slots(const void *handle) {
  const TcLaunchData *d = (const TcLaunchData *)handle;
  return (int64_t)d->prm.tiles_m * d->prm.tiles_n * d->epi;
}

cudaError_t launch_contract_tc(void *handle, const StepItem *d_items, int n_items,
                               const OpDesc *d_ops, Rec *d_recs, DeviceStatus *st,
                               int64_t watchdog_ns, int sm_count, cudaStream_t s,
                               double2 *dot_partials) {
  TcLaunchData *d = (TcLaunchData *)handle;
  TcParams prm = d->prm;
  prm.dot_partials = dot_partials;
  if (prm.sh.dot && !dot_partials) return cudaErrorInvalidValue;
  prm.items = d_items;
  prm.n_items = n_items;
  prm.ops = d_ops;
  prm.recs = d_recs;
  prm.st = st;
  prm.watchdog_ns = watchdog_ns;
  const int cg = d->cg;
  const int pair_tiles = n_items * (prm.tiles_m / cg) * prm.tiles_n;
  if (pair_tiles < 1) return cudaSuccess;
  const int units = pair_tiles * cg < sm_count ? pair_tiles * cg : sm_count;
  const int np = np_of(prm.sh.fmt);
  const size_t smem = (size_t)prm.stages * np * (BM + prm.BN / cg) * d->rowb + 1024 +
                      (2 * prm.stages + 6) * 8 + 16;
  return with_kernel_of(d, LaunchKernel{prm, units, smem, s});
}

// ---------------------------------------------------------------------------
// Tensor-core operand build: the real embedding of E (scaled by 2^b_t), split
// into the form's planes, K-major [Nr][Kr].  Also the bound beta_t.
// ---------------------------------------------------------------------------
// Tiles first, first + step, ... below last of one operand: 32 x 32 entries of
// Ec each, through shared memory.
__device__ __forceinline__ int bt_tiles(const OpDesc &op, bool marked) {   // none if no lane reads it
  if (op.Bt[0] == nullptr || (marked && !op.used)) return 0;
  return ((op.K + 31) / 32) * ((op.N + 31) / 32);
}
template <int FMT>
__device__ __forceinline__ void bt_operand_tiles(OpDesc &op, int first, int last, int step) {
  const int K = op.K, N = op.N;
  const float sc = ldexpf(1.f, op.b_t);
  const float2 *const Ec = op.Ec;
  void *const hi = const_cast<void *>(op.Bt[0]), *const lo = const_cast<void *>(op.Bt[1]);
  // 32 x 32 complex tiles of Ec through shared memory: read along n, written
  // along k, two real columns (a = 0, 1 of one k) per store
  __shared__ float2 tile[32][33];
  const int tn = (N + 31) / 32;
  const int64_t Kr = 2 * (int64_t)K;
  for (int t = first; t < last; t += step) {
    const int k0 = (t / tn) * 32, n0 = (t % tn) * 32;
    for (int e = threadIdx.x; e < 32 * 32; e += blockDim.x) {
      const int kk = e >> 5, nn = e & 31;
      tile[kk][nn] = (k0 + kk < K && n0 + nn < N) ? Ec[(int64_t)(k0 + kk) * N + n0 + nn]
                                                    : make_float2(0.f, 0.f);
    }
    __syncthreads();
    if (FMT != FMT_TF32 && K % 4 == 0) {
      // four neighbouring k per thread: 16-byte stores, four rows per warp
      const int k4 = (threadIdx.x & 7) * 4;
      for (int r = threadIdx.x >> 3; r < 64; r += blockDim.x >> 3) {
        const int nn = r >> 1, b = r & 1, n = n0 + nn;
        if (k0 + k4 >= K || n >= N) continue;
        uint32_t h[4], l[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float2 e = tile[k4 + j][nn];
          const float v0 = (b == 0 ? e.x : e.y) * sc, v1 = (b == 0 ? -e.y : e.x) * sc;
          if (FMT == FMT_BF16) h[j] = pack_bf16(v0, v1);
          else if (FMT == FMT_FP16) h[j] = pack_f16(v0, v1);
          else split16<FMT == FMT_BF16X2>(make_float2(v0, v1), h[j], l[j]);
        }
        const int64_t w = (((int64_t)(2 * n + b) * Kr) >> 1) + k0 + k4;   // in column pairs
        *(uint4 *)((uint32_t *)hi + w) = make_uint4(h[0], h[1], h[2], h[3]);
        if (FMT == FMT_BF16X2 || FMT == FMT_FP16X2)
          *(uint4 *)((uint32_t *)lo + w) = make_uint4(l[0], l[1], l[2], l[3]);
      }
      __syncthreads();
      continue;
    }
    const int kk = threadIdx.x & 31, k = k0 + kk;
    for (int r = threadIdx.x >> 5; r < 64; r += blockDim.x >> 5) {
      const int nn = r >> 1, b = r & 1, n = n0 + nn;
      if (k >= K || n >= N) continue;
      // row 2n holds (re, -im) at columns 2k, 2k+1; row 2n+1 holds (im, re)
      const float2 e = tile[kk][nn];
      const float v0 = (b == 0 ? e.x : e.y) * sc, v1 = (b == 0 ? -e.y : e.x) * sc;
      const int64_t w = ((int64_t)(2 * n + b) * Kr + 2 * (int64_t)k) >> 1;   // in column pairs
      if (FMT == FMT_TF32) {
        ((float2 *)hi)[w] = make_float2(round_tf32(v0), round_tf32(v1));
      } else if (FMT == FMT_BF16) {
        ((uint32_t *)hi)[w] = pack_bf16(v0, v1);
      } else if (FMT == FMT_FP16) {
        ((uint32_t *)hi)[w] = pack_f16(v0, v1);
      } else {
        constexpr bool BF = FMT == FMT_BF16X2;
        uint32_t h, l;
        split16<BF>(make_float2(v0, v1), h, l);
        ((uint32_t *)hi)[w] = h;
        ((uint32_t *)lo)[w] = l;
      }
    }
    __syncthreads();
  }
  if (first == 0 && threadIdx.x == 0) {
    // beta_t = beta_c * 2^b_t (beta_c already carries a rounding margin; the
    // rounded planes differ from the scaled values by at most 2^-8 relative)
    const float bc = __uint_as_float(op.beta_c_bits);
    op.beta_t_bits = __float_as_uint(bc * sc * (1.0f + 1.0f / 128.0f));
  }
}

template <int FMT>
__global__ void __launch_bounds__(256) k_build_bt(const OpList list, int n, OpDesc *ops,
                                                  bool marked) {
  pdl_trigger();
  pdl_wait();
  if (gridDim.y > 1 || n == 1) {   // by operand
    OpDesc &op = ops[list.op(blockIdx.y)];
    const int nt = bt_tiles(op, marked);
    if ((int)blockIdx.x < nt) bt_operand_tiles<FMT>(op, blockIdx.x, nt, gridDim.x);
    return;
  }
  auto tiles = [&](int j) { return bt_tiles(ops[list.op(j)], marked); };
  for_block_share(n, (int)threadIdx.x < n ? tiles(threadIdx.x) : 0, tiles,
                  [&](int j, int a, int b) { bt_operand_tiles<FMT>(ops[list.op(j)], a, b, 1); });
}

// A merge operand straight from a stored tensor G whose k index is contiguous:
// Ec[k][n] = G[k + nh ns_hi + nl ns] 2^-target (n = nh Nlo + nl) is never
// written out.  One pass over G gives the column bound beta_c = max_n sum_k
// |Ec[k][n]|_1 and the complex-as-real planes Bt[(n, b)][(k, a)]; reads and
// writes both run along k.  Bound by memory: 8 bytes read and 16 written per
// entry (FP16X3).  16 operands of 4096 x 4096: bound and planes in two passes
// 2380 us, in this one 1086 us (5.9 TB/s).  Same values as Ec -> k_beta_ops -> k_build_bt.
__global__ void k_tensor_init(const TensorOpEntry *__restrict__ e, int n, OpDesc *ops,
                              const Rec *recs) {
  pdl_trigger();
  pdl_wait();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const TensorOpEntry g = e[i];
  OpDesc &op = ops[g.op];
  op.beta_c_bits = 0u;
  op.beta_t_bits = 0u;
  op.e_c = recs[g.rec].exp - g.target;
}

// Entry k of column n (ek = its value 2^-target 2^b_t) into both rows of the planes.
template <int FMT>
__device__ __forceinline__ void put_bt(void *hi, void *lo, int64_t n, int64_t K, int64_t k,
                                       float re, float im) {
  // row 2n holds (re, -im) at columns 2k, 2k+1; row 2n+1 holds (im, re)
  const float2 r0 = make_float2(re, -im), r1 = make_float2(im, re);
  const int64_t w0 = 2 * n * K + k, w1 = w0 + K;   // in column pairs
  if (FMT == FMT_TF32) {
    ((float2 *)hi)[w0] = make_float2(round_tf32(r0.x), round_tf32(r0.y));
    ((float2 *)hi)[w1] = make_float2(round_tf32(r1.x), round_tf32(r1.y));
  } else if (FMT == FMT_BF16) {
    ((uint32_t *)hi)[w0] = pack_bf16(r0.x, r0.y);
    ((uint32_t *)hi)[w1] = pack_bf16(r1.x, r1.y);
  } else if (FMT == FMT_FP16) {
    ((uint32_t *)hi)[w0] = pack_f16(r0.x, r0.y);
    ((uint32_t *)hi)[w1] = pack_f16(r1.x, r1.y);
  } else {
    constexpr bool BF = FMT == FMT_BF16X2;
    uint32_t h0, l0, h1, l1;
    split16<BF>(r0, h0, l0);
    split16<BF>(r1, h1, l1);
    ((uint32_t *)hi)[w0] = h0;
    ((uint32_t *)hi)[w1] = h1;
    ((uint32_t *)lo)[w0] = l0;
    ((uint32_t *)lo)[w1] = l1;
  }
}

// COL = 1: a block per column (threads along k), COL = 0: a warp per column (K
// too short for a block).  Either way a column's sum is eight partial sums (k
// mod 256 in [32 w, 32 w + 32), each the tree of 32 lane sums over k ascending)
// added in order.
template <int FMT, int COL>
__global__ void __launch_bounds__(256) k_tensor_bt(const TensorOpEntry *__restrict__ e,
                                                   int64_t plane, OpDesc *ops) {
  pdl_trigger();
  const TensorOpEntry g = e[blockIdx.y];   // one entry per grid row
  pdl_wait();
  OpDesc &op = ops[g.op];
  const int64_t K = g.K, N = g.N;
  void *const hi = const_cast<void *>(op.Bt[0]), *const lo = const_cast<void *>(op.Bt[1]);
  const float sc = pow2f(-g.target), sb = ldexpf(1.f, op.b_t);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  __shared__ float red[8];
  float best = 0.f;
  // the lane sum over k = k0, k0 + 256, ..., four loads in flight
  auto lane_sum = [&](int64_t n, int64_t base, int64_t k0) {
    float s = 0.f;
    for (int64_t k = k0; k < K; k += 1024) {
      float2 v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (k + 256 * u < K) v[u] = load_g<FMT>(g.G, base + (k + 256 * u) * g.ks, plane);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (k + 256 * u >= K) break;
        const float re = v[u].x * sc, im = v[u].y * sc;
        s += fabsf(re) + fabsf(im);
        put_bt<FMT>(hi, lo, n, K, k + 256 * u, re * sb, im * sb);
      }
    }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
  };
  auto column = [&](int64_t n) {
    const int64_t nh = n / g.Nlo, nl = n - nh * g.Nlo;
    return nh * g.ns_hi + nl * g.ns;
  };
  if (COL) {
    for (int64_t n = blockIdx.x; n < N; n += gridDim.x) {
      const float s = lane_sum(n, column(n), threadIdx.x);
      if (lane == 0) red[warp] = s;
      __syncthreads();
      if (threadIdx.x == 0) {
        float t = 0.f;
        for (int w = 0; w < 8; ++w) t += red[w];
        best = fmaxf(best, t);
      }
      __syncthreads();
    }
  } else {
    for (int64_t n = (int64_t)blockIdx.x * 8 + warp; n < N; n += (int64_t)gridDim.x * 8) {
      const int64_t base = column(n);
      float t = 0.f;
      for (int w = 0; w < 8 && 32 * w < K; ++w) t += lane_sum(n, base, 32 * w + lane);
      best = fmaxf(best, t);
    }
    if (lane == 0) red[warp] = best;
    __syncthreads();
    if (threadIdx.x == 0)
      for (int w = 0; w < 8; ++w) best = fmaxf(best, red[w]);
  }
  if (threadIdx.x == 0) {
    // beta_t = beta_c 2^b_t with its margin: increasing in beta_c, so the
    // blocks' largest is that of the largest beta_c
    const float bc = best * (1.0f + 1.0f / 256.0f);
    atomicMax(&op.beta_c_bits, __float_as_uint(bc));
    atomicMax(&op.beta_t_bits, __float_as_uint(bc * sb * (1.0f + 1.0f / 128.0f)));
  }
}

template <int FMT>
static cudaError_t tensor_bt(const TensorOpEntry *d_entry, int n_entries, int K, int N,
                             int64_t plane, OpDesc *d_ops, cudaStream_t s) {
  // some 16 blocks per SM in all, each with several columns
  const bool col = K >= 1024;
  const int units = col ? N : (N + 7) / 8;
  int gx = (16 * 152 + n_entries - 1) / n_entries;
  if (gx > units) gx = units;
  const dim3 grid((unsigned)gx, (unsigned)n_entries);
  return col ? launch_dependent(k_tensor_bt<FMT, 1>, grid, dim3(256), 0, s, d_entry, plane, d_ops)
             : launch_dependent(k_tensor_bt<FMT, 0>, grid, dim3(256), 0, s, d_entry, plane, d_ops);
}

cudaError_t launch_tensor_operand_tc(const TensorOpEntry *d_entry, int n_entries, int K, int N,
                                     int fmt, int64_t plane, OpDesc *d_ops, const Rec *d_recs,
                                     cudaStream_t s) {
  if (n_entries <= 0) return cudaSuccess;
  const cudaError_t r = launch_dependent(k_tensor_init, dim3((n_entries + 127) / 128), dim3(128), 0, s,
                                         d_entry, n_entries, d_ops, d_recs);
  if (r != cudaSuccess) return r;
  switch (fmt) {
    case FMT_TF32: return tensor_bt<FMT_TF32>(d_entry, n_entries, K, N, plane, d_ops, s);
    case FMT_BF16: return tensor_bt<FMT_BF16>(d_entry, n_entries, K, N, plane, d_ops, s);
    case FMT_FP16: return tensor_bt<FMT_FP16>(d_entry, n_entries, K, N, plane, d_ops, s);
    case FMT_BF16X2: return tensor_bt<FMT_BF16X2>(d_entry, n_entries, K, N, plane, d_ops, s);
    case FMT_FP16X2: return tensor_bt<FMT_FP16X2>(d_entry, n_entries, K, N, plane, d_ops, s);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_build_tc_operands(int n, const OpList &list, int64_t max_kn, OpDesc *d_ops,
                                     int fmt, bool marked, int sm_count, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  // the list of all operands' tiles, or by operand where that gives about
  // every tile its own block
  const int64_t tiles = (max_kn + 1023) / 1024 + 2;
  const dim3 grid = n == 1 || n * tiles <= 2048 ? dim3((unsigned)(tiles < 2048 ? tiles : 2048), n)
                                                : dim3(6 * sm_count);
  switch (fmt) {
    case FMT_TF32: return launch_dependent(k_build_bt<FMT_TF32>, grid, dim3(256), 0, s, list, n, d_ops, marked);
    case FMT_BF16: return launch_dependent(k_build_bt<FMT_BF16>, grid, dim3(256), 0, s, list, n, d_ops, marked);
    case FMT_FP16: return launch_dependent(k_build_bt<FMT_FP16>, grid, dim3(256), 0, s, list, n, d_ops, marked);
    case FMT_BF16X2: return launch_dependent(k_build_bt<FMT_BF16X2>, grid, dim3(256), 0, s, list, n, d_ops, marked);
    case FMT_FP16X2: return launch_dependent(k_build_bt<FMT_FP16X2>, grid, dim3(256), 0, s, list, n, d_ops, marked);
  }
  return cudaErrorInvalidValue;
}

}  // namespace peps
