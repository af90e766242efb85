// Prefill GEMM of the PolyQ mixed-bit layer on the 5th-generation tensor
// cores (tcgen05, tensor memory), on pairs of SMs:
//
//   Y[m][n] = sum_p X[m][gather[p]] * W'[n][p]        (Section 4.1 product)
//
// The contraction runs over K tiles of 32 or 64 (half or all of a quantisation
// group); every tile lies inside one bit block (Section 4.2) and one group, so
// each weight row of a tile has one (scale, zero).
//  1. A pre-pass (gemm_prep_rows, or gemm_prep_small for a few rows) gathers X
//     through `gather` into a clustered fp16 matrix Xg (workspace),
//     zero-padded at block ends, with the K order inside each tile permuted
//     the same way the dequantiser emits codes.  Xg is stored as the
//     shared-memory images of the producer's copies: per (CTA's tokens, 32 K
//     slots) one block of R rows of 64 bytes in the 64-byte swizzle, so that
//     one contiguous bulk copy fetches a stage's X.  Each row m is scaled by
//     the power of two 2^-e_m that brings its largest |x * t| into
//     [2^14, 2^15), so that any finite bf16 row rounds to fp16 without
//     overflow and without dropping small values into subnormals; the
//     epilogue multiplies row m of Y by 2^e_m.
//  2. gemm_main: persistent clusters of two CTAs, one CTA per SM.  A work unit
//     is 256 weight rows by T tokens; CTA r of the pair holds weight rows
//     128 r.. and half of the tokens, and one tcgen05.mma.cta_group::2
//     (M = 256, N = 32..256, K = 16, fp16 in, fp32 accumulate) multiplies all
//     rows with all tokens, so each weight is dequantised by one SM only and
//     each operand byte is read from shared memory once per SM pair.  The
//     weights are the A operand, so a TMEM lane holds one output column.
//       warp 0      TMA producer: Xg blocks (bulk copies), packed code bytes
//                   and meta of the CTA's 128 weight rows, or for 16-bit
//                   blocks the fp16 weights straight into the operand buffer;
//       warp 1      allocates 512 TMEM columns; in the leader CTA it issues
//                   the MMAs;
//       warps 2..   groups of four warps dequantise, one weight row per
//                   thread, alternating over the stages: (q - z) * s in fp16,
//                   written in the UMMA 64-byte-swizzle K-major layout;
//       last four   drain the accumulators with tcgen05.ld and store fp32 Y,
//                   each warp store covering 32 consecutive columns of a row.
//     When the (M, N) tiles cannot fill the GPU the K range is split,
//     uniformly or stream-K (each pair an equal contiguous share of all (tile,
//     K tile) pairs, or of those left after full waves of whole tiles), and the
//     pieces are added into a zeroed Y (so the order of those additions
//     varies); otherwise Y is stored directly.  Every wait is bounded and
//     reports through the workspace status word.
// Bound by the tensor pipe at large M (13824 x 5120, M = 2048, B = 3: 174 us for
// both kernels, 1660 TFLOP/s, the pipe active 83% of the cycles; on single SMs
// 273 us, 50%) and by the dequantisers' stages and the fixed time of the two
// launches at small M (5120 x 5120, M = 16: 14.6 us, before 27).
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cstring>

#include "polyq.h"
#ifdef POLYQ_DEBUG
#include "polyq_debug.h"
#include "polyq_debug_gemm.h"
#endif
#include "polyq_dev.cuh"
#include "polyq_gemv_dev.cuh"
#include "polyq_internal.h"

namespace {

using namespace polyq;

constexpr int kRowsN = 256;       // weight rows per work unit
constexpr int kRowsCta = 128;     // of which each CTA of a pair holds half
constexpr int kSlots = 32;        // K slots of an Xg block and of a 64-byte operand row
constexpr int kCodeBox = 32;      // code bytes per row of one code box: the codes of a tile of 32
                                  // from a 16-byte aligned start (offset <= 12 with at most 16
                                  // bytes of codes, or 32 bytes of 8-bit codes at offset 0), or of
                                  // a tile of 64 at 2 to 4 bits (24 bytes at offset 0 or 8, else
                                  // at offset 0); one TMA row request each (48-byte rows take two)
constexpr int kBoxBytes = kRowsCta * kCodeBox;  // 4 KB
constexpr int kMetaBytes = kRowsCta * 16;       // 2 KB
constexpr int kHalfTile = kRowsCta * kSlots * 2;  // 8 KB: 128 operand rows of 64 bytes
constexpr double kZeroBytesPerS = 5e12;  // the pre-pass zeroing Y
constexpr uint32_t kTmemCols = 512;
// Cost model of the split of K (plan_split), seconds: one stage of a pair and
// the overhead of a piece, by token tile.
// (Stages as traced in short runs, at about 1.9 GHz: with 512 tokens the MMAs'
// 512 cycles.  Long runs, under the power cap, take 0.33 to 0.36 us for those.
// Pieces set so that the model picks the faster of both splits and both tiles on
// 5120 x 5120, 13824 x 5120 and 5120 x 13824 from M = 16 to 4096, to 2%: 5120 x
// 5120, M = 512 34.5 us with 4.5 and 5.5, 32.2 with 3.5 and 6.5; 13824 x 5120,
// M = 256 36.3 and 34.4.)
constexpr double kStage32 = 0.23e-6, kPiece32 = 1.5e-6;
constexpr double kStage64 = 0.24e-6, kPiece64 = 1.5e-6;
constexpr double kStage128 = 0.26e-6, kPiece128 = 2e-6;
constexpr double kStage256 = 0.31e-6, kPiece256 = 3.5e-6;
constexpr double kStage512 = 0.27e-6, kPiece512 = 6.5e-6;

// One kernel per token count T of a work unit.
//   TN      tokens per MMA (its N); CTA r of the pair holds TN / 2 of them
//   NACC    accumulators of a unit (T = NACC * TN); with one, two units'
//           accumulators alternate, so that one drains while the next fills
//   BK      K of a stage
//   OPS     weight slots: a dequantised tile
//   XS      token slots: the tile's X
//   CODES   code slots: packed codes and meta, free again once a dequantiser
//           holds them in registers, so that the copies of the packed weights
//           run CODES stages ahead whatever the MMAs do
//   GROUPS  dequantiser groups (CODES and OPS multiples of it): the twelve warps as three of
//           four, a weight row per thread, or as six of two, two rows per thread.  Two rows
//           share a stage's waits, fence and arrivals (M = 16: 26.0 -> 24.7 us for 13824 x
//           5120, M = 96: 30.2 -> 29.4); with 512 tokens the MMAs set the pace either way
//   EPI     epilogue warps (a multiple of four)
template <int TN_, int NACC_, int BK_, int OPS_, int XS_, int CODES_, int GROUPS_, int EPI_>
struct Cfg {
  static constexpr int TN = TN_, NACC = NACC_, BK = BK_, OPS = OPS_, XS = XS_;
  static constexpr int CODES = CODES_, GROUPS = GROUPS_, EPI = EPI_;
  static constexpr int T = TN * NACC;
  static constexpr bool kWhole = T == 512;  // see plan_split
  static constexpr int R = T / 2;           // tokens (rows of X) per CTA
  static constexpr int NBUF = NACC == 1 ? 2 : 1;
  static constexpr int HALVES = BK / kSlots;
  static constexpr int kA = HALVES * kHalfTile;
  static constexpr int kX = HALVES * R * kSlots * 2;
  static constexpr int kCodes = HALVES * kBoxBytes;
  static constexpr int kCode = kCodes + kMetaBytes;
  static constexpr int kCodeProd = 2;  // producer warps of the codes
  static constexpr int kDqGroup = 12 / GROUPS, kDqRows = kRowsCta / (32 * kDqGroup);  // warps, rows a thread
  static constexpr int kEpiWarp = 16, kWarps = kEpiWarp + EPI;
  static constexpr int kThreads = 32 * kWarps;
  static constexpr int kXOff = OPS * kA, kCodeOff = kXOff + XS * kX;  // in shared memory
  static constexpr size_t kSmem = (size_t)kCodeOff + CODES * kCode + 1024;
  static constexpr uint32_t kIdesc = umma_idesc_f16(kRowsN, TN);
  static_assert(kX % 1024 == 0 && kSmem <= 225 * 1024 + 512 && NACC * NBUF * TN <= (int)kTmemCols, "");
  static_assert((GROUPS == 3 || GROUPS == 6) && CODES % GROUPS == 0 && OPS % GROUPS == 0 && kCodeProd <= CODES &&
                OPS <= 32, "");  // a parity bit per weight slot
};
using Cfg32 = Cfg<32, 1, 64, 6, 16, 6, 6, 4>;
using Cfg64 = Cfg<64, 1, 64, 6, 8, 6, 6, 4>;
using Cfg128 = Cfg<128, 1, 64, 6, 6, 6, 6, 4>;
using Cfg256 = Cfg<256, 1, 64, 6, 4, 6, 6, 4>;
using Cfg512 = Cfg<256, 2, 32, 6, 7, 9, 3, 8>;
// Warps 0, 4, 8 and 12, which share a scheduler, are the lone-thread roles
// (two code producers, the X producer, the MMA issuer), the other twelve of
// the first sixteen the dequantisers: their long unrolled code would evict a
// role's few instructions from the scheduler's instruction cache every stage
// (gate at M = 2048: 186 us with the roles spread over all schedulers, 180 us).
enum Role { kRoleCode0 = 0, kRoleCode1, kRoleX, kRoleMma, kRoleDequant, kRoleEpilogue };

struct GmBlock {
  int bits, n_ch, pos0, seg_off, grp_off;
  int kt0;  // first K tile of the block
};

struct GmParams {
  CUtensorMap tm_codes;  // packed [N][S] u8, box {kCodeBox, 128}
  CUtensorMap tm_meta;   // meta [N][meta_stride] u32, box {4, 128}
  CUtensorMap tm_w16;    // packed [N][S/2] u16, box {32, 128}, 64B swizzle
  GmBlock blk[POLYQ_MAX_BLOCKS];
  int n_blocks;
  int M, N, K, KT;  // KT: K tiles of BK
  int bk;           // 32 or 64
  int r_log2;       // rows of X per CTA and unit: 2^r_log2
  int units_m, units_n, ksplit, units;  // work units: (token tile, N tile, K split)
  int zero_col0;  // first column of Y that the pre-pass zeroes for a split of K
  int whole;    // units that one pair computes alone (all, or with streamk the first ones)
  int streamk;  // 1: each pair takes an equal contiguous range of (unit, K tile) pairs:
  int sk_share, sk_extra;  // sk_share of them, the first sk_extra pairs one more
  int has_meta;
  int prep_seg;     // gemm_prep_small: CTAs per row
  int prep_rows;    // gemm_prep_small: CTAs that gather rows (the others zero Y)
  const __nv_bfloat16* x;
  const int32_t* gather;
  const float* xscale;  // Section 3.4 activation factors (clustered order) or NULL
  __half* xg;
  float* rowscale;      // [M]: 2^e_m, the power of two row m of Xg was divided by
  float* y;
  int* status;
};

// ---------------------------------------------------------------------------
// CTA pairs
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t cluster_ctarank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t mapa(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release;\n barrier.cluster.wait.acquire;" ::: "memory");
}
// Arrive on a barrier of a CTA of the cluster (address from mapa).  With the
// default scope: what such an arrival announces (weights and X in this CTA's
// shared memory, drained tensor memory) reaches the other side only through
// the tensor core, which fence.proxy.async and the tcgen05 fences order (by the
// letter of the memory model the arrival would be at cluster scope too).  A
// release at cluster scope waits for all of the warp's memory traffic at every
// stage: gate at M = 2048 took 352 us with it and 281 us without.
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tmem_alloc2(uint32_t dst_smem, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst_smem),
               "r"(ncols)
               : "memory");
}
__device__ __forceinline__ void tmem_relinquish2() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc2(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols)
               : "memory");
}
// D[tmem of both CTAs] (+)= A * B^T over the pair's operands: descriptors are
// this CTA's, and the peer's operands lie at the same offsets.
__device__ __forceinline__ void tc_mma2_f16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc,
                                            uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d_tmem),
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// Arrive (once) on the barrier at this offset in both CTAs when all tcgen05
// operations issued so far by this thread have completed.
__device__ __forceinline__ void tc_commit2(uint32_t bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64"
      " [%0], %1;" ::"r"(bar),
      "h"((uint16_t)3)
      : "memory");
}

// try_wait that lets the hardware suspend the thread for up to `hint_ns`
// (it wakes when the phase completes) instead of returning at once.
__device__ __forceinline__ bool mbar_try_wait_hint(uint32_t bar, uint32_t parity,
                                                   uint32_t hint_ns) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n"
      " mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity), "r"(hint_ns)
      : "memory");
  return ok != 0;
}

// Bounded waits that also give up once another role of the pair has failed:
// 0 when the phase completed, 1 on a timeout, 2 when `abort` was raised.  The
// flag is read only after a poll has failed, so that a stage whose barrier
// has already completed costs one poll and no shared load.  The lone producer
// and MMA threads poll with a suspend hint of up to 1 us, so that their
// polling does not take issue slots from the dequantisation warps that share
// their schedulers: at most 2^22 such polls, a few seconds.
constexpr uint32_t kWaitLimitSleep = 1u << 22;
constexpr long long kAbortStayCycles = 1 << 21;  // a millisecond
constexpr uint32_t kSuspendHintNs = 1000;
constexpr int kWaitOk = 0, kWaitTimeout = 1, kWaitAborted = 2;
__device__ __forceinline__ int wait_ab(uint32_t bar, uint32_t parity, const volatile int* abort) {
  for (uint32_t it = 0; it < kWaitLimit; ++it) {
    if (mbar_try_wait(bar, parity)) return kWaitOk;
    if (*abort) return kWaitAborted;
  }
  return kWaitTimeout;
}
__device__ __forceinline__ int wait_sleep_ab(uint32_t bar, uint32_t parity,
                                             const volatile int* abort) {
  for (uint32_t it = 0; it < kWaitLimitSleep; ++it) {
    if (mbar_try_wait_hint(bar, parity, kSuspendHintNs)) return kWaitOk;
    if (*abort) return kWaitAborted;
  }
  return kWaitTimeout;
}

// The same without a way out but the limit.
__device__ __forceinline__ void mbar_wait_sleep(uint32_t bar, uint32_t parity, uint32_t limit) {
  for (uint32_t it = 0; it < limit && !mbar_try_wait_hint(bar, parity, kSuspendHintNs); ++it) {
  }
}

__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bit i: whether the phase of the i-th slot from `s` on, every STEP-th of N,
// has completed (parity `ph` up to the ring's end, the other after it).  A
// poll's answer takes 200 to 300 cycles here, behind the dequantisers' shared
// memory traffic, but polls follow each other every 15: a lone thread that
// polls B stages at once pays that latency once for all that are ready.
template <int B, int N, int STEP = 1>
__device__ __forceinline__ uint32_t poll_ahead(uint32_t bar0, int s, uint32_t ph) {
  static_assert((B - 1) * STEP < N, "one phase per slot");
  uint32_t ok = 0;
#pragma unroll
  for (int i = 0; i < B; ++i) {
    int k = s + i * STEP;
    uint32_t p = ph;
    if (k >= N) {
      k -= N;
      p ^= 1u;
    }
    ok |= (mbar_test(bar0 + 8 * k, p) ? 1u : 0u) << i;
  }
  return ok;
}
// Stages ready in a row.
__device__ __forceinline__ int leading(uint32_t ok) { return __ffs(~ok) - 1; }

// The pieces of work a CTA pair takes, in order: an output tile (um, un) and a
// range [kt_lo, kt_hi) of its K tiles.  Units are strided over the pairs, each
// with its K split's range; with `streamk`, units below `whole` are, and of the
// (unit, K tile) pairs of the others, in unit-major order, a CTA pair takes an
// equal contiguous share (to one), which cuts at most two units per pair short.
// Every role of both CTAs walks the same sequence.
template <bool WHOLE>  // the kernel takes whole units before a stream-K
struct Pieces {
  int g, g_hi;  // stream-K: (unit, K tile) pairs, g_hi -1 before them; else: unit
  __device__ __forceinline__ void init(const GmParams& P) {
    g = blockIdx.x >> 1;
    g_hi = -1;
    if (!WHOLE && P.streamk) share(P);
  }
  __device__ __forceinline__ void share(const GmParams& P) {
    const int b = blockIdx.x >> 1;
    g = (WHOLE ? P.whole * P.KT : 0) + b * P.sk_share + min(b, P.sk_extra);
    g_hi = g + P.sk_share + (b < P.sk_extra ? 1 : 0);
  }
  // After next(): the piece is one of several of its tile, to be added.
  __device__ __forceinline__ bool adds(const GmParams& P) const {
    return P.ksplit > 1 || (WHOLE ? g_hi >= 0 : P.streamk);
  }
  __device__ __forceinline__ bool next(const GmParams& P, int& um, int& un, int& kt_lo,
                                       int& kt_hi) {
    int uu, ks = 0;
    if (WHOLE ? g_hi < 0 && g < P.whole : !P.streamk) {
      if (g >= P.whole) return false;
      uu = g;
      g += gridDim.x >> 1;
      kt_lo = 0;
      kt_hi = P.KT;
    } else {
      if (WHOLE && g_hi < 0) {
        if (!P.streamk) return false;
        share(P);
      }
      if (g >= g_hi) return false;
      uu = g / P.KT;
      kt_lo = g - uu * P.KT;
      kt_hi = min(P.KT, kt_lo + (g_hi - g));
      g += kt_hi - kt_lo;
    }
    const int q = uu / P.units_m;
    um = uu - q * P.units_m;
    un = q;
    if (P.ksplit > 1) {
      ks = q / P.units_n;
      un = q - ks * P.units_n;
      kt_lo = ks * P.KT / P.ksplit;
      kt_hi = (ks + 1) * P.KT / P.ksplit;
    }
    return true;
  }
};

__device__ __forceinline__ int find_kblock(const GmBlock* blk, int nblk, int kt) {
  int b = 0;
  while (b + 1 < nblk && kt >= blk[b + 1].kt0) ++b;
  return b;
}

// The block of the current K tile with its fields in registers.  K tiles
// only increase within a piece, so after a seek at the piece's first tile the
// cursor advances with one comparison per tile instead of a search through
// the block table in shared memory.
struct BlockCursor {
  int bi, kt0, next_kt0, bits, seg_off, grp_off;
  __device__ __forceinline__ void load(const GmBlock* sblk, int nblk) {
    const GmBlock& B = sblk[bi];
    kt0 = B.kt0;
    bits = B.bits;
    seg_off = B.seg_off;
    grp_off = B.grp_off;
    next_kt0 = bi + 1 < nblk ? sblk[bi + 1].kt0 : 0x7FFFFFFF;
  }
  __device__ __forceinline__ void seek(const GmBlock* sblk, int nblk, int kt) {
    bi = find_kblock(sblk, nblk, kt);
    load(sblk, nblk);
  }
  __device__ __forceinline__ void advance(const GmBlock* sblk, int nblk, int kt) {
    while (kt >= next_kt0) {
      ++bi;
      load(sblk, nblk);
    }
  }
};

// Position inside a 32-code half group of the code that fills K slot `s`
// (0..31) of a tile: the halves of the decoder's pair s / 2 (2, 3 and 4 bits:
// the pair tables of the GEMV's decoder; 8 and 16 bits: natural order).
__host__ __device__ inline int slot_code(int bits, int s) {
  if (bits > 4) return s;
  const int gp = gv::group_pairs(bits), j = s >> 1;
  const gv::PairDef d = gv::pair_def(bits, j % gp);
  return (j / gp) * gv::group_units(bits) + ((s & 1) ? d.hi : d.lo);
}

// Shared copy of the block table and of slot_code for every width.
struct PrepTables {
  GmBlock blk[POLYQ_MAX_BLOCKS];
  alignas(8) uint8_t code[5][kSlots];
};
__device__ __forceinline__ int width_index(int bits) {
  return bits <= 4 ? bits - 2 : (bits == 8 ? 3 : 4);
}
__device__ __forceinline__ void load_blocks(const GmParams& P, GmBlock* sblk) {
  if (threadIdx.x < POLYQ_MAX_BLOCKS) {  // constant-offset parameter reads only
    switch (threadIdx.x) {
      case 0: sblk[0] = P.blk[0]; break;
      case 1: sblk[1] = P.blk[1]; break;
      case 2: sblk[2] = P.blk[2]; break;
      case 3: sblk[3] = P.blk[3]; break;
      default: sblk[4] = P.blk[4]; break;
    }
  }
}
__device__ __forceinline__ void load_tables(const GmParams& P, PrepTables* S) {
  load_blocks(P, S->blk);
  if (threadIdx.x < 5 * kSlots) {
    const int w = threadIdx.x / kSlots;
    const int bits = w < 3 ? w + 2 : (w == 3 ? 8 : 16);
    S->code[w][threadIdx.x % kSlots] = (uint8_t)slot_code(bits, threadIdx.x % kSlots);
  }
}

// ---------------------------------------------------------------------------
// pre-pass: Xg(m, k) = fp16(X[m][gather[p]] * xscale[p] * 2^-e_m), p the
// position that fills K slot k (slot_pos).
// ---------------------------------------------------------------------------
constexpr int kRowExp = 14;       // a row's largest magnitude becomes [2^14, 2^15)
constexpr int kRowExpMin = -126;  // 2^e stays a normal float
constexpr int kPrepThreads = 256;
constexpr int kPrepMaxSmem = 200 * 1024;
constexpr int kSmallOcts = 2;                 // 8-slot pieces per thread of gemm_prep_small
constexpr int kSmallMaxK = 32768;             // widest row it stages
// Most rows it is used for: 13824 x 5120 / 5120 x 13824 at M = 256 36.1 / 40.1
// us for the call, 37.1 / 45.8 with gemm_prep_rows; at M = 512 59.4 / 66.2 and
// 60.3 / 58.6.
constexpr int kSmallMaxM = 256;

// Element offset of Xg(m, k) in the blocked layout: block (m / R, k / 32) of
// R rows x 32 fp16, row m % R at 64 bytes each, its 16-byte chunks in the
// 64-byte swizzle (chunk index XOR bits 7..8 of the byte address).
__device__ __forceinline__ size_t xg_off(int m, int k, int kslots, int r_log2) {
  const int r = m & ((1 << r_log2) - 1), c = (k >> 3) & 3;
  return ((((size_t)(m >> r_log2) * kslots + (k >> 5)) << r_log2) + r) * kSlots +
         ((c ^ ((r >> 1) & 3)) << 3) + (k & 7);
}

// Clustered K slot k of a row: the position p it takes its value from, or -1
// past the end of a block.
__device__ __forceinline__ int slot_pos(const PrepTables& S, int nblk, int bk, int k) {
  const int kt = bk == 64 ? k >> 6 : k >> 5;
  const GmBlock& B = S.blk[find_kblock(S.blk, nblk, kt)];
  const int o = k - B.kt0 * bk;
  const int w = (o & ~(kSlots - 1)) + S.code[width_index(B.bits)][o & (kSlots - 1)];
  return w < B.n_ch ? B.pos0 + w : -1;
}

// Source channels (-1 past the end of the block) and, for a scaled layer,
// activation factors of the 8 slots from k on (k a multiple of 8: they lie in
// one block and half group, so that finding them takes 11 instructions a slot
// and not the 60 of slot_pos).
template <bool XS>
__device__ __forceinline__ void slot_sources(const GmParams& P, const PrepTables& S, int k,
                                             int (&src)[8], float (&fac)[8]) {
  const GmBlock& B = S.blk[find_kblock(S.blk, P.n_blocks, P.bk == 64 ? k >> 6 : k >> 5)];
  const int o = k - B.kt0 * P.bk;
  const uint2 c8 = *reinterpret_cast<const uint2*>(&S.code[width_index(B.bits)][o & (kSlots - 1)]);
  const int base = o & ~(kSlots - 1);
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const int w = base + (int)(((u < 4 ? c8.x : c8.y) >> (8 * (u & 3))) & 0xFFu);
    const int p = B.pos0 + w;
    const bool in = w < B.n_ch;
    src[u] = !in ? -1 : (P.gather ? __ldg(P.gather + p) : p);
    fac[u] = (XS && in) ? __ldg(P.xscale + p) : 0.f;
  }
}

// Y = 0 by CTA `cta` of `n_cta` (Y is 16-byte aligned).
template <bool COLS>  // perhaps only the columns from zero_col0 on
__device__ __forceinline__ void zero_y(const GmParams& P, int cta, int n_cta) {
  const int col0 = P.zero_col0;
  if (COLS && col0 > 0) {  // the columns from the first tile on that is added up
    const int w = P.N - col0;
    const bool vec = P.N % 4 == 0;
    const int cw = vec ? w / 4 : w;
    for (int m = cta; m < P.M; m += n_cta) {
      float* row = P.y + (size_t)m * P.N + col0;
      for (int c = threadIdx.x; c < cw; c += blockDim.x) {
        if (vec) reinterpret_cast<float4*>(row)[c] = make_float4(0.f, 0.f, 0.f, 0.f);
        else row[c] = 0.f;
      }
    }
    return;
  }
  const long long total = (long long)P.M * P.N, total4 = total / 4;
  for (long long e = (long long)cta * blockDim.x + threadIdx.x; e < total4;
       e += (long long)n_cta * blockDim.x)
    reinterpret_cast<float4*>(P.y)[e] = make_float4(0.f, 0.f, 0.f, 0.f);
  if (cta == 0 && threadIdx.x < (int)(total & 3)) P.y[total4 * 4 + threadIdx.x] = 0.f;
}

// e_m = floor(log2(max)) - kRowExp of a row whose largest magnitude has the
// fp32 bits mx, an fp32 subnormal maximum counting as 2^-127.  2^e and 2^-e
// are normal floats (-126 <= e <= 113), so the products with 2^-e are exact
// scalings (rounded like any product where they fall below the normal range).
__device__ __forceinline__ int row_exp(uint32_t mx) {
  return mx ? max((int)(mx >> 23) - 127 - kRowExp, kRowExpMin) : 0;
}
// Largest magnitudes of the low and of the high halves of eight bf16 (their bit
// patterns without the sign order as integers), and the larger of the two.
__device__ __forceinline__ uint32_t bf16x8_max(const uint4& v, uint32_t mx2) {
  constexpr uint32_t kAbs = 0x7FFF7FFFu;
  return __vmaxu2(__vmaxu2(__vmaxu2(mx2, v.x & kAbs), v.y & kAbs),
                  __vmaxu2(v.z & kAbs, v.w & kAbs));
}
__device__ __forceinline__ uint32_t max_halves(uint32_t mx2) {
  return max(mx2 & 0xFFFFu, mx2 >> 16);
}

// Many rows, RW (1, 2 or 4) at a time: a CTA stages RW rows of X in shared
// memory interleaved, one word of RW bf16 values per channel, and gathers from
// there, so that one index read and one word read serve RW values.  Bound by
// shared-memory wavefronts (62-75% of the pipe) and issue (60%); one row at a
// time, with an index, a value, a test and 64-bit address arithmetic per
// element, it was bound by 25 to 34 instructions an element.  K = 5120, M =
// 8192: 49 -> 37 us; K = 13824, M = 2048: 48 -> 31 us (cold cache).  16-byte
// pieces of RW words lie in planes, so that the staging stores of a warp are
// contiguous; the slot map holds positions in that layout and is built, from
// static layer data, before the wait for the previous kernel.
constexpr int kRowsThreads = 512;
constexpr int kRowsMaxK = 65520;  // staged positions and the zero word fit 16 bits

// Words (of RW bf16) per 16-byte piece.
template <int RW>
__host__ __device__ constexpr int piece_words() {
  return 8 / RW;
}
// Position of channel k among the staged words: the 8 channels of a 16-byte
// piece of X fill RW staged pieces, one in each of RW planes of n8.  The words
// after them, from 8 n8 on, are zero: the source of slots past a block's end.
template <int RW>
__device__ __forceinline__ uint32_t staged_pos(int k, int n8) {
  constexpr int PW = piece_words<RW>();
  return (uint32_t)(((k & 7) / PW * n8 + (k >> 3)) * PW + (k & (PW - 1)));
}
template <int RW>
__host__ __device__ constexpr size_t rows_smem(int K, int Kp, bool xscale) {
  return (size_t)((K + 7) / 8) * 16 * RW + 16 + (size_t)Kp * 2 + (xscale ? (size_t)Kp * 4 : 0);
}

template <int RW, bool XS>  // XS: scaled layer
__global__ void __launch_bounds__(kRowsThreads) gemm_prep_rows(const __grid_constant__ GmParams P) {
  extern __shared__ __align__(16) uint8_t psm[];
  constexpr int PW = piece_words<RW>();
  pdl_trigger();
  __shared__ PrepTables S;
  __shared__ uint32_t s_max[2][RW];
  load_tables(P, &S);
  if (threadIdx.x < 2 * RW) s_max[threadIdx.x / RW][threadIdx.x % RW] = 0;
  __syncthreads();
  const int Kp = P.KT * P.bk, ks = Kp / kSlots, n8 = (P.K + 7) / 8;
  uint4* s_x = reinterpret_cast<uint4*>(psm);
  uint16_t* s_map = reinterpret_cast<uint16_t*>(psm + (size_t)n8 * 16 * RW + 16);
  float* s_fac = reinterpret_cast<float*>(s_map + Kp);
  {
    for (int k = 8 * threadIdx.x; k < Kp; k += 8 * kRowsThreads) {
      int src[8];
      float fac[8];
      slot_sources<XS>(P, S, k, src, fac);
      uint32_t m[4];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const uint32_t v = src[u] < 0 ? 8u * n8 : staged_pos<RW>(src[u], n8);
        m[u >> 1] = (u & 1) ? m[u >> 1] | (v << 16) : v;
        if (XS) s_fac[k + u] = fac[u];
      }
      *reinterpret_cast<uint4*>(s_map + k) = make_uint4(m[0], m[1], m[2], m[3]);
    }
    if (threadIdx.x == 0) s_x[n8 * RW] = make_uint4(0u, 0u, 0u, 0u);
  }
  pdl_wait();  // X comes from the previous kernel; Y and the workspace may still be in use
  if (blockIdx.x == 0 && threadIdx.x == 0) *P.status = 0;
  if (P.ksplit > 1 || P.streamk) zero_y<true>(P, blockIdx.x, gridDim.x);
  const int lane = threadIdx.x & 31;
  const int Mp = P.units_m << (P.r_log2 + 1);  // rows past M are zero: their MMA columns must be finite
  const bool vec = (P.K & 7) == 0 && (reinterpret_cast<uintptr_t>(P.x) & 15) == 0;
  const uint16_t* x = reinterpret_cast<const uint16_t*>(P.x);
  int it = 0;
  for (int m0 = blockIdx.x * RW; m0 < Mp; m0 += gridDim.x * RW, it ^= 1) {
    uint32_t mx[RW];
#pragma unroll
    for (int r = 0; r < RW; ++r) mx[r] = 0;
    constexpr int U = 4 / RW;  // pieces of a thread in flight: four 16-byte loads
    for (int i0 = threadIdx.x; i0 < n8; i0 += U * kRowsThreads) {
      uint4 v[U][RW];  // 8 channels of each row
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int r = 0; r < RW; ++r) {
          const int i = i0 + u * kRowsThreads;
          v[u][r] = make_uint4(0u, 0u, 0u, 0u);
          if (m0 + r < P.M && i < n8) {
            const size_t o = (size_t)(m0 + r) * P.K + 8 * i;
            if (vec) {
              v[u][r] = __ldcg(reinterpret_cast<const uint4*>(x + o));
            } else {
              uint32_t e[8];
#pragma unroll
              for (int c = 0; c < 8; ++c) e[c] = 8 * i + c < P.K ? (uint32_t)__ldcg(x + o + c) : 0u;
              v[u][r] = make_uint4(e[0] | e[1] << 16, e[2] | e[3] << 16, e[4] | e[5] << 16,
                                   e[6] | e[7] << 16);
            }
          }
        }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int i = i0 + u * kRowsThreads;
        if (i >= n8) break;
        uint32_t w[RW][4];
#pragma unroll
        for (int r = 0; r < RW; ++r) {
          mx[r] = bf16x8_max(v[u][r], mx[r]);
          w[r][0] = v[u][r].x; w[r][1] = v[u][r].y; w[r][2] = v[u][r].z; w[r][3] = v[u][r].w;
        }
#pragma unroll
        for (int j = 0; j < RW; ++j) {  // piece j: channels j * PW.., row-fastest
          uint32_t o[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            if (RW == 1) {
              o[q] = w[0][q];
            } else {
              const int c = j * PW + (2 * q) / RW, r = (2 * q) % RW;
              o[q] = __byte_perm(w[r][c >> 1], w[r + (RW > 1)][c >> 1], (c & 1) ? 0x7632 : 0x5410);
            }
          }
          s_x[j * n8 + i] = make_uint4(o[0], o[1], o[2], o[3]);
        }
      }
    }
    if (!XS) {  // without factors the largest |X| of the raw row, as the gather is a permutation
#pragma unroll
      for (int r = 0; r < RW; ++r) {
        const uint32_t v = __reduce_max_sync(0xffffffffu, max_halves(mx[r])) << 16;  // bf16 -> fp32
        if (lane == 0) atomicMax(&s_max[it][r], v);
      }
    }
    __syncthreads();  // the rows (and, on the first pass, the map) are complete
    // the RW values of a slot
    auto values = [&](uint32_t pos, float (&v)[RW]) {
      if constexpr (RW == 4) {
        const uint2 a = reinterpret_cast<const uint2*>(s_x)[pos];
        v[0] = bf16_lo(a.x); v[1] = bf16_hi(a.x); v[2] = bf16_lo(a.y); v[3] = bf16_hi(a.y);
      } else if constexpr (RW == 2) {
        const uint32_t a = reinterpret_cast<const uint32_t*>(s_x)[pos];
        v[0] = bf16_lo(a); v[1] = bf16_hi(a);
      } else {
        v[0] = bf16_lo(reinterpret_cast<const uint16_t*>(s_x)[pos]);
      }
    };
    if (XS) {
#pragma unroll
      for (int r = 0; r < RW; ++r) mx[r] = 0;
      for (int k = threadIdx.x; k < Kp; k += kRowsThreads) {
        float v[RW];
        values(s_map[k], v);
#pragma unroll
        for (int r = 0; r < RW; ++r) mx[r] = max(mx[r], __float_as_uint(fabsf(v[r] * s_fac[k])));
      }
#pragma unroll
      for (int r = 0; r < RW; ++r) {
        const uint32_t v = __reduce_max_sync(0xffffffffu, mx[r]);
        if (lane == 0) atomicMax(&s_max[it][r], v);
      }
      __syncthreads();
    }
    float inv[RW];
#pragma unroll
    for (int r = 0; r < RW; ++r) {
      const int e = row_exp(s_max[it][r]);
      if ((int)threadIdx.x == r && m0 + r < P.M) P.rowscale[m0 + r] = __int_as_float((127 + e) << 23);
      inv[r] = __int_as_float((127 - e) << 23);
    }
    if (threadIdx.x < RW) s_max[it ^ 1][threadIdx.x] = 0;  // for the next pass
    // rows m0.. of one block of R rows: addresses as in xg_off
    __half* dst = P.xg + xg_off(m0, 0, ks, P.r_log2);  // its swizzle undone below
    const int r0 = m0 & ((1 << P.r_log2) - 1);
    dst -= ((r0 >> 1) & 3) << 3;
    for (int i = threadIdx.x; i < Kp / 4; i += kRowsThreads) {
      const uint2 mp = reinterpret_cast<const uint2*>(s_map)[i];
      const uint32_t pos[4] = {mp.x & 0xFFFFu, mp.x >> 16, mp.y & 0xFFFFu, mp.y >> 16};
      float v[4][RW];
#pragma unroll
      for (int e = 0; e < 4; ++e) values(pos[e], v[e]);
      if (XS) {
        const float4 f = reinterpret_cast<const float4*>(s_fac)[i];
        const float fac[4] = {f.x, f.y, f.z, f.w};
#pragma unroll
        for (int e = 0; e < 4; ++e)
#pragma unroll
          for (int r = 0; r < RW; ++r) v[e][r] *= fac[e];
      }
      const uint32_t at = ((uint32_t)(i >> 3) << (P.r_log2 + 5)) + 4 * (i & 1);
      const int c = (i >> 1) & 3;
#pragma unroll
      for (int r = 0; r < RW; ++r) {
        const __half2 a = __floats2half2_rn(v[0][r] * inv[r], v[1][r] * inv[r]);
        const __half2 b = __floats2half2_rn(v[2][r] * inv[r], v[3][r] * inv[r]);
        *reinterpret_cast<uint2*>(dst + at + (r * kSlots + ((c ^ (((r0 + r) >> 1) & 3)) << 3))) =
            make_uint2(*reinterpret_cast<const uint32_t*>(&a), *reinterpret_cast<const uint32_t*>(&b));
      }
    }
    __syncthreads();  // the staged rows are replaced by the next pass
  }
}

// Layers too wide to stage a row (see rows_smem): gathered from global memory.
__global__ void __launch_bounds__(kPrepThreads) gemm_prep_wide(const __grid_constant__ GmParams P) {
  pdl_trigger();
  __shared__ PrepTables S;
  __shared__ uint32_t s_wmax[kPrepThreads / 32];
  load_tables(P, &S);
  __syncthreads();
  const int Kp = P.KT * P.bk, ks = Kp / kSlots;
  pdl_wait();  // X comes from the previous kernel; Y and the workspace may still be in use
  if (blockIdx.x == 0 && threadIdx.x == 0) *P.status = 0;
  if (P.ksplit > 1 || P.streamk) zero_y<true>(P, blockIdx.x, gridDim.x);
  const int Mp = P.units_m << (P.r_log2 + 1);
  for (int m = blockIdx.x; m < Mp; m += gridDim.x) {
    auto value = [&](int k) -> float {  // at clustered slot k
      const int p = m < P.M ? slot_pos(S, P.n_blocks, P.bk, k) : -1;
      if (p < 0) return 0.f;
      const int src = P.gather ? __ldg(P.gather + p) : p;
      const uint16_t b = __ldcg(reinterpret_cast<const uint16_t*>(P.x) + (size_t)m * P.K + src);
      const float v = __uint_as_float((uint32_t)b << 16);
      return P.xscale ? v * __ldg(P.xscale + p) : v;
    };
    uint32_t mx = 0;
    for (int k = threadIdx.x; k < Kp; k += kPrepThreads)
      mx = max(mx, __float_as_uint(fabsf(value(k))));
    mx = __reduce_max_sync(0xffffffffu, mx);
    if ((threadIdx.x & 31) == 0) s_wmax[threadIdx.x >> 5] = mx;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < kPrepThreads / 32; ++w) mx = max(mx, s_wmax[w]);
    const int e = row_exp(mx);
    if (threadIdx.x == 0 && m < P.M) P.rowscale[m] = __int_as_float((127 + e) << 23);
    const float inv = __int_as_float((127 - e) << 23);
    for (int i = threadIdx.x; i < Kp / 2; i += kPrepThreads)
      *reinterpret_cast<__half2*>(P.xg + xg_off(m, 2 * i, ks, P.r_log2)) =
          __floats2half2_rn(value(2 * i) * inv, value(2 * i + 1) * inv);
    __syncthreads();  // s_wmax is reused by the next row
  }
}

// A few rows: prep_seg CTAs per row (of all rows of the token tiles), each
// gathering a segment of the row's slots, so that even one row is spread over
// the GPU; further CTAs zero Y.  Every CTA stages the whole row in shared
// memory and finds its largest magnitude itself.  A thread's gather indices
// (and factors) are loaded before the wait for the previous kernel.  Bound by
// latency and by the instructions of the slot look-up: with eight slots a look-
// up and 16-byte stores the call takes 25.8 instead of 28.1 us at 13824 x 5120,
// M = 96, 27.0 instead of 30.7 at 5120 x 13824.
template <bool XS>
__global__ void __launch_bounds__(kPrepThreads) gemm_prep_small(const __grid_constant__ GmParams P) {
  extern __shared__ __align__(16) uint8_t psm[];
  pdl_trigger();
  if ((int)blockIdx.x >= P.prep_rows) {
    pdl_wait();  // Y may still be in use
    zero_y<false>(P, (int)blockIdx.x - P.prep_rows, (int)gridDim.x - P.prep_rows);
    return;
  }
  __shared__ PrepTables S;
  __shared__ uint32_t s_wmax[kPrepThreads / 32];
  load_tables(P, &S);
  __syncthreads();
  const int m = blockIdx.x / P.prep_seg, seg = blockIdx.x % P.prep_seg;
  const int octs = P.KT * P.bk / 8, ks = P.KT * P.bk / kSlots;
  const int o_lo = (int)((long long)seg * octs / P.prep_seg);
  const int o_hi = (int)((long long)(seg + 1) * octs / P.prep_seg);
  int src[kSmallOcts][8];
  float fac[kSmallOcts][8];
#pragma unroll
  for (int u = 0; u < kSmallOcts; ++u) {
    const int i = o_lo + u * kPrepThreads + threadIdx.x;
    if (i < o_hi && m < P.M) slot_sources<XS>(P, S, 8 * i, src[u], fac[u]);
  }
  pdl_wait();  // X comes from the previous kernel; the workspace may still be in use
  if (blockIdx.x == 0 && threadIdx.x == 0) *P.status = 0;
  if (m >= P.M) {  // a row that pads the token tile: its MMA columns must be finite
    for (int i = o_lo + threadIdx.x; i < o_hi; i += kPrepThreads)
      *reinterpret_cast<uint4*>(P.xg + xg_off(m, 8 * i, ks, P.r_log2)) = make_uint4(0u, 0u, 0u, 0u);
    return;
  }
  const uint16_t* s_row = reinterpret_cast<const uint16_t*>(psm);
  const uint16_t* row = reinterpret_cast<const uint16_t*>(P.x) + (size_t)m * P.K;
  uint32_t mx = 0;
  if ((P.K & 7) == 0 && (reinterpret_cast<uintptr_t>(row) & 15) == 0) {
    constexpr int U = 4;  // a thread's 16-byte loads in flight
    const int n8 = P.K / 8;
    for (int i0 = threadIdx.x; i0 < n8; i0 += U * kPrepThreads) {
      uint4 v[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int i = i0 + u * kPrepThreads;
        v[u] = i < n8 ? __ldcg(reinterpret_cast<const uint4*>(row) + i) : make_uint4(0u, 0u, 0u, 0u);
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int i = i0 + u * kPrepThreads;
        if (i < n8) reinterpret_cast<uint4*>(psm)[i] = v[u];
        mx = bf16x8_max(v[u], mx);
      }
    }
  } else {
    for (int i = threadIdx.x; i < P.K; i += kPrepThreads) {
      const uint16_t v = __ldcg(row + i);
      reinterpret_cast<uint16_t*>(psm)[i] = v;
      mx = max(mx, (uint32_t)(v & 0x7FFFu));
    }
  }
  mx = max_halves(mx) << 16;  // bf16 magnitude bits -> fp32 bits
  __syncthreads();
  if (XS) {  // the largest |x * t| over the whole row
    mx = 0;
    for (int p = threadIdx.x; p < P.K; p += kPrepThreads) {
      const int c = P.gather ? __ldg(P.gather + p) : p;
      mx = max(mx, __float_as_uint(fabsf(__uint_as_float((uint32_t)s_row[c] << 16) *
                                         __ldg(P.xscale + p))));
    }
  }
  mx = __reduce_max_sync(0xffffffffu, mx);
  if ((threadIdx.x & 31) == 0) s_wmax[threadIdx.x >> 5] = mx;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < kPrepThreads / 32; ++w) mx = max(mx, s_wmax[w]);
  const int e = row_exp(mx);
  if (seg == 0 && threadIdx.x == 0) P.rowscale[m] = __int_as_float((127 + e) << 23);
  const float inv = __int_as_float((127 - e) << 23);
#pragma unroll
  for (int u = 0; u < kSmallOcts; ++u) {
    const int i = o_lo + u * kPrepThreads + threadIdx.x;
    if (i >= o_hi) break;
    uint32_t w[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      float v[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int c = src[u][2 * q + h];
        const float x = c < 0 ? 0.f : __uint_as_float((uint32_t)s_row[c] << 16);
        v[h] = (XS ? x * fac[u][2 * q + h] : x) * inv;
      }
      const __half2 p = __floats2half2_rn(v[0], v[1]);
      w[q] = *reinterpret_cast<const uint32_t*>(&p);
    }
    *reinterpret_cast<uint4*>(P.xg + xg_off(m, 8 * i, ks, P.r_log2)) =
        make_uint4(w[0], w[1], w[2], w[3]);
  }
}

// ---------------------------------------------------------------------------
// dequantisation of one weight row of one tile into the swizzled A operand
// ---------------------------------------------------------------------------
__device__ __forceinline__ void red_add_f32(float* p, float a) {
  asm volatile("red.global.add.f32 [%0], %1;" ::"l"(p), "f"(a) : "memory");
}

__device__ __forceinline__ __half2 half2_bits(uint32_t v) {
  return *reinterpret_cast<const __half2*>(&v);
}
// fp16 bits of 2^-p and of -1024 * 2^-p (0 <= p <= 8)
__host__ __device__ constexpr uint32_t h_pow2(int p) { return (uint32_t)(15 - p) << 10; }
__host__ __device__ constexpr uint32_t h_neg_magic(int p) {
  return 0x8000u | ((uint32_t)(25 - p) << 10);
}

// Dequantise the 32 codes of a half group (w: its code words, from the first
// code's bit 0) into the 16 fp16 pairs of an operand row.  A code pair is cut out of the
// stream as two fp16 values 1024 + q * 2^p with one LOP3 (the GEMV decoder's
// windows); an FMA by 2^-p with -(1024 * 2^-p + z) gives q - z exactly (every
// intermediate is an integer or a short binary fraction of at most 11 bits),
// and the product with s is rounded once to fp16.  Three instructions a pair
// and seven window shifts per 32 codes at 3 bits, instead of six a pair with
// every code shifted to bit 0.
template <int BITS>
__device__ __forceinline__ void dequant_half(const uint32_t* w, __half2 zz, __half2 ss,
                                             uint32_t magic, uint32_t* p) {
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    __half2 d;
    if constexpr (BITS == 8) {
      const uint32_t v = __byte_perm(w[j >> 1], 0x64646464u, (j & 1) ? 0x4342 : 0x4140);
      d = __hadd2(half2_bits(v), __hsub2(half2_bits(h_neg_magic(0) * 0x10001u), zz));
    } else {
      const gv::PairDef pd = gv::pair_def(BITS, j % gv::group_pairs(BITS));
      const uint32_t v = gv::make_pair<BITS>(w, j, magic);
      const uint32_t mul = h_pow2(pd.plo) | (h_pow2(pd.phi) << 16);
      const uint32_t neg = h_neg_magic(pd.plo) | (h_neg_magic(pd.phi) << 16);
      d = __hfma2(half2_bits(v), half2_bits(mul), __hsub2(half2_bits(neg), zz));
    }
    const __half2 q = __hmul2(d, ss);
    p[j] = *reinterpret_cast<const uint32_t*>(&q);
  }
}

template <int V>
struct IntC {
  static constexpr int value = V;
};

// Shared memory by 32-bit address (the tile pointers, aligned by hand, are
// generic to the compiler, and generic accesses cost it 64-bit arithmetic).
__device__ __forceinline__ uint32_t lds32(uint32_t a) {
  uint32_t v;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ void lds128(uint32_t a, uint32_t* v) {
  asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
               : "r"(a)
               : "memory");
}
__device__ __forceinline__ void sts128(uint32_t a, const uint32_t* v) {
  asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};" ::"r"(a), "r"(v[0]), "r"(v[1]), "r"(v[2]),
               "r"(v[3])
               : "memory");
}

// The code words of a tile row in registers, from the first code's bit 0: the
// codes start `off` bytes (uniform over the CTA) into the row's box row at
// address `a`: at 0 or (3 bits) 8 for a tile of 64, also at 4 or 12 for one of
// 32.  An 8-bit tile of 64 has a second box, read by the caller.
template <int BITS, int HALVES>
struct CodeWords {
  static constexpr int N = BITS == 8 ? 8 : BITS * HALVES;
  uint32_t w[N];
  __device__ __forceinline__ void load(uint32_t a, int off) {
    constexpr bool kShift = BITS == 3 || (BITS == 2 && HALVES == 1);
    uint32_t cw[8];
    lds128(a, cw);
    if (kShift || N > 4) lds128(a + 16, cw + 4);
    const int sh = kShift ? off >> 2 : 0;
#pragma unroll
    for (int k = 0; k < N; ++k) {
      uint32_t v = cw[k];
      if (kShift) v = sh >= 2 ? cw[k + 2] : v;
      if (BITS == 3 && HALVES == 1) {
        const uint32_t o = sh >= 2 ? cw[k + 3] : cw[k + 1];
        v = (sh & 1) ? o : v;
      }
      w[k] = v;
    }
  }
};

#ifdef POLYQ_DEBUG
// Debug build only: every fp16 weight the dequantisers (or, for 16-bit
// blocks, TMA) place in an A tile is written to g_dbg_w[n][position] (the
// layer's clustered order), read back from the swizzled tile.
__device__ uint16_t* g_dbg_w;
__device__ long long g_dbg_wK;

// Half tile `tile` holds the block's half group hg.
__device__ __forceinline__ void dbg_row(const uint8_t* tile, int r, int n, int N,
                                        const GmBlock& B, int hg) {
  uint16_t* out = g_dbg_w;
  if (!out || n >= N) return;
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const uint16_t* src =
        reinterpret_cast<const uint16_t*>(tile + r * 64 + ((c ^ ((r >> 1) & 3)) << 4));
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const int w = 32 * hg + slot_code(B.bits, 8 * c + e);
      if (w < B.n_ch) out[(long long)n * g_dbg_wK + B.pos0 + w] = src[e];
    }
  }
}
#endif

// One chunk of 32 accumulator columns (tokens m0.., lane j holding token j's
// row scale) of the warp's 32 output columns into Y: v * 2^e_m, stored or
// (split K) added.  Nothing here depends from token to token (a token's
// address is one multiply), because a warp runs this alone and waits out
// every dependent instruction: with a running 64-bit pointer and a test per
// token the chunk took 2500 cycles whatever the number of warps, now 1100.
template <bool ADD>
__device__ __forceinline__ void store_chunk(float* __restrict__ y, uint32_t N, bool ok, int jn,
                                            const uint32_t (&v)[32], float rs_l) {
  float f[32];
#pragma unroll
  for (int j = 0; j < 32; ++j)
    f[j] = __uint_as_float(v[j]) * __shfl_sync(0xffffffffu, rs_l, j);
  if (!ok) return;
  if (jn == 32) {
#pragma unroll
    for (int j = 0; j < 32; ++j) {
      float* dst = y + (size_t)N * (uint32_t)j;
      if (ADD) red_add_f32(dst, f[j]);
      else *dst = f[j];
    }
  } else {
#pragma unroll
    for (int j = 0; j < 32; ++j) {
      float* dst = y + (size_t)N * (uint32_t)j;
      if (j < jn) {
        if (ADD) red_add_f32(dst, f[j]);
        else *dst = f[j];
      }
    }
  }
}

// What bounds it, by token tile (13824 x 5120 at B = 3, one call): with 512
// tokens the tensor core: a stage of 32 K takes the MMAs' 512 cycles (8192
// multiply-adds a cycle and pair; traced to 1%), an accumulator drain 9400
// cycles per 95000 of a unit (M = 2048: 277 -> 171 us; M = 4096: 529 -> 349 us,
// 1660 TFLOP/s).  With 256 and fewer the latency
// of a stage of 64 K through its rings, 440 to 590 cycles (M = 256: 53.6 -> 37
// us, M = 96: 54 -> 28 us, M = 16: 53 -> 24 us): the arrival at the leader
// (1300 cycles of a weight slot's turn of 2640), the commit back (400), and
// dequantisation; the copy of 128 code rows and 128 meta rows takes 325 cycles
// of the TMA unit (a row a cycle, 32 bytes across a 32-byte boundary two).  "Before" is one CTA per tile of 256 x 256
// whatever M, which dequantised every weight once per SM and 256 tokens.
template <class C>
__global__ void __launch_bounds__(C::kThreads, 1) gemm_main(const __grid_constant__ GmParams P,
                                                            uint32_t magic) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  // 1024-byte alignment of the operand tiles; both CTAs of the pair have the
  // same layout, so the offsets agree, as the MMA's descriptors need
  uint8_t* smem = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint8_t* smem_codes = smem + C::kCodeOff;
  __shared__ uint64_t bar_cfull[C::CODES];  // a code slot's copies have landed
  __shared__ uint64_t bar_cfree[C::CODES];  // its dequantisers hold the codes in registers
  __shared__ uint64_t bar_xfull[C::XS];     // a token slot's copy has landed (leader: both CTAs')
  __shared__ uint64_t bar_xfree[C::XS];     // its MMAs are done
  __shared__ uint64_t bar_bready[C::OPS];   // leader: both CTAs' weights are in place
  __shared__ uint64_t bar_sfree[C::OPS];    // a weight slot's MMAs are done
  __shared__ uint64_t bar_w16[C::OPS];      // a weight slot's tile of fp16 weights has landed
  __shared__ uint64_t bar_accf[C::NBUF];    // an accumulator is complete
  __shared__ uint64_t bar_acce[C::NBUF];    // leader: both CTAs have drained it
  __shared__ uint64_t bar_done;             // every MMA is done (both CTAs wait for it)
  __shared__ uint32_t tmem_base_slot;
  __shared__ GmBlock sblk[POLYQ_MAX_BLOCKS];
  __shared__ volatile int s_abort;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  const int role = warp >= C::kEpiWarp ? kRoleEpilogue : (warp & 3) == 0 ? warp >> 2 : kRoleDequant;

  load_blocks(P, sblk);
  if (threadIdx.x == 0) {
    s_abort = 0;
    for (int s = 0; s < C::CODES; ++s) {
      mbar_init(smem_u32(&bar_cfull[s]), 1);
      mbar_init(smem_u32(&bar_cfree[s]), C::kDqGroup);
    }
    for (int s = 0; s < C::OPS; ++s) {
      mbar_init(smem_u32(&bar_bready[s]), 2 * C::kDqGroup);  // a group of each CTA
      mbar_init(smem_u32(&bar_sfree[s]), 1);
      mbar_init(smem_u32(&bar_w16[s]), 1);
    }
    for (int s = 0; s < C::XS; ++s) {
      mbar_init(smem_u32(&bar_xfull[s]), rank == 0 ? 2 : 1);  // the producer; the peer's relay
      mbar_init(smem_u32(&bar_xfree[s]), 1);
    }
    for (int b = 0; b < C::NBUF; ++b) {
      mbar_init(smem_u32(&bar_accf[b]), 1);
      mbar_init(smem_u32(&bar_acce[b]), 2 * C::EPI);
    }
    mbar_init(smem_u32(&bar_done), 1);
    mbar_fence_init();
  }
  // one warp of each CTA of the pair allocates, and later frees, for the pair
  if (role == kRoleMma) {
    tmem_alloc2(smem_u32(&tmem_base_slot), kTmemCols);
    tmem_relinquish2();
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync();  // the peer's barriers are initialised too
  tc_fence_after();
  const uint32_t tmem = tmem_base_slot;
  pdl_trigger();

  const int nblk = P.n_blocks;
  // A role gives up.  Then nobody waits for the copies of X in the leader and
  // those of fp16 weights: by staying a thousand times their own time it keeps
  // both CTAs, which leave together.  (Waits by the roles that asked for them,
  // or a test at the kernel's end, cost every call 0.1 us.)
  auto fail = [&](int code) {
    s_abort = 1;
    const uint32_t peer = mapa(smem_u32((const void*)&s_abort), rank ^ 1u);
    asm volatile("st.relaxed.cluster.shared::cluster.u32 [%0], %1;" ::"r"(peer), "r"(1) : "memory");
    atomicExch(P.status, code);
    for (const long long t0 = clock64(); clock64() - t0 < kAbortStayCycles;) __nanosleep(1000);
  };
  Pieces<C::kWhole> pc;
  pc.init(P);
  int um, un, kt_lo, kt_hi;
  BlockCursor B;

  if (role <= kRoleCode1) {
    // ---------------- code producers: stages k with k % kCodeProd == role ----------------
    // The packed weights do not depend on earlier kernels, so these copies
    // start before the pre-pass is done.
    if (elect_one()) {
      prefetch_tmap(&P.tm_codes);
      if (P.has_meta) prefetch_tmap(&P.tm_meta);
      constexpr int kAhead = C::CODES / C::kCodeProd / 2;  // stages polled at once
      int kg = 0, last = -1;  // stages before this piece; last stage issued
      int s = role, free = 0;
      uint32_t ph = 1;  // a fresh barrier's parity-1 phase counts as complete
      while (!s_abort && pc.next(P, um, un, kt_lo, kt_hi)) {
        B.seek(sblk, nblk, kt_lo);
        const int n_row = un * kRowsN + (int)rank * kRowsCta;
        int kt = kt_lo + (role + C::kCodeProd - kg % C::kCodeProd) % C::kCodeProd;
        for (; kt < kt_hi; kt += C::kCodeProd) {
          if (free == 0) {
            free = leading(poll_ahead<kAhead, C::CODES, C::kCodeProd>(smem_u32(&bar_cfree[0]), s, ph));
            if (free == 0) {
              const int w = wait_sleep_ab(smem_u32(&bar_cfree[s]), ph, &s_abort);
              if (w != kWaitOk) {
                if (w == kWaitTimeout) fail(kStatusTimeoutEmpty);
                break;
              }
              free = 1;
            }
          }
          --free;
          B.advance(sblk, nblk, kt);
          const uint32_t bar = smem_u32(&bar_cfull[s]);
          if (B.bits == 16) {  // no codes: the weights go straight to the weight slot
            mbar_arrive(bar);
          } else {
            const uint32_t st = smem_u32(smem_codes + s * C::kCode);
            const int tb = kt - B.kt0;  // tile of the block
            const int boxes = B.bits == 8 ? C::HALVES : 1;
            const int start = B.seg_off + (C::BK / 8) * B.bits * tb;
            mbar_expect_tx(bar, boxes * kBoxBytes + kMetaBytes);
            tma_load_2d(st, &P.tm_codes, start & ~15, n_row, bar);
            if (boxes == 2) tma_load_2d(st + kBoxBytes, &P.tm_codes, start + kCodeBox, n_row, bar);
            tma_load_2d(st + C::kCodes, &P.tm_meta, (B.grp_off + tb * C::BK / 64) & ~3, n_row, bar);
          }
          last = kg + (kt - kt_lo);
          s += C::kCodeProd;
          if (s >= C::CODES) {
            s -= C::CODES;
            ph ^= 1u;
          }
        }
        kg += kt_hi - kt_lo;
      }
      // wait (bounded) for the copies still in flight: only a slot's last use,
      // whose phase no other producer has moved on
      for (int k = last; k >= 0 && k > (s_abort ? last : kg - 1) - C::CODES; k -= C::kCodeProd)
        mbar_wait(smem_u32(&bar_cfull[k % C::CODES]), (k / C::CODES) & 1);
    }
  } else if (role == kRoleX) {
    // ---------------- X producer ----------------
    if (elect_one()) {
      pdl_wait();  // Xg comes from the pre-pass
      constexpr int kAhead = C::XS / 2;
      int k = 0, s = 0, free = 0;
      uint32_t ph = 1;
      while (!s_abort && pc.next(P, um, un, kt_lo, kt_hi)) {
        const __half* xg = P.xg + (size_t)(um * 2 + (int)rank) * P.KT * (C::BK * C::R);
        for (int kt = kt_lo; kt < kt_hi; ++kt, ++k) {
          if (free == 0) {
            free = leading(poll_ahead<kAhead, C::XS>(smem_u32(&bar_xfree[0]), s, ph));
            if (free == 0) {
              const int w = wait_sleep_ab(smem_u32(&bar_xfree[s]), ph, &s_abort);
              if (w != kWaitOk) {
                if (w == kWaitTimeout) fail(kStatusTimeoutEmpty);
                break;
              }
              free = 1;
            }
          }
          --free;
          // this CTA's tokens: one contiguous block of Xg, already swizzled
          const uint32_t bar = smem_u32(&bar_xfull[s]);
          mbar_expect_tx(bar, C::kX);
          bulk_load(smem_u32(smem + C::kXOff + s * C::kX), xg + (size_t)kt * (C::BK * C::R), C::kX,
                    bar);
          if (++s == C::XS) {
            s = 0;
            ph ^= 1u;
          }
        }
      }
      if (rank != 0)  // copies still in flight (the leader's MMA thread waits for its own)
        for (int j = max(0, k - C::XS); j < k; ++j)
          mbar_wait(smem_u32(&bar_xfull[j % C::XS]), (j / C::XS) & 1);
    }
  } else if (role == kRoleMma && rank != 0) {
    // ---------------- X relay (second CTA) ----------------
    // Tells the leader's MMA thread that this CTA's X of a stage has landed.
    if (elect_one()) {
      const uint32_t xfull0 = mapa(smem_u32(&bar_xfull[0]), 0);
      constexpr int kAhead = C::XS / 2;
      int s = 0, ready = 0;
      uint32_t ph = 0;
      while (!s_abort && pc.next(P, um, un, kt_lo, kt_hi)) {
        for (int kt = kt_lo; kt < kt_hi; ++kt) {
          if (ready == 0) {
            ready = leading(poll_ahead<kAhead, C::XS>(smem_u32(&bar_xfull[0]), s, ph));
            if (ready == 0) {
              const int w = wait_sleep_ab(smem_u32(&bar_xfull[s]), ph, &s_abort);
              if (w != kWaitOk) {
                if (w == kWaitTimeout) fail(kStatusTimeoutFull);
                break;
              }
              ready = 1;
            }
          }
          --ready;
          mbar_arrive_cluster(xfull0 + 8 * s);
          if (++s == C::XS) {
            s = 0;
            ph ^= 1u;
          }
        }
      }
      // The leader's commits arrive in this CTA's shared memory too, where no
      // role waits for those of the last stages: stay for the last of all.
      mbar_wait_sleep(smem_u32(&bar_done), 0, kWaitLimitSleep);
    }
  } else if (role == kRoleMma) {
    // ---------------- MMA issuer (leader CTA) ----------------
    if (elect_one()) {
      constexpr int kAhead = C::OPS / 2;
      int uc = 0, s = 0, xs = 0, ready = 0;
      uint32_t ph = 0, xph = 0;
      const uint64_t da0 = umma_desc_sw64(smem_u32(smem));
      const uint64_t dx0 = umma_desc_sw64(smem_u32(smem + C::kXOff));
      for (; !s_abort && pc.next(P, um, un, kt_lo, kt_hi); ++uc) {
        const int buf = uc % C::NBUF;
        if (uc >= C::NBUF) {
          const int w =
              wait_sleep_ab(smem_u32(&bar_acce[buf]), (uc / C::NBUF - 1) & 1, &s_abort);
          if (w != kWaitOk) {
            if (w == kWaitTimeout) fail(kStatusTimeoutEmpty);
            break;
          }
        }
        tc_fence_after();
        const uint32_t acc = tmem + buf * (C::NACC * C::TN);
        for (int kt = kt_lo; kt < kt_hi; ++kt) {
          if (ready == 0) {
            ready = leading(poll_ahead<kAhead, C::OPS>(smem_u32(&bar_bready[0]), s, ph) &
                            poll_ahead<kAhead, C::XS>(smem_u32(&bar_xfull[0]), xs, xph));
            if (ready == 0) {
              int w = wait_sleep_ab(smem_u32(&bar_bready[s]), ph, &s_abort);
              if (w == kWaitOk) w = wait_sleep_ab(smem_u32(&bar_xfull[xs]), xph, &s_abort);
              if (w != kWaitOk) {
                if (w == kWaitTimeout) fail(kStatusTimeoutFull);
                break;
              }
              ready = 1;
            }
          }
          --ready;
          tc_fence_after();
          // A: the pair's 256 weight rows; B: accumulator a's TN tokens.  The
          // slots' descriptors are those of slot 0 plus an offset (>> 4).
          const uint64_t da = da0 + (uint64_t)((s * C::kA) >> 4);
          const uint64_t dx = dx0 + (uint64_t)((xs * C::kX) >> 4);
#pragma unroll
          for (int a = 0; a < C::NACC; ++a)
#pragma unroll
            for (int kk = 0; kk < C::BK / 16; ++kk)
              tc_mma2_f16(acc + a * C::TN,
                          da + (uint64_t)((kk / 2) * (kHalfTile >> 4) + 2 * (kk & 1)),
                          dx + (uint64_t)((kk / 2) * ((C::R * 64) >> 4) + a * ((C::TN / 2 * 64) >> 4) +
                                          2 * (kk & 1)),
                          C::kIdesc, (kt > kt_lo || kk > 0) ? 1u : 0u);
          tc_commit2(smem_u32(&bar_sfree[s]));
          tc_commit2(smem_u32(&bar_xfree[xs]));
          if (++s == C::OPS) {
            s = 0;
            ph ^= 1u;
          }
          if (++xs == C::XS) {
            xs = 0;
            xph ^= 1u;
          }
        }
        tc_commit2(smem_u32(&bar_accf[buf]));
      }
      // the pair's shared and tensor memory stay in use until the last MMA is done
      tc_commit2(smem_u32(&bar_done));
      mbar_wait(smem_u32(&bar_done), 0);
    }
  } else if (role == kRoleDequant) {
    // ---------------- dequantisation ----------------
    // Group g takes the stages k with k % GROUPS == g, thread r of the group
    // weight row r of the CTA.  (Copies may land out of order, and a parity
    // wait cannot tell a phase from the last but one: a code slot always
    // belongs to one group, as GROUPS divides CODES.  For the same reason no
    // barrier of the group may get two phases ahead of a warp that still waits
    // there.  cfull, sfree and w16 of a slot cannot: the slot's next use
    // needs its MMAs, so an arrival of every warp of the group after its wait.
    // One w16 barrier for a group's two slots could: with the other slot free,
    // the warp that asks for the copies passes stage j and completes stage
    // j + GROUPS on it while another warp has still to look at stage j.)
    const int dq = (warp >> 2) * 3 + (warp & 3) - 1;  // 0..11
    constexpr int RW = C::kDqRows, kRowStep = 32 * C::kDqGroup;
    const int grp = dq / C::kDqGroup;
    const int r = dq % C::kDqGroup * 32 + lane;  // the thread's rows: r, r + kRowStep
    const uint32_t code_row = smem_u32(smem_codes) + r * kCodeBox;
    const uint32_t meta_row = smem_u32(smem_codes) + C::kCodes + r * 16;
    // 16-byte chunk c of operand row r lies at (c XOR bits 7..8 of the row's
    // address) under the 64-byte swizzle
    const uint32_t op_row = smem_u32(smem) + r * 64 + (((r >> 1) & 3) << 4);
    const uint32_t bready0 = mapa(smem_u32(&bar_bready[0]), 0);  // the leader's
    int sc = grp, s = grp;  // code and weight slot of the group's next stage
    uint32_t cph = 0, sph = 1;
    uint32_t w16_ph = 0;  // bit s: parity of slot s's next fp16 tile
    int skip = grp;  // stages until the group's next one
    while (!s_abort && pc.next(P, um, un, kt_lo, kt_hi)) {
      B.seek(sblk, nblk, kt_lo);
      int kt = kt_lo + skip;
      for (; kt < kt_hi; kt += C::GROUPS) {
        int w = wait_ab(smem_u32(&bar_cfull[sc]), cph, &s_abort);
        if (w != kWaitOk) {
          if (w == kWaitTimeout) fail(kStatusTimeoutFull);
          break;
        }
        // polled once while the codes are on their way to registers; the slot
        // is waited for only before the stores
        const bool free = mbar_test(smem_u32(&bar_sfree[s]), sph);
        B.advance(sblk, nblk, kt);
        const int tb = kt - B.kt0;
        bool early = false;  // the code slot has been released
        const uint32_t op = op_row + s * C::kA;
        const uint32_t codes = code_row + sc * C::kCode;
        auto dequant = [&](auto bits) {
          constexpr int BITS = decltype(bits)::value;
          const uint32_t ma = meta_row + sc * C::kCode + ((B.grp_off + tb * C::BK / 64) & 3) * 4;
          const int off = (B.seg_off + (C::BK / 8) * BITS * tb) & 15;
          CodeWords<BITS, C::HALVES> cw[RW];
          __half2 ss[RW], zz[RW];
#pragma unroll
          for (int i = 0; i < RW; ++i) {
            const uint32_t meta = lds32(ma + i * kRowStep * 16);
            cw[i].load(codes + i * kRowStep * kCodeBox, off);
            const __half s16 = __ushort_as_half((uint16_t)(meta & 0xFFFFu));
            const __half z16 = __ushort_as_half((uint16_t)(meta >> 16));
            ss[i] = __halves2half2(s16, s16);
            zz[i] = __halves2half2(z16, z16);
          }
#pragma unroll 1  // one copy of the code for both halves
          for (int h = 0;;) {
            uint32_t p[RW][16];
#pragma unroll
            for (int i = 0; i < RW; ++i) dequant_half<BITS>(cw[i].w, zz[i], ss[i], magic, p[i]);
            if (h == 0 && !free) {
              w = wait_ab(smem_u32(&bar_sfree[s]), sph, &s_abort);
              if (w != kWaitOk) break;
            }
#pragma unroll
            for (int i = 0; i < RW; ++i)
#pragma unroll
              for (int c = 0; c < 4; ++c)
                sts128((op + h * kHalfTile + i * kRowStep * 64) ^ (c << 4), p[i] + 4 * c);
            if (++h == C::HALVES) break;
            if constexpr (BITS != 8) {
              // every code word is in registers (the stores above follow the
              // reads in the shared-memory pipe): the slot is free half a tile
              // early, which the ring of six needs (its turn, 2930 cycles with
              // the slot held to the tile's end, set the stage)
              __syncwarp();
              if (lane == 0) mbar_arrive(smem_u32(&bar_cfree[sc]));
              early = true;
            }
#pragma unroll
            for (int i = 0; i < RW; ++i) {
              if constexpr (BITS == 8) {
                cw[i].load(codes + kBoxBytes + i * kRowStep * kCodeBox, 0);
              } else if constexpr (C::HALVES == 2) {
#pragma unroll
                for (int k = 0; k < BITS; ++k) cw[i].w[k] = cw[i].w[k + BITS];
              }
            }
          }
          fence_proxy_async_smem();
        };
        switch (B.bits) {
          case 2: dequant(IntC<2>()); break;
          case 3: dequant(IntC<3>()); break;
          case 4: dequant(IntC<4>()); break;
          case 8: dequant(IntC<8>()); break;
          default:  // fp16 weights: copied straight into the weight slot
            if (!free) w = wait_ab(smem_u32(&bar_sfree[s]), sph, &s_abort);
            if (w != kWaitOk) break;
            if (r == 0) {
              const uint32_t bar = smem_u32(&bar_w16[s]);
              mbar_expect_tx(bar, C::kA);
#pragma unroll
              for (int h = 0; h < C::HALVES; ++h)
                tma_load_2d(smem_u32(smem) + s * C::kA + h * kHalfTile, &P.tm_w16,
                            B.seg_off / 2 + C::BK * tb + kSlots * h,
                            un * kRowsN + (int)rank * kRowsCta, bar);
            }
            w = wait_ab(smem_u32(&bar_w16[s]), (w16_ph >> s) & 1u, &s_abort);
            w16_ph ^= 1u << s;
            break;
        }
        if (w != kWaitOk) {
          if (w == kWaitTimeout) fail(kStatusTimeoutEmpty);
          break;
        }
#ifdef POLYQ_DEBUG
        for (int h = 0; h < C::HALVES; ++h)
          for (int q = r; q < kRowsCta; q += kRowStep)
            dbg_row(smem + s * C::kA + h * kHalfTile, q, un * kRowsN + (int)rank * kRowsCta + q, P.N,
                    sblk[B.bi], tb * C::HALVES + h);
#endif
        __syncwarp();
        if (lane == 0) {
          mbar_arrive_cluster(bready0 + 8 * s);
          if (!early) mbar_arrive(smem_u32(&bar_cfree[sc]));
        }
        sc += C::GROUPS;
        if (sc >= C::CODES) {
          sc = grp;
          cph ^= 1u;
        }
        s += C::GROUPS;
        if (s >= C::OPS) {
          s = grp;
          sph ^= 1u;
        }
      }
      skip = kt - kt_hi;
    }
  } else {
    // ---------------- epilogue ----------------
    // Lane i of a warp owns output column n = weight row 128 rank + 32 q + i
    // of the unit, and each TMEM column one token, so every store of a warp
    // writes 32 consecutive floats of one row of Y, 32 tokens at a time.
    const int q = warp & 3;  // TMEM lane quarter this warp may access
    const int e0 = (warp - C::kEpiWarp) >> 2;  // chunks e0, e0 + EPI / 4, ...
    constexpr int kChunks = C::T / 32 / (C::EPI / 4);
    const uint32_t acce0 = mapa(smem_u32(&bar_acce[0]), 0);
    pdl_wait();  // the row scales come from the pre-pass
    for (int uc = 0; !s_abort && pc.next(P, um, un, kt_lo, kt_hi); ++uc) {
      const int buf = uc % C::NBUF;
      const bool add = pc.adds(P);  // Y was zeroed by the pre-pass
      // column 32 c of the unit's accumulators: with two, columns [0, TN / 2)
      // of accumulator a are tokens a * TN / 2.. of CTA 0's R, the others of
      // CTA 1's
      auto token0 = [&](int c) {
        const int a = 32 * c / C::TN, col = 32 * c % C::TN;
        return um * C::T + (col / (C::TN / 2)) * C::R + a * (C::TN / 2) + col % (C::TN / 2);
      };
      float rs[kChunks];  // 2^e_m of the pre-pass, token token0 + lane of each chunk
#pragma unroll
      for (int i = 0; i < kChunks; ++i) {
        const int m = token0(e0 + i * (C::EPI / 4)) + lane;
        rs[i] = m < P.M ? __ldcg(P.rowscale + m) : 0.f;
      }
      {
        const int w = wait_sleep_ab(smem_u32(&bar_accf[buf]), (uc / C::NBUF) & 1, &s_abort);
        if (w != kWaitOk) {
          if (w == kWaitTimeout) fail(kStatusTimeoutFull);
          break;
        }
      }
      tc_fence_after();
      const int n = un * kRowsN + (int)rank * kRowsCta + 32 * q + lane;
      const uint32_t t0 = tmem + ((uint32_t)(32 * q) << 16) + buf * (C::NACC * C::TN);
#pragma unroll 1
      for (int i = 0; i < kChunks; ++i) {
        const int c = e0 + i * (C::EPI / 4);
        const int m0 = token0(c);
        const int jn = min(32, P.M - m0);  // tokens of this chunk inside M
        if (jn > 0) {
          uint32_t v[32];
          tc_ld_32x32b_x32(t0 + 32 * c, v);
          float rs_l = rs[0];
#pragma unroll
          for (int k = 1; k < kChunks; ++k) rs_l = k == i ? rs[k] : rs_l;
          tc_wait_ld();
          tc_regs_ready(v);
          float* dst = P.y + (size_t)m0 * P.N + n;
          if (add) store_chunk<true>(dst, P.N, n < P.N, jn, v, rs_l);
          else store_chunk<false>(dst, P.N, n < P.N, jn, v, rs_l);
          __syncwarp();
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(acce0 + 8 * buf);
    }
  }

  // all roles of both CTAs done (or aborted): free TMEM; neither CTA exits
  // while its peer may still reach its shared memory
  __syncthreads();
  cluster_sync();
  if (role == kRoleMma) {
    tc_fence_after();
    tmem_dealloc2(tmem, kTmemCols);
  }
  cluster_sync();
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
int k_tiles(const polyq_dev_layer* L, int bk, GmBlock* blk) {
  int kt = 0;
  for (int i = 0; i < L->n_blocks; ++i) {
    const polyq_block& b = L->blocks[i];
    GmBlock g;
    g.bits = b.bits;
    g.n_ch = b.n_ch;
    g.pos0 = b.pos0;
    g.seg_off = b.seg_off;
    g.grp_off = b.grp_off;
    g.kt0 = kt;
    kt += (b.n_ch + bk - 1) / bk;
    if (blk) blk[i] = g;
  }
  return kt;
}

// Workspace: Xg fp16 (M rounded up to a token tile of any kernel that may
// take it, K slots padded to 64 per block), the row scales [M] fp32, then 256
// bytes holding the status word; each part starts on a 256-byte boundary.
// Grows with M, so that a workspace made for M serves fewer rows too.
size_t gemm_xg_rows(int64_t M) {
  size_t Mp = 32;
  while (Mp < 512 && Mp < (size_t)M) Mp *= 2;
  return Mp == 512 ? ((size_t)M + 511) / 512 * 512 : Mp;
}
size_t gemm_xg_bytes(const polyq_dev_layer* L, int64_t M) {
  return gemm_xg_rows(M) * k_tiles(L, 64, nullptr) * 64 * 2;
}
size_t gemm_workspace(const polyq_dev_layer* L, int64_t M) {
  return gemm_xg_bytes(L, M) + ((size_t)M * 4 + 255) / 256 * 256 + 256;
}

// CTA pairs resident at once for a kernel (per device, queried once), after
// its shared-memory limit has been raised.
constexpr int kMaxDevices = 64;
template <class C>
int resident_pairs(int dev, int* pairs) {
  static std::atomic<int> cached[kMaxDevices];
  int n = cached[dev].load(std::memory_order_acquire);
  if (n == 0) {
    cudaError_t e = cudaFuncSetAttribute(gemm_main<C>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)C::kSmem);
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 2;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2);
    cfg.blockDim = dim3(C::kThreads);
    cfg.dynamicSmemBytes = C::kSmem;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&n, gemm_main<C>, &cfg);
    if (e != cudaSuccess || n < 1)
      return polyq_set_error(POLYQ_ECUDA, "polyq_linear_gemm: %d CTA pairs fit: %s", n,
                             cudaGetErrorString(e));
    cached[dev].store(n, std::memory_order_release);
  }
  *pairs = n;
  return POLYQ_OK;
}

// Modelled time (s) of a kernel on this problem and the K split it would use.
// A unit's K tile takes `stage` seconds of a pair; a piece costs `piece` more
// (pipeline fill, draining the accumulator) and splitting adds the zeroing of
// Y.  Uniform split into k ranges: whole waves of units.  Stream-K: one
// pair's equal share plus the pieces it touches; with `whole`, also after the
// full waves of units that pairs compute alone, so that only the last wave is
// shared.  Near ties go to the simpler choice (a gain of 3% promised to 13824 x
// 5120, M = 8192 by a shared last wave did not show).  (5120 x 5120, M = 2048 / 4096 /
// 8192: 87 / 163 / 314 us without the shared last wave, 84 / 150 / 296 with;
// 13824 x 5120, M = 1536: 153 and 139; 5120 x 13824, M = 4096: 398 and 377.
// The 256-token kernel is left without: 13824 x 5120, M = 512 59.9 us against
// 57.5, but 1% slower at M = 256 and 1024 and 8% faster only for 5120 x 5120 at
// M = 1024.)
struct Split {
  double t;
  int ksplit, streamk;
  long long whole;  // stream-K: units before it
};
Split plan_split(int64_t M, int64_t N, int T, int KT, int bk, int pairs, double stage,
                 double piece, bool whole) {
  const long long mn = ((M + T - 1) / T) * ((N + kRowsN - 1) / kRowsN);
  const double zero = (double)M * N * 4.0 / kZeroBytesPerS;
  Split s = {1e300, 1, 0, 0};
  const int kmax = std::max(1, std::min(64, KT * bk / 512));
  for (int k = 1; k <= kmax; ++k) {
    const long long waves = (mn * k + pairs - 1) / pairs;
    const double t = waves * ((double)KT / k * stage + piece) + (k > 1 ? zero : 0.0);
    if (t < 0.98 * s.t) s = {t, k, 0, 0};
  }
  for (long long w : {0ll, whole ? mn / pairs : 0ll}) {  // whole waves before the shared units
    const long long rest = mn - w * pairs;
    const double share = std::ceil((double)rest * KT / pairs);
    const double t_sk = w * (KT * stage + piece) + share * stage +
                        piece * (std::ceil(share / KT) + 1.0) + zero * rest / mn;
    if (rest * KT >= pairs && mn * KT < (1ll << 31) && t_sk < (w > 0 ? 0.95 : 0.98) * s.t)
      s = {t_sk, 1, 1, w * pairs};
  }
  return s;
}

template <class C>
int launch_main(GmParams& P, const Split& sp, int pairs, cudaStream_t st) {
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = 2;
  at[1].val.clusterDim.y = at[1].val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.stream = st;
  cfg.attrs = at;
  cfg.numAttrs = 2;
  cfg.gridDim = dim3((unsigned)(2 * (sp.streamk ? pairs : std::min(P.units, pairs))));
  cfg.blockDim = dim3(C::kThreads);
  cfg.dynamicSmemBytes = C::kSmem;
  cudaError_t e = cudaLaunchKernelEx(&cfg, gemm_main<C>, P, gv::kMagic);
  if (e != cudaSuccess)
    return polyq_set_error(POLYQ_ECUDA, "polyq_linear_gemm: launch: %s", cudaGetErrorString(e));
  return POLYQ_OK;
}

// The row-staging pre-pass with RW rows at a time: as many CTAs as are resident
// at once.
template <int RW, bool XS>
int launch_prep_rows(const GmParams& P, int sms, int dev, cudaLaunchConfig_t cfg) {
  static std::atomic<bool> attr_done[kMaxDevices];
  if (!attr_done[dev].load(std::memory_order_acquire)) {
    cudaError_t e = cudaFuncSetAttribute(gemm_prep_rows<RW, XS>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, kPrepMaxSmem);
    if (e != cudaSuccess)
      return polyq_set_error(POLYQ_ECUDA, "polyq_linear_gemm: prep smem attribute: %s",
                             cudaGetErrorString(e));
    attr_done[dev].store(true, std::memory_order_release);
  }
  cfg.blockDim = dim3(kRowsThreads);
  cfg.dynamicSmemBytes = rows_smem<RW>(P.K, P.KT * P.bk, P.xscale != nullptr);
  int per_sm = 0;
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, gemm_prep_rows<RW, XS>,
                                                                kRowsThreads, cfg.dynamicSmemBytes);
  if (e != cudaSuccess || per_sm < 1)
    return polyq_set_error(POLYQ_ECUDA, "polyq_linear_gemm: prep occupancy: %s",
                           cudaGetErrorString(e));
  const int Mp = P.units_m << (P.r_log2 + 1);
  cfg.gridDim = dim3((unsigned)std::min<long long>(Mp / RW, (long long)sms * per_sm));
  e = cudaLaunchKernelEx(&cfg, gemm_prep_rows<RW, XS>, P);
  if (e != cudaSuccess)
    return polyq_set_error(POLYQ_ECUDA, "polyq_linear_gemm: prep launch: %s", cudaGetErrorString(e));
  return POLYQ_OK;
}

// The pre-pass of a few rows: about two CTAs per SM, each with half to
// kSmallOcts pieces per thread, and CTAs that zero Y.  (Four per SM: the same
// up to M = 64, M = 128 0.3 us slower; eight 0.8 to 2.6 us slower.)
template <bool XS>
int launch_prep_small(GmParams& P, int sms, int dev, cudaLaunchConfig_t cfg) {
  static std::atomic<bool> attr_done[kMaxDevices];
  cudaError_t e;
  if (!attr_done[dev].load(std::memory_order_acquire)) {
    e = cudaFuncSetAttribute(gemm_prep_small<XS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             kSmallMaxK * 2);
    if (e != cudaSuccess)
      return polyq_set_error(POLYQ_ECUDA, "polyq_linear_gemm: prep smem attribute: %s",
                             cudaGetErrorString(e));
    attr_done[dev].store(true, std::memory_order_release);
  }
  const int Mp = P.units_m << (P.r_log2 + 1);
  const int octs = P.KT * P.bk / 8;
  const int lo = (octs + kSmallOcts * kPrepThreads - 1) / (kSmallOcts * kPrepThreads);
  const int hi = (2 * octs + kPrepThreads - 1) / kPrepThreads;  // half of the threads at work
  P.prep_seg = std::max(lo, std::min(hi, 2 * sms / Mp));
  P.prep_rows = Mp * P.prep_seg;
  int n_zero = 0;
  if (P.ksplit > 1 || P.streamk)  // eight float4 per thread, at most two CTAs per SM
    n_zero = (int)std::min<long long>(2 * sms, ((long long)P.M * P.N + 32 * kPrepThreads - 1) /
                                                   (32 * kPrepThreads));
  cfg.gridDim = dim3((unsigned)(P.prep_rows + n_zero));
  cfg.blockDim = dim3(kPrepThreads);
  cfg.dynamicSmemBytes = ((size_t)P.K * 2 + 15) / 16 * 16;
  e = cudaLaunchKernelEx(&cfg, gemm_prep_small<XS>, P);
  if (e != cudaSuccess)
    return polyq_set_error(POLYQ_ECUDA, "polyq_linear_gemm: prep launch: %s", cudaGetErrorString(e));
  return POLYQ_OK;
}

int launch_prep(GmParams& P, int sms, int dev, cudaStream_t st) {
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.stream = st;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  const int Kp = P.KT * P.bk;
  const int Mp = P.units_m << (P.r_log2 + 1);
  cudaError_t e;
  if (P.M <= kSmallMaxM && P.K <= kSmallMaxK)
    return P.xscale ? launch_prep_small<true>(P, sms, dev, cfg)
                    : launch_prep_small<false>(P, sms, dev, cfg);
  // Four rows at a time when two CTAs of that size share an SM and the rows
  // then still fill the GPU twice, else two, else one (K = 5120, M = 768: 81 us
  // for the whole call at two, 85 at four).
  const bool xs = P.xscale != nullptr;
  const size_t half_sm = 112 * 1024;
  if (P.K <= kRowsMaxK) {
    if (rows_smem<4>(P.K, Kp, xs) <= half_sm && Mp / 4 >= 2 * sms)
      return xs ? launch_prep_rows<4, true>(P, sms, dev, cfg)
                : launch_prep_rows<4, false>(P, sms, dev, cfg);
    if (rows_smem<2>(P.K, Kp, xs) <= half_sm && Mp / 2 >= sms)
      return xs ? launch_prep_rows<2, true>(P, sms, dev, cfg)
                : launch_prep_rows<2, false>(P, sms, dev, cfg);
    if (rows_smem<1>(P.K, Kp, xs) <= (size_t)kPrepMaxSmem)
      return xs ? launch_prep_rows<1, true>(P, sms, dev, cfg)
                : launch_prep_rows<1, false>(P, sms, dev, cfg);
  }
  cfg.gridDim = dim3((unsigned)std::min<long long>(Mp, 8ll * sms));
  cfg.blockDim = dim3(kPrepThreads);
  e = cudaLaunchKernelEx(&cfg, gemm_prep_wide, P);
  if (e != cudaSuccess)
    return polyq_set_error(POLYQ_ECUDA, "polyq_linear_gemm: prep launch: %s", cudaGetErrorString(e));
  return POLYQ_OK;
}

// One kernel's candidacy: its modelled time and split.
struct Choice {
  int cfg, pairs;
  Split split;
};
template <class C>
int consider(const polyq_dev_layer* L, int64_t M, int dev, int id, double stage, double piece,
             Choice* best) {
  int pairs = 0;
  int rc = resident_pairs<C>(dev, &pairs);
  if (rc) return rc;
  const Split s = plan_split(M, L->N, C::T, k_tiles(L, C::BK, nullptr), C::BK, pairs, stage, piece,
                             C::kWhole);
  if (best->cfg < 0 || s.t < 0.98 * best->split.t) *best = {id, pairs, s};
  return POLYQ_OK;
}

// The smallest token tile that holds M (a wider one would multiply padding:
// 13824 x 5120 takes 24 / 28 / 37 us at M = 16 / 96 / 256, and took 53 us at
// each with 256), or for more than 256 tokens the cheaper of 256 and 512 by
// the model (stage and piece times measured).  `tokens` > 0: that tile.
int choose(const polyq_dev_layer* L, int64_t M, int dev, int tokens, Choice* ch) {
  const int t = tokens ? tokens : M <= 32 ? 32 : M <= 64 ? 64 : M <= 128 ? 128 : 256;
  if (t == 32) return consider<Cfg32>(L, M, dev, 32, kStage32, kPiece32, ch);
  if (t == 64) return consider<Cfg64>(L, M, dev, 64, kStage64, kPiece64, ch);
  if (t == 128) return consider<Cfg128>(L, M, dev, 128, kStage128, kPiece128, ch);
  int rc = POLYQ_OK;
  if (t == 256) rc = consider<Cfg256>(L, M, dev, 256, kStage256, kPiece256, ch);
  if (!rc && (t == 512 || (!tokens && M > 256)))
    rc = consider<Cfg512>(L, M, dev, 512, kStage512, kPiece512, ch);
  return rc;
}

template <class C>
int run(const polyq_dev_layer* L, GmParams& P, const Choice& ch, int sms, int dev,
        cudaStream_t st) {
  P.bk = C::BK;
  P.KT = k_tiles(L, C::BK, P.blk);
  P.r_log2 = 0;
  while ((1 << P.r_log2) < C::R) ++P.r_log2;
  P.units_m = (P.M + C::T - 1) / C::T;
  P.units_n = (P.N + kRowsN - 1) / kRowsN;
  P.ksplit = ch.split.ksplit;
  P.streamk = ch.split.streamk;
  P.units = P.units_m * P.units_n * P.ksplit;
  P.whole = P.units;
  if (P.streamk) {
    P.whole = (int)ch.split.whole;
    P.zero_col0 = P.whole / P.units_m * kRowsN;
    const int total = (P.units - P.whole) * P.KT;  // below 2^31, see plan_split
    P.sk_share = total / ch.pairs;
    P.sk_extra = total % ch.pairs;
  }
  int rc = launch_prep(P, sms, dev, st);
  if (rc) return rc;
  // The main kernel may launch while the pre-pass runs (programmatic
  // dependent launch): its set-up overlaps the pre-pass, and its producer
  // waits for the pre-pass before the first load of Xg.  It allocates all of
  // an SM's tensor memory, which is safe because two of its CTAs (more than
  // half of an SM's shared memory each) never share an SM.
  return launch_main<C>(P, ch.split, ch.pairs, st);
}

}  // namespace

extern "C" int polyq_gemm_workspace_bytes(const polyq_dev_layer* L, int64_t M, size_t* bytes) {
  polyq_clear_error();
  int rc = polyq_check_dev_layer(L, "polyq_gemm_workspace_bytes");
  if (rc) return rc;
  if (!bytes) return polyq_set_error(POLYQ_EINVAL, "polyq_gemm_workspace_bytes: bytes is NULL");
  if (M < 1 || M > (1 << 24))
    return polyq_set_error(POLYQ_EINVAL, "polyq_gemm_workspace_bytes: M=%lld", (long long)M);
  *bytes = gemm_workspace(L, M);
  return POLYQ_OK;
}

namespace {

int device_index(int* dev) {
  *dev = 0;
  cudaGetDevice(dev);
  if (*dev < 0 || *dev >= kMaxDevices)
    return polyq_set_error(POLYQ_EUNSUPPORTED, "polyq_linear_gemm: device %d >= %d", *dev,
                           kMaxDevices);
  return POLYQ_OK;
}

// polyq_linear_gemm; tokens > 0 (debug build): with this token tile.
int gemm_call(const polyq_dev_layer* L, const void* X, int64_t M, float* Y, void* workspace,
              size_t ws_bytes, int tokens, void* stream) {
  int rc = polyq_check_dev_layer(L, "polyq_linear_gemm");
  if (rc) return rc;
  if (!X || !Y) return polyq_set_error(POLYQ_EINVAL, "polyq_linear_gemm: X or Y is NULL");
  if ((uintptr_t)Y % 16)  // Y is zeroed for split K with 16-byte stores
    return polyq_set_error(POLYQ_EINVAL, "polyq_linear_gemm: Y must be 16-byte aligned");
  if (M < 1 || M > (1 << 24))
    return polyq_set_error(POLYQ_EINVAL, "polyq_linear_gemm: M=%lld", (long long)M);
  const size_t need = gemm_workspace(L, M);
  if (!workspace || ws_bytes < need)
    return polyq_set_error(POLYQ_ENOMEM, "polyq_linear_gemm: workspace needs %zu bytes, got %zu",
                           need, ws_bytes);
  if ((uintptr_t)workspace % 256)
    return polyq_set_error(POLYQ_EINVAL, "polyq_linear_gemm: workspace must be 256-byte aligned");
  if (L->row_stride % 16)
    return polyq_set_error(POLYQ_EINVAL, "polyq_linear_gemm: row_stride must be a multiple of 16");

  GmParams P;
  memset(&P, 0, sizeof P);
  P.n_blocks = L->n_blocks;
  P.M = (int)M;
  P.N = (int)L->N;
  P.K = (int)L->K;
  P.x = (const __nv_bfloat16*)X;
  P.gather = L->gather;
  P.xscale = L->xscale;
  P.xg = (__half*)workspace;
  P.rowscale = (float*)((uint8_t*)workspace + gemm_xg_bytes(L, M));
  P.y = Y;
  P.status = (int*)((uint8_t*)workspace + need - 256);
  rc = polyq_tensor_map_2d(&P.tm_codes, L->packed, 1, (uint64_t)L->row_stride, (uint64_t)L->N,
                           (uint64_t)L->row_stride, kCodeBox, kRowsCta);
  if (rc) return rc;
  rc = polyq_tensor_map_2d(&P.tm_w16, L->packed, 2, (uint64_t)L->row_stride / 2, (uint64_t)L->N,
                           (uint64_t)L->row_stride, kSlots, kRowsCta, 64);
  if (rc) return rc;
  if (L->n_groups > 0) {
    rc = polyq_tensor_map_2d(&P.tm_meta, L->meta, 4, (uint64_t)L->meta_stride, (uint64_t)L->N,
                             (uint64_t)L->meta_stride * 4, 4, kRowsCta);
    if (rc) return rc;
    P.has_meta = 1;
  }

  cudaStream_t st = (cudaStream_t)stream;
  int sms = 0, dev = 0;
  rc = polyq_sm_count(&sms);
  if (rc) return rc;
  rc = device_index(&dev);
  if (rc) return rc;
  Choice ch = {-1, 0, {}};
  rc = choose(L, M, dev, tokens, &ch);
  if (rc) return rc;
  switch (ch.cfg) {
    case 32: return run<Cfg32>(L, P, ch, sms, dev, st);
    case 64: return run<Cfg64>(L, P, ch, sms, dev, st);
    case 128: return run<Cfg128>(L, P, ch, sms, dev, st);
    case 256: return run<Cfg256>(L, P, ch, sms, dev, st);
    default: return run<Cfg512>(L, P, ch, sms, dev, st);
  }
}

}  // namespace

extern "C" int polyq_linear_gemm(const polyq_dev_layer* L, const void* X, int64_t M, float* Y,
                                 void* workspace, size_t ws_bytes, void* stream) {
  polyq_clear_error();
  return gemm_call(L, X, M, Y, workspace, ws_bytes, 0, stream);
}

#ifdef POLYQ_DEBUG
// Debug build only: polyq_linear_gemm with a given token tile and, if w_out is
// not NULL, every weight placed in an A tile written to it ([N][K] fp16 bits,
// clustered order).
extern "C" int polyq_debug_linear_gemm(const polyq_dev_layer* L, const void* X, int64_t M,
                                       float* Y, void* workspace, size_t ws_bytes, int tokens,
                                       uint16_t* w_out, void* stream) {
  polyq_clear_error();
  if (tokens != 0 && tokens != 32 && tokens != 64 && tokens != 128 && tokens != 256 && tokens != 512)
    return polyq_set_error(POLYQ_EINVAL, "debug: no kernel of %d tokens", tokens);
  if (tokens && M > 0 && ((size_t)M + tokens - 1) / tokens * tokens > gemm_xg_rows(M))
    return polyq_set_error(POLYQ_EINVAL, "debug: the workspace of M=%lld holds no tile of %d tokens",
                           (long long)M, tokens);
  cudaStream_t st = (cudaStream_t)stream;
  const long long K = L ? L->K : 0;
  cudaError_t e = cudaMemcpyToSymbolAsync(g_dbg_w, &w_out, sizeof w_out, 0,
                                          cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess)
    e = cudaMemcpyToSymbolAsync(g_dbg_wK, &K, sizeof K, 0, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return polyq_set_error(POLYQ_ECUDA, "debug: %s", cudaGetErrorString(e));
  const int rc = gemm_call(L, X, M, Y, workspace, ws_bytes, tokens, stream);
  uint16_t* none = nullptr;
  cudaMemcpyToSymbolAsync(g_dbg_w, &none, sizeof none, 0, cudaMemcpyHostToDevice, st);
  cudaStreamSynchronize(st);
  return rc;
}

extern "C" int polyq_debug_gemm_weights(const polyq_dev_layer* L, const void* X, int64_t M,
                                        float* Y, void* workspace, size_t ws_bytes,
                                        uint16_t* w_out, void* stream) {
  return polyq_debug_linear_gemm(L, X, M, Y, workspace, ws_bytes, 0, w_out, stream);
}

// Debug build only: what polyq_linear_gemm would launch.
extern "C" int polyq_debug_gemm_choice(const polyq_dev_layer* L, int64_t M, polyq_gemm_choice* out) {
  polyq_clear_error();
  int rc = polyq_check_dev_layer(L, "polyq_debug_gemm_choice");
  if (rc) return rc;
  if (!out || M < 1 || M > (1 << 24))
    return polyq_set_error(POLYQ_EINVAL, "polyq_debug_gemm_choice: M=%lld", (long long)M);
  int dev = 0;
  rc = device_index(&dev);
  if (rc) return rc;
  Choice ch = {-1, 0, {}};
  rc = choose(L, M, dev, 0, &ch);
  if (rc) return rc;
  *out = {ch.cfg, ch.pairs, ch.split.ksplit, ch.split.streamk, (int64_t)ch.split.whole};
  return POLYQ_OK;
}
#endif
