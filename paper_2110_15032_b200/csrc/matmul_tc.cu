// Tensor-core MatMul for sm_100a: bf16 operands, fp32 accumulation in tensor memory.
//
// Pairs of CTAs (a cluster of two SMs) walk the (group, m-tile, n-tile) list of a grouped-GEMM
// plan (matmul_plan.h).  A pair owns one 256 x 256 output tile at a time: CTA r of the pair
// holds rows 128 r .. 128 r + 127 of the A tile, columns 128 r .. 128 r + 127 of the B tile and
// rows 128 r .. of the accumulator in its own tensor memory; one tcgen05.mma.cta_group::2
// instruction, issued by the pair's first CTA, multiplies across both.  Per CTA and 64-deep
// K-block that is 16 KiB of A and 16 KiB of B through TMA for 2 x 128 x 256 x 64 MACs, two
// thirds of what two independent 128 x 256 CTAs would pull from L2.
//
//   warp 0     producer   TMA loads of this CTA's A and B halves into a kStages-deep ring; the
//                         transaction bytes of both CTAs land on the first CTA's "full" barrier
//   warp 1     MMA        (first CTA only) an elected lane issues four M256 N256 K16 MMAs per K-block
//                         into one of two 256-column accumulators; tcgen05.commit, delivered to
//                         both CTAs, frees the ring slot / publishes the accumulator
//   warps 2-9  epilogue   warp w drains lanes 32 (w mod 4) .. +31, columns 128 ((w-2)/4) .. +127
//                         of its CTA's accumulator (tcgen05.ld), applies GeLU when asked, rounds
//                         to the output type, stages 32 x 128-byte slabs in swizzled shared memory
//                         and writes them with TMA stores, once per destination replica, while
//                         the next tile's MMAs fill the other accumulator
//
// A fused "P(sum) product written as B / S(i)" plan simply chains the K-blocks of all shards'
// operands, in rank order, into the same accumulator: the partial products are never stored.
//
// Every barrier wait is bounded in time (the one wait that is not is the allocation of tensor memory
// at the start, which cannot block: the shared-memory footprint keeps the kernel to one CTA per SM,
// so the CTA is alone on its SM's tensor memory).  A wait that expires raises a flag that
// sbp_check_device_errors() reports; the CTA then stops issuing work, waits (bounded) for the
// loads it still has in flight, meets its partner at the closing cluster barrier, frees its
// tensor memory and returns.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cstdlib>
#include <mutex>
#include <type_traits>

#include "boxing_shift.h"
#include "bounds_check.h"
#include "matmul_plan.h"
#include "sbp_internal.h"
#include "tc_ptx.h"

namespace sbp {

constexpr int BM = 256, BN = 256, BK = 64;      // tile of a CTA pair
constexpr int BMH = BM / 2, BNH = BN / 2;       // what one CTA of the pair loads
constexpr int kStages = 6;                        // 6 slots + 1 staging slab per warp beat 5 + 2 once the hand-back of an accumulator was cheap
constexpr int kStageA = BMH * BK * 2;             // 16 KiB
constexpr int kStageB = BK * BNH * 2;             // 16 KiB
constexpr int kStageBytes = kStageA + kStageB;    // 32 KiB per CTA
constexpr int kEpiWarps = 8;
constexpr int kSlabBytes = 32 * 128;              // one epilogue slab: 32 rows x 128 bytes
constexpr int kEpiBufs = 1;                       // staging slabs per epilogue warp
constexpr int kEpiBytes = kEpiWarps * kEpiBufs * kSlabBytes;
constexpr int kSmemBytes = kStages * kStageBytes + kEpiBytes + 1024;   // + alignment slack
// The tall form (MH = 2): a CTA pair owns a 512 x 256 tile -- two m-halves of 256 rows that share
// every B slice -- with BOTH 256-column accumulators in use at once.  A 64-deep K-block then brings
// 48 KiB per CTA into shared memory for 2 x 4 MMAs (1024 clocks) instead of 32 KiB for 4 MMAs
// (512 clocks): a quarter less operand traffic per MMA clock, both from L2 and through shared
// memory.  At the square form's rate the shared-memory data path has to carry one 128-byte
// wavefront every clock (TMA writes + MMA reads) and the tensor pipe reaches 76 %; with the
// slack the tall form leaves it runs the main loop at full rate.  The price is that the
// epilogue of a tile no longer overlaps the next tile's MMAs in full (the second accumulator is
// not a spare any more), which a long contraction repays many times over and a short one does not:
// the host picks the form per product.
constexpr int kStagesTall = 4;
constexpr int kStageBytesTall = 2 * kStageA + kStageB;     // 48 KiB per CTA
constexpr int kEpiBufsTall = 1;
constexpr int kSmemBytesTall = kStagesTall * kStageBytesTall + kEpiWarps * kEpiBufsTall * kSlabBytes + 1024;
// The short form (MH = 3): the square tile with four ring slots and three staging slabs a warp.  Where the contraction is
// short the tile is its epilogue: with one slab a warp waits for each store to have read it before it stages the next.
// (us, square / short, products over 2^19 to 2^20 classes: 1 K-block, 176 rows 56 / 50, 232 rows 108 / 103; gradient with 2
// K-blocks 137 / 129; 3 K-blocks 39 / 35; softmax partials with 2 K-blocks 132 / 125, 3 37.7 / 35.9, 4 89 / 84.  With 5 and
// 8 K-blocks four slots are too few: 29.0 / 32.4, 521 / 544.)
constexpr int kStagesShort = 4, kEpiBufsShort = 3, kShortBlocks = 4;
static_assert(kStagesShort * kStageBytes + kEpiWarps * kEpiBufsShort * kSlabBytes + 1024 <= kSmemBytes, "the short form fits where the square one does");
constexpr int kMaxStages = kStages > kStagesTall ? kStages : kStagesTall;
constexpr int kThreadsTc = 32 * (2 + kEpiWarps);
constexpr int kTmemCols = 512;

struct TcParams {
  CUtensorMap map_a[SBP_MAX_K];
  CUtensorMap map_b[SBP_MAX_K];
  CUtensorMap map_y[SBP_MAX_K];
  CUtensorMap map_rep[SBP_MAX_K];
  long long m[SBP_MAX_K], n[SBP_MAX_K], row_off[SBP_MAX_K], col_off[SBP_MAX_K];
  int kblocks[SBP_MAX_K];       // per segment
  int tile_begin[SBP_MAX_K + 1];   // prefix sum of tiles per group
  int tiles_m[SBP_MAX_K];
  int tiles_n[SBP_MAX_K];
  int mt_begin[SBP_MAX_K + 1];     // stacked == 1: prefix sum of m-tiles per group; == 2: of n-tiles
  int stacked;                     // the groups are row (1) / column (2) blocks of one result and are walked as one grid
  int ngroups, nseg, chain, gelu, n_rep;
  int out_f32;
  int total_tiles;
  unsigned panel_magic[SBP_MAX_K];   // floor(2^32 / (kPanelM * n-tiles)) of the group (stacked walks: entry 0, of the whole list)
  int walk_m;                   // rows of a walked tile: 256, or 512 (tall form and the square remainder of a mixed run)
  int tile_first;               // index of the first walked tile of this launch
  int half_split;               // square form over 512-row walked tiles: launch tile 2t + h is m-half h of walked tile t
  int xent;                     // 1: softmax partials instead of stored logits
  XentFusion xf;
  // Results the copy engine cannot address (a base or a row pitch that is not a multiple of 16
  // bytes): the epilogue then writes its staged slabs itself, row by row, with element-wise stores.
  int y_direct;
  void* y_ptr[SBP_MAX_K];
  void* rep_ptr[SBP_MAX_K];
  long long ldy[SBP_MAX_K];
};

// Instruction descriptor: D fp32, A and B bf16, M = 256 (pair), N = `n`.  Bit 15 / bit 16 say
// that A / B lies in shared memory with its M / N index contiguous ("MN-major") instead of its
// K index.  Operands as given: A [M,K] row-major is K-major, B [K,N] row-major is N-major; a
// transposed operand is the other way round.
constexpr unsigned kIdescBase = (1u << 4) | (1u << 7) | (1u << 10) | ((BM >> 4) << 24);
__host__ __device__ constexpr unsigned make_idesc(int a_trans, int b_trans, int n = BN) {
  return kIdescBase | ((unsigned)(n >> 3) << 17) | ((a_trans ? 1u : 0u) << 15) | ((b_trans ? 0u : 1u) << 16);
}

// Two numbers in one register pair.
__device__ __forceinline__ unsigned long long two(float x, float y) {
  unsigned long long v;
  asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(x), "f"(y));
  return v;
}
__device__ __forceinline__ unsigned long long two(float x) { return two(x, x); }
__device__ __forceinline__ unsigned long long fma_two(unsigned long long a, unsigned long long b, unsigned long long c) {
  unsigned long long v;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(v) : "l"(a), "l"(b), "l"(c));
  return v;
}
__device__ __forceinline__ unsigned long long mul_two(unsigned long long a, unsigned long long b) {
  unsigned long long v;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(v) : "l"(a), "l"(b));
  return v;
}

__device__ __forceinline__ unsigned long long add_two(unsigned long long a, unsigned long long b) {
  unsigned long long v;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(v) : "l"(a), "l"(b));
  return v;
}

// 2^((a - m) log2e + c) and the same of b: the difference is exact in m, and in pairs it costs no more than one multiply-add an
// element.  (m log2e folded into c: its rounding is a factor on the whole row, 3e-4 at a maximum of 1e4, 4 % at 1e6.)
__device__ __forceinline__ void exp_two(float& a, float& b, unsigned long long neg_m, unsigned long long c) {
  const unsigned long long v = fma_two(add_two(two(a, b), neg_m), two(1.4426950408889634f), c);
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(a) : "f"(__uint_as_float((unsigned)v)));
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(b) : "f"(__uint_as_float((unsigned)(v >> 32))));
}
__device__ __forceinline__ float exp_one(float a, float m, float c) {
  float e;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(fmaf(a - m, 1.4426950408889634f, c)));
  return e;
}

// GeLU(v) = 0.5 v (1 + erf(v / sqrt 2)) of two numbers, erf by the rational approximation 7.1.26 of Abramowitz & Stegun
// (|error| <= 1.5e-7), which is far below the rounding of the bf16 / fp32 store that follows and costs two special-function
// operations where erff costs a long polynomial.  Each number goes through the operations of the formula in its order, so the
// bits are those of the scalar form; in pairs they are ten and a half instructions a number where that takes twenty.  The
// epilogue of a tile that nothing overlaps is these instructions.
__device__ __forceinline__ void gelu_two(float& a, float& b) {
  const unsigned long long v = two(a, b), x = mul_two(v, two(0.70710678118654752440f));
  const unsigned x0 = (unsigned)x, x1 = (unsigned)(x >> 32);
  const unsigned long long ax = two(fabsf(__uint_as_float(x0)), fabsf(__uint_as_float(x1)));
  const unsigned long long d = fma_two(two(0.3275911f), ax, two(1.0f)), y = mul_two(mul_two(ax, ax), two(-1.4426950408889634f));
  float ta, tb, ea, eb;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(ta) : "f"(__uint_as_float((unsigned)d)));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(tb) : "f"(__uint_as_float((unsigned)(d >> 32))));
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(ea) : "f"(__uint_as_float((unsigned)y)));
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(eb) : "f"(__uint_as_float((unsigned)(y >> 32))));
  const unsigned long long t = two(ta, tb);
  unsigned long long q = fma_two(t, two(-1.061405429f), two(1.453152027f));      // the polynomial, negated
  q = fma_two(q, t, two(-1.421413741f));
  q = fma_two(q, t, two(0.284496736f));
  q = fma_two(q, t, two(-0.254829592f));
  q = fma_two(mul_two(q, t), two(ea, eb), two(1.0f));
  const unsigned r0 = ((unsigned)q & 0x7fffffffu) | (x0 & 0x80000000u), r1 = ((unsigned)(q >> 32) & 0x7fffffffu) | (x1 & 0x80000000u);
  const unsigned long long g = mul_two(mul_two(v, two(0.5f)), add_two(two(1.0f), two(__uint_as_float(r0), __uint_as_float(r1))));
  a = __uint_as_float((unsigned)g);
  b = __uint_as_float((unsigned)(g >> 32));
}

struct TileCoord {
  int g, m0, n0;
};

// Tiles of a group are walked in panels of kPanelM m-tiles: inside a panel the m-tile index varies
// fastest and the n-tile index steps once per column of the panel, so that the CTA pairs running at
// the same time cover a roughly square patch of the output and share both their A rows and their B
// columns in L2.
constexpr int kPanelM = 8;

// n / d for 0 <= n < 2^31 and d >= 2 with magic = floor(2^32 / d): the high product is short of the
// quotient by at most one or two, which the loop makes up.  (The tile walk divides twice per tile
// in each of three roles; the generic division is a few hundred clocks of the one thread that
// issues the MMAs.)
__device__ __forceinline__ int div_by(int n, int d, unsigned magic) {
  int q = (int)__umulhi((unsigned)n, magic);
  while (n - q * d >= d) ++q;
  return q;
}

// position inside a panel of pm m-tiles: pm is kPanelM everywhere but in a group's last panel
__device__ __forceinline__ int div_panel(int rem, int pm) { return pm == kPanelM ? rem / kPanelM : rem / pm; }

__device__ __forceinline__ TileCoord tile_coord(const TcParams& p, int tile) {
  int half_m = 0;
  if (p.half_split) {
    half_m = (tile & 1) * BM;
    tile >>= 1;
  }
  tile += p.tile_first;
  if (p.stacked == 2) {
    // The same for a fused product written as S(1): column blocks of one result, which share every
    // A row block; the n-tiles of all groups form one list.
    const int tm = p.tiles_m[0], tn = p.mt_begin[p.ngroups];
    const int panel = div_by(tile, kPanelM * tn, p.panel_magic[0]);
    const int rem = tile - panel * (kPanelM * tn);
    const int pm = min(kPanelM, tm - panel * kPanelM);
    const int nt = div_panel(rem, pm), mt = panel * kPanelM + (rem - nt * pm);
    int g = 0;
    while (g + 1 < p.ngroups && nt >= p.mt_begin[g + 1]) ++g;
    return TileCoord{g, mt * p.walk_m + half_m, (nt - p.mt_begin[g]) * BN};
  }
  if (p.stacked) {
    // A fused product written as S(0): the groups are the row blocks of ONE result and share every
    // B column block.  Walking them one after the other would stream the whole B operand once per
    // group; instead the m-tiles of all groups form one list and the panel walk runs over that.
    const int tm = p.mt_begin[p.ngroups], tn = p.tiles_n[0];
    const int panel = div_by(tile, kPanelM * tn, p.panel_magic[0]);
    const int rem = tile - panel * (kPanelM * tn);
    const int pm = min(kPanelM, tm - panel * kPanelM);
    const int nt = div_panel(rem, pm), mt = panel * kPanelM + (rem - nt * pm);
    int g = 0;
    while (g + 1 < p.ngroups && mt >= p.mt_begin[g + 1]) ++g;
    return TileCoord{g, (mt - p.mt_begin[g]) * p.walk_m + half_m, nt * BN};
  }
  int g = 0;
  while (g + 1 < p.ngroups && tile >= p.tile_begin[g + 1]) ++g;
  const int local = tile - p.tile_begin[g];
  const int tm = p.tiles_m[g], tn = p.tiles_n[g];
  const int panel = div_by(local, kPanelM * tn, p.panel_magic[g]);
  const int rem = local - panel * (kPanelM * tn);
  const int pm = min(kPanelM, tm - panel * kPanelM);   // m-tiles in this (possibly last) panel
  const int nt = div_panel(rem, pm), mt = panel * kPanelM + (rem - nt * pm);
  return TileCoord{g, mt * p.walk_m + half_m, nt * BN};
}

// Part `lane` of `lanes` of a row of `bytes` bytes that starts at dst, which need not be 16-byte aligned, from shared
// memory (`at`: where a byte of the row lies; 16-byte chunks are whole): a whole aligned vector of the destination, two
// chunks shifted together, and every lanes-th element of those before the first and after the last such vector.
// (A result [1500 x 4832] over eight devices, rows of 604: 40.0 us so, 45.8 with an element a lane and store; [585 x 1204] over four 14.2, 17.9; [4000 x 4091] 60, 73.)
template <int ESZ, typename At>
__device__ __forceinline__ void store_shifted(unsigned char* dst, int bytes, int lane, int lanes, At at) {
  const int to_line = (int)(-reinterpret_cast<long long>(dst) & 15), head = to_line < bytes ? to_line : bytes;
  const int nvec = (bytes - head) >> 4;
  if (lane < nvec && SBP_GUARD(dst + head + lane * 16, 16)) {
    uint4 v = *reinterpret_cast<const uint4*>(at(lane * 16));
    if (head) v = shift_pair<ESZ>(v, *reinterpret_cast<const uint4*>(at(lane * 16 + 16)), (unsigned)head);
    *reinterpret_cast<uint4*>(dst + head + lane * 16) = v;
  }
  using E = typename ShiftElem<ESZ>::type;
  for (int e = lane * ESZ; e < bytes - nvec * 16; e += lanes * ESZ) {
    const int off = e < head ? e : nvec * 16 + e;
    if (SBP_GUARD(dst + off, ESZ)) *reinterpret_cast<E*>(dst + off) = *reinterpret_cast<const E*>(at(off));
  }
}

// ------------------------------------------------------------------ the kernel

// AT / BT: operand A / B is stored transposed.  They are compile-time so that the usual
// (untransposed) form carries no trace of the other three: as run-time switches they cost the
// MMA-issuing thread and the producer enough to slow every product by 6 %.
// MH: 1 = square form, 2 = tall form (two m-halves of 256 rows per pair tile, see kStageBytesTall), 3 = short form.
template <int AT, int BT, int MH>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreadsTc, 1)
    matmul_tc_kernel(const __grid_constant__ TcParams p) {
  constexpr int kHalves = MH == 2 ? 2 : 1;
  constexpr int kSt = MH == 2 ? kStagesTall : (MH == 3 ? kStagesShort : kStages);      // ring depth
  constexpr int kStA = kHalves * kStageA;                                    // bytes of A per ring slot
  constexpr int kStBytes = kStA + kStageB;
  constexpr int kEB = MH == 2 ? kEpiBufsTall : (MH == 3 ? kEpiBufsShort : kEpiBufs);                // staging slabs per epilogue warp
  extern __shared__ unsigned char smem_raw[];
  __shared__ __align__(8) unsigned long long bar_full[kMaxStages], bar_empty[kMaxStages], bar_acc_full[2], bar_acc_empty[2];
  __shared__ unsigned tmem_base_slot;
  __shared__ int abort_flag_s;
  volatile int* abort_flag = &abort_flag_s;

  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  unsigned char* epi = smem + kSt * kStBytes;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const unsigned rank = cluster_ctarank();     // 0 = the CTA that issues the pair's MMAs

  if (threadIdx.x == 0) {
    abort_flag_s = 0;
    for (int i = 0; i < kSt; ++i) {
      mbar_init(smem_addr(&bar_full[i]), 1);      // used in CTA 0 only: one arrive + both CTAs' bytes
      mbar_init(smem_addr(&bar_empty[i]), 1);     // one commit per use, delivered to both CTAs
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(smem_addr(&bar_acc_full[i]), 1);
      mbar_init(smem_addr(&bar_acc_empty[i]), 2 * kEpiWarps);   // used in CTA 0 only: both CTAs' epilogue warps
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&tmem_base_slot)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  cluster_arrive();
  const int first = blockIdx.x >> 1, stride = gridDim.x >> 1;   // tiles are dealt to CTA pairs
  TileCoord tc = tile_coord(p, first);
  if (warp == 2 && lane == 0) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(&p.map_a[p.chain ? 0 : tc.g]) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&p.map_b[p.chain ? 0 : tc.g]) : "memory");
    if (p.xent != 1 && !p.y_direct) asm volatile("prefetch.tensormap [%0];" ::"l"(&p.map_y[tc.g]) : "memory");
  }
  cluster_wait();                                // both CTAs' barriers exist before anyone signals them
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const unsigned tmem_base = tmem_base_slot;
  // A kernel launched behind this one as its programmatic dependent may be set up from here on;
  // it waits on the device for this grid to finish before it reads what this grid writes.  This
  // kernel is launched the same way: barriers and TMEM are set up under the end of the kernel before.
  SBP_PDL_RELEASE();
  // The first tile's place and descriptors are there before the wait: the first operands land 1.25 us after it, 2.2 to 2.9
  // where both came after it (500 x 1024 x 1024 over eight devices; 2048 x 1024 x 4096 2.2, 3.3).
  SBP_PDL_WAIT();

  if (warp == 0) {
    // ------------------------------------------------ producer (both CTAs)
    //
    // Both single-issue roles run as whole warps: every lane walks the loop and waits on the barriers, one
    // elected lane issues.  Ring position, addresses and descriptors are then the same in all lanes of a
    // converged warp and can live in uniform registers, which the copy and MMA instructions take their
    // operands from; with one lane alone inside the loop each operand was moved there per instruction.
    // [8192,4096] x [4096,16384] + GeLU 755 -> 709 us back to back, fused classifier forward (512 x 512 x
    // 2^20) 489 -> 456 us, its backward 577 -> 527 us (same GPU, MMA warp and producer about half each).
    const bool leader = elect_one();
    // ring position kept as (slot, round parity) and stepped, not divided out of a running count:
    // with a slot count that is not a power of two the division is a long instruction sequence,
    // once per K-block
    long long kb_iter = 0;
    int slot = 0;
    unsigned round = 0;
    for (int tile = first; tile < p.total_tiles; tile += stride) {
      if (tile != first) tc = tile_coord(p, tile);
      const int s_lo = p.chain ? 0 : tc.g, s_hi = p.chain ? p.nseg : tc.g + 1;
      for (int s = s_lo; s < s_hi; ++s) {
        const int nkb = p.kblocks[s];
        for (int kb = 0; kb < nkb; ++kb, ++kb_iter, slot = slot + 1 == kSt ? 0 : slot + 1, round ^= (slot == 0)) {
          const unsigned parity = round ^ 1;
          if (!mbar_wait_warp(smem_addr(&bar_empty[slot]), parity, abort_flag)) goto producer_done;
          if (leader) {
            const unsigned full0 = map_to_cta(smem_addr(&bar_full[slot]), 0);
            if (rank == 0) mbar_expect_tx(smem_addr(&bar_full[slot]), 2 * kStBytes);
            unsigned char* sa0 = smem + slot * kStBytes;
            unsigned char* sb = sa0 + kStA;
            const int bcol = (int)p.col_off[tc.g] + tc.n0 + (int)rank * BNH;
#pragma unroll
            for (int h = 0; h < kHalves; ++h) {       // this CTA's 128 rows of every m-half
              unsigned char* sa = sa0 + h * kStageA;
              const int arow = (int)p.row_off[tc.g] + tc.m0 + h * BM + (int)rank * BMH;
              if constexpr (!AT) {   // [rows, K] in memory: one box of 128 rows x 64 K
                tma_load_2d(smem_addr(sa), &p.map_a[s], kb * BK, arow, full0);
              } else {            // [K, rows] in memory: two boxes of 64 K x 64 rows
#pragma unroll
                for (int c = 0; c < BMH / 64; ++c)
                  tma_load_2d(smem_addr(sa + c * (BK * 128)), &p.map_a[s], arow + c * 64, kb * BK, full0);
              }
            }
            if constexpr (!BT) {   // [K, cols] in memory: two boxes of 64 K x 64 columns
#pragma unroll
              for (int c = 0; c < BNH / 64; ++c)
                tma_load_2d(smem_addr(sb + c * (BK * 128)), &p.map_b[s], bcol + c * 64, kb * BK, full0);
            } else {            // [cols, K] in memory: one box of 128 columns x 64 K
              tma_load_2d(smem_addr(sb), &p.map_b[s], kb * BK, bcol, full0);
            }
          }
          __syncwarp();
        }
      }
    }
  producer_done:
    if (*abort_flag && rank == 0 && leader) {
      // give the loads still in flight a bounded chance to land before the CTA goes away
      const long long issued = kb_iter;
      for (long long i = issued > kSt ? issued - kSt : 0; i < issued; ++i) {
        const unsigned long long t0 = now_ns();
        while (!mbar_try(smem_addr(&bar_full[i % kSt]), (unsigned)((i / kSt) & 1)) && now_ns() - t0 < 100000000ull) {
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------ MMA issuer (first CTA of the pair only)
    if (rank == 0) {
      const bool leader = elect_one();
      int slot = 0;
      unsigned round = 0;
      int tile_iter = 0;
      constexpr unsigned idesc = make_idesc(AT, BT);
      for (int tile = first; tile < p.total_tiles; tile += stride, ++tile_iter) {
        if (tile != first) tc = tile_coord(p, tile);
        // Square form: the two accumulators take turns, so a tile's MMAs run while the tile before
        // it is drained.  Tall form: accumulator h belongs to m-half h of every tile; the first
        // m-half may start as soon as ITS accumulator has been drained, the second waits for its own.
        const int acc = MH == 2 ? 0 : (tile_iter & 1);
        const unsigned empty_parity = MH == 2 ? (unsigned)((tile_iter & 1) ^ 1) : (unsigned)(((tile_iter >> 1) & 1) ^ 1);
        if (!mbar_wait_warp(smem_addr(&bar_acc_empty[acc]), empty_parity, abort_flag)) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const int s_lo = p.chain ? 0 : tc.g, s_hi = p.chain ? p.nseg : tc.g + 1;
        unsigned accumulate = 0;
        bool ok = true;
        for (int s = s_lo; s < s_hi && ok; ++s) {
          const int nkb = p.kblocks[s];
          for (int kb = 0; kb < nkb; ++kb, slot = slot + 1 == kSt ? 0 : slot + 1, round ^= (slot == 0)) {
            if (!mbar_wait_warp(smem_addr(&bar_full[slot]), round, abort_flag)) {
              ok = false;
              break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const unsigned sa0 = smem_addr(smem + slot * kStBytes);
            const unsigned sb = sa0 + kStA;
#pragma unroll
            for (int h = 0; h < kHalves; ++h) {
              if (MH == 2 && h == 1 && accumulate == 0) {      // first K-block of the tile: the second accumulator must be free too
                if (!mbar_wait_warp(smem_addr(&bar_acc_empty[1]), empty_parity, abort_flag)) {
                  ok = false;
                  break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
              }
              const unsigned sa = sa0 + h * kStageA;
              const unsigned d_tmem = tmem_base + (MH == 2 ? h : acc) * BN;
              if (leader) {
#pragma unroll
                for (int kk = 0; kk < BK / 16; ++kk) {
                  // K-major tile (A as given, B transposed): rows of 128 bytes = 64 K-elements, 8-row
                  //    groups 1024 bytes apart; 16 K-elements = 32 bytes.
                  // MN-major tile (B as given, A transposed): 64-element chunks of the M / N index
                  //    BK*128 bytes apart, 8-row K groups 1024 bytes apart; 16 K-rows = 2048 bytes.
                  // Each CTA holds its 128 of the pair's 256 rows (A) or columns (B).
                  // (shared-memory addresses are below 256 KiB and the tiles 1024-byte aligned, so the
                  //  start-address field is address >> 4 and stepping it cannot carry out of the field)
                  constexpr unsigned a_lo = desc_lo_fixed(AT ? BK * 128 : 16), b_lo = desc_lo_fixed(BT ? 16 : BK * 128);
                  constexpr unsigned hi = desc_hi_fixed(1024);
                  const unsigned long long da = desc_pack(a_lo + (sa >> 4) + kk * (AT ? 128 : 2), hi);
                  const unsigned long long db = desc_pack(b_lo + (sb >> 4) + kk * (BT ? 2 : 128), hi);
                  umma_bf16(d_tmem, da, db, idesc, kk == 0 ? accumulate : 1u);
                }
              }
              __syncwarp();
            }
            if (!ok) break;
            accumulate = 1;
            if (leader) umma_commit_pair(smem_addr(&bar_empty[slot]));   // slot reusable in both CTAs
            __syncwarp();
          }
        }
        if (!ok) break;
        if (leader) umma_commit_pair(smem_addr(&bar_acc_full[acc]));      // accumulator(s) complete in both CTAs
        __syncwarp();
      }
    }
  } else {
    // ------------------------------------------------ epilogue (warps 2..9, both CTAs)
    const int q = warp & 3;                       // the 32 tensor-memory lanes this warp may read
    const int half = (warp - 2) >> 2;             // which 128 of the 256 columns
    unsigned char* my_epi = epi + (warp - 2) * kEB * kSlabBytes;
    const int cols_per_slab = p.out_f32 ? 32 : 64;
    const int nslabs = (BN / 2) / cols_per_slab;
    const unsigned acc_empty0[2] = {map_to_cta(smem_addr(&bar_acc_empty[0]), 0), map_to_cta(smem_addr(&bar_acc_empty[1]), 0)};
    int tile_iter = 0;
    unsigned slab_iter = 0;
    for (int tile = first; tile < p.total_tiles; tile += stride, ++tile_iter) {
      if (*abort_flag) break;
      if (tile != first) tc = tile_coord(p, tile);
      const int facc = MH == 2 ? 0 : (tile_iter & 1);
      bool ok = true;
      if (lane == 0)
        ok = mbar_wait(smem_addr(&bar_acc_full[facc]), MH == 2 ? (unsigned)(tile_iter & 1) : (unsigned)((tile_iter >> 1) & 1), abort_flag);
      ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
      if (!ok) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const long long Mg = p.m[tc.g], Ng = p.n[tc.g];
      // tall form: the accumulator of the first m-half is drained (and handed back) before the second
#pragma unroll 1
      for (int h = 0; h < kHalves; ++h) {
      const int acc = MH == 2 ? h : facc;
      const int row0 = tc.m0 + h * BM + (int)rank * BMH + q * 32;
      const unsigned taddr = tmem_base + ((unsigned)(q * 32) << 16) + acc * BN + half * (BN / 2);
      if (p.xent == 1) {
        // Softmax partials of this warp's 32 rows x 128 columns; one thread owns one row, so
        // nothing crosses lanes.  Columns are taken 32 at a time: batch max, then the running
        // (m, s) is rescaled and the batch's exponentials are added.
        const int colbase = tc.n0 + half * (BN / 2);
        const long long row = row0 + lane;
        if (row0 < Mg && colbase < Ng) {            // warp-uniform
          float m = -INFINITY, s = 0.f, t = 0.f;
          long long want = -1;
          if (row < Mg && SBP_GUARD(p.xf.labels + row, 8)) want = p.xf.labels[row] - p.xf.class_start[tc.g] - colbase;
          for (int b = 0; b < 4; ++b) {
            const int c0 = colbase + b * 32;
            if (c0 >= Ng) break;                      // warp-uniform
            float v[32];
            tmem_ld32(taddr + b * 32, v);
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
            const int nvalid = (int)min((long long)32, Ng - c0);
            if (nvalid < 32) {
#pragma unroll
              for (int i = 0; i < 32; ++i)
                if (i >= nvalid) v[i] = -INFINITY;
            }
            float bm = v[0];
#pragma unroll
            for (int i = 1; i < 32; ++i) bm = fmaxf(bm, v[i]);
            const float mm = fmaxf(m, bm);
            const float carried = m != -INFINITY ? s * exp_one(m, mm, 0.f) : 0.f;
            const unsigned long long neg = two(-mm);
            float s0 = 0.f, s1 = 0.f;
#pragma unroll
            for (int i = 0; i < 32; i += 2) {
              exp_two(v[i], v[i + 1], neg, 0ull);
              s0 += v[i];
              s1 += v[i + 1];
            }
            s = carried + (s0 + s1);
            m = mm;
          }
          // The label's logit: rows whose label falls inside this chunk (rare) re-read that one
          // column from tensor memory, one row at a time so the load stays warp-uniform.
          const long long ncols = min((long long)(BN / 2), Ng - colbase);
          unsigned hits = __ballot_sync(0xffffffffu, want >= 0 && want < ncols);
          while (hits) {
            const int src_lane = __ffs(hits) - 1;
            hits &= hits - 1;
            const int col = __shfl_sync(0xffffffffu, (int)want, src_lane);
            unsigned bitsv;
            asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(bitsv) : "r"(taddr + col) : "memory");
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
            if (lane == src_lane) t = __uint_as_float(bitsv);
          }
          if (row < Mg) {
            const long long slot = (long long)(p.xf.part_base[tc.g] + colbase / 128) * p.xf.rows + row;
            if (SBP_GUARD(p.xf.part_m + slot, 4)) p.xf.part_m[slot] = m;
            if (SBP_GUARD(p.xf.part_s + slot, 4)) p.xf.part_s[slot] = s;
            if (SBP_GUARD(p.xf.part_t + slot, 4)) p.xf.part_t[slot] = t;
          }
        }
      } else {
      // The element-wise modes are compiled apart (MODE 0 plain, 1 GeLU, 2 softmax - onehot of the
      // recomputed logits) so that the plain store, which the short-K classifier product leans
      // on, carries none of the others' instructions.
      auto slabs = [&](auto mode_tag) {
        constexpr int MODE = decltype(mode_tag)::value;
        // softmax = 2^((z - m) log2e - log2 S): the division by the row sum is folded into the exponent
        float g_max = 0.f, g_neg = 0.f;       // this thread's row
        long long g_lab = -1;
        if constexpr (MODE == 2) {
          const long long row = row0 + lane;
          if (row < Mg && SBP_GUARD(p.xf.row_max + row, 4) && SBP_GUARD(p.xf.row_sum + row, 4) && SBP_GUARD(p.xf.labels + row, 8)) {
            g_max = p.xf.row_max[row];
            g_neg = -log2f(p.xf.row_sum[row]);
            g_lab = p.xf.labels[row] - p.xf.class_start[tc.g];
          }
        }
        int lab_rel = -1;   // the label's column inside the current slab, if it lies there
        auto xform = [&](float& a, float& b) {
          if constexpr (MODE == 1) gelu_two(a, b);
          if constexpr (MODE == 2) {      // (as a pair its constants took two registers more: the kernel spilled, GeLU was 2 % slower)
            a = exp_one(a, g_max, g_neg);
            b = exp_one(b, g_max, g_neg);
          }                               // the label's column gets its -1 below
        };
        for (int sl = 0; sl < nslabs; ++sl) {
          const int col0 = tc.n0 + half * (BN / 2) + sl * cols_per_slab;
          const bool live = row0 < Mg && col0 < Ng;   // warp-uniform
          if constexpr (MODE == 2) lab_rel = (g_lab >= col0 && g_lab < col0 + cols_per_slab) ? (int)(g_lab - col0) : -1;
          float v[64];
          if (live) {
            tmem_ld32(taddr + sl * cols_per_slab, v);
            if (!p.out_f32) tmem_ld32(taddr + sl * cols_per_slab + 32, v + 32);
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
            unsigned char* buf = my_epi + (slab_iter % kEB) * kSlabBytes;
            // the store that last used this buffer must have finished reading it
            if (lane == 0) asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(kEB - 1) : "memory");
            __syncwarp();
            unsigned char* rowp = buf + lane * 128;
            if (p.out_f32) {
#pragma unroll
              for (int c = 0; c < 8; ++c) {
                float4 o;
                xform(v[4 * c], v[4 * c + 1]);
                xform(v[4 * c + 2], v[4 * c + 3]);
                o.x = v[4 * c]; o.y = v[4 * c + 1]; o.z = v[4 * c + 2]; o.w = v[4 * c + 3];
                *reinterpret_cast<float4*>(rowp + ((c ^ (lane & 7)) << 4)) = o;
              }
            } else {
#pragma unroll
              for (int c = 0; c < 8; ++c) {
                float f[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) f[e] = v[8 * c + e];
#pragma unroll
                for (int e = 0; e < 8; e += 2) xform(f[e], f[e + 1]);
                uint4 o;
                __nv_bfloat162 h;
                h = __floats2bfloat162_rn(f[0], f[1]); o.x = *reinterpret_cast<unsigned*>(&h);
                h = __floats2bfloat162_rn(f[2], f[3]); o.y = *reinterpret_cast<unsigned*>(&h);
                h = __floats2bfloat162_rn(f[4], f[5]); o.z = *reinterpret_cast<unsigned*>(&h);
                h = __floats2bfloat162_rn(f[6], f[7]); o.w = *reinterpret_cast<unsigned*>(&h);
                *reinterpret_cast<uint4*>(rowp + ((c ^ (lane & 7)) << 4)) = o;
              }
            }
            if constexpr (MODE == 2) {
              // softmax - onehot: a row's label falls into this slab once in 2^14 slabs, so the -1 is
              // not a compare and a select on every element but a rare fix-up: the column is read
              // again from tensor memory (one row at a time, so the load stays warp-uniform) and the
              // staged element rewritten with exp - 1 computed in fp32 as before.
              unsigned hits = __ballot_sync(0xffffffffu, lab_rel >= 0);
              while (hits) {
                const int src_lane = __ffs(hits) - 1;
                hits &= hits - 1;
                const int col = __shfl_sync(0xffffffffu, lab_rel, src_lane);
                unsigned bitsv;
                asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(bitsv) : "r"(taddr + sl * cols_per_slab + col) : "memory");
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                if (lane == src_lane) {
                  const float e = exp_one(__uint_as_float(bitsv), g_max, g_neg) - 1.0f;
                  if (p.out_f32) *reinterpret_cast<float*>(rowp + (((col >> 2) ^ (lane & 7)) << 4) + ((col & 3) << 2)) = e;
                  else *reinterpret_cast<__nv_bfloat16*>(rowp + (((col >> 3) ^ (lane & 7)) << 4) + ((col & 7) << 1)) = __float2bfloat16_rn(e);
                }
              }
              __syncwarp();
            }
            if (p.y_direct) {
              // eight lanes to a row of the slab, four rows at a time
              __syncwarp();
              const int n_out = (tc.g == 0 ? p.n_rep : 0) + 1, esz = p.out_f32 ? 4 : 2;
              const int bytes = (int)min((long long)cols_per_slab, Ng - col0) * esz;
              for (int o = 0; o < n_out; ++o) {
                unsigned char* yb = static_cast<unsigned char*>(o == 0 ? p.y_ptr[tc.g] : p.rep_ptr[o - 1]) + col0 * esz;
                const long long ld = p.ldy[tc.g];
#pragma unroll 4
                for (int r = lane >> 3; r < 32; r += 4) {
                  if (row0 + r >= Mg) break;
                  auto at = [&](int off) { return buf + r * 128 + ((((off >> 4) ^ (r & 7)) << 4) | (off & 15)); };
                  if (p.out_f32) store_shifted<4>(yb + (row0 + r) * ld * 4, bytes, lane & 7, 8, at);
                  else store_shifted<2>(yb + (row0 + r) * ld * 2, bytes, lane & 7, 8, at);
                }
              }
              __syncwarp();      // every lane has read the slab before its buffer is staged again
            } else {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) {
              tma_store_2d(&p.map_y[tc.g], col0, row0, smem_addr(buf));
              if (tc.g == 0)
                for (int r = 0; r < p.n_rep; ++r) tma_store_2d(&p.map_rep[r], col0, row0, smem_addr(buf));
              asm volatile("cp.async.bulk.commit_group;" ::: "memory");
            }
            }
            ++slab_iter;
          }
        }
      };
      if (p.xent == 2) slabs(std::integral_constant<int, 2>{});
      else if (p.gelu) slabs(std::integral_constant<int, 1>{});
      else slabs(std::integral_constant<int, 0>{});
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(acc_empty0[acc]);   // tells CTA 0's MMA thread
      }
    }
    // done with tensor memory and barriers; what is left is the stores
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncwarp();
    cluster_arrive();
    if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    __syncwarp();
    cluster_wait();
    return;
  }

  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncwarp();
  cluster_arrive();
  cluster_wait();              // the partner may still signal this CTA's barriers or read its tiles
  if (warp == 1) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kTmemCols) : "memory");
  }
}

// ------------------------------------------------------------------ the split form
//
// A product with fewer 256 x 256 tiles than the device has CTA pairs leaves pairs idle for its whole
// contraction (a fused P(sum) product of 512 x 512 over 2^20 classes: 4 tiles of 16384 K-blocks, 4.6 ms on
// four of 74 pairs), and one with few rows multiplies padding.  Here a tile belongs to a CLUSTER of
// `splits` pairs, each of which multiplies its own range of the K-blocks into its own tensor memory; the
// partial accumulators are then added up through distributed shared memory: the tile's columns are dealt
// out to the pairs, every other pair pushes its partial sums of those columns into the owner's shared
// memory (which its ring no longer needs), and the owner adds the slices in ascending order (the same bits
// every time), applies GeLU and stores.  No workspace and no atomics.  Where even eight pairs a tile leave
// pairs idle and the caller gave a workspace, the K-blocks are cut further, over several clusters, whose fp32
// results matmul_parts_kernel adds up in order (512 x 512 over 2^20 classes: 72 pairs instead of 40).
//   NB  columns of a tile.  A tile is 256 rows x NB; narrower ones give more tiles, or less padding.
//   SW  the operands are exchanged by the host, Y^T = W^T X^T: the tile's rows are then columns of the
//       result and its NB columns are rows of it.  A product of few rows so spends its tile on them: the
//       weight streams through shared memory as the 256-row operand with NB = 32 columns beside it, 18 KiB
//       a K-block and CTA of which 16 are weight, ten K-blocks deep.
// One tile per cluster, so nothing is persistent; results leave through shared memory as whole 16-byte
// pieces of rows (element by element where base or pitch is not aligned).
struct TcSplitParams {
  CUtensorMap map_a[SBP_MAX_K];
  CUtensorMap map_b[SBP_MAX_K];
  long long m[SBP_MAX_K], n[SBP_MAX_K], row_off[SBP_MAX_K], col_off[SBP_MAX_K], ldy[SBP_MAX_K];
  void* y_ptr[SBP_MAX_K];
  void* rep_ptr[SBP_MAX_K];
  int kblocks[SBP_MAX_K];
  int tile_begin[SBP_MAX_K + 1];
  int tiles_m[SBP_MAX_K];
  int ngroups, nseg, chain, gelu, n_rep, out_f32;
  int splits;
  int y_vec;                     // 16-byte stores are possible everywhere
  // row blocks of one fused result, as S(0) cuts it: multiplied as one product (group 0), block b's rows from
  // block_row[b] on stored to block_y[b].  0: every group has a result of its own
  int blocks;
  long long block_row[SBP_MAX_K + 1];
  void* block_y[SBP_MAX_K];
  int tiles, outer;              // outer > 1: cluster c works on tile c mod tiles and part c / tiles of its K-blocks ...
  long long part_bytes;          // ... and writes fp32 partial results this far apart, which a second kernel adds up
};

// A ring slot holds kGroup K-blocks behind one pair of barriers: whatever its size, a round of waits, issue and
// bookkeeping costs either single-issue role some 480 clocks, and a K-block of a narrow tile is worth 64-256
// clocks of the tensor pipe.
constexpr int kGroup = 2;
constexpr int kMaxSplits = 8;         // a cluster has at most 16 CTAs
template <int NB>
constexpr int split_block_bytes() { return kStageA + BK * NB; }        // B: 64 x NB/2 elements of 2 bytes per CTA
constexpr int kSplitRing = 192 * 1024;
template <int NB>
constexpr int split_stages() { return kSplitRing / (kGroup * split_block_bytes<NB>()); }      // 3 (NB = 256), 4, 4, 5 (NB = 32)
constexpr int kSmemSplit = kSplitRing + 1024;                                       // + alignment slack

template <int AT, int BT, int NB, int SW>
__global__ void __launch_bounds__(kThreadsTc, 1) matmul_tc_split_kernel(const __grid_constant__ TcSplitParams p) {
  constexpr int kSt = split_stages<NB>(), kBlk = split_block_bytes<NB>(), kBH = NB / 2;
  static_assert(BT || kBH % 64 == 0, "an N-major B tile comes in boxes of 64 columns");
  extern __shared__ unsigned char smem_raw[];
  __shared__ __align__(8) unsigned long long bar_full[kSt], bar_empty[kSt], bar_acc;
  __shared__ unsigned tmem_base_slot;
  __shared__ int abort_flag_s;
  volatile int* abort_flag = &abort_flag_s;

  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const unsigned crank = cluster_ctarank(), rank = crank & 1, even = crank & ~1u;      // `even` issues its pair's MMAs
  const int S = p.splits, slice = (int)(crank >> 1);

  if (threadIdx.x == 0) {
    abort_flag_s = 0;
    for (int i = 0; i < kSt; ++i) {
      mbar_init(smem_addr(&bar_full[i]), 1);      // used in the even CTA only
      mbar_init(smem_addr(&bar_empty[i]), 1);
    }
    mbar_init(smem_addr(&bar_acc), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&tmem_base_slot)), "r"(NB)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncwarp();
  cluster_arrive();            // and under this barrier: this cluster's tile and this pair's range of its K-blocks
  const int cluster = (int)(blockIdx.x / (unsigned)(2 * S)), part = p.outer > 1 ? cluster / p.tiles : 0;
  const int tile = cluster - part * p.tiles;
  int g = 0;
  while (g + 1 < p.ngroups && tile >= p.tile_begin[g + 1]) ++g;
  const int local = tile - p.tile_begin[g], nt = local / p.tiles_m[g], mt = local - nt * p.tiles_m[g];
  const int m0 = mt * BM, n0 = nt * NB;
  const int s_lo = p.chain ? 0 : g, s_hi = p.chain ? p.nseg : g + 1;
  long long total = 0;
  for (int s = s_lo; s < s_hi; ++s) total += p.kblocks[s];
  const int cuts = S * p.outer, cut = part * S + slice;
  const int it0 = (int)(total * cut / cuts), iters = (int)(total * (cut + 1) / cuts) - it0;
  if (warp == 2 && lane == 0) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(&p.map_a[s_lo]) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&p.map_b[s_lo]) : "memory");
  }
  cluster_wait();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const unsigned tmem_base = tmem_base_slot;
  bool ok = true;
  // Everything up to here overlaps the kernel before this one, the fetch of the descriptors included: a layer step of
  // 147 x 584 x 416 takes 22.3 us so, 23.9 with the wait after the set-up and the prefetch after that.  (Letting the next
  // kernel in at the start, where a product has few CTAs, gave nothing more.)
  SBP_PDL_WAIT();

  if (warp == 0) {
    // ------------------------------------------------ producer (both CTAs of every pair)
    const bool leader = elect_one();
    int seg = s_lo, kb = it0, slot = 0, rounds = 0;
    unsigned round = 0;
    while (seg < s_hi && kb >= p.kblocks[seg]) kb -= p.kblocks[seg++];
    int nkb = seg < s_hi ? p.kblocks[seg] : 0;
    const int arow = (int)p.row_off[g] + m0 + (int)rank * BMH, bcol = (int)p.col_off[g] + n0 + (int)rank * kBH;
    for (int left = iters; left > 0; left -= kGroup, ++rounds) {
      if (!mbar_wait_warp(smem_addr(&bar_empty[slot]), round ^ 1, abort_flag)) break;
      const unsigned full0 = map_to_cta(smem_addr(&bar_full[slot]), even);
      if (leader && rank == 0) mbar_expect_tx(smem_addr(&bar_full[slot]), 2 * kBlk * (left < kGroup ? left : kGroup));
#pragma unroll
      for (int b = 0; b < kGroup; ++b) {
        if (b >= left) break;
        if (leader) {
          unsigned char* sa = smem + (slot * kGroup + b) * kBlk;
          unsigned char* sb = sa + kStageA;
          if constexpr (!AT) {
            tma_load_2d(smem_addr(sa), &p.map_a[seg], kb * BK, arow, full0);
          } else {
#pragma unroll
            for (int c = 0; c < BMH / 64; ++c) tma_load_2d(smem_addr(sa + c * (BK * 128)), &p.map_a[seg], arow + c * 64, kb * BK, full0);
          }
          if constexpr (!BT) {
#pragma unroll
            for (int c = 0; c < kBH / 64; ++c) tma_load_2d(smem_addr(sb + c * (BK * 128)), &p.map_b[seg], bcol + c * 64, kb * BK, full0);
          } else {
            tma_load_2d(smem_addr(sb), &p.map_b[seg], kb * BK, bcol, full0);
          }
        }
        __syncwarp();
        if (++kb >= nkb) {
          kb = 0;
          do nkb = ++seg < s_hi ? p.kblocks[seg] : 1; while (nkb == 0);      // steps over empty segments
        }
      }
      slot = slot + 1 == kSt ? 0 : slot + 1;
      round ^= (slot == 0);
    }
    if (*abort_flag && rank == 0 && leader) {
      // give the loads still in flight a bounded chance to land before the CTA goes away
      for (int i = rounds > kSt ? rounds - kSt : 0; i < rounds; ++i) {
        const unsigned long long t0 = now_ns();
        while (!mbar_try(smem_addr(&bar_full[i % kSt]), (unsigned)((i / kSt) & 1)) && now_ns() - t0 < 100000000ull) {
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------ MMA issuer (the even CTA of every pair)
    if (rank == 0) {
      const bool leader = elect_one();
      const unsigned short pair_mask = (unsigned short)(3u << even);
      constexpr unsigned idesc = make_idesc(AT, BT, NB);
      int slot = 0;
      unsigned round = 0, accumulate = 0;
      for (int left = iters; left > 0; left -= kGroup) {
        if (!mbar_wait_warp(smem_addr(&bar_full[slot]), round, abort_flag)) {
          ok = false;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        // a shared-memory address carries the CTA's rank in its high bits; a descriptor takes the offset alone
        const unsigned s0 = smem_addr(smem + slot * kGroup * kBlk) & 0x3ffffu;
        if (leader) {
#pragma unroll
          for (int b = 0; b < kGroup; ++b) {
            if (b >= left) break;
            const unsigned sa = s0 + b * kBlk, sb = sa + kStageA;
#pragma unroll
            for (int kk = 0; kk < BK / 16; ++kk) {        // descriptors as in the persistent kernel
              constexpr unsigned a_lo = desc_lo_fixed(AT ? BK * 128 : 16), b_lo = desc_lo_fixed(BT ? 16 : BK * 128);
              constexpr unsigned hi = desc_hi_fixed(1024);
              umma_bf16(tmem_base, desc_pack(a_lo + (sa >> 4) + kk * (AT ? 128 : 2), hi), desc_pack(b_lo + (sb >> 4) + kk * (BT ? 2 : 128), hi),
                        idesc, (b > 0 || kk > 0) ? 1u : accumulate);
            }
          }
          umma_commit_pair(smem_addr(&bar_empty[slot]), pair_mask);
        }
        __syncwarp();
        accumulate = 1;
        slot = slot + 1 == kSt ? 0 : slot + 1;
        round ^= (slot == 0);
      }
      if (leader && ok) umma_commit_pair(smem_addr(&bar_acc), pair_mask);
      __syncwarp();
    }
  }

  // Epilogue warps 2..9: tensor-memory lanes 32 q .. 32 q + 31.  The tile's columns are dealt to the pairs in groups
  // of 8, `per` groups each (the last owner may have fewer, the last pairs none); of an owner's groups the first
  // warp of a lane quadrant takes the first half, the second warp the rest.
  constexpr int kCg = NB / 8;
  const int q = warp & 3, half = (warp - 2) >> 2;
  const long long Mg = p.m[g], Ng = p.n[g];
  const int row0 = m0 + (int)rank * BMH + q * 32;
  const int per = (kCg + S - 1) / S;
  const bool rows_live = warp >= 2 && row0 < Mg;       // warp-uniform
  const unsigned tq = tmem_base + ((unsigned)(q * 32) << 16);
  // this warp's column groups of owner o, counted from the owner's first
  auto mine = [&](int o, int* lo, int* hi) {
    const int have = kCg - o * per < per ? kCg - o * per : per;
    *lo = half ? (have + 1) / 2 : 0;
    *hi = half ? have : (have + 1) / 2;
  };
  if (warp >= 2) {
    ok = lane != 0 || mbar_wait(smem_addr(&bar_acc), 0, abort_flag);
    ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  }
  SBP_PDL_RELEASE();
  if (S > 1) {
    cluster_sync_all();                                // every pair is done with its ring
    if (rows_live && ok) {
      for (int d = 1; d < S; ++d) {
        const int o = slice + d < S ? slice + d : slice + d - S;
        int lo, hi;
        mine(o, &lo, &hi);
        if (lo >= hi) continue;
        const int from = slice < o ? slice : slice - 1;              // my place among o's S - 1 sources
        const unsigned dst = map_to_cta(smem_addr(smem) + (unsigned)(from * per * (BMH * 32)), (unsigned)(2 * o) + rank);
        for (int c = lo; c < hi; ++c) {
          float v[8];
          tmem_ld8(tq + (o * per + c) * 8, v);
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
          const unsigned at = dst + (unsigned)(2 * c * BMH + q * 32 + lane) * 16u;      // [4-column group][row]
#pragma unroll
          for (int e = 0; e < 2; ++e)
            asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(at + e * BMH * 16u), "f"(v[4 * e]), "f"(v[4 * e + 1]),
                         "f"(v[4 * e + 2]), "f"(v[4 * e + 3])
                         : "memory");
        }
      }
    }
    cluster_sync_all();                                // all partial sums have arrived
  }
  int lo, hi;
  mine(slice, &lo, &hi);
  const int col0 = n0 + (slice * per + lo) * 8;
  const bool mine_live = rows_live && ok && lo < hi && col0 < Ng;      // warp-uniform
  const int esz = p.out_f32 ? 4 : 2, cols = (hi - lo) * 8;
  const int pitch = SW ? 32 * esz : cols * esz + 16;
  unsigned char* stage = smem + (S - 1) * per * (BMH * 32) + (warp - 2) * (32 * ((per + 1) / 2 * 8 * esz + 16));
  if (mine_live) {
    // Staged per warp as rows of the RESULT: 32 rows of `cols` elements, 16 bytes apart so that 32 rows written at
    // once spread over the banks (SW: `cols` rows of 32 elements).
    // eight finished sums of this lane's row, columns cc .. cc + 7 of the warp's
    auto put = [&](int cc, float* v) {
      if (p.gelu) {
#pragma unroll
        for (int e = 0; e < 8; e += 2) gelu_two(v[e], v[e + 1]);
      }
      if constexpr (SW) {
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          unsigned char* at = stage + (cc + e) * pitch + lane * esz;
          if (p.out_f32) *reinterpret_cast<float*>(at) = v[e];
          else *reinterpret_cast<__nv_bfloat16*>(at) = __float2bfloat16_rn(v[e]);
        }
      } else {
        unsigned char* at = stage + lane * pitch + cc * esz;
        if (p.out_f32) {
          *reinterpret_cast<float4*>(at) = make_float4(v[0], v[1], v[2], v[3]);
          *reinterpret_cast<float4*>(at + 16) = make_float4(v[4], v[5], v[6], v[7]);
        } else {
          uint4 o;
          __nv_bfloat162 h;
          h = __floats2bfloat162_rn(v[0], v[1]); o.x = *reinterpret_cast<unsigned*>(&h);
          h = __floats2bfloat162_rn(v[2], v[3]); o.y = *reinterpret_cast<unsigned*>(&h);
          h = __floats2bfloat162_rn(v[4], v[5]); o.z = *reinterpret_cast<unsigned*>(&h);
          h = __floats2bfloat162_rn(v[6], v[7]); o.w = *reinterpret_cast<unsigned*>(&h);
          *reinterpret_cast<uint4*>(at) = o;
        }
      }
    };
    if (S == 1) {            // nothing to add: up to 32 columns a load
      constexpr int kG = NB / 16 < 4 ? NB / 16 : 4;
      for (int c = lo; c < hi; c += kG) {
        float v[8 * kG];
        if constexpr (kG == 4) {
          tmem_ld32(tq + c * 8, v);
        } else {
#pragma unroll
          for (int i = 0; i < kG; ++i) tmem_ld8(tq + (c + i) * 8, v + 8 * i);
        }
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
        for (int i = 0; i < kG; ++i) put((c + i - lo) * 8, v + 8 * i);
      }
    } else {
      for (int c = lo; c < hi; ++c) {
        float v[8], own[8];
        tmem_ld8(tq + (slice * per + c) * 8, own);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        for (int s = 0; s < S; ++s) {
          float x[8];
          if (s == slice) {
#pragma unroll
            for (int e = 0; e < 8; ++e) x[e] = own[e];
          } else {
            const int from = s < slice ? s : s - 1;
            const unsigned char* at = smem + from * per * (BMH * 32) + (2 * c * BMH + q * 32 + lane) * 16;
            *reinterpret_cast<float4*>(x) = *reinterpret_cast<const float4*>(at);
            *reinterpret_cast<float4*>(x + 4) = *reinterpret_cast<const float4*>(at + BMH * 16);
          }
#pragma unroll
          for (int e = 0; e < 8; ++e) v[e] = s == 0 ? x[e] : v[e] + x[e];
        }
        put((c - lo) * 8, v);
      }
    }
  }
  // done with tensor memory and with what the other CTAs may signal or write; what is left is the stores
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncwarp();
  cluster_arrive();
  if (mine_live) {
    // Out: consecutive lanes take consecutive 16-byte pieces of a row of the result.  Where a row lies is worked out once, by
    // the lane of its number, and handed round; row and piece are stepped, not divided out.  (Both for every piece of every
    // row: the stores of [2048 x 1024]^T [2048 x 4096] in 256 x 256 tiles to eight row blocks took 9.9 us, 3.7 so; one
    // result a device, 256 x 128 tiles 3.9, 2.5.)
    const int el = 16 / esz, pieces = (SW ? 4 : hi - lo) << (p.out_f32 ? 1 : 0), nrows = SW ? cols : 32;
    const long long yr0 = SW ? col0 : row0, yc0 = SW ? row0 : col0, yrows = SW ? Ng : Mg, ycols = SW ? Mg : Ng;
    const int n_out = (g == 0 ? p.n_rep : 0) + 1;
    const long long row_bytes = p.ldy[g] * esz;
    const int left = (int)min((long long)pieces * el, ycols - yc0);      // columns this warp has
    // where row r starts, from the start of the result (row blocks: its address)
    auto row_at = [&](int r) -> unsigned long long {
      const long long row = yr0 + r;
      if (!p.blocks) return (unsigned long long)(row * row_bytes + yc0 * esz);
      int b = 0;
      while (b + 1 < p.blocks && row >= p.block_row[b + 1]) ++b;
      return reinterpret_cast<unsigned long long>(p.block_y[b]) + (unsigned long long)((row - p.block_row[b]) * row_bytes + yc0 * esz);
    };
    const unsigned long long at0 = row_at(lane), at1 = SW && NB > 64 ? row_at(lane + 32) : 0ull;
    unsigned char* const y0 = p.blocks ? nullptr : static_cast<unsigned char*>(p.y_ptr[g]) + part * p.part_bytes;
    const int log2p = 31 - __clz(pieces);
    const bool pow2 = (1 << log2p) == pieces;
    int r = pow2 ? lane >> log2p : lane / pieces, ch = lane - r * pieces;
    const int dr = pow2 ? 32 >> log2p : 32 / pieces, dc = 32 - dr * pieces;
    const int total = (int)min((long long)nrows, yrows - yr0) * pieces;
    auto step = [&](auto vec, auto one) {
#pragma unroll 4
      for (int i = 0; i < total; i += 32) {
        unsigned long long off = __shfl_sync(0xffffffffu, at0, r & 31);
        if (SW && NB > 64) {
          const unsigned long long far = __shfl_sync(0xffffffffu, at1, r & 31);
          if (r >= 32) off = far;
        }
        if (i + lane < total) {
          uint4 v;
          if constexpr (decltype(vec)::value) v = *reinterpret_cast<const uint4*>(stage + r * pitch + ch * 16);
          for (int o = 0; o < (decltype(one)::value ? 1 : n_out); ++o) {
            unsigned char* at = (o == 0 ? y0 : static_cast<unsigned char*>(p.rep_ptr[o - 1])) + off;
            if constexpr (!decltype(vec)::value) {
              auto in = [&](int b) { return stage + r * pitch + b; };
              if (p.out_f32) store_shifted<4>(at, left * 4, ch, pieces, in);
              else store_shifted<2>(at, left * 2, ch, pieces, in);
            } else {
              at += ch * 16;
              if ((ch + 1) * el <= left) {
                if (SBP_GUARD(at, 16)) *reinterpret_cast<uint4*>(at) = v;
              } else if (p.out_f32) {
                const float* f = reinterpret_cast<const float*>(&v);
#pragma unroll
                for (int e = 0; e < 3; ++e)
                  if (ch * el + e < left && SBP_GUARD(at + 4 * e, 4)) reinterpret_cast<float*>(at)[e] = f[e];
              } else {
                const unsigned short* f = reinterpret_cast<const unsigned short*>(&v);
#pragma unroll
                for (int e = 0; e < 7; ++e)
                  if (ch * el + e < left && SBP_GUARD(at + 2 * e, 2)) reinterpret_cast<unsigned short*>(at)[e] = f[e];
              }
            }
          }
        }
        r += dr;
        ch += dc;
        if (ch >= pieces) {
          ch -= pieces;
          ++r;
        }
      }
    };
    if (!p.y_vec) step(std::false_type{}, std::false_type{});
    else if (n_out == 1) step(std::true_type{}, std::true_type{});
    else step(std::true_type{}, std::false_type{});
  }
  __syncwarp();
  cluster_wait();
  if (warp == 1) {
    __syncwarp();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(NB) : "memory");
  }
}

// Adds up the fp32 results of a contraction cut over several clusters, in order, applies GeLU and stores the
// result and its replicas.  Four columns a thread; eight parts are in flight at once.
struct PartsParams {
  const float* part[SBP_MAX_K];        // group g's first part: rows of ld[g] floats
  long long m[SBP_MAX_K], n[SBP_MAX_K], ld[SBP_MAX_K], ldy[SBP_MAX_K];
  void* y_ptr[SBP_MAX_K];
  void* rep_ptr[SBP_MAX_K];
  long long stride;                    // floats between parts
  int parts, gelu, n_rep, out_f32, y_vec;
};

__global__ void __launch_bounds__(256) matmul_parts_kernel(const __grid_constant__ PartsParams p) {
  SBP_PDL_RELEASE();
  const int g = blockIdx.y;
  const long long quads = p.ld[g] / 4, total = p.m[g] * quads;
  SBP_PDL_WAIT();
  for (long long i = (long long)blockIdx.x * 256 + threadIdx.x; i < total; i += (long long)gridDim.x * 256) {
    const long long row = i / quads, c = (i - row * quads) * 4;
    const float* at = p.part[g] + row * p.ld[g] + c;
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int q0 = 0; q0 < p.parts; q0 += 8) {
      float4 x[8];
#pragma unroll
      for (int q = 0; q < 8; ++q)
        if (q0 + q < p.parts && SBP_GUARD(at + (q0 + q) * p.stride, 16)) x[q] = __ldcg(reinterpret_cast<const float4*>(at + (q0 + q) * p.stride));
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        if (q0 + q >= p.parts) continue;
        if (q0 + q == 0) {
          v = x[0];
        } else {
          v.x += x[q].x; v.y += x[q].y; v.z += x[q].z; v.w += x[q].w;
        }
      }
    }
    float f[4] = {v.x, v.y, v.z, v.w};
    if (p.gelu) {
#pragma unroll
      for (int e = 0; e < 4; e += 2) gelu_two(f[e], f[e + 1]);
    }
    const int n_out = (g == 0 ? p.n_rep : 0) + 1;
    for (int o = 0; o < n_out; ++o) {
      void* y = o == 0 ? p.y_ptr[g] : p.rep_ptr[o - 1];
      if (p.out_f32) {
        float* d = static_cast<float*>(y) + row * p.ldy[g] + c;
        if (p.y_vec && c + 4 <= p.n[g]) {
          if (SBP_GUARD(d, 16)) *reinterpret_cast<float4*>(d) = make_float4(f[0], f[1], f[2], f[3]);
        } else {
#pragma unroll
          for (int e = 0; e < 4; ++e)
            if (c + e < p.n[g] && SBP_GUARD(d + e, 4)) d[e] = f[e];
        }
      } else {
        __nv_bfloat16* d = static_cast<__nv_bfloat16*>(y) + row * p.ldy[g] + c;
        if (p.y_vec && c + 4 <= p.n[g]) {
          const __nv_bfloat162 lo = __floats2bfloat162_rn(f[0], f[1]), hi = __floats2bfloat162_rn(f[2], f[3]);
          if (SBP_GUARD(d, 8))
            *reinterpret_cast<uint2*>(d) = make_uint2(*reinterpret_cast<const unsigned*>(&lo), *reinterpret_cast<const unsigned*>(&hi));
        } else {
#pragma unroll
          for (int e = 0; e < 4; ++e)
            if (c + e < p.n[g] && SBP_GUARD(d + e, 2)) d[e] = __float2bfloat16_rn(f[e]);
        }
      }
    }
  }
}

// ------------------------------------------------------------------ the fused classifier for few rows
//
// Softmax partials or gradient of the class-split logits, operands exchanged: a tile is 256 CLASSES (128 per CTA of the
// pair) by all NB >= rows rows.  The weight is read once whatever is done, 2 * feat bytes a class, and is the floor for
// few rows; in the persistent kernel above a tile of 256 rows costs its epilogue all the same, of whose warps only
// those that hold the few rows work (14 rows, 176 features, 475 696 classes: 77 us forward, 83 backward, where the
// weight takes 26; here 40 and 39 with what follows the product).  Here the features stay in shared memory, the weight streams past them in K-blocks of
// 16 KB a CTA, and every epilogue warp has 32 classes.
//   forward   a warp turns its 32 classes x 32 rows over in shared memory, so that a lane holds a row: maximum, sum and
//             the label's logit without a shuffle; the four warps of a 128-class chunk are merged through shared memory.
//   backward  a lane is a class; four lanes exchange their rows so that each stores four classes of one.
// With many rows and few features the epilogue is the bound again (its shared-memory and exponential phases, some 1850
// clocks a batch): 192 features, 161 472 classes, forward / backward: 32 rows 20.5 / 17.9 (persistent kernel 35.7 / 36.2),
// 64 rows 23.5 / 21.4 (36 / 37), 128 rows 33 / 30 (37 / 38.5), where the line is; above it the rows need a second tile.
// 512 features, 2^20 classes, 64 rows: 171 / 192 (223 / 225), the weight's 164 us and the gradient's 21.
struct NarrowParams {
  CUtensorMap map_w[SBP_MAX_K];       // [feat, classes of shard g], boxes of 64 x 64
  CUtensorMap map_f;                  // [rows, feat], boxes of NB / 2 rows x 64
  long long n[SBP_MAX_K], ldy[SBP_MAX_K], class_start[SBP_MAX_K];
  void* y[SBP_MAX_K];
  int tile_begin[SBP_MAX_K + 1];
  int ngroups, kblocks, rows, out_f32, stages;
  int y_quads;                        // bf16 gradient whose rows take 8-byte stores, classes by the four
  XentFusion xf;
};

constexpr int kNarrowRows = 128;
constexpr int kNarrowMaxStages = 12;
constexpr int kNarrowAccs = 4;                                 // accumulators of NB columns in flight
constexpr int kNarrowFeatures = 64 * 1024;                     // most shared memory the features may take
constexpr int kNarrowPitch = 36;                               // floats between the staged classes of a warp
constexpr int kNarrowStageBytes = kEpiWarps * 32 * kNarrowPitch * 4;
constexpr int kNarrowRedBytes = 2 * 2 * 4 * 3 * 32 * 4;        // [half][parity][quadrant][m, s, t][row]
constexpr int kNarrowSmem = 220 * 1024;
template <int NB>
constexpr int narrow_feature_block() { return NB / 2 * 128; }  // one CTA's half of the rows, 64 features

template <int NB, int MODE>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreadsTc, 1) xent_narrow_kernel(const __grid_constant__ NarrowParams p) {
  constexpr int kFb = narrow_feature_block<NB>();
  extern __shared__ unsigned char smem_raw[];
  __shared__ __align__(8) unsigned long long bar_full[kNarrowMaxStages], bar_empty[kNarrowMaxStages], bar_feat, bar_acc_full[kNarrowAccs],
      bar_acc_empty[kNarrowAccs];
  __shared__ unsigned tmem_base_slot;
  __shared__ int abort_flag_s;
  __shared__ __align__(16) float less_s[MODE == 2 ? NB : 4], neg_s[MODE == 2 ? NB : 4];
  __shared__ long long lab_s[NB];
  volatile int* abort_flag = &abort_flag_s;

  unsigned char* feat = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  unsigned char* ring = feat + (p.kblocks * kFb + 1023) / 1024 * 1024;
  float* staging = reinterpret_cast<float*>(ring + p.stages * kStageA);
  float* red = staging + kEpiWarps * 32 * kNarrowPitch;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const unsigned rank = cluster_ctarank();

  if (threadIdx.x == 0) {
    abort_flag_s = 0;
    for (int i = 0; i < p.stages; ++i) {
      mbar_init(smem_addr(&bar_full[i]), 1);
      mbar_init(smem_addr(&bar_empty[i]), 1);
    }
    mbar_init(smem_addr(&bar_feat), 1);
    for (int i = 0; i < kNarrowAccs; ++i) {
      mbar_init(smem_addr(&bar_acc_full[i]), 1);
      mbar_init(smem_addr(&bar_acc_empty[i]), NB == 32 ? kEpiWarps : 2 * kEpiWarps);      // used in CTA 0: both CTAs' warps
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&tmem_base_slot)),
                 "r"(kNarrowAccs * NB)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  SBP_PDL_RELEASE();
  SBP_PDL_WAIT();
  if (threadIdx.x < NB) {
    const int row = threadIdx.x;
    lab_s[row] = row < p.rows && SBP_GUARD(p.xf.labels + row, 8) ? p.xf.labels[row] : -1;
    // softmax = 2^((z - m) log2e - log2 S): the division by the row sum is folded into the exponent
    if (MODE == 2 && row < p.rows && SBP_GUARD(p.xf.row_max + row, 4) && SBP_GUARD(p.xf.row_sum + row, 4)) {
      less_s[row] = -p.xf.row_max[row];
      neg_s[row] = -log2f(p.xf.row_sum[row]);
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  cluster_sync_all();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const unsigned tmem_base = tmem_base_slot;

  const int first = blockIdx.x >> 1, stride = gridDim.x >> 1, tiles = p.tile_begin[p.ngroups];
  if (warp == 0) {
    // ------------------------------------------------ producer (both CTAs)
    const bool leader = elect_one();
    if (leader) {
      if (rank == 0) mbar_expect_tx(smem_addr(&bar_feat), 2 * p.kblocks * kFb);
      const unsigned feat0 = map_to_cta(smem_addr(&bar_feat), 0);
      for (int kb = 0; kb < p.kblocks; ++kb) tma_load_2d(smem_addr(feat + kb * kFb), &p.map_f, kb * BK, (int)rank * (NB / 2), feat0);
    }
    __syncwarp();
    int slot = 0, rounds = 0, g = 0;
    unsigned round = 0;
    for (int tile = first; tile < tiles && !*abort_flag; tile += stride) {
      while (tile >= p.tile_begin[g + 1]) ++g;
      const int col = (tile - p.tile_begin[g]) * BM + (int)rank * BMH;
      for (int kb = 0; kb < p.kblocks; ++kb, ++rounds) {
        if (!mbar_wait_warp(smem_addr(&bar_empty[slot]), round ^ 1, abort_flag)) break;
        if (leader) {
          const unsigned full0 = map_to_cta(smem_addr(&bar_full[slot]), 0);
          if (rank == 0) mbar_expect_tx(smem_addr(&bar_full[slot]), 2 * kStageA);
#pragma unroll
          for (int c = 0; c < BMH / 64; ++c)
            tma_load_2d(smem_addr(ring + slot * kStageA + c * (BK * 128)), &p.map_w[g], col + c * 64, kb * BK, full0);
        }
        __syncwarp();
        slot = slot + 1 == p.stages ? 0 : slot + 1;
        round ^= (slot == 0);
      }
    }
    if (*abort_flag && rank == 0 && leader) {
      // give the loads still in flight a bounded chance to land before the CTA goes away
      for (int i = rounds > p.stages ? rounds - p.stages : 0; i < rounds; ++i) {
        const unsigned long long t0 = now_ns();
        while (!mbar_try(smem_addr(&bar_full[i % p.stages]), (unsigned)((i / p.stages) & 1)) && now_ns() - t0 < 100000000ull) {
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------ MMA issuer (CTA 0)
    if (rank == 0) {
      const bool leader = elect_one();
      constexpr unsigned idesc = make_idesc(1, 1, NB);
      bool ok = mbar_wait_warp(smem_addr(&bar_feat), 0, abort_flag);
      int slot = 0, it = 0;
      unsigned round = 0;
      for (int tile = first; tile < tiles && ok; tile += stride, ++it) {
        const int buf = it % kNarrowAccs;
        ok = mbar_wait_warp(smem_addr(&bar_acc_empty[buf]), (unsigned)((it / kNarrowAccs) & 1) ^ 1, abort_flag);
        for (int kb = 0; kb < p.kblocks && ok; ++kb) {
          ok = mbar_wait_warp(smem_addr(&bar_full[slot]), round, abort_flag);
          if (!ok) break;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          if (leader) {
            const unsigned sa = smem_addr(ring + slot * kStageA) & 0x3ffffu, sb = smem_addr(feat + kb * kFb) & 0x3ffffu;
#pragma unroll
            for (int kk = 0; kk < BK / 16; ++kk) {
              constexpr unsigned a_lo = desc_lo_fixed(BK * 128), b_lo = desc_lo_fixed(16), hi = desc_hi_fixed(1024);
              umma_bf16(tmem_base + buf * NB, desc_pack(a_lo + (sa >> 4) + kk * 128, hi), desc_pack(b_lo + (sb >> 4) + kk * 2, hi), idesc,
                        (kb > 0 || kk > 0) ? 1u : 0u);
            }
            umma_commit_pair(smem_addr(&bar_empty[slot]));
          }
          __syncwarp();
          slot = slot + 1 == p.stages ? 0 : slot + 1;
          round ^= (slot == 0);
        }
        if (leader && ok) umma_commit_pair(smem_addr(&bar_acc_full[buf]));
        __syncwarp();
      }
    }
  } else {
    // ------------------------------------------------ epilogue (both CTAs): 32 classes and 32 rows a warp and batch
    // After a wait that ran out the warps go on without waiting: they still meet at their barriers.
    const int q = warp & 3, half = (warp - 2) >> 2;
    const unsigned tq = tmem_base + ((unsigned)(q * 32) << 16);
    float* mine = staging + (warp - 2) * (32 * kNarrowPitch);
    int it = 0, g = 0, met = 0;
    for (int tile = first; tile < tiles; tile += stride, ++it) {
      if (NB == 32 && (it & 1) != half) continue;      // one batch a tile: the two warps of a quadrant take turns
      while (tile >= p.tile_begin[g + 1]) ++g;
      const int buf = it % kNarrowAccs;
      bool ok = !*abort_flag;
      if (ok && lane == 0) ok = mbar_wait(smem_addr(&bar_acc_full[buf]), (unsigned)((it / kNarrowAccs) & 1), abort_flag);
      __syncwarp();
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const long long chunk0 = (long long)(tile - p.tile_begin[g]) * BM + rank * BMH;      // this CTA's first class in the shard
      const long long cls = chunk0 + q * 32 + lane, Ng = p.n[g];
      constexpr int kBatches = NB / 32, kStep = NB == 32 ? 1 : 2;
#pragma unroll(MODE == 1 ? 2 : 1)
      for (int b0 = 0; b0 < kBatches; b0 += kStep) {
        const int b = NB == 32 ? 0 : b0 + half, r0 = b * 32;
        float v[32];
        tmem_ld32(tq + buf * NB + r0, v);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        if (b0 + kStep >= kBatches) {                  // the accumulator is free again
          asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
          __syncwarp();
          if (lane == 0) mbar_arrive_cluster(map_to_cta(smem_addr(&bar_acc_empty[buf]), 0));
        }
        if (r0 >= p.rows || chunk0 >= Ng) continue;    // the same for the four warps of a half
        if constexpr (MODE == 1) {
#pragma unroll
          for (int c = 0; c < 8; ++c) {
            float4 f = make_float4(v[4 * c], v[4 * c + 1], v[4 * c + 2], v[4 * c + 3]);
            if (cls >= Ng) f = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
            *reinterpret_cast<float4*>(mine + lane * kNarrowPitch + 4 * c) = f;
          }
          __syncwarp();
          float x[32];                                  // this lane's row, 32 classes
#pragma unroll
          for (int i = 0; i < 32; ++i) x[i] = mine[i * kNarrowPitch + lane];
          float top[4] = {x[0], x[1], x[2], x[3]};
#pragma unroll
          for (int i = 4; i < 32; ++i) top[i & 3] = fmaxf(top[i & 3], x[i]);
          const float m = fmaxf(fmaxf(top[0], top[1]), fmaxf(top[2], top[3]));
          const unsigned long long neg = two(m == -INFINITY ? 0.f : -m);      // no class of the shard here: sum 0
          float sum[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
          for (int i = 0; i < 32; i += 2) {
            exp_two(x[i], x[i + 1], neg, 0ull);
            sum[i & 3] += x[i];
            sum[(i & 3) + 1] += x[i + 1];
          }
          const long long want = lab_s[r0 + lane] - p.class_start[g] - chunk0 - q * 32;
          const float t = want >= 0 && want < 32 && want < Ng - chunk0 - q * 32 ? mine[(int)want * kNarrowPitch + lane] : 0.f;
          float* out = red + ((half * 2 + (met & 1)) * 4) * 96 + lane;
          out[q * 96] = m;
          out[q * 96 + 32] = (sum[0] + sum[1]) + (sum[2] + sum[3]);
          out[q * 96 + 64] = t;
          asm volatile("bar.sync %0, 128;" ::"r"(1 + half) : "memory");
          if (q == (met & 3) && r0 + lane < p.rows) {
            float M = fmaxf(fmaxf(out[0], out[96]), fmaxf(out[192], out[288])), S = 0.f, T = 0.f;
#pragma unroll
            for (int w = 0; w < 4; ++w) {
              S = fmaf(out[w * 96 + 32], exp_one(out[w * 96], M, 0.f), S);
              T += out[w * 96 + 64];
            }
            const long long at = (long long)(p.xf.part_base[g] + chunk0 / BMH) * p.rows + r0 + lane;
            if (SBP_GUARD(p.xf.part_m + at, 4)) p.xf.part_m[at] = M;
            if (SBP_GUARD(p.xf.part_s + at, 4)) p.xf.part_s[at] = S;
            if (SBP_GUARD(p.xf.part_t + at, 4)) p.xf.part_t[at] = T;
          }
          ++met;
        } else {
          const long long first_class = p.class_start[g] + chunk0 + q * 32, step = p.ldy[g];
#pragma unroll
          for (int c = 0; c < 32; c += 4) {
            const ulonglong2 less = *reinterpret_cast<const ulonglong2*>(less_s + r0 + c), neg = *reinterpret_cast<const ulonglong2*>(neg_s + r0 + c);
            exp_two(v[c], v[c + 1], less.x, neg.x);
            exp_two(v[c + 2], v[c + 3], less.y, neg.y);
          }
          // rows whose label is one of this warp's 32 classes are rare
          const long long want = lab_s[r0 + lane] - first_class;
          if (__any_sync(0xffffffffu, want >= 0 && want < 32)) {
#pragma unroll
            for (int c = 0; c < 32; ++c)
              if (lab_s[r0 + c] == first_class + lane) v[c] -= 1.0f;
          }
          if (p.y_quads) {
            // bf16 in pieces of four classes: lanes 4 i .. 4 i + 3 hold 4 x 4 elements of four rows, and after two
            // exchanges lane 4 i + r has row r's four
            const bool odd = lane & 1, high = lane & 2;
            unsigned char* at = static_cast<unsigned char*>(p.y[g]) + ((r0 + (lane & 3)) * step + (cls & ~3ll)) * 2;
#pragma unroll
            for (int c = 0; c < 32; c += 4, at += 8 * step) {
              if (r0 + c >= p.rows) break;
              unsigned w[2];
#pragma unroll
              for (int h = 0; h < 2; ++h) {
                const __nv_bfloat162 two = __floats2bfloat162_rn(v[c + 2 * h], v[c + 2 * h + 1]);
                const unsigned own = *reinterpret_cast<const unsigned*>(&two), other = __shfl_xor_sync(0xffffffffu, own, 1);
                w[h] = odd ? __byte_perm(other, own, 0x7632) : __byte_perm(own, other, 0x5410);      // row 2 h + odd, two classes
              }
              const unsigned other = __shfl_xor_sync(0xffffffffu, high ? w[0] : w[1], 2);
              const uint2 o = high ? make_uint2(other, w[1]) : make_uint2(w[0], other);
              if (cls < Ng && r0 + c + (lane & 3) < p.rows && SBP_GUARD(at, 8)) *reinterpret_cast<uint2*>(at) = o;
            }
          } else if (cls < Ng) {
            const int esz = p.out_f32 ? 4 : 2;
            unsigned char* at = static_cast<unsigned char*>(p.y[g]) + (r0 * step + cls) * esz;
#pragma unroll
            for (int c = 0; c < 32; ++c, at += step * esz) {
              if (r0 + c >= p.rows) break;
              if (p.out_f32) {
                if (SBP_GUARD(at, 4)) *reinterpret_cast<float*>(at) = v[c];
              } else {
                if (SBP_GUARD(at, 2)) *reinterpret_cast<__nv_bfloat16*>(at) = __float2bfloat16_rn(v[c]);
              }
            }
          }
        }
      }
    }
  }

  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  cluster_sync_all();
  if (warp == 1) {
    __syncwarp();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kNarrowAccs * NB) : "memory");
  }
}

// ------------------------------------------------------------------ host side

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* ptr = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &qres) == cudaSuccess &&
        qres == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(ptr);
  });
  return fn;
}

// Tensor maps already encoded by this process, keyed by everything that goes into one.  A map holds
// nothing but the address and the layout, so an entry stays valid for as long as its key recurs: a
// product that is called again on the same buffers (every step of a training loop) encodes nothing.
// Two-way set-associative; used with the parameter block's lock held.
struct MapKey {
  const void* base;
  long long rows, cols, ld;
  int esz, box_rows, box_cols;
  bool operator==(const MapKey& o) const {
    return base == o.base && rows == o.rows && cols == o.cols && ld == o.ld && esz == o.esz && box_rows == o.box_rows &&
           box_cols == o.box_cols;
  }
};
struct MapSlot {
  CUtensorMap map;
  MapKey key;
  bool used;
};
constexpr int kMapCacheSets = 2048, kMapCacheWays = 2;
static MapSlot g_map_cache[kMapCacheSets][kMapCacheWays];
static unsigned char g_map_victim[kMapCacheSets];
static unsigned long long g_map_hits = 0, g_map_encodes = 0;

static unsigned map_slot_of(const MapKey& k) {
  unsigned long long h = reinterpret_cast<uintptr_t>(k.base) >> 4;
  auto mix = [&](unsigned long long v) { h = (h ^ v) * 0x9E3779B97F4A7C15ull; h ^= h >> 29; };
  mix((unsigned long long)k.rows);
  mix((unsigned long long)k.cols);
  mix((unsigned long long)k.ld);
  mix((unsigned long long)(k.esz | (k.box_rows << 8) | (k.box_cols << 20)));
  return (unsigned)(h % kMapCacheSets);
}

void tensor_map_cache_stats(unsigned long long* hits, unsigned long long* encodes) {
  *hits = g_map_hits;
  *encodes = g_map_encodes;
}

// launches of the kernel by form: square or split, tall, square over the halves that a mixed run leaves; and the split ones
static std::atomic<unsigned long long> g_form_launches[3], g_split_launches;

// Overrides of the form choice and of the CTA pairs a launch may use (tests and measurements):
// set by tc_set_form, else taken once from SBP_TC_FORM (square | tall | mixed | split) and SBP_TC_PAIRS.
static std::atomic<int> g_forced_form{-1}, g_pair_cap{-1};

static int forced_form() {
  int v = g_forced_form.load();
  if (v < 0) {
    const char* e = getenv("SBP_TC_FORM");
    v = e ? (e[0] == 's' ? (e[1] == 'p' ? 4 : 1) : (e[0] == 't' ? 2 : (e[0] == 'm' ? 3 : 0))) : 0;
    g_forced_form.store(v);
  }
  return v;
}

static int pair_cap() {
  int v = g_pair_cap.load();
  if (v < 0) {
    const char* e = getenv("SBP_TC_PAIRS");
    v = e ? std::max(0, atoi(e)) : 0;
    g_pair_cap.store(v);
  }
  return v;
}

void tc_set_form(int form, int max_pairs) {
  g_forced_form.store(form >= 0 && form <= 4 ? form : 0);
  g_pair_cap.store(max_pairs > 0 ? max_pairs : 0);
}

void tc_form_stats(unsigned long long out[3]) {
  for (int i = 0; i < 3; ++i) out[i] = g_form_launches[i].load();
}

unsigned long long tc_split_launches() { return g_split_launches.load(); }

// 2-D row-major tensor [rows, cols] with leading dimension ld (elements), box [box_rows, box_cols].
static bool make_map(CUtensorMap* map, const void* base, int esz, long long rows, long long cols, long long ld,
                     int box_rows, int box_cols) {
  const MapKey key{base, rows, cols, ld, esz, box_rows, box_cols};
  const unsigned set = map_slot_of(key);
  for (int w = 0; w < kMapCacheWays; ++w) {
    const MapSlot& hit = g_map_cache[set][w];
    if (hit.used && hit.key == key) {
      *map = hit.map;
      ++g_map_hits;
      return true;
    }
  }
  int way = (g_map_victim[set] + 1) % kMapCacheWays;      // the way not written last ...
  for (int w = kMapCacheWays - 1; w >= 0; --w)
    if (!g_map_cache[set][w].used) way = w;                 // ... unless one is still unused
  g_map_victim[set] = (unsigned char)way;
  MapSlot& slot = g_map_cache[set][way];
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)ld * esz};
  cuuint32_t box[2] = {(cuuint32_t)box_cols, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUtensorMapDataType dt = esz == 2 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32;
  if (fn(map, dt, 2, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
         CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return false;
  ++g_map_encodes;
  slot.map = *map;
  slot.key = key;
  slot.used = true;
  return true;
}

static bool aligned16(const void* p) { return reinterpret_cast<uintptr_t>(p) % 16 == 0; }

// Launch of one compiled form of the kernel (called with the parameter block's lock held), or,
// with p == nullptr, only the number of CTA pairs of that form the device holds at once.
template <int AT, int BT, int MH>
static sbp_status launch_tc_form(const TcParams* p, cudaStream_t st, int* capacity) {
  constexpr int kSmem = MH == 2 ? kSmemBytesTall : kSmemBytes;
  // per device: the kernel's shared-memory opt-in and the number of CTA pairs that fit at once
  static int pairs_on_device[64] = {};
  int dev = 0;
  SBP_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return fail(SBP_ERR_UNSUPPORTED, "device ordinal %d out of range", dev);
  if (pairs_on_device[dev] == 0) {
    SBP_CUDA_TRY(cudaFuncSetAttribute(matmul_tc_kernel<AT, BT, MH>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem));
    int sms = 0;
    SBP_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    // how many CTA pairs the device can hold at once (pairs must sit in one GPC)
    cudaLaunchConfig_t probe = {};
    probe.gridDim = dim3((unsigned)(2 * (sms / 2)));
    probe.blockDim = dim3(kThreadsTc);
    probe.dynamicSmemBytes = kSmem;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = 2;
    attr.val.clusterDim.y = 1;
    attr.val.clusterDim.z = 1;
    probe.attrs = &attr;
    probe.numAttrs = 1;
    int clusters = 0;
    if (cudaOccupancyMaxActiveClusters(&clusters, matmul_tc_kernel<AT, BT, MH>, &probe) != cudaSuccess || clusters < 1) {
      cudaGetLastError();
      clusters = sms / 2;
    }
    pairs_on_device[dev] = clusters;
  }
  // a cap on the pairs (test and measurement switch): a small one makes small products run many
  // waves, and so take the mixed route
  const int cap = pair_cap();
  const int max_pairs = cap > 0 && cap < pairs_on_device[dev] ? cap : pairs_on_device[dev];
  if (capacity) *capacity = max_pairs;
  if (!p) return SBP_OK;
  const int pairs = p->total_tiles < max_pairs ? p->total_tiles : max_pairs;
  SBP_BOUNDS_UPLOAD(st);
  const cudaError_t e = launch_dependent(matmul_tc_kernel<AT, BT, MH>, dim3((unsigned)(2 * pairs)), dim3(kThreadsTc), kSmem, st, *p);
  if (e != cudaSuccess) return cuda_fail(e, "tensor-core matmul launch");
  count_launch();
  g_form_launches[MH == 2 ? 1 : (p->half_split ? 2 : 0)]++;
  return SBP_OK;
}

enum TcForm { kFormSquare = 0, kFormTall = 1, kFormShort = 2 };

static sbp_status launch_tc(TcForm form, bool a_trans, bool b_trans, const TcParams* p, cudaStream_t st, int* capacity) {
  switch (4 * form + ((a_trans ? 2 : 0) | (b_trans ? 1 : 0))) {
    case 0: return launch_tc_form<0, 0, 1>(p, st, capacity);
    case 1: return launch_tc_form<0, 1, 1>(p, st, capacity);
    case 2: return launch_tc_form<1, 0, 1>(p, st, capacity);
    case 3: return launch_tc_form<1, 1, 1>(p, st, capacity);
    case 8: return launch_tc_form<0, 0, 3>(p, st, capacity);
    case 9: return launch_tc_form<0, 1, 3>(p, st, capacity);
    case 10: return launch_tc_form<1, 0, 3>(p, st, capacity);
    case 11: return launch_tc_form<1, 1, 3>(p, st, capacity);
    case 4: return launch_tc_form<0, 0, 2>(p, st, capacity);
    case 5: return launch_tc_form<0, 1, 2>(p, st, capacity);
    case 6: return launch_tc_form<1, 0, 2>(p, st, capacity);
    default: return launch_tc_form<1, 1, 2>(p, st, capacity);
  }
}

// Which form runs a product.  Times in microseconds per wave (one tile on every CTA pair), fitted
// to this kernel's measured times on B200 under its power cap (the clock settles lower the busier
// the tensor pipe is -- about 1.6 GHz in the square form, 1.4 GHz in the tall one -- which is why
// these are times and not clock counts):
//   square form  0.388 per 64-deep K-block (about 590 clocks); the epilogue is hidden unless it is store-bound;
//   tall form    0.70 per K-block (1024 clocks) for twice the rows, plus an exposed epilogue of about 2.6.
// A run may be mixed: whole waves of tall tiles, then the rest of the walk in the square form (two
// 256-row halves per walked tile) -- a last wave that only half fills the device costs a whole
// tall wave otherwise.
struct FormChoice {
  bool walk_tall;      // tiles are walked 512 rows at a time
  int tall_tiles;      // the first so many walked tiles run in the tall form
  double cost;         // the model's time for it, without what every launch pays
};

// What the copy engine needs for the rows of 128 bytes that a CTA loads per K-block, us: 64 bytes a clock, and a
// row that starts off a 128-byte boundary of memory is two requests (a [5696 x 2280]^T [5696 x 632] product took
// 44.7 us where [5696 x 2304]^T [5696 x 640] took 28.1).  A long product of such pitches wants wide tiles; the first
// K-blocks only fill the ring.  Operands whose rows lie along K do not pay it: the next K-block finds the other half of the
// line in L2 (dX of [6000 x 4000] by [2000 x 4000], both pitches misaligned: 72.8 us, 79.5 where the square form paid it).
struct OperandRows {
  double a = 1.0e-3, b = 1.0e-3;      // us per row
  // time of kb K-blocks beyond `per_kb` each, which they take otherwise
  double extra(int rows_a, int rows_b, double kb, double per_kb) const {
    return std::max(0.0, kb - 8.0) * std::max(0.0, a * rows_a + b * rows_b - per_kb);
  }
};

static OperandRows operand_rows(const MatmulPlan& p) {
  OperandRows r;
  for (int s = 0; s < p.nseg; ++s) {
    if ((!p.chain && s >= p.ngroups) || p.kseg[s] == 0) continue;
    if (p.a_trans && (p.lda[s] % 64 != 0 || reinterpret_cast<uintptr_t>(p.a[s]) % 128 != 0)) r.a = 1.9e-3;
    if (!p.b_trans && (p.ldb[s] % 64 != 0 || reinterpret_cast<uintptr_t>(p.b[s]) % 128 != 0)) r.b = 1.9e-3;
  }
  return r;
}

static FormChoice choose_form(long long tiles_sq, long long tiles_tall, long long kb, int cap_sq, int cap_tall, bool gelu, int n_rep,
                              bool out_f32, const OperandRows& rows, int forced) {
  const double wave_sq = 0.388 * kb + rows.extra(BMH, BNH, (double)kb, 0.388) + (gelu ? 1.3 : 0.0) + 1.2 * n_rep + (out_f32 ? 1.0 : 0.0);
  const double wave_tall = 0.70 * kb + rows.extra(2 * BMH, BNH, (double)kb, 0.70) + 2.6 + (gelu ? 8.6 : 0.0) + 2.5 * n_rep + (out_f32 ? 3.0 : 0.0);
  const double kRelaunch = 5.0;
  auto waves = [](long long tiles, int cap) { return (double)((tiles + cap - 1) / cap); };
  const double cost_sq = waves(tiles_sq, cap_sq) * wave_sq;
  const double cost_tall = waves(tiles_tall, cap_tall) * wave_tall;
  const long long full = tiles_tall / cap_tall * cap_tall;       // tall tiles in whole waves
  const double cost_mixed = full == 0 || full == tiles_tall
                                ? 1e30
                                : (double)(full / cap_tall) * wave_tall + waves(2 * (tiles_tall - full), cap_sq) * wave_sq + kRelaunch;
  int pick;      // 0 square, 1 tall, 2 mixed
  if (forced) pick = forced - 1;
  else {
    pick = 0;
    double best = cost_sq * 0.98;                                // ties go to the square form
    if (cost_tall < best) { best = cost_tall; pick = 1; }
    if (cost_mixed < best) { best = cost_mixed; pick = 2; }
  }
  if (pick == 2 && (full == 0 || full == tiles_tall)) pick = full == 0 ? 0 : 1;
  if (pick == 0) return FormChoice{false, 0, cost_sq};
  return FormChoice{true, (int)(pick == 1 ? tiles_tall : full), pick == 1 ? cost_tall : cost_mixed};
}

// choose_form for callers outside this file (the C ABI's planning query): 0 square, 1 tall, 2 mixed.
int tc_route(long long tiles_sq, long long tiles_tall, long long kb, int pairs, bool gelu, int n_rep, bool out_f32, int forced,
             long long* tall_tiles) {
  const FormChoice f = choose_form(tiles_sq, tiles_tall, kb, pairs, pairs, gelu, n_rep, out_f32, OperandRows{}, forced);
  if (tall_tiles) *tall_tiles = f.walk_tall ? f.tall_tiles : 0;
  return !f.walk_tall ? 0 : (f.tall_tiles == tiles_tall ? 1 : 2);
}

// One split product, or, with p == nullptr, only the clusters of this size the device holds at once.
template <int AT, int BT, int NB, int SW>
static sbp_status launch_split_form(const TcSplitParams* p, int splits, int tiles, cudaStream_t st, int* capacity) {
  static std::atomic<unsigned long long> opted{0};      // one bit per device
  int dev = 0;
  SBP_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return fail(SBP_ERR_UNSUPPORTED, "device ordinal %d out of range", dev);
  auto* kernel = matmul_tc_split_kernel<AT, BT, NB, SW>;
  if (!(opted.load(std::memory_order_relaxed) >> dev & 1)) {
    SBP_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemSplit));
    SBP_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    opted.fetch_or(1ull << dev, std::memory_order_relaxed);
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(2 * splits * tiles * (p ? p->outer : 1)));
  cfg.blockDim = dim3(kThreadsTc);
  cfg.dynamicSmemBytes = kSmemSplit;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)(2 * splits);
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (capacity) {
    *capacity = 0;
    if (cudaOccupancyMaxActiveClusters(capacity, kernel, &cfg) != cudaSuccess) {
      cudaGetLastError();
      *capacity = 0;
    }
    return SBP_OK;
  }
  cfg.numAttrs = 2;
  SBP_BOUNDS_UPLOAD(st);
  cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, *p);
  if (e != cudaSuccess) return cuda_fail(e, "tensor-core matmul launch");
  count_launch();
  g_form_launches[0]++;
  g_split_launches++;
  return SBP_OK;
}

// How a split product is cut: NB columns a tile, `splits` pairs a tile (0: the persistent kernel runs it),
// operands exchanged or not, `outer` clusters a tile.
struct SplitChoice {
  int nb, splits, swap, outer;
};

static long long pad4(long long v) { return (v + 3) / 4 * 4; }

// Floats of one set of partial results.
static long long part_floats(const MatmulPlan& plan) {
  long long v = 0;
  for (int g = 0; g < plan.ngroups; ++g) v += plan.m[g] * pad4(plan.n[g]);
  return v;
}

static sbp_status launch_split_any(bool a_trans, bool b_trans, SplitChoice c, const TcSplitParams* p, int tiles, cudaStream_t st) {
  const int s = c.splits;
  if (c.swap) {            // b_trans holds: the exchanged operand is X as given
    switch (c.nb | (a_trans ? 1 : 0)) {
      case 32: return launch_split_form<0, 1, 32, 1>(p, s, tiles, st, nullptr);
      case 33: return launch_split_form<1, 1, 32, 1>(p, s, tiles, st, nullptr);
      case 64: return launch_split_form<0, 1, 64, 1>(p, s, tiles, st, nullptr);
      case 65: return launch_split_form<1, 1, 64, 1>(p, s, tiles, st, nullptr);
      case 128: return launch_split_form<0, 1, 128, 1>(p, s, tiles, st, nullptr);
      default: return launch_split_form<1, 1, 128, 1>(p, s, tiles, st, nullptr);
    }
  }
  switch (c.nb | (a_trans ? 2 : 0) | (b_trans ? 1 : 0)) {
    case 128: return launch_split_form<0, 0, 128, 0>(p, s, tiles, st, nullptr);
    case 129: return launch_split_form<0, 1, 128, 0>(p, s, tiles, st, nullptr);
    case 130: return launch_split_form<1, 0, 128, 0>(p, s, tiles, st, nullptr);
    case 131: return launch_split_form<1, 1, 128, 0>(p, s, tiles, st, nullptr);
    case 256: return launch_split_form<0, 0, 256, 0>(p, s, tiles, st, nullptr);
    case 257: return launch_split_form<0, 1, 256, 0>(p, s, tiles, st, nullptr);
    case 258: return launch_split_form<1, 0, 256, 0>(p, s, tiles, st, nullptr);
    default: return launch_split_form<1, 1, 256, 0>(p, s, tiles, st, nullptr);
  }
}

// Clusters of 2 * splits CTAs that the current device holds at once (every instance of the kernel fills an SM).
static int split_capacity(int splits) {
  static std::atomic<int> known[64][kMaxSplits + 1];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  int v = known[dev][splits].load(std::memory_order_relaxed);
  if (v == 0) {
    if (launch_split_form<0, 0, 256, 0>(nullptr, splits, 1, nullptr, &v) != SBP_OK || v < 1) v = -1;
    known[dev][splits].store(v, std::memory_order_relaxed);
  }
  return v;
}

// Whether a product runs in the split form, and how it is cut: the smallest estimated time in us.  Per wave of
// clusters: a K-block takes 0.32 us with 256 columns (the tensor pipe's 512 clocks and a little), 0.19-0.20
// with 128 and fewer (the single-issue roles); set-up, drain and stores 9.6 / 6.6 us (256 / 128 columns),
// 6.5 / 5.3 / 4.4 for the exchanged form (128 / 64 / 32).  Fitted to 1208 timings of 54 products (rms error
// 12 %; the pick within 8 % of the best cut of each).  The persistent kernel keeps what it does as well:
// `cost_persistent` includes the 5.5 us it takes besides its waves, and a split has to win by 8 %.  An fp32 result is
// twice the stores, like another replica ([16384 x 512] x [512 x 64] over four devices to fp32 S(0): 12.3 us split, which
// the rule took without that term, 7.9 persistent; three [333 x 333] x [333 x 111] to fp32 14.0 / 18.4).
// (us, persistent / split, one product in a row of them: 16 rows [4096 x 16384] 31 / 24 and [16384 x 4096]
// 79 / 26; 1000 rows [4096 x 1024] written to four replicas 28 / 16; 500 rows [1024 x 4096] + GeLU 15 / 11;
// 512 x 512 over 2^20 classes 4569 / 621; 64 x 256 over 2^17 578 / 48.)
static SplitChoice choose_split(const MatmulPlan& plan, const int* kblocks, double cost_persistent, int forced, size_t ws_bytes) {
  long long kb_max = 0, kb_min = -1, chain_kb = 0, m_max = 0;
  for (int s = 0; s < plan.nseg; ++s) chain_kb += kblocks[s];
  for (int g = 0; g < plan.ngroups; ++g) {
    if (plan.m[g] <= 0 || plan.n[g] <= 0) continue;
    m_max = plan.m[g] > m_max ? plan.m[g] : m_max;
    const long long kb = plan.chain ? chain_kb : kblocks[g];
    kb_max = kb > kb_max ? kb : kb_max;
    kb_min = kb_min < 0 || kb < kb_min ? kb : kb_min;
  }
  SplitChoice best{0, 0, 0, 1}, cut{0, 0, 0, 1};
  const OperandRows rows = operand_rows(plan);
  const long long pf = part_floats(plan);
  const long long room = pf > 0 ? (long long)std::min<size_t>(ws_bytes / 4, size_t(1) << 60) / pf : 0;      // sets of partial results the workspace holds
  double best_cost = forced == 4 ? 1e300 : cost_persistent, cut_cost = 1e300, any_cut_cost = 1e300;
  for (int swap = 0; swap < 2; ++swap) {
    if (swap && plan.a_trans) continue;      // X would be the N-major operand: boxes of 64 rows and more
    if (swap && m_max > 192) continue;       // its tiles read the weight once per 128 rows, the plain ones once per 256
    for (int nb = swap ? 128 : 256; nb >= (swap ? 32 : 128); nb /= 2) {
      long long tiles = 0;
      for (int g = 0; g < plan.ngroups; ++g) {
        const long long rows = swap ? plan.n[g] : plan.m[g], cols = swap ? plan.m[g] : plan.n[g];
        if (rows > 0 && cols > 0) tiles += (rows + BM - 1) / BM * ((cols + nb - 1) / nb);
      }
      if (tiles > 4096) continue;
      for (int s = 1; s <= kMaxSplits; ++s) {
        if (kb_min < s) break;
        const int cap = split_capacity(s);
        if (cap < 1) continue;
        const double waves = (double)((tiles + cap - 1) / cap), kb = (double)((kb_max + s - 1) / s);
        const double per_kb = nb == 256 ? 0.323 : (nb == 128 ? 0.2 : 0.187);
        auto k_time = [&](double kbs) { return kbs * per_kb + (swap ? rows.extra(nb / 2, BMH, kbs, per_kb) : rows.extra(BMH, nb / 2, kbs, per_kb)); };
        const double per_wave = nb == 256 ? 9.6 : (nb == 128 ? 6.6 : (nb == 64 ? 5.3 : 4.4));
        const double cost = waves * (k_time(kb) + per_wave + (s > 1 ? 0.8 + 0.08 * s : 0.0) + (plan.gelu ? 0.4 : 0.0) +
                                     (plan.n_rep + (plan.out_dtype == SBP_F32 ? 1 : 0)) * 2.0 * nb / (256.0 * s));
        if (cost < best_cost) {
          best_cost = cost;
          best = SplitChoice{nb, s, swap, 1};
        }
        // as many clusters a tile as run at once; adding their results up is a launch, one write and one read
        auto cut_over = [&](long long outer) {
          const double kbo = (double)((kb_max + s * outer - 1) / (s * outer));
          const double sum = 4.0 + (double)pf * (8.0 * outer + (plan.out_dtype == SBP_F32 ? 4.0 : 2.0) * (1 + plan.n_rep)) / 5e6;
          return k_time(kbo) + per_wave + (s > 1 ? 0.8 + 0.08 * s : 0.0) + sum;
        };
        const long long all = std::min({tiles > 0 ? cap / tiles : 0, kb_min / (8 * s), 128LL}), outer = std::min(all, room);
        if (all >= 2) any_cut_cost = std::min(any_cut_cost, cut_over(all));
        if (outer >= 2) {
          const double co = cut_over(outer);
          if (co < cut_cost) {
            cut_cost = co;
            cut = SplitChoice{nb, s, swap, (int)outer};
          }
        }
      }
    }
  }
  // The workspace is used only where the size query reports room for it: not where a cut pays with less room alone.
  if (any_cut_cost < best_cost && cut_cost < best_cost) return cut;
  return best;
}

// The row blocks of one fused result as one product, where their results share a pitch; false where they are none.
// (A block of 34 rows has a tile of 256 to itself otherwise, and one that starts off a multiple of 8 rows of a
// transposed X needs a repacked copy.  us, separate and repacked / as one: [6838 x 136]^T [6838 x 1808] over four
// devices 37.6 / 15.4; [5293 x 2488]^T [5293 x 544] over two 38 / 26.)
static bool merge_row_blocks(const MatmulPlan& plan, MatmulPlan* merged) {
  if (!plan.chain || plan.ngroups < 2 || plan.n_rep != 0) return false;
  long long rows = 0;
  for (int g = 0; g < plan.ngroups; ++g) {
    if (plan.row_off[g] != rows || plan.col_off[g] != 0 || plan.n[g] != plan.n[0] || plan.ldy[g] != plan.ldy[0]) return false;
    rows += plan.m[g];
  }
  *merged = plan;
  merged->ngroups = 1;
  merged->m[0] = rows;
  return true;
}

static sbp_status launch_split(const MatmulPlan& given, const MatmulPlan* merged, const int* kblocks, SplitChoice c, bool y_vec, float* ws,
                               cudaStream_t st, bool* taken) {
  MatmulPlan plan = merged ? *merged : given;
  if (c.swap) {            // Y^T = W^T X^T
    for (int i = 0; i < SBP_MAX_K; ++i) {
      std::swap(plan.a[i], plan.b[i]);
      std::swap(plan.lda[i], plan.ldb[i]);
      std::swap(plan.m[i], plan.n[i]);
      std::swap(plan.row_off[i], plan.col_off[i]);
    }
    plan.a_trans = !given.b_trans;
    plan.b_trans = !given.a_trans;
  }
  TcSplitParams p;
  p.blocks = 0;
  if (merged && c.outer == 1) {
    p.blocks = given.ngroups;
    for (int g = 0; g < given.ngroups; ++g) {
      p.block_row[g] = given.row_off[g];
      p.block_y[g] = given.y[g];
    }
  }
  int tiles = 0;
  for (int g = 0; g < plan.ngroups; ++g) {
    p.m[g] = plan.m[g];
    p.n[g] = plan.n[g];
    p.row_off[g] = plan.row_off[g];
    p.col_off[g] = plan.col_off[g];
    p.ldy[g] = plan.ldy[g];
    p.y_ptr[g] = plan.y[g];
    p.tile_begin[g] = tiles;
    const int tm = (int)((plan.m[g] + BM - 1) / BM);
    p.tiles_m[g] = tm > 0 ? tm : 1;
    if (plan.m[g] > 0 && plan.n[g] > 0) tiles += tm * (int)((plan.n[g] + c.nb - 1) / c.nb);
  }
  for (int g = plan.ngroups; g <= SBP_MAX_K; ++g) p.tile_begin[g] = tiles;
  for (int r = 0; r < plan.n_rep; ++r) p.rep_ptr[r] = plan.y_rep[r];
  for (int s = 0; s < plan.nseg; ++s) {
    p.kblocks[s] = kblocks[s];
    if (!(plan.chain || s < plan.ngroups) || kblocks[s] == 0) continue;
    long long rows_a = plan.chain ? 0 : plan.m[s], cols_b = plan.chain ? 0 : plan.n[s];
    for (int g = 0; plan.chain && g < plan.ngroups; ++g) {
      rows_a = std::max(rows_a, plan.row_off[g] + plan.m[g]);
      cols_b = std::max(cols_b, plan.col_off[g] + plan.n[g]);
    }
    if (rows_a == 0 || cols_b == 0) continue;
    const bool ok_a = plan.a_trans ? make_map(&p.map_a[s], plan.a[s], 2, plan.kseg[s], rows_a, plan.lda[s], BK, 64)
                                   : make_map(&p.map_a[s], plan.a[s], 2, rows_a, plan.kseg[s], plan.lda[s], BMH, BK);
    const bool ok_b = plan.b_trans ? make_map(&p.map_b[s], plan.b[s], 2, cols_b, plan.kseg[s], plan.ldb[s], c.nb / 2, BK)
                                   : make_map(&p.map_b[s], plan.b[s], 2, plan.kseg[s], cols_b, plan.ldb[s], BK, 64);
    if (!ok_a || !ok_b) return fail(SBP_ERR_CUDA, "cuTensorMapEncodeTiled failed for an operand of shard %d", s);
  }
  p.ngroups = plan.ngroups;
  p.nseg = plan.nseg;
  p.chain = plan.chain;
  p.gelu = plan.gelu;
  p.n_rep = plan.n_rep;
  p.out_f32 = plan.out_dtype == SBP_F32;
  p.splits = c.splits;
  p.y_vec = y_vec ? 1 : 0;
  p.tiles = tiles;
  p.outer = c.outer;
  p.part_bytes = 0;
  *taken = true;
  if (tiles == 0) return SBP_OK;
  if (c.outer == 1) return launch_split_any(plan.a_trans, plan.b_trans, c, &p, tiles, st);

  PartsParams q;
  float* at = ws;
  long long quads = 0;
  for (int g = 0; g < given.ngroups; ++g) {
    q.part[g] = at;
    q.m[g] = given.m[g];
    q.n[g] = given.n[g];
    q.ld[g] = pad4(given.n[g]);
    q.ldy[g] = given.ldy[g];
    q.y_ptr[g] = given.y[g];
    p.y_ptr[g] = at;          // of row blocks multiplied as one, the first: the others follow it
    p.ldy[g] = q.ld[g];
    at += given.m[g] * q.ld[g];
    quads = std::max(quads, given.m[g] * q.ld[g] / 4);
  }
  for (int r = 0; r < given.n_rep; ++r) q.rep_ptr[r] = given.y_rep[r];
  q.stride = at - ws;
  q.parts = c.outer;
  q.gelu = given.gelu;
  q.n_rep = given.n_rep;
  q.out_f32 = p.out_f32;
  q.y_vec = p.y_vec;
  p.part_bytes = q.stride * 4;
  p.gelu = 0;
  p.n_rep = 0;
  p.out_f32 = 1;
  p.y_vec = 1;
  const sbp_status rs = launch_split_any(plan.a_trans, plan.b_trans, c, &p, tiles, st);
  if (rs != SBP_OK) return rs;
  const long long blocks = std::min(8LL * device_sms(), (quads + 255) / 256);
  const cudaError_t e = launch_dependent(matmul_parts_kernel, dim3((unsigned)blocks, (unsigned)given.ngroups), dim3(256), 0, st, q);
  if (e != cudaSuccess) return cuda_fail(e, "matmul partial sums launch");
  count_launch();
  return SBP_OK;
}

template <int NB, int MODE>
static sbp_status launch_narrow_form(NarrowParams& p, cudaStream_t st) {
  static std::atomic<int> pairs_on_device[64];
  int dev = 0;
  SBP_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return fail(SBP_ERR_UNSUPPORTED, "device ordinal %d out of range", dev);
  auto* kernel = xent_narrow_kernel<NB, MODE>;
  int pairs = pairs_on_device[dev].load(std::memory_order_relaxed);
  if (pairs == 0) {
    SBP_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kNarrowSmem));
    int sms = 0;
    SBP_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    cudaLaunchConfig_t probe = {};
    probe.gridDim = dim3((unsigned)(2 * (sms / 2)));
    probe.blockDim = dim3(kThreadsTc);
    probe.dynamicSmemBytes = kNarrowSmem;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = 2;
    attr.val.clusterDim.y = 1;
    attr.val.clusterDim.z = 1;
    probe.attrs = &attr;
    probe.numAttrs = 1;
    if (cudaOccupancyMaxActiveClusters(&pairs, kernel, &probe) != cudaSuccess || pairs < 1) {
      cudaGetLastError();
      pairs = sms / 2;
    }
    pairs_on_device[dev].store(pairs, std::memory_order_relaxed);
  }
  const int features = (p.kblocks * narrow_feature_block<NB>() + 1023) / 1024 * 1024;
  const int room = kNarrowSmem - 1024 - features - (MODE == 1 ? kNarrowStageBytes + kNarrowRedBytes : 0);
  p.stages = std::min(kNarrowMaxStages, room / kStageA);
  const int tiles = p.tile_begin[p.ngroups];
  SBP_BOUNDS_UPLOAD(st);
  const cudaError_t e = launch_dependent(kernel, dim3((unsigned)(2 * std::min(tiles, pairs))), dim3(kThreadsTc), kNarrowSmem, st, p);
  if (e != cudaSuccess) return cuda_fail(e, "fused classifier launch");
  count_launch();
  return SBP_OK;
}

// The fused classifier for at most kNarrowRows rows; *taken stays false where the features do not fit.
static sbp_status launch_narrow(const MatmulPlan& plan, const XentFusion& xf, cudaStream_t st, bool* taken) {
  const int nb = xf.rows <= 32 ? 32 : (xf.rows <= 64 ? 64 : 128);
  const long long kb = (plan.kseg[0] + BK - 1) / BK;
  if (xf.rows > kNarrowRows || kb * (nb / 2 * 128) > kNarrowFeatures) return SBP_OK;
  NarrowParams p;
  p.ngroups = plan.ngroups;
  p.kblocks = (int)kb;
  p.rows = (int)xf.rows;
  p.out_f32 = plan.out_dtype == SBP_F32;
  p.y_quads = !p.out_f32;
  p.xf = xf;
  int tiles = 0;
  for (int g = 0; g < plan.ngroups; ++g) {
    p.tile_begin[g] = tiles;
    p.n[g] = plan.n[g];
    p.ldy[g] = plan.ldy[g];
    p.y[g] = plan.y[g];
    p.class_start[g] = xf.class_start[g];
    if (plan.n[g] % 4 != 0 || plan.ldy[g] % 4 != 0 || reinterpret_cast<uintptr_t>(plan.y[g]) % 8 != 0) p.y_quads = 0;
    if (plan.n[g] <= 0) continue;
    if (plan.n[g] / BM + tiles > 0x3fffffffLL) return SBP_OK;
    tiles += (int)((plan.n[g] + BM - 1) / BM);
    if (!make_map(&p.map_w[g], plan.b[g], 2, plan.kseg[g], plan.n[g], plan.ldb[g], BK, 64))
      return fail(SBP_ERR_CUDA, "cuTensorMapEncodeTiled failed for the weight of shard %d", g);
  }
  for (int g = plan.ngroups; g <= SBP_MAX_K; ++g) p.tile_begin[g] = tiles;
  // the replicas of the features are equal: the first serves every shard
  if (!make_map(&p.map_f, plan.a[0], 2, xf.rows, plan.kseg[0], plan.lda[0], nb / 2, BK))
    return fail(SBP_ERR_CUDA, "cuTensorMapEncodeTiled failed for the features");
  *taken = true;
  if (tiles == 0) return SBP_OK;
  switch (nb | (xf.grad ? 1 : 0)) {
    case 32: return launch_narrow_form<32, 1>(p, st);
    case 33: return launch_narrow_form<32, 2>(p, st);
    case 64: return launch_narrow_form<64, 1>(p, st);
    case 65: return launch_narrow_form<64, 2>(p, st);
    case 128: return launch_narrow_form<128, 1>(p, st);
    default: return launch_narrow_form<128, 2>(p, st);
  }
}

// room != nullptr: nothing is launched; *room is the workspace that the product would use if it were given all it can use.
static sbp_status run_matmul_tc(const MatmulPlan& plan, const XentFusion* xf, void* ws, size_t ws_bytes, cudaStream_t st, bool* taken, size_t* room) {
  *taken = false;
  if (plan.in_dtype != SBP_BF16) return SBP_ERR_UNSUPPORTED;
  const int oesz = plan.out_dtype == SBP_F32 ? 4 : 2;
  const bool stores_y = !xf || xf->grad;      // the softmax-partials mode writes no product

  // the rules of the TMA path: 16-byte aligned bases, leading dimensions and column offsets
  for (int s = 0; s < plan.nseg; ++s) {
    const bool used = plan.chain || s < plan.ngroups;
    if (!used) continue;
    if (plan.kseg[s] > 0 && (!aligned16(plan.a[s]) || !aligned16(plan.b[s]))) return SBP_ERR_UNSUPPORTED;
    if (plan.lda[s] % 8 != 0 || plan.ldb[s] % 8 != 0) return SBP_ERR_UNSUPPORTED;
    if (plan.lda[s] == 0 || plan.ldb[s] == 0) return SBP_ERR_UNSUPPORTED;
  }
  MatmulPlan merged;
  const bool as_one = merge_row_blocks(plan, &merged);
  bool y_direct = false, rows_aligned = true;
  long long ktotal_chain = 0;
  for (int s = 0; s < plan.nseg; ++s) ktotal_chain += plan.kseg[s];
  for (int g = 0; g < plan.ngroups; ++g) {
    if (plan.m[g] == 0 || plan.n[g] == 0) continue;
    if (stores_y && (!aligned16(plan.y[g]) || (plan.ldy[g] * oesz) % 16 != 0)) y_direct = true;
    if (!plan.b_trans && plan.col_off[g] % 8 != 0) return SBP_ERR_UNSUPPORTED;   // the x coordinate of a TMA load
    if (plan.a_trans && plan.row_off[g] % 8 != 0) rows_aligned = false;
    const long long kg = plan.chain ? ktotal_chain : plan.kseg[g];
    if (kg == 0) return SBP_ERR_UNSUPPORTED;   // an all-zero result: left to the FMA kernel
    if (plan.m[g] > 0x7fffffffLL || plan.n[g] > 0x7fffffffLL) return SBP_ERR_UNSUPPORTED;
  }
  for (int r = 0; r < plan.n_rep; ++r)
    if (!aligned16(plan.y_rep[r])) y_direct = true;
  if (!encode_fn()) return SBP_ERR_UNSUPPORTED;
  if (!rows_aligned && !as_one) return SBP_ERR_UNSUPPORTED;

  int kblocks[SBP_MAX_K];
  long long kb_tile = 0, tiles_sq = 0, tiles_tall = 0;
  for (int s = 0; s < plan.nseg; ++s) {
    kblocks[s] = (int)((plan.kseg[s] + BK - 1) / BK);
    if (plan.chain || s < plan.ngroups) kb_tile = plan.chain ? kb_tile + kblocks[s] : std::max<long long>(kb_tile, kblocks[s]);
  }
  for (int g = 0; g < plan.ngroups; ++g) {
    if (plan.m[g] <= 0 || plan.n[g] <= 0) continue;
    const long long tn = (plan.n[g] + BN - 1) / BN;
    tiles_sq += (plan.m[g] + BM - 1) / BM * tn;
    tiles_tall += (plan.m[g] + 2 * BM - 1) / (2 * BM) * tn;
  }

  static TcParams p;          // large; filled under a lock and copied by value at launch
  static std::mutex mu;
  std::lock_guard<std::mutex> lock(mu);

  if (xf && forced_form() == 0 && pair_cap() == 0) {
    const sbp_status ns = launch_narrow(plan, *xf, st, taken);
    if (ns != SBP_OK || *taken) return ns;
  }

  // Which form (see choose_form).  The softmax epilogues are written for the square form, and so is
  // the element-wise store of a result the copy engine cannot address.
  FormChoice form{false, 0, 0.0};
  if (!xf && tiles_tall > 0 && tiles_sq <= 0x1fffffffLL) {
    int cap_sq = 0, cap_tall = 0;
    sbp_status qs = launch_tc(kFormSquare, plan.a_trans, plan.b_trans, nullptr, st, &cap_sq);
    if (qs == SBP_OK) qs = launch_tc(kFormTall, plan.a_trans, plan.b_trans, nullptr, st, &cap_tall);
    if (qs != SBP_OK) return qs;
    const int forced = forced_form();
    OperandRows rows = operand_rows(plan);
    if (!rows_aligned) {      // it would run on a repacked copy of X, whose pitch is another
      long long pitch = 0;
      for (int g = 0; g < plan.ngroups; ++g) pitch += (plan.m[g] + 7) / 8 * 8;
      rows.a = pitch % 64 != 0 ? 1.9e-3 : 1.0e-3;
    }
    form = choose_form(tiles_sq, tiles_tall, kb_tile, cap_sq, cap_tall, plan.gelu != 0, plan.n_rep, plan.out_dtype == SBP_F32, rows,
                       forced == 4 ? 0 : forced);
    if (y_direct) {      // its shifted row stores are exposed at the end, where a split deals them out to its pairs
      form.walk_tall = false;
      form.cost += 1.0;
    }
    if (!rows_aligned) {      // the copy: a launch, one read and one write
      form.cost += 4.0;
      for (int s = 0; s < plan.nseg; ++s) form.cost += (double)plan.kseg[s] * merged.m[0] * 4.0 / 4e6;
    }
    if (forced == 4 || (forced == 0 && pair_cap() == 0)) {
      const SplitChoice sc = choose_split(as_one ? merged : plan, kblocks, 0.92 * (form.cost + 5.5), forced, aligned16(ws) ? ws_bytes : 0);
      if (room) {
        *taken = sc.splits > 0 || rows_aligned;
        *room = sc.outer > 1 ? (size_t)sc.outer * (size_t)part_floats(plan) * 4 : 0;
        return SBP_OK;
      }
      if (sc.splits > 0) return launch_split(plan, as_one ? &merged : nullptr, kblocks, sc, !y_direct, static_cast<float*>(ws), st, taken);
    }
  }
  if (!rows_aligned) return SBP_ERR_UNSUPPORTED;
  if (room) {
    *taken = true;
    return SBP_OK;
  }

  p.ngroups = plan.ngroups;
  p.nseg = plan.nseg;
  p.chain = plan.chain;
  p.gelu = plan.gelu;
  p.n_rep = plan.n_rep;
  p.out_f32 = plan.out_dtype == SBP_F32;
  p.xent = xf ? (xf->grad ? 2 : 1) : 0;
  if (xf) p.xf = *xf;
  p.y_direct = y_direct ? 1 : 0;

  for (int s = 0; s < plan.nseg; ++s) {
    p.kblocks[s] = kblocks[s];
    const bool used = plan.chain || s < plan.ngroups;
    if (!used || plan.kseg[s] == 0) continue;
    long long rows_a = 0, cols_b = 0;
    if (plan.chain) {
      for (int g = 0; g < plan.ngroups; ++g) {
        rows_a = std::max(rows_a, plan.row_off[g] + plan.m[g]);
        cols_b = std::max(cols_b, plan.col_off[g] + plan.n[g]);
      }
    } else {
      rows_a = plan.m[s];
      cols_b = plan.n[s];
    }
    if (rows_a == 0 || cols_b == 0) { p.kblocks[s] = plan.chain ? p.kblocks[s] : 0; continue; }
    // as stored: A [rows, K] (transposed [K, rows]), B [K, cols] (transposed [cols, K])
    const bool ok_a = plan.a_trans ? make_map(&p.map_a[s], plan.a[s], 2, plan.kseg[s], rows_a, plan.lda[s], BK, 64)
                                   : make_map(&p.map_a[s], plan.a[s], 2, rows_a, plan.kseg[s], plan.lda[s], BMH, BK);
    if (!ok_a) return fail(SBP_ERR_CUDA, "cuTensorMapEncodeTiled failed for operand x of shard %d", s);
    const bool ok_b = plan.b_trans ? make_map(&p.map_b[s], plan.b[s], 2, cols_b, plan.kseg[s], plan.ldb[s], BNH, BK)
                                   : make_map(&p.map_b[s], plan.b[s], 2, plan.kseg[s], cols_b, plan.ldb[s], BK, 64);
    if (!ok_b) return fail(SBP_ERR_CUDA, "cuTensorMapEncodeTiled failed for operand w of shard %d", s);
  }
  const int tile_m = form.walk_tall ? 2 * BM : BM;
  p.walk_m = tile_m;
  p.tile_first = 0;
  p.half_split = 0;

  int tiles = 0;
  const int box_cols = p.out_f32 ? 32 : 64;
  for (int g = 0; g < plan.ngroups; ++g) {
    p.m[g] = plan.m[g];
    p.n[g] = plan.n[g];
    p.row_off[g] = plan.row_off[g];
    p.col_off[g] = plan.col_off[g];
    p.tile_begin[g] = tiles;
    const long long tm = (plan.m[g] + tile_m - 1) / tile_m, tn = (plan.n[g] + BN - 1) / BN;
    p.tiles_m[g] = (int)std::max(1LL, tm);
    p.tiles_n[g] = (int)std::max(1LL, tn);
    if (plan.m[g] > 0 && plan.n[g] > 0) {
      if (tm * tn + tiles > 0x3fffffffLL) return SBP_ERR_UNSUPPORTED;
      tiles += (int)(tm * tn);
      p.y_ptr[g] = plan.y[g];
      p.ldy[g] = plan.ldy[g];
      if (stores_y && !y_direct && !make_map(&p.map_y[g], plan.y[g], oesz, plan.m[g], plan.n[g], plan.ldy[g], 32, box_cols))
        return fail(SBP_ERR_CUDA, "cuTensorMapEncodeTiled failed for the result of group %d", g);
    }
  }
  // row-block (or column-block) groups of one fused result: one grid for the walk
  bool rows_stack = plan.chain && plan.ngroups > 1, cols_stack = rows_stack;
  for (int g = 0; g < plan.ngroups; ++g) {
    if (plan.n[g] != plan.n[0] || plan.col_off[g] != 0 || plan.n[g] == 0) rows_stack = false;
    if (plan.m[g] != plan.m[0] || plan.row_off[g] != 0 || plan.m[g] == 0) cols_stack = false;
  }
  p.stacked = rows_stack ? 1 : (cols_stack ? 2 : 0);
  p.mt_begin[0] = 0;
  for (int g = 0; g < plan.ngroups; ++g) {
    const bool live = plan.m[g] > 0 && plan.n[g] > 0;
    p.mt_begin[g + 1] = p.mt_begin[g] + (live ? (p.stacked == 2 ? p.tiles_n[g] : p.tiles_m[g]) : 0);
  }
  for (int g = 0; g < plan.ngroups; ++g) {
    const long long tn_walk = p.stacked == 2 ? p.mt_begin[plan.ngroups] : (p.stacked ? p.tiles_n[0] : p.tiles_n[g]);
    p.panel_magic[g] = (unsigned)((1ull << 32) / (unsigned long long)(kPanelM * std::max(1LL, tn_walk)));
  }
  p.tile_begin[plan.ngroups] = tiles;
  for (int g = plan.ngroups + 1; g <= SBP_MAX_K; ++g) p.tile_begin[g] = tiles;
  p.total_tiles = tiles;
  for (int r = 0; r < plan.n_rep; ++r) {
    p.rep_ptr[r] = plan.y_rep[r];
    if (!y_direct && !make_map(&p.map_rep[r], plan.y_rep[r], oesz, plan.m[0], plan.n[0], plan.ldy[0], 32, box_cols))
      return fail(SBP_ERR_CUDA, "cuTensorMapEncodeTiled failed for a result replica");
  }
  *taken = true;
  if (tiles == 0) return SBP_OK;

  if (!form.walk_tall) return launch_tc(kb_tile <= kShortBlocks ? kFormShort : kFormSquare, plan.a_trans, plan.b_trans, &p, st, nullptr);
  // tall form over the first walked tiles, then (mixed run) the square form over the halves of the rest
  const int tall_tiles = std::min(form.tall_tiles, tiles);
  p.total_tiles = tall_tiles;
  sbp_status rs = launch_tc(kFormTall, plan.a_trans, plan.b_trans, &p, st, nullptr);
  if (rs != SBP_OK || tall_tiles == tiles) return rs;
  p.tile_first = tall_tiles;
  p.half_split = 1;
  p.total_tiles = 2 * (tiles - tall_tiles);
  return launch_tc(kFormSquare, plan.a_trans, plan.b_trans, &p, st, nullptr);
}

sbp_status launch_matmul_tc(const MatmulPlan& plan, const XentFusion* xf, void* ws, size_t ws_bytes, cudaStream_t st, bool* taken) {
  return run_matmul_tc(plan, xf, ws, ws_bytes, st, taken, nullptr);
}

bool matmul_tc_room(const MatmulPlan& plan, size_t* room) {
  *room = 0;
  bool taken = false;
  return run_matmul_tc(plan, nullptr, nullptr, ~size_t(0), nullptr, &taken, room) == SBP_OK && taken;
}

sbp_status read_and_clear_tc_timeout(bool* timed_out) { return read_and_clear_timeout_flag(timed_out); }

}  // namespace sbp
