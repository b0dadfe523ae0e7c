// fp32 MatMul on the tensor cores: executes a grouped-GEMM plan (matmul_plan.h) with the accuracy of fp32 arithmetic.
//
// An fp32 number from 2^-110 on is the sum of three bf16 numbers, x = h + m + l, each the rounding of what the ones before it
// leave; below, bits would fall under bf16's smallest step of 2^-133.  So every operand is taken 2^39 times, which brings fp32's
// smallest step to 2^-110 and the results, 2^78 times as large, clear of where low products would be lost, and the sums are put
// back at the end.  What that carries past fp32's range, operands from 2^88 and sums from 2^49 on, is found like infinities.
// A product of two numbers is then hh + (hm + mh) + (hl + mm + lh) + terms below 2^-24 of it, that is six products of bf16
// numbers, each exact in fp32.  The tensor cores sum them up over a slot of 32 K-steps, the smallest products first: their
// accumulator cuts off what an addition shifts out, and over longer runs that would show.  The slot's sum is then added to
// fp32 registers with IEEE additions.  (The split and the six products: Henry, Tang and Heinecke, Leveraging the bfloat16
// artificial intelligence datatype for higher-precision computations, 2019; sums outside the tensor cores: Ootomo and Yokota,
// Recovering single precision accuracy from tensor cores, 2022.)
// Error against fp64, root mean square, relative, this / the tiled FMA kernel as it would be cut:
//   1024 x K x 1024, K =      64               128              1024             2048 (2048^3)
//   normal operands           6.3e-8 / 14e-8   7.0e-8 / 11e-8   10e-8 / 29e-8    12e-8 / 41e-8
//   their magnitudes          6.4e-8 / 12e-8   6.6e-8 / 5.8e-8  7.7e-8 / 13e-8   8.8e-8 / 18e-8
//   log-normal, sigma 2       29e-8 / 14e-8    27e-8 / 13e-8    22e-8 / 32e-8    20e-8 / 55e-8
// Operands of one sign show what the cut-off leaves (slots of 64: 3.2e-7 at any K), sums of a few large terms what it takes from the
// small ones.  Over 92 drawn products that run here, normal operands: 0.36 of the FMA kernel's error on the geometric mean and
// 0.60 at most; their magnitudes 0.64 and 1.35 (948 x 1877 x 1769, which that kernel cuts in eight: 13e-8 / 9.6e-8).  (hh in an
// accumulator of its own: 5.6e-8 at K = 64, log-normal as before; left there for 64 K-steps 9.0e-8 and 4.9e-7.)
//
//   warps 0-7   the accumulators: they add a slot's sum, 32 rows x half of the columns a warp, out of one of two buffers
//               in tensor memory
//   warps 8-15  the operands: they load fp32 quads into registers a slot ahead, split them and put the parts into the
//               six planes of a ring slot in shared memory
//   warp 16     one elected lane issues the slot's twelve M128 N16..192 K16 MMAs and commits slot and buffer
//
// Operands keep the order they have in memory: K-contiguous ones become K-major tiles with 64-byte rows, the others
// MN-major tiles in chunks of 64 columns.  A tile whose K is long and whose device is otherwise idle is cut along K
// over the CTAs of a cluster, whose partial tiles are added in order through distributed shared memory.
//
// Bound: no one unit.  At 2048^3 the data path of shared memory is busy 67 % of the clocks (per slot of a 128 x 128 tile the
// MMAs read 768 lines of 128 bytes, the planes take 384, the loads pass 256 to 512, in some 2200 clocks), the schedulers issue in
// 49 %, the tensor pipe works in 31 %; a slot's round through loads, splitting, barriers and accumulators sets the pace.
// A wider tile shares the A operand (192 columns 2800 clocks, 1870 for 128 of them); 16 warps for the operands instead of 8 change
// nothing (2048^3 157 and 153 us).
// 1000 x 1024 x 1500 on four shards 33 us, 1000 x 1500 x 777 40, 2048^3 166 (103 TFLOP/s); FMA kernel 87, 92, 422.
//
// A result that is not finite (operands or sums that are not, or not once scaled, or a bf16 part that rounds to infinity) is found
// in the accumulators; the CTA then multiplies its tile again with fp32 multiply-adds (multiply_again).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <type_traits>

#include "bounds_check.h"
#include "matmul_plan.h"
#include "sbp_internal.h"
#include "tc_ptx.h"

namespace sbp {

namespace {

constexpr int kTM = 128;                 // rows of a tile
constexpr int kTN = 192;                 // columns of a tile, at most
constexpr int kSK = 32;                  // K-steps of a ring slot
constexpr int kMaxSlots = 8;
constexpr int kDrain = 256;              // threads that keep the accumulators, threads that split operands
constexpr int kWorkers = 256;
constexpr int kThreads = kDrain + kWorkers + 128;      // and a warpgroup one warp of which issues the MMAs
constexpr int kMmaWarp = (kDrain + kWorkers) / 32;
constexpr int kPlaneA = kTM * kSK * 2;   // one bf16 part of an A slot
constexpr int kRing = 198 * 1024;
constexpr int kSmem = kRing + 1024;      // + alignment slack
constexpr int kAccs = 2;                 // accumulators in tensor memory
constexpr int kAccCols = 256;            // columns from one to the other

struct F32TcParams {
  MatmulPlan plan;
  int splits;                            // CTAs per tile (cluster size)
  int nb;                                // columns of a tile, a multiple of 16
  int slots;                             // ring slots
};

__device__ __forceinline__ float gelu_erf(float v) { return 0.5f * v * (1.0f + erff(v * 0.70710678118654752440f)); }

__device__ __forceinline__ unsigned long long pack(float x, float y) {
  unsigned long long v;
  asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(x), "f"(y));
  return v;
}

// Two numbers, scaled, as three bf16 each, packed.
constexpr float kScale = 0x1p39f;
__device__ __forceinline__ unsigned bf16_pair(float lo, float hi) {
  unsigned r;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
  return r;
}
// (x, y) less the two bf16 of h: exact
__device__ __forceinline__ void less_pair(float& x, float& y, unsigned h) {
  asm("{\n\t.reg .b64 v, w;\n\tmov.b64 v, {%0, %1};\n\tmov.b64 w, {%2, %3};\n\tfma.rn.f32x2 v, w, %4, v;\n\tmov.b64 {%0, %1}, v;\n\t}"
      : "+f"(x), "+f"(y)
      : "r"(h << 16), "r"(h & 0xffff0000u), "l"(0xbf800000bf800000ull));
}
__device__ __forceinline__ void split_pair(float x, float y, unsigned& h, unsigned& m, unsigned& l) {
  asm("{\n\t.reg .b64 v;\n\tmov.b64 v, {%0, %1};\n\tmul.rn.f32x2 v, v, %2;\n\tmov.b64 {%0, %1}, v;\n\t}"
      : "+f"(x), "+f"(y)
      : "l"(pack(kScale, kScale)));
  h = bf16_pair(x, y);
  less_pair(x, y, h);
  m = bf16_pair(x, y);
  less_pair(x, y, m);
  l = bf16_pair(x, y);
}

// A worker's share of an operand: Q quads of consecutive elements a slot, kept in registers between their load and
// their way into the ring slot's planes.  KC: K is contiguous in memory; quad j of thread t is quad t mod 8 of row
// t / 8 + 32 j.  Otherwise a K-step has 2^SH quads, and quad j is one of K-step (t >> SH) + j (256 >> SH).
// The loads are predicated instructions: where a branch stood around them each was waited for before the next was made
// (300 to 430 clocks a quad).
template <int Q, bool KC, int SH>
struct Share {
  static constexpr int kApart = KC ? kWorkers / 8 : kWorkers >> SH;      // rows (K-steps) from quad j to quad j + 1
  static constexpr int kHop = kApart * (KC ? 64 : 128);                  // bytes
  static constexpr unsigned kOdd = !KC && SH == 6 ? 64 : 0;              // four K-steps on, the 128-byte swizzle is another one
  float4 r[Q];
  const float* at;               // quad 0 of the next slot to load
  int step;                      // elements from quad j to quad j + 1
  int limit;                     // KC: K in the slot before the quad; else elements from it to the operand's edge
  int first;                     // row (K-step) of quad 0
  int rows, tile_rows;           // rows of the operand / of the tile from there on (KC)
  unsigned off;                  // where quad 0 goes in a plane

  __device__ __forceinline__ void init(int t, int ext, int width) {
    if constexpr (KC) {          // rows of 64 bytes, 64-byte swizzle
      const int row = t >> 3, c = t & 7;
      first = row;
      limit = c * 4;
      rows = ext - row;
      tile_rows = width - row;
      off = row * 64 + (((c >> 1) ^ ((row >> 1) & 3)) << 4) + (c & 1) * 8;
    } else {                     // chunks of 64 positions: rows of 128 bytes, 128-byte swizzle
      const int k = t >> SH, c = t & ((1 << SH) - 1);
      first = k;
      limit = ext - c * 4;
      rows = 0;
      tile_rows = c * 4 < width ? kSK : 0;
      off = (c >> 4) * (kSK * 128) + k * 128 + ((((c >> 1) & 7) ^ (k & 7)) << 4) + (c & 1) * 8;
    }
  }
  // g: position (0, 0) of the slot that is loaded next
  __device__ __forceinline__ void point(const float* g, long long ld, int t) {
    at = g + first * ld + (KC ? limit : (t & ((1 << SH) - 1)) * 4);
    step = kApart * (int)ld;
  }
  // VEC: every quad lies inside as a whole or not at all, and 16-byte aligned.  count: quads a slot
  template <bool VEC>
  __device__ __forceinline__ void load(int left, int count) {
#pragma unroll
    for (int j = 0; j < Q; ++j) {
      if (j >= count) break;
      const float* src = at + (long long)j * step;
      int have;                  // elements of the quad that lie inside
      if constexpr (KC) have = j * kApart < rows ? left - limit : 0;
      else have = first + j * kApart < left ? limit : 0;
      r[j] = make_float4(0.f, 0.f, 0.f, 0.f);
      if constexpr (VEC) {
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %5, 0;\n\t@p ld.global.L1::no_allocate.v4.f32 {%0, %1, %2, %3}, [%4];\n\t}"
                     : "+f"(r[j].x), "+f"(r[j].y), "+f"(r[j].z), "+f"(r[j].w)
                     : "l"(src), "r"(have > 0 && SBP_GUARD(src, 16) ? 1 : 0));
      } else {
        float* e[4] = {&r[j].x, &r[j].y, &r[j].z, &r[j].w};
#pragma unroll
        for (int i = 0; i < 4; ++i)
          asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %2, 0;\n\t@p ld.global.f32 %0, [%1];\n\t}"
                       : "+f"(*e[i])
                       : "l"(src + i), "r"(have > i && SBP_GUARD(src + i, 4) ? 1 : 0));
      }
    }
  }
  __device__ __forceinline__ void store(unsigned base, int plane, int count) {
#pragma unroll
    for (int j = 0; j < Q; ++j) {
      if (j >= count) break;
      const unsigned to = base + ((j & 1) ? off ^ kOdd : off) + j * kHop;
      uint2 h, m, l;
      split_pair(r[j].x, r[j].y, h.x, m.x, l.x);
      split_pair(r[j].z, r[j].w, h.y, m.y, l.y);
      asm volatile(
          "{\n\t.reg .pred p;\n\tsetp.gt.s32 p, %9, %10;\n\t@p st.shared.v2.b32 [%0], {%3, %4};\n\t@p st.shared.v2.b32 [%1], {%5, %6};\n\t"
          "@p st.shared.v2.b32 [%2], {%7, %8};\n\t}" ::"r"(to),
          "r"(to + plane), "r"(to + 2 * plane), "r"(h.x), "r"(h.y), "r"(m.x), "r"(m.y), "r"(l.x), "r"(l.y), "r"(tile_rows), "r"(KC ? j * kApart : 0));
    }
  }
};

// a += b on two packed numbers
__device__ __forceinline__ void add2(unsigned long long& a, unsigned long long b) { asm("add.rn.f32x2 %0, %0, %1;" : "+l"(a) : "l"(b)); }
__device__ __forceinline__ float lo(unsigned long long v) { return __uint_as_float((unsigned)v); }
__device__ __forceinline__ float hi(unsigned long long v) { return __uint_as_float((unsigned)(v >> 32)); }

// 16 accumulator columns of this warp's 32 rows, in pairs
__device__ __forceinline__ void tmem_ld16_wait(unsigned taddr, unsigned long long (&v)[8]) {
  unsigned r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
#pragma unroll
  for (int i = 0; i < 8; ++i) asm("mov.b64 %0, {%1, %2};" : "=l"(v[i]) : "r"(r[2 * i]), "r"(r[2 * i + 1]));
}

// 4 * QUARTERS bytes, or as many zeros
template <int QUARTERS>
__device__ __forceinline__ void copy_async(const float* to, const float* from, const float* somewhere, bool in) {
  if constexpr (QUARTERS == 4)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_addr(to)), "l"(in ? from : somewhere), "r"(in ? 16u : 0u) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(smem_addr(to)), "l"(in ? from : somewhere), "r"(in ? 4u : 0u) : "memory");
}

// Whole aligned quads everywhere, or element by element?
template <int AT, int BT>
__device__ __forceinline__ void whole_quads(const MatmulPlan& p, int g, int s_lo, int s_hi, int rows, int cols, bool& a, bool& b) {
  a = AT ? (rows & 3) == 0 && (p.row_off[g] & 3) == 0 : true;
  b = BT ? true : (cols & 3) == 0 && (p.col_off[g] & 3) == 0;
  for (int s = s_lo; s < s_hi; ++s) {
    a = a && (reinterpret_cast<unsigned long long>(p.a[s]) & 15) == 0 && (p.lda[s] & 3) == 0 && (AT || (p.kseg[s] & 3) == 0);
    b = b && (reinterpret_cast<unsigned long long>(p.b[s]) & 15) == 0 && (p.ldb[s] & 3) == 0 && (!BT || (p.kseg[s] & 3) == 0);
  }
}

// The slots of CTA `slice` of the `splits` that share a tile of group g: segment and K inside it where they start, and how many.
__device__ __forceinline__ void slots_of(const MatmulPlan& p, int g, int slice, int splits, int& seg, long long& k, int& n) {
  const int s_lo = p.chain ? 0 : g, s_hi = p.chain ? p.nseg : g + 1;
  long long total = 0;
  for (int s = s_lo; s < s_hi; ++s) total += (p.kseg[s] + kSK - 1) / kSK;
  const long long first = total * slice / splits;
  n = (int)(total * (slice + 1) / splits - first);
  seg = s_lo;
  k = first;
  while (seg < s_hi) {
    const long long slots = (p.kseg[seg] + kSK - 1) / kSK;
    if (k < slots) break;
    k -= slots;
    ++seg;
  }
  k *= kSK;
}

// A slot of an operand on its way into shared memory, in the order it has: K-contiguous as rows of kSK + 4, else `width` positions a
// K-step, `pitch` apart.  Q elements at once.
constexpr int kAll = kDrain + kWorkers, kPitchK = kSK + 4;
template <int Q, bool KC>
__device__ __forceinline__ void fill_slot(float* to, const float* from, long long ld, int ext, int left, int width, int pitch, int tid) {
  if constexpr (KC) {
    constexpr int kPer = kSK / Q;
    for (int r = tid / kPer; r < width; r += kAll / kPer) {
      const int k = tid % kPer * Q;
      const float* src = from + r * ld + k;
      copy_async<Q>(to + r * kPitchK + k, src, from, r < ext && k < left && SBP_GUARD(src, Q * 4));
    }
  } else {
    for (int k = tid >> 5; k < kSK; k += kAll / 32)
      for (int c = (tid & 31) * Q; c < width; c += 32 * Q) {
        const float* src = from + k * ld + c;
        copy_async<Q>(to + k * pitch + c, src, from, k < left && c < ext && SBP_GUARD(src, Q * 4));
      }
  }
}

// A tile that bf16 parts do not serve, once more with fp32 multiply-adds, by the warps of the accumulators and of the operands:
// 4 x 12 elements a thread, slots of fp32 operands in two buffers at the ring's end.  A chain is four slots, its sum goes to the
// tile.  Bound: the FMA pipe, 64 clocks a K-step and 64 columns.
// (us, a product on the tensor cores / with every tile once more / on the FMA kernel, whose tiles fill the device more evenly:
// 1024^3 27 / 123 / 61, 2048^3 165 / 908 / 422, 1000 x 1500 x 777 36 / 168 / 95; one chain of loads an element: 4740, 35200, 3200.  Over 21 drawn products that run here 1.65
// times the FMA kernel's time on the geometric mean, 2.7 at most, 40 x 2500 x 24.)
template <int AT, int BT>
__device__ __forceinline__ void multiply_again(const F32TcParams& P, unsigned char* smem, int tid) {
  // Where the tile lies, once more: kept from the start it would take registers from the operands' loop.
  unsigned bx, by, bz;
  asm volatile("mov.u32 %0, %%ctaid.x;\n\tmov.u32 %1, %%ctaid.y;\n\tmov.u32 %2, %%ctaid.z;" : "=r"(bx), "=r"(by), "=r"(bz));
  const MatmulPlan& p = P.plan;
  const int g = (int)bz, nb = P.nb;
  const long long m0 = (long long)by * kTM, n0 = (long long)(bx / (unsigned)P.splits) * nb;
  const int rows = (int)min((long long)kTM, p.m[g] - m0), cols = (int)min((long long)nb, p.n[g] - n0);
  const int s_hi = p.chain ? p.nseg : g + 1;
  int s, iters;
  long long k;
  slots_of(p, g, (int)(bx % (unsigned)P.splits), P.splits, s, k, iters);
  bool a_vec, b_vec;
  whole_quads<AT, BT>(p, g, p.chain ? 0 : g, s_hi, rows, cols, a_vec, b_vec);
  constexpr bool AKC = !AT, BKC = BT;
  constexpr int kPitchA = kTM + 4, kPitchB = kTN + 4, kChain = 4;
  constexpr int kA = AKC ? kTM * kPitchK : kSK * kPitchA, kB = BKC ? kTN * kPitchK : kSK * kPitchB;
  static_assert(kTM * (kTN + 4) * 4 + 2 * (kA + kB) * 4 <= kRing, "tile and two buffers");
  float* const buffers = reinterpret_cast<float*>(smem + kRing) - 2 * (kA + kB);
  const int ty = tid >> 4, tx = tid & 15;
  float* const out = reinterpret_cast<float*>(smem) + ty * 4 * (nb + 4) + (BKC ? tx : tx * 4);
  auto fill = [&](int b) {
    while (s < s_hi && k >= p.kseg[s]) { ++s; k = 0; }      // also steps over empty segments
    const int left = (int)min((long long)kSK, p.kseg[s] - k);
    const long long lda = p.lda[s], ldb = p.ldb[s];
    const float* A = static_cast<const float*>(p.a[s]) + (AT ? k * lda + p.row_off[g] + m0 : (p.row_off[g] + m0) * lda + k);
    const float* B = static_cast<const float*>(p.b[s]) + (BT ? (p.col_off[g] + n0) * ldb + k : k * ldb + p.col_off[g] + n0);
    float* to = buffers + b * (kA + kB);
    if (a_vec) fill_slot<4, AKC>(to, A, lda, rows, left, kTM, kPitchA, tid);
    else fill_slot<1, AKC>(to, A, lda, rows, left, kTM, kPitchA, tid);
    if (b_vec) fill_slot<4, BKC>(to + kA, B, ldb, cols, left, nb, kPitchB, tid);
    else fill_slot<1, BKC>(to + kA, B, ldb, cols, left, nb, kPitchB, tid);
    k += kSK;
  };
  unsigned long long acc[4][6];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 6; ++j) acc[i][j] = 0ull;
  if (iters > 0) fill(0);
  asm volatile("cp.async.commit_group;" ::: "memory");
#pragma unroll 1
  for (int it = 0; it < iters; ++it) {
    if (it + 1 < iters) fill((it + 1) & 1);
    asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 1;" ::: "memory");
    asm volatile("bar.sync 2, 512;" ::: "memory");
    const float* sa = buffers + (it & 1) * (kA + kB) + ty * 4 * (AKC ? kPitchK : 1);
    const float* sb = buffers + (it & 1) * (kA + kB) + kA + tx * (BKC ? kPitchK : 4);
#pragma unroll 2
    for (int k0 = 0; k0 < kSK; k0 += 2) {
      float2 x[4];                                     // of row i, two K-steps
      if constexpr (AKC) {
#pragma unroll
        for (int i = 0; i < 4; ++i) x[i] = *reinterpret_cast<const float2*>(sa + i * kPitchK + k0);
      } else {
        const float4 u = *reinterpret_cast<const float4*>(sa + k0 * kPitchA), v = *reinterpret_cast<const float4*>(sa + (k0 + 1) * kPitchA);
        x[0] = make_float2(u.x, v.x); x[1] = make_float2(u.y, v.y); x[2] = make_float2(u.z, v.z); x[3] = make_float2(u.w, v.w);
      }
#pragma unroll
      for (int j = 0; j < 3; ++j) {                    // columns past nb: whatever lies there, never stored
        if (j * 64 >= nb) break;
        unsigned long long w[2][2];                    // K-step, pair of columns
        if constexpr (BKC) {
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const float2 u = *reinterpret_cast<const float2*>(sb + (j * 64 + e * 32) * kPitchK + k0);
            const float2 v = *reinterpret_cast<const float2*>(sb + (j * 64 + e * 32 + 16) * kPitchK + k0);
            w[0][e] = pack(u.x, v.x);
            w[1][e] = pack(u.y, v.y);
          }
        } else {
#pragma unroll
          for (int kk = 0; kk < 2; ++kk) {
            const ulonglong2 u = *reinterpret_cast<const ulonglong2*>(sb + (k0 + kk) * kPitchB + j * 64);
            w[kk][0] = u.x;
            w[kk][1] = u.y;
          }
        }
#pragma unroll
        for (int kk = 0; kk < 2; ++kk)
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const unsigned long long a = kk ? pack(x[i].y, x[i].y) : pack(x[i].x, x[i].x);
            asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc[i][2 * j]) : "l"(a), "l"(w[kk][0]));
            asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc[i][2 * j + 1]) : "l"(a), "l"(w[kk][1]));
          }
      }
    }
    if ((it + 1) % kChain == 0 || it + 1 == iters) {
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          const float v[4] = {lo(acc[i][2 * j]), hi(acc[i][2 * j]), lo(acc[i][2 * j + 1]), hi(acc[i][2 * j + 1])};
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            float* at = out + i * (nb + 4) + j * 64 + (BKC ? e * 16 : e);
            if (j * 64 + (BKC ? e * 16 + tx : tx * 4 + e) < nb) *at = it >= kChain ? *at + v[e] : v[e];
          }
          acc[i][2 * j] = acc[i][2 * j + 1] = 0ull;
        }
    }
    asm volatile("bar.sync 2, 512;" ::: "memory");      // the buffer has been read
  }
}

// AT / BT: the operand is stored transposed.  A as given and B transposed are K-contiguous.
template <int AT, int BT>
__global__ void __launch_bounds__(kThreads, 1) matmul_f32_tc_kernel(const __grid_constant__ F32TcParams P) {
  constexpr bool AKC = !AT, BKC = BT;
  extern __shared__ unsigned char smem_raw[];
  __shared__ __align__(8) unsigned long long bar_full[kMaxSlots], bar_empty[kMaxSlots], bar_acc_full[kAccs], bar_acc_empty[kAccs];
  __shared__ unsigned tmem_base_slot;
  __shared__ int abort_flag_s, again_s;
  volatile int* abort_flag = &abort_flag_s;

  const MatmulPlan& p = P.plan;
  const int g = blockIdx.z, splits = P.splits, slice = (int)(blockIdx.x % (unsigned)splits), nb = P.nb;
  const long long M = p.m[g], N = p.n[g];
  const long long m0 = (long long)blockIdx.y * kTM, n0 = (long long)(blockIdx.x / (unsigned)splits) * nb;
  if (m0 >= M || n0 >= N) return;                  // the whole cluster
  const int rows = (int)min((long long)kTM, M - m0), cols = (int)min((long long)nb, N - n0);
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int plane_b = (nb + 63) / 64 * (64 * kSK * 2), slot_bytes = 3 * (kPlaneA + plane_b), slots = P.slots;

  if (tid == 0) {
    abort_flag_s = 0;
    again_s = 0;
    for (int i = 0; i < slots; ++i) {
      mbar_init(smem_addr(&bar_full[i]), kWorkers / 32);
      mbar_init(smem_addr(&bar_empty[i]), 1);
    }
    for (int i = 0; i < kAccs; ++i) {
      mbar_init(smem_addr(&bar_acc_full[i]), 1);
      mbar_init(smem_addr(&bar_acc_empty[i]), kDrain / 32);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kMmaWarp) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&tmem_base_slot)), "r"(kAccs * kAccCols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }

  // this CTA's range of slots over all segments
  const int s_lo = p.chain ? 0 : g, s_hi = p.chain ? p.nseg : g + 1;
  int seg0, iters;
  long long k0;
  slots_of(p, g, slice, splits, seg0, k0, iters);

  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const unsigned tmem_base = tmem_base_slot;
  SBP_PDL_WAIT();                                  // everything up to here overlaps the kernel before this one

  const int q = warp & 3, half = (warp >> 2) & 1, width = nb / 2;      // a draining warp's tensor-memory lanes and columns
  if (warp < kMmaWarp) {                           // two roles that end with the same registers
  if (warp < kDrain / 32) {
    // ------------------------------------------------ accumulators
    asm volatile("setmaxnreg.inc.sync.aligned.u32 128;");        // 2 x 128 + 2 x 88 + 48 = 5 x 96
    unsigned long long acc[kTN / 4];
#pragma unroll
    for (int i = 0; i < kTN / 4; ++i) acc[i] = 0ull;
    bool ok = true;
    for (int c = 0; c < iters; ++c) {
      ok = mbar_wait_warp(smem_addr(&bar_acc_full[c % kAccs]), (unsigned)(c / kAccs & 1), abort_flag);
      if (!ok) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const unsigned at = tmem_base + ((unsigned)(q * 32) << 16) + (c % kAccs) * kAccCols + half * width;
#pragma unroll
      for (int b = 0; b < kTN / 4; b += 8) {
        if (2 * b >= width) break;
        unsigned long long v[8];
        tmem_ld16_wait(at + 2 * b, v);
#pragma unroll
        for (int i = 0; i < 8; ++i) add2(acc[b + i], v[i]);
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_addr(&bar_acc_empty[c % kAccs]));
    }
    // every product has been made: the ring becomes the tile
    SBP_PDL_RELEASE();
    float zero = 0.f;                              // stays so unless something is not finite
    float* tile = reinterpret_cast<float*>(smem) + (q * 32 + lane) * (nb + 4) + half * width;
#pragma unroll
    for (int i = 0; i < kTN / 4; i += 4) {
      if (2 * i >= width) break;
#pragma unroll
      for (int e = 0; e < 4; ++e) zero = fmaf(hi(acc[i + e]), 0.f, fmaf(lo(acc[i + e]), 0.f, zero));
    }
    if (zero != 0.f) again_s = 1;
    asm volatile("bar.sync 1, 256;" ::: "memory");      // every warp has seen its last chunk
#pragma unroll
    for (int i = 0; i < kTN / 4; i += 2) {
      if (2 * i >= width) break;
      constexpr float kBack = 1.0f / (kScale * kScale);
      *reinterpret_cast<float4*>(tile + 2 * i) = make_float4(lo(acc[i]) * kBack, hi(acc[i]) * kBack, lo(acc[i + 1]) * kBack, hi(acc[i + 1]) * kBack);
    }
    asm volatile("setmaxnreg.dec.sync.aligned.u32 88;");         // as the others that go on
  } else {
    // ------------------------------------------------ operands
    asm volatile("setmaxnreg.dec.sync.aligned.u32 88;");
    const int t = tid - kDrain;
    bool a_vec, b_vec;
    whole_quads<AT, BT>(p, g, s_lo, s_hi, rows, cols, a_vec, b_vec);
    constexpr int kQA = kTM * kSK / 4 / kWorkers;
    // sh: log2 of the quads of a K-step of an MN-contiguous B
    auto run = [&](auto av, auto bv, auto sh) {
      constexpr bool AV = decltype(av)::value, BV = decltype(bv)::value;
      constexpr int SH = decltype(sh)::value, kQB = BKC ? kTN * kSK / 4 / kWorkers : kSK / (kWorkers >> SH);
      Share<kQA, AKC, 5> A;
      Share<kQB, BKC, SH> B;
      A.init(t, rows, kTM);
      B.init(t, cols, nb);
      const int count_b = BKC ? (nb + 31) / 32 : kQB;
      int ls = seg0, left = 0, lk = (int)k0;
      // the next slot to load: afresh at the start of a segment, else one step on
      auto next_slot = [&](bool start) {
        if (!start) {
          lk += kSK;
          if (lk < (int)p.kseg[ls]) {
            A.at += AKC ? kSK : kSK * (int)p.lda[ls];
            B.at += BKC ? kSK : kSK * (int)p.ldb[ls];
            left = min(kSK, (int)p.kseg[ls] - lk);
            return;
          }
        }
        while (ls < s_hi && lk >= p.kseg[ls]) { ++ls; lk = 0; }      // also steps over empty segments
        const long long lda = p.lda[ls], ldb = p.ldb[ls];
        A.point(static_cast<const float*>(p.a[ls]) + (AT ? lk * lda + p.row_off[g] + m0 : (p.row_off[g] + m0) * lda + lk), lda, t);
        B.point(static_cast<const float*>(p.b[ls]) + (BT ? (p.col_off[g] + n0) * ldb + lk : lk * ldb + p.col_off[g] + n0), ldb, t);
        left = min(kSK, (int)p.kseg[ls] - lk);
      };
      if (iters > 0) {
        next_slot(true);
        A.template load<AV>(left, kQA);
        B.template load<BV>(left, count_b);
      }
      int slot = 0;
      unsigned round = 0;
      for (int it = 0; it < iters; ++it) {
        if (!mbar_wait_warp(smem_addr(&bar_empty[slot]), round ^ 1, abort_flag)) break;
        const unsigned to = smem_addr(smem) + slot * slot_bytes;
        if (it + 1 < iters) next_slot(false);
        else left = 0;
        A.store(to, kPlaneA, kQA);                 // and the next slot's quads take the registers
        A.template load<AV>(left, kQA);
        B.store(to + 3 * kPlaneA, plane_b, count_b);
        B.template load<BV>(left, count_b);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_addr(&bar_full[slot]));
        slot = slot + 1 == slots ? 0 : slot + 1;
        round ^= (slot == 0);
      }
    };
    auto run_b = [&](auto av, auto sh) {
      if (b_vec) run(av, std::true_type{}, sh);
      else run(av, std::false_type{}, sh);
    };
    auto run_a = [&](auto sh) {
      if (a_vec) run_b(std::true_type{}, sh);
      else run_b(std::false_type{}, sh);
    };
    if constexpr (BKC) {
      run_a(std::integral_constant<int, 5>{});
    } else {
      if (nb > 128) run_a(std::integral_constant<int, 6>{});
      else if (nb > 64) run_a(std::integral_constant<int, 5>{});
      else run_a(std::integral_constant<int, 4>{});
    }
  }
  asm volatile("bar.sync 2, 512;" ::: "memory");
  if (again_s) multiply_again<AT, BT>(P, smem, tid);
  } else {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 48;");
    if (warp == kMmaWarp) {
    // ------------------------------------------------ MMA issuer
    const bool leader = elect_one();
    const unsigned idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((AT ? 1u : 0u) << 15) | ((BT ? 0u : 1u) << 16) | ((unsigned)(nb >> 3) << 17) |
                           ((unsigned)(kTM >> 4) << 24);
    constexpr unsigned a_lo = desc_lo_fixed(AKC ? 16 : kSK * 128), b_lo = desc_lo_fixed(BKC ? 16 : kSK * 128);
    constexpr unsigned a_hi = AKC ? desc_hi_fixed(512, 4) : desc_hi_fixed(1024), b_hi = BKC ? desc_hi_fixed(512, 4) : desc_hi_fixed(1024);
    constexpr unsigned a_step = AKC ? 2 : 128, b_step = BKC ? 2 : 128;      // 16 K-steps, in 16-byte units
    int slot = 0;
    unsigned round = 0;
    for (int it = 0; it < iters; ++it) {
      const int c = it;
      if (!mbar_wait_warp(smem_addr(&bar_acc_empty[c % kAccs]), (unsigned)((c / kAccs & 1) ^ 1), abort_flag)) break;
      if (!mbar_wait_warp(smem_addr(&bar_full[slot]), round, abort_flag)) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      if (leader) {
        const unsigned sa = (smem_addr(smem) + slot * slot_bytes) & 0x3ffffu, sb = sa + 3 * kPlaneA;
        const unsigned d = tmem_base + (c % kAccs) * kAccCols;
        unsigned accumulate = 0;
        // parts of A and B, the smallest products first
        constexpr int pa[6] = {2, 0, 1, 1, 0, 0}, pb[6] = {0, 2, 1, 0, 1, 0};
#pragma unroll
        for (int t = 0; t < 6; ++t)
#pragma unroll
          for (int kk = 0; kk < kSK / 16; ++kk) {
            umma_bf16_cta(d, desc_pack(a_lo + ((sa + pa[t] * kPlaneA) >> 4) + kk * a_step, a_hi),
                          desc_pack(b_lo + ((sb + pb[t] * plane_b) >> 4) + kk * b_step, b_hi), idesc, accumulate);
            accumulate = 1;
          }
        umma_commit_cta(smem_addr(&bar_empty[slot]));
        umma_commit_cta(smem_addr(&bar_acc_full[c % kAccs]));
      }
      __syncwarp();
      slot = slot + 1 == slots ? 0 : slot + 1;
      round ^= (slot == 0);
    }
    if (*abort_flag && leader) {                   // products in flight get a bounded chance to finish
      umma_commit_cta(smem_addr(&bar_acc_full[0]));
      const unsigned long long t0 = now_ns();
      const unsigned parity = 0;
      while (!mbar_try(smem_addr(&bar_acc_full[0]), parity) && now_ns() - t0 < 100000000ull) {
      }
    }
    __syncwarp();
    }
  }

  // The tile is in shared memory: each CTA of the cluster adds up the partial sums of its rows, slice by slice, and stores them.
  if (splits > 1) cluster_sync_all();
  else __syncthreads();
  if (warp < kMmaWarp) {
    const int r_lo = kTM * slice / splits, r_hi = min(rows, kTM * (slice + 1) / splits);
    const long long ldy = p.ldy[g];
    const int n_out = (g == 0 ? p.n_rep : 0) + 1;
    bool y_vec = (reinterpret_cast<unsigned long long>(p.y[g]) & 15) == 0 && (ldy & 3) == 0;
    for (int o = 1; o < n_out; ++o) y_vec = y_vec && (reinterpret_cast<unsigned long long>(p.y_rep[o - 1]) & 15) == 0;
    for (int r = r_lo + warp; r < r_hi; r += kMmaWarp) {
      for (int c = lane * 4; c < cols; c += 128) {
        const unsigned at = smem_addr(smem) + (unsigned)(r * (nb + 4) + c) * 4;
        float v[4];
        if (splits == 1) {
          *reinterpret_cast<float4*>(v) = *reinterpret_cast<const float4*>(reinterpret_cast<const float*>(smem) + r * (nb + 4) + c);
        } else {
#pragma unroll 1
          for (int s = 0; s < splits; s += 4) {      // four at a time, in ascending order
            float x[4][4];
#pragma unroll
            for (int i = 0; i < 4; ++i)
              if (s + i < splits)
                asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                             : "=f"(x[i][0]), "=f"(x[i][1]), "=f"(x[i][2]), "=f"(x[i][3])
                             : "r"(map_to_cta(at, s + i))
                             : "memory");
#pragma unroll
            for (int i = 0; i < 4; ++i)
              if (s + i < splits) {
#pragma unroll
                for (int e = 0; e < 4; ++e) v[e] = s + i == 0 ? x[i][e] : v[e] + x[i][e];
              }
          }
        }
        if (p.gelu) {
#pragma unroll
          for (int e = 0; e < 4; ++e) v[e] = gelu_erf(v[e]);
        }
        for (int o = 0; o < n_out; ++o) {
          float* y = static_cast<float*>(o == 0 ? p.y[g] : p.y_rep[o - 1]) + (m0 + r) * ldy + n0 + c;
          if (y_vec && c + 3 < cols) {
            if (SBP_GUARD(y, 16)) *reinterpret_cast<float4*>(y) = make_float4(v[0], v[1], v[2], v[3]);
          } else {
#pragma unroll
            for (int e = 0; e < 4; ++e)
              if (c + e < cols && SBP_GUARD(y + e, 4)) y[e] = v[e];
          }
        }
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  if (splits > 1) cluster_sync_all();              // nobody leaves while its tile may still be read
  else __syncthreads();
  if (warp == kMmaWarp) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kAccs * kAccCols) : "memory");
  }
}

template <int AT, int BT>
cudaError_t launch_form(const F32TcParams* P, int splits, dim3 grid, cudaStream_t st, int* capacity) {
  static std::atomic<unsigned long long> opted{0};      // one bit per device
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const unsigned long long bit = 1ull << (dev & 63);
  if (dev >= 64 || !(opted.load(std::memory_order_relaxed) & bit)) {
    e = cudaFuncSetAttribute(matmul_f32_tc_kernel<AT, BT>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
    if (e != cudaSuccess) return e;
    if (dev < 64) opted.fetch_or(bit, std::memory_order_relaxed);
  }
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = kSmem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)splits;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (capacity) return cudaOccupancyMaxActiveClusters(capacity, matmul_f32_tc_kernel<AT, BT>, &cfg);
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, matmul_f32_tc_kernel<AT, BT>, *P);
}

constexpr int kCuts[6] = {1, 2, 3, 4, 6, 8};      // CTAs that may share a tile

// Clusters of kCuts[i] CTAs that the current device holds at once (a CTA fills its SM), asked once a device.
bool cluster_capacities(int (&cap)[6]) {
  static std::atomic<int> known[64][6];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return false;
  for (int i = 0; i < 6; ++i) {
    cap[i] = known[dev][i].load(std::memory_order_relaxed);
    if (cap[i] == 0) {
      if (launch_form<0, 0>(nullptr, kCuts[i], dim3((unsigned)kCuts[i]), nullptr, &cap[i]) != cudaSuccess || cap[i] < 1) {
        cudaGetLastError();
        cap[i] = -1;
      }
      known[dev][i].store(cap[i], std::memory_order_relaxed);
    }
  }
  return true;
}

}  // namespace

// The best cut of a plan for this kernel: estimated time in us (negative: it does not take the plan), columns of a tile, CTAs a
// tile.  Per wave of clusters: a slot takes 0.705 us and 0.0034 more a column (all of its warps' round: loads, splitting,
// twelve MMAs, the accumulators' turn), 0.15 and 0.001 a column more where A / B come element by element, set-up, drain and
// stores 6 and 0.016 a column.  Fitted to 823 timings of 30 products (rms error 8 %; the pick within 1.5 % of the best cut on
// the average); the exchange is set dearer than in a row of equal calls, between others large clusters wait for their SMs.
// Nothing is looked for (negative) where the least that any cut takes is not below `limit`.
double f32_tc_cost(const MatmulPlan& plan, double limit, int* nb, int* splits) {
  long long slots = 0, mmax = 0, nmax = 0;
  bool a_vec = true, b_vec = true;
  for (int s = 0; s < plan.nseg; ++s) {
    if (!plan.chain && s >= plan.ngroups) continue;
    if (plan.lda[s] % 4 != 0) a_vec = false;
    if (plan.ldb[s] % 4 != 0) b_vec = false;
    if (plan.kseg[s] > 0x7fffff00LL || plan.lda[s] > (1 << 25) || plan.ldb[s] > (1 << 25)) return -1;      // 32-bit steps
    const long long n = (plan.kseg[s] + kSK - 1) / kSK;
    slots = plan.chain ? slots + n : std::max(slots, n);
  }
  for (int g = 0; g < plan.ngroups; ++g) {
    mmax = std::max(mmax, plan.m[g]);
    nmax = std::max(nmax, plan.n[g]);
  }
  if ((mmax + kTM - 1) / kTM > 65535 || slots == 0 || slots > 0x7fffffffLL || nmax == 0) return -1;
  if ((double)((slots + 7) / 8) * 0.76 + 6.2 >= limit) return -1;
  int cap[6];
  if (!cluster_capacities(cap)) return -1;
  double best = -1;
  const long long least = (nmax + kTN - 1) / kTN;
  for (long long t = least; t <= least + 12; ++t) {
    const int w = (int)(((nmax + t - 1) / t + 15) / 16 * 16);
    long long tiles = 0, of_one = 0;
    for (int g = 0; g < plan.ngroups; ++g) {
      if (g == 0 || plan.m[g] != plan.m[g - 1] || plan.n[g] != plan.n[g - 1]) of_one = ((plan.m[g] + kTM - 1) / kTM) * ((plan.n[g] + w - 1) / w);
      tiles += of_one;
    }
    const double per_slot = 0.705 + 0.0034 * w + (a_vec ? 0 : 0.15) + (b_vec ? 0 : 0.001 * w);
    for (int i = 0; i < 6; ++i) {
      const int s = kCuts[i];
      if (slots < s) break;
      if (cap[i] < 1) continue;
      const double waves = (double)((tiles + cap[i] - 1) / cap[i]);
      const double cost = waves * ((double)((slots + s - 1) / s) * per_slot + 6.0 + 0.016 * w + (s > 1 ? 0.25 * s : 0.0));
      if (best < 0 || cost < best) {
        best = cost;
        *nb = w;
        *splits = s;
      }
    }
    if (w <= 32) break;
  }
  return best;
}

sbp_status launch_matmul_f32_tc(const MatmulPlan& plan, int nb, int splits, cudaStream_t st) {
  F32TcParams P;
  P.plan = plan;
  P.nb = nb;
  P.splits = splits;
  P.slots = std::min(kMaxSlots, kRing / (3 * (kPlaneA + (nb + 63) / 64 * (64 * kSK * 2))));
  long long mmax = 0, nmax = 0;
  for (int g = 0; g < plan.ngroups; ++g) {
    mmax = std::max(mmax, plan.m[g]);
    nmax = std::max(nmax, plan.n[g]);
  }
  const long long gx = (nmax + nb - 1) / nb * splits;
  if (gx > 0x7fffffffLL || (mmax + kTM - 1) / kTM > 65535) return fail(SBP_ERR_UNSUPPORTED, "matrix too large for one launch");
  const dim3 grid((unsigned)gx, (unsigned)((mmax + kTM - 1) / kTM), (unsigned)plan.ngroups);
  SBP_BOUNDS_UPLOAD(st);
  cudaError_t e;
  switch ((plan.a_trans ? 2 : 0) | (plan.b_trans ? 1 : 0)) {
    case 0: e = launch_form<0, 0>(&P, splits, grid, st, nullptr); break;
    case 1: e = launch_form<0, 1>(&P, splits, grid, st, nullptr); break;
    case 2: e = launch_form<1, 0>(&P, splits, grid, st, nullptr); break;
    default: e = launch_form<1, 1>(&P, splits, grid, st, nullptr); break;
  }
  if (e != cudaSuccess) return cuda_fail(e, "matmul launch");
  return SBP_OK;
}

sbp_status read_and_clear_f32_tc_timeout(bool* timed_out) { return read_and_clear_timeout_flag(timed_out); }

}  // namespace sbp
