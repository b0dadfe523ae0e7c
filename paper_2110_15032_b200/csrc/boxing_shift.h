// The 16-byte path of the boxing kernels for data that is not 16-byte aligned (device code; shared by the
// same-placement and the different-placement transforms).
//
// A task moves segments (contiguous runs) from one place to another, and where a shard's rows have an odd
// length every segment starts at an address of its own on either side.  Moving such a task in vectors that
// both sides can address means 2-, 4- or 8-byte accesses: an eighth to a half of the bytes in flight per thread,
// and the index arithmetic once per element.  Here a team of threads takes a piece of one segment: where the
// segment lies is worked out once per thread, then each thread writes J whole ALIGNED 16-byte vectors of the
// destination.  The 16 source bytes under one lie in two aligned source vectors (one when the two sides agree
// modulo 16), which are read and shifted together.  The up to 31 bytes before the first and after the last such
// vector are moved element by element, one element a thread, beside the vectors.
// Values and their order are those of the plain kernels, so the results are the same bits.
#pragma once

#include "bounds_check.h"
#include "boxing_arith.h"
#include "sbp_internal.h"

namespace sbp {

// The segments of one task: segment i = (x, ia, m) with i = (x * la + ia) * M + m; byte offsets inside the source
// and the destination local tensor.
struct SegView {
  long long nseg, la, M, seg_bytes;
  bool flat;                                 // one loop level only: x = m = 0
  long long s0, sx, si, sm;                  // source: first segment, and what a step of x, ia, m adds
  long long d0, dx, di, dm;
};

// Segments shorter than this (bytes) are mostly incomplete vectors: they keep the element-wise kernels.
constexpr long long kShiftMinSegment = 64;
// Tensors below this many elements too: bf16 [60, 8001] takes 2.0-3.1 us either way, fp32 [100, 777] 1.2 us element
// by element and 1.6-2.9 in shifted vectors.
constexpr long long kShiftMinElements = 400000;

// How the segments of a transform are dealt out: teams of 1 << team_log2 threads (16 to 256), `chunks` units per segment.
struct ShiftPlan {
  int team_log2;
  unsigned chunks;
};

// Vectors per thread and sources at once: 4 to 8 loads of 16 bytes in flight whatever the transform.
constexpr int kShiftJCopy = 4;
constexpr int shift_kb(int k) { return k <= 2 ? 2 : (k == 3 ? 3 : 4); }
constexpr int shift_j(int kb, int esz) { return (kb == 2 ? 2 : 1) * (esz == 4 ? 2 : 1); }
// CTAs per SM the registers are held to (fp32 [4096, 4097] P(sum) -> S(1) over two shards 50 us with two, 68 with
// three, 76 with four; bf16 [4001, 3333] over eight 84 us with four, 94 with three, 124 with two).
constexpr int shift_ctas(int op, int kb, int esz) { return op == OP_COPY || esz != 4 ? 4 : (kb == 2 ? 2 : 3); }

inline ShiftPlan shift_plan(long long seg_bytes, int J) {
  const long long nv = seg_bytes / 16 > 0 ? seg_bytes / 16 : 1;
  int t = 4;      // at least as many threads as elements beside the whole vectors
  while (t < 8 && (J << t) < nv) ++t;
  return ShiftPlan{t, (unsigned)((nv + ((long long)J << t) - 1) / ((long long)J << t))};
}

template <int ESZ>
struct ShiftElem;
template <>
struct ShiftElem<2> { using type = uint16_t; };
template <>
struct ShiftElem<4> { using type = uint32_t; };
template <>
struct ShiftElem<8> { using type = uint2; };

__device__ __forceinline__ uint4 ld_keep(const void* p) {      // read again by the neighbouring lane: keep it in L1
  uint4 r;
  asm volatile("ld.global.nc.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w) : "l"(p));
  return r;
}

// Bytes sh .. sh + 15 of the 32 bytes (a, b), 0 < sh < 16, sh a multiple of ESZ.
template <int ESZ>
__device__ __forceinline__ uint4 shift_pair(uint4 a, uint4 b, unsigned sh) {
  unsigned w0 = a.x, w1 = a.y, w2 = a.z, w3 = a.w, w4 = b.x, w5 = b.y;
  if (sh & 8) { w0 = a.z; w1 = a.w; w2 = b.x; w3 = b.y; w4 = b.z; w5 = b.w; }
  if (ESZ < 8 && (sh & 4)) { w0 = w1; w1 = w2; w2 = w3; w3 = w4; w4 = w5; }
  if (ESZ < 4 && (sh & 2)) {
    w0 = __funnelshift_r(w0, w1, 16);
    w1 = __funnelshift_r(w1, w2, 16);
    w2 = __funnelshift_r(w2, w3, 16);
    w3 = __funnelshift_r(w3, w4, 16);
  }
  return make_uint4(w0, w1, w2, w3);
}

// One unit of a task (a team of threads and J vectors for each of them).  Sources first, first + stride, ...
// (`count` of them, one for a copy), KB at a time, combined in that order; those of a reduction have one size and
// bases that agree modulo 16.  The result goes to n_dst destinations whose bases agree modulo 16.
template <int ESZ, int OP, int J, int KB>
__device__ __forceinline__ void shift_unit(const SegView& g, ShiftPlan sp, unsigned tile, const char* const* src, const long long* src_bytes,
                                           int first, int stride, int count, char* const* dst, int n_dst) {
  using E = typename ShiftElem<ESZ>::type;
  const unsigned T = 1u << sp.team_log2, tl = threadIdx.x & (T - 1);
  const unsigned unit = tile * (256u >> sp.team_log2) + (threadIdx.x >> sp.team_log2);
  const unsigned seg = sp.chunks == 1 ? unit : unit / sp.chunks, c = unit - seg * sp.chunks;
  if (seg >= g.nseg) return;
  unsigned x = 0, ia = seg, m = 0;
  if (!g.flat) {
    const unsigned q = seg / (unsigned)g.M;
    m = seg - q * (unsigned)g.M;
    x = q / (unsigned)g.la;
    ia = q - x * (unsigned)g.la;
  }
  const long long so = g.s0 + x * g.sx + ia * g.si + m * g.sm, dofs = g.d0 + x * g.dx + ia * g.di + m * g.dm;
  const int to_line = (int)((0ull - (reinterpret_cast<unsigned long long>(dst[0]) + (unsigned long long)dofs)) & 15);
  int head = to_line < g.seg_bytes ? to_line : (int)g.seg_bytes;
  long long nbody = (g.seg_bytes - head) >> 4;
  // where the source stands under a whole vector; a first or last one whose aligned source pair would reach beyond
  // the tensor joins the elements before or after the whole vectors
  const unsigned sh = (unsigned)((reinterpret_cast<unsigned long long>(src[first]) + (unsigned long long)(so + head)) & 15);
  if (sh != 0 && nbody > 0 && so + head - (int)sh < 0) {
    head += 16;
    --nbody;
  }
  if (sh != 0 && nbody > 0 && so + head - (int)sh + nbody * 16 + 16 > src_bytes[first]) --nbody;
  const int tail = (int)(g.seg_bytes - head - nbody * 16);
  const long long v0 = (long long)c * (J * T) + tl;
  // this thread's elements before the first and after the last whole vector (offsets in the segment, -1: none)
  const int eo0 = c == 0 && (int)tl * ESZ < head ? (int)tl * ESZ : -1;
  const long long eo1 = c == sp.chunks - 1 && (int)tl * ESZ < tail ? g.seg_bytes - tail + (long long)tl * ESZ : -1;
  const long long eo[2] = {eo0, eo1};
  bool in[J];
#pragma unroll
  for (int j = 0; j < J; ++j) in[j] = v0 + j * T < nbody;

  SBP_PDL_WAIT();      // the kernel before this one has finished

  if constexpr (OP == OP_COPY) {
    const char* base = src[first] + so;
    E ev[2];
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      ev[e] = E{};
      if (eo[e] >= 0 && SBP_GUARD(base + eo[e], ESZ)) ev[e] = *reinterpret_cast<const E*>(base + eo[e]);
    }
    const char* at = base + head + v0 * 16;
    uint4 val[J];
    if (sh == 0) {
#pragma unroll
      for (int j = 0; j < J; ++j)
        if (in[j] && SBP_GUARD(at + j * T * 16, 16)) val[j] = ld_stream(reinterpret_cast<const uint4*>(at + j * T * 16));
    } else {
      uint4 a[J], b[J];
#pragma unroll
      for (int j = 0; j < J; ++j)
        if (in[j] && SBP_GUARD(at - sh + j * T * 16, 32)) {
          a[j] = ld_keep(at - sh + j * T * 16);
          b[j] = ld_keep(at - sh + j * T * 16 + 16);
        }
#pragma unroll
      for (int j = 0; j < J; ++j)
        if (in[j]) val[j] = shift_pair<ESZ>(a[j], b[j], sh);
    }
    for (int r = 0; r < n_dst; ++r) {
      char* d = dst[r] + dofs;
#pragma unroll
      for (int j = 0; j < J; ++j)
        if (in[j] && SBP_GUARD(d + head + (v0 + j * T) * 16, 16)) st_stream(reinterpret_cast<uint4*>(d + head + (v0 + j * T) * 16), val[j]);
#pragma unroll
      for (int e = 0; e < 2; ++e)
        if (eo[e] >= 0 && SBP_GUARD(d + eo[e], ESZ)) *reinterpret_cast<E*>(d + eo[e]) = ev[e];
    }
  } else {
    using L = typename Lanes<OP, uint4>::type;
    using LE = typename Lanes<OP, E>::type;
    L acc[J];
    const long long off = so + head + v0 * 16;
    for (int r0 = 0; r0 < count; r0 += KB) {
      uint4 a[KB][J], b[KB][J];
#pragma unroll
      for (int i = 0; i < KB; ++i) {
        if (r0 + i >= count) continue;
        const char* at = src[first + (r0 + i) * stride] + off;
#pragma unroll
        for (int j = 0; j < J; ++j) {
          if (!in[j]) continue;
          if (sh == 0) {
            if (SBP_GUARD(at + j * T * 16, 16)) a[i][j] = ld_stream(reinterpret_cast<const uint4*>(at + j * T * 16));
          } else if (SBP_GUARD(at - sh + j * T * 16, 32)) {
            a[i][j] = ld_keep(at - sh + j * T * 16);
            b[i][j] = ld_keep(at - sh + j * T * 16 + 16);
          }
        }
      }
#pragma unroll
      for (int i = 0; i < KB; ++i) {
        if (r0 + i >= count) continue;
#pragma unroll
        for (int j = 0; j < J; ++j) {
          if (!in[j]) continue;
          L t;
          t.load(sh != 0 ? shift_pair<ESZ>(a[i][j], b[i][j], sh) : a[i][j]);
          if (r0 + i == 0) acc[j] = t;
          else combine<OP>(acc[j], t);
        }
      }
    }
    uint4 val[J];
#pragma unroll
    for (int j = 0; j < J; ++j)
      if (in[j]) val[j] = count > 0 ? acc[j].store() : make_uint4(0u, 0u, 0u, 0u);
    for (int r = 0; r < n_dst; ++r) {
      char* d = dst[r] + dofs + head + v0 * 16;
#pragma unroll
      for (int j = 0; j < J; ++j)
        if (in[j] && SBP_GUARD(d + j * T * 16, 16)) st_stream(reinterpret_cast<uint4*>(d + j * T * 16), val[j]);
    }
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      if (eo[e] < 0) continue;
      LE acc;
      for (int r0 = 0; r0 < count; r0 += KB) {
        E xs[KB];
#pragma unroll
        for (int i = 0; i < KB; ++i) {
          xs[i] = E{};
          const char* at = r0 + i < count ? src[first + (r0 + i) * stride] + so + eo[e] : nullptr;
          if (at && SBP_GUARD(at, ESZ)) xs[i] = *reinterpret_cast<const E*>(at);
        }
#pragma unroll
        for (int i = 0; i < KB; ++i) {
          if (r0 + i >= count) continue;
          LE t;
          t.load(xs[i]);
          if (r0 + i == 0) acc = t;
          else combine<OP>(acc, t);
        }
      }
      const E val = count > 0 ? acc.store() : E{};
      for (int r = 0; r < n_dst; ++r) {
        E* d = reinterpret_cast<E*>(dst[r] + dofs + eo[e]);
        if (SBP_GUARD(d, ESZ)) *d = val;
      }
    }
  }
}

}  // namespace sbp
