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
// A reduction adds up the sources' own aligned vectors and shifts the sums (shift_reduce_unit).
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

// How the segments of a transform are dealt out: teams of 1 << team_log2 threads (16 to 256), `chunks` units per segment.
struct ShiftPlan {
  int team_log2;
  unsigned chunks;
};

// Vectors per thread and sources at once: 4 to 8 loads of 16 bytes in flight whatever the transform.  A copy that fills the
// device only once or twice, or that writes each value to eight places, takes one vector a thread: more CTAs, whose stores
// begin earlier (us, four vectors / one: bf16 [60, 8001] S(0) -> B over three 2.6 / 1.8, fp32 [129, 65, 97] over six 6.8 / 4.4,
// over eight 9.1 / 5.5, bf16 [17, 300001] S(1) -> B over eight 18.7 / 13.3; fp32 [4096, 4096] over three 42 / 82, [3000, 3001]
// over six 41 / 45).  elements: of the tensor; n_dst: destinations of each value (0 or 1: one).
inline int shift_copy_j(int esz, int n_dst, long long elements) {
  const long long bytes = elements * esz;
  return n_dst >= 8 || (n_dst >= 4 && bytes < 6400000) || (n_dst > 1 && bytes < 2000000) ? 1 : 4;
}
constexpr int shift_kb(int k) { return k <= 2 ? 2 : (k == 3 ? 3 : 4); }
constexpr int shift_j(int kb) { return kb == 2 ? 4 : 2; }
// When a transform of unaligned data takes this path, from both paths timed on the device over some 700 transforms of 14
// shapes (us, element-wise tiles / this path):
//   copies      segments of 32 elements and more, 64 where several destinations take four vectors a thread: i64 [200001, 33]
//               over three S(1) -> S(0), segments of 11, 38 / 144, [129, 65, 97] over eight S(0) -> S(2), of 12, 8.2 / 20; over
//               three, of 32, 11.3 / 7.5.  Aligned pairs in segments of up to 32 of them fill half a row of a tile and stay
//               there: [20001, 100] over two S(0) -> S(1), bf16 5.5 / 11.2, fp32 5.5 / 11.6
//   reductions  of one placement keep the tiles up to 64 units (what a tile moves per access) a segment, which is one pass of a
//               row: [50, 200, 100] bf16 over two P(sum) -> S(2) 4.7 / 13.6, [60001, 127] 42 / 67, [50, 200, 301] over five 21 / 24,
//               over eight 33 / 45, of 65 units 62 / 50; the same with 120 to 128 units of pairs (fp32 [50, 100, 500] over two 7.5 /
//               11.0).  Three sources, and the last three of seven, the tiles read one after the other, and are slower: fp32
//               [50, 200, 301] over seven 38 / 33, [50, 200, 106] over three 12.3 / 10.6.
//               The eight sources of one placement they read all at once: long segments pay only from 1.2 M elements on
//               ([513, 1025] P(sum) -> B 4.4 / 7.1, [1021, 1537] bf16 11.8 / 9.7), and never in fp32 pairs ([50, 100, 2000] 52 / 66)
//               or 4 bytes and more that go to several destinations ([200001, 33] 65 / 71, bf16 [1429, 4726] 35 / 42)
//               Between different placements the tiles read a few sources at a time as well and only two keep them: bf16
//               [50, 200, 306] over two to three 17 / 19, over eight to seven, of 38, 45 / 40; [4095, 8193] over five to two 320 / 144
//   where the tiles move several elements an access they are as good: up to 1.2 M bf16 or fp32 elements ([60, 8001] bf16
//               P(sum) -> B over three 2.6 / 3.8), and 8 bytes an access are enough for i64 gathers to few replicas unless
//               the rows are short and many ([1021, 1537] over three S(0) -> B 7.4 / 8.1, S(1) -> B 12 / 9.4)
// Below 400 000 elements (500 000 of those eight sources, 800 000 of more than four sources and eight destinations: [513, 1025]
// over eight to nine P(sum) -> B 6.2 / 8.4) a call is all latency: bf16 [60, 8001] takes 2.0-3.1 us either way, fp32 [100, 777]
// 1.2 us element by element and 1.6-2.9 in shifted vectors.
// same: one placement on both sides.
// vbytes: what the tiles would move per access.
inline bool shift_pays(bool copy, bool same, int esz, int vbytes, int k, int n_dst, long long seg_bytes, long long elements) {
  const long long seg = seg_bytes / esz;
  const long long units = seg_bytes / vbytes;
  const bool eight = !copy && same && k == 8, small = elements < 1200000;
  if (vbytes >= 16 || elements < (eight ? 500000 : 400000) || seg < 32) return false;
  if (copy) {
    if (vbytes > esz && units <= 32) return false;
  } else if (!same) {
    if (units <= 64 && k == 2) return false;
  } else {
    const bool one_by_one = k % 4 == 3 && (vbytes == esz ? k == 3 || esz > 2 : units > 32 && units <= 56);
    if ((units <= 64 && !one_by_one) || (vbytes > esz && units > 120 && units <= 128)) return false;
    if (eight && esz == 4 && vbytes == 8) return false;
  }
  if (esz < 8 && vbytes > esz && small) return false;
  if (copy) {
    if (n_dst > 1 && seg < 64 && shift_copy_j(esz, n_dst, elements) > 1) return false;
    if (esz < 8 || n_dst <= 1 || n_dst >= 8) return true;
    return n_dst >= 4 ? seg < (1 << 17) || elements < 800000 : seg < 2048 || (seg < (1 << 17) && elements >= 2000000);
  }
  if (!eight) return k <= 4 || n_dst < 8 || elements >= 800000;
  return seg < 4096 || (!small && !(vbytes >= 4 && n_dst > 1));
}

// CTAs per SM the registers are held to (P(sum) -> S(1), us with 2 / 3 / 4: bf16 [1429, 4727] over two shards, four
// vectors a thread, 13.2 / 11.9, with two vectors and four CTAs 12.0; bf16 [1249, 6988] over three 19.4 / 19.7 / 17.3; bf16
// [7894, 4206] over eight 169 / 136 / 128).
constexpr int shift_ctas(int op, int kb) { return op != OP_COPY && kb == 2 ? 3 : 4; }

// How the segments of a copy are dealt out.
inline ShiftPlan shift_plan_copy(long long seg_bytes, int J) {
  const long long nv = seg_bytes / 16 > 0 ? seg_bytes / 16 : 1;
  int t = 4;      // at least as many threads as elements beside the whole vectors
  while (t < 8 && ((long long)J << t) < nv) ++t;
  return ShiftPlan{t, (unsigned)((nv + ((long long)J << t) - 1) / ((long long)J << t))};
}

// The same for a reduction: the team whose lanes are busiest on segments of this length, the largest of equals.
inline ShiftPlan shift_plan_reduce(long long seg_bytes, int J) {
  const long long nv = seg_bytes / 16 + 2;      // destination vectors, incomplete ones included
  ShiftPlan best{4, 1};
  double best_use = 0.0;
  for (int t = 4; t <= 8; ++t) {
    const long long T = 1 << t, W = T < 32 ? T : 32, per = (long long)J * (T / W) * (W - 1), chunks = (nv + per - 1) / per;
    const double use = (double)nv / (double)(chunks * J * T);
    if (use >= best_use) {
      best_use = use;
      best = ShiftPlan{t, (unsigned)chunks};
    }
  }
  return best;
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

// One unit of a copy (a team of threads and J vectors for each of them) to n_dst destinations whose bases agree modulo 16.
template <int ESZ, int J>
__device__ __forceinline__ void shift_copy_unit(const SegView& g, ShiftPlan sp, unsigned tile, const char* src, long long src_bytes,
                                                char* const* dst, int n_dst) {
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
  const unsigned sh = (unsigned)((reinterpret_cast<unsigned long long>(src) + (unsigned long long)(so + head)) & 15);
  if (sh != 0 && nbody > 0 && so + head - (int)sh < 0) {
    head += 16;
    --nbody;
  }
  if (sh != 0 && nbody > 0 && so + head - (int)sh + nbody * 16 + 16 > src_bytes) --nbody;
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

  const char* base = src + so;
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
}

// Bytes lo .. hi - 1 of the 16 at p, the others zero.
template <int ESZ>
__device__ __forceinline__ uint4 load_part(const char* p, int lo, int hi) {
  using E = typename ShiftElem<ESZ>::type;
  unsigned long long w[2] = {0ull, 0ull};
#pragma unroll 1
  for (int e = lo; e < hi; e += ESZ) {
    if (!SBP_GUARD(p + e, ESZ)) continue;
    const E x = *reinterpret_cast<const E*>(p + e);
    unsigned long long v;
    if constexpr (ESZ == 8) v = ((unsigned long long)x.y << 32) | x.x;
    else v = x;
    if (e < 8) w[0] |= v << (8 * e);
    else w[1] |= v << (8 * (e - 8));
  }
  return make_uint4((unsigned)w[0], (unsigned)(w[0] >> 32), (unsigned)w[1], (unsigned)(w[1] >> 32));
}

// One vector of a unit whose sources reach beyond their tensors, which hold `bytes` bytes: 16 at `at`.
template <int ESZ, int OP>
__device__ __noinline__ uint4 shift_part(const char* const* src, int first, int stride, int count, long long at, long long bytes) {
  const int lo = at < 0 ? (int)-at : 0, hi = at + 16 <= bytes ? 16 : (int)(bytes - at);
  typename Lanes<OP, uint4>::type acc, t;
#pragma unroll 1
  for (int r = 0; r < count; ++r) {
    t.load(load_part<ESZ>(src[first + r * stride] + at, lo, hi));
    if (r == 0) acc = t;
    else combine<OP>(acc, t);
  }
  return count > 0 ? acc.store() : make_uint4(0u, 0u, 0u, 0u);
}

template <int ESZ>
__device__ __noinline__ void store_part(char* p, uint4 v, int lo, int hi) {
  using E = typename ShiftElem<ESZ>::type;
  const unsigned long long w[2] = {((unsigned long long)v.y << 32) | v.x, ((unsigned long long)v.w << 32) | v.z};
#pragma unroll 1
  for (int e = lo; e < hi; e += ESZ) {
    const unsigned long long x = e < 8 ? w[0] >> (8 * e) : w[1] >> (8 * (e - 8));
    if (!SBP_GUARD(p + e, ESZ)) continue;
    if constexpr (ESZ == 8) *reinterpret_cast<E*>(p + e) = make_uint2((unsigned)x, (unsigned)(x >> 32));
    else *reinterpret_cast<E*>(p + e) = (E)x;
  }
}

// One unit of a reduction (a team of threads and J vectors for each of them).  Sources first, first + stride, ...
// (`count` of them) have one size and bases that agree modulo 16, and are combined KB at a time in that order, as aligned
// vectors of the SOURCES: each is loaded once, by one lane.  The sums are shifted, not the sources: a lane gets the vector
// after its own from the next lane, so of W lanes W - 1 store.  Incomplete vectors at a segment's ends are summed like the
// others and stored element by element.  The result goes to n_dst destinations whose bases agree modulo 16.
template <int ESZ, int OP, int J, int KB>
__device__ __forceinline__ void shift_reduce_unit(const SegView& g, ShiftPlan sp, unsigned tile, const char* const* src, const long long* src_bytes,
                                           int first, int stride, int count, char* const* dst, int n_dst) {
  const unsigned T = 1u << sp.team_log2, tl = threadIdx.x & (T - 1), W = T < 32 ? T : 32, lw = tl & (W - 1);
  const unsigned unit = tile * (256u >> sp.team_log2) + (threadIdx.x >> sp.team_log2);
  unsigned seg = sp.chunks == 1 ? unit : unit / sp.chunks;
  const unsigned c = unit - seg * sp.chunks;
  const bool live = seg < g.nseg;              // a warp may hold teams on both sides of the end
  if (!live) seg = 0;
  unsigned x = 0, ia = seg, m = 0;
  if (!g.flat) {
    const unsigned q = seg / (unsigned)g.M;
    m = seg - q * (unsigned)g.M;
    x = q / (unsigned)g.la;
    ia = q - x * (unsigned)g.la;
  }
  const long long so = g.s0 + x * g.sx + ia * g.si + m * g.sm, dofs = g.d0 + x * g.dx + ia * g.di + m * g.dm;
  // the segment begins `lead` bytes into the first aligned vector of the destination; the source bytes under that
  // vector begin `sh` into an aligned vector of the source, `from` bytes from the source's base
  const int lead = (int)((reinterpret_cast<unsigned long long>(dst[0]) + (unsigned long long)dofs) & 15);
  const unsigned sh = (unsigned)((reinterpret_cast<unsigned long long>(src[first]) + (unsigned long long)(so - lead)) & 15);
  const long long from = so - lead - sh, end = lead + g.seg_bytes, bytes = src_bytes[first];
  const long long nv = live ? (end + 15) >> 4 : 0;
  const unsigned per_sub = W - 1, subs = T / W;
  const long long v0 = (long long)(c * J * subs + tl / W) * per_sub + lw;      // and subs * per_sub further for each j
  const int step = (int)(subs * per_sub);
  const long long at0 = from + v0 * 16;        // where source vector 0's bytes begin
  bool in[J], part[J];
#pragma unroll
  for (int j = 0; j < J; ++j) {
    const long long at = at0 + (long long)j * step * 16;
    const bool wanted = v0 + (long long)j * step < nv + (sh != 0 ? 1 : 0) && at < bytes && at + 16 > 0;
    in[j] = wanted && at >= 0 && at + 16 <= bytes;
    part[j] = wanted && !in[j];
  }

  SBP_PDL_WAIT();      // the kernel before this one has finished

  uint4 val[J];
  using L = typename Lanes<OP, uint4>::type;
  L acc[J];
  for (int r0 = 0; r0 < count; r0 += KB) {
    uint4 a[KB][J];
#pragma unroll
    for (int i = 0; i < KB; ++i) {
      if (r0 + i >= count) continue;
      const char* base = src[first + (r0 + i) * stride] + at0;
#pragma unroll
      for (int j = 0; j < J; ++j) {
        a[i][j] = make_uint4(0u, 0u, 0u, 0u);
        if (in[j] && SBP_GUARD(base + j * step * 16, 16)) a[i][j] = ld_keep(base + j * step * 16);
      }
    }
#pragma unroll
    for (int i = 0; i < KB; ++i) {
      if (r0 + i >= count) continue;
#pragma unroll
      for (int j = 0; j < J; ++j) {
        L t;
        t.load(a[i][j]);
        if (r0 + i == 0) acc[j] = t;
        else combine<OP>(acc[j], t);
      }
    }
  }
#pragma unroll
  for (int j = 0; j < J; ++j) val[j] = count > 0 ? acc[j].store() : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
  for (int j = 0; j < J; ++j)
    if (part[j]) val[j] = shift_part<ESZ, OP>(src, first, stride, count, at0 + (long long)j * step * 16, bytes);
#pragma unroll
  for (int j = 0; j < J; ++j) {
    uint4 next;                                // the vector after this lane's
    next.x = __shfl_down_sync(0xffffffffu, val[j].x, 1, W);
    next.y = __shfl_down_sync(0xffffffffu, val[j].y, 1, W);
    next.z = __shfl_down_sync(0xffffffffu, val[j].z, 1, W);
    next.w = __shfl_down_sync(0xffffffffu, val[j].w, 1, W);
    if (sh != 0) val[j] = shift_pair<ESZ>(val[j], next, sh);
  }
  for (int r = 0; r < n_dst; ++r) {
    char* d = dst[r] + dofs - lead;
#pragma unroll
    for (int j = 0; j < J; ++j) {
      const long long v = v0 + (long long)j * step, o = v * 16;
      if (v >= nv || lw == per_sub) continue;
      if (o >= lead && o + 16 <= end) {
        if (SBP_GUARD(d + o, 16)) st_stream(reinterpret_cast<uint4*>(d + o), val[j]);
      } else {
        store_part<ESZ>(d + o, val[j], o < lead ? (int)(lead - o) : 0, o + 16 <= end ? 16 : (int)(end - o));
      }
    }
  }
}

}  // namespace sbp
