// Class-split softmax cross entropy (Section 6.3: classifier weight S(1) => logits S(1)).
//
// The paper's plan has two reductions inside the softmax, max and sum, each done locally per
// shard first and then across shards.  Here:
//   partial kernel   one CTA per (row, shard, column chunk) streams its piece of the logits
//                    once and leaves a local max m_p, a local exp-sum s_p = sum exp(z - m_p)
//                    and the label's logit t_p (0 when the label lies elsewhere);
//   (or, with many rows, one kernel whose teams of threads finish a row each: xent_rows_kernel)
//   combine kernel   per row, over the pieces p (one warp per row: the pieces of a lane in
//                    ascending order, then the lanes by a butterfly):
//                    m = max_p m_p            (the P(max) -> B boxing of the local maxima)
//                    S = sum_p s_p exp(m_p-m) (the P(sum) -> B boxing, after rescaling)
//                    loss = log S + m - sum_p t_p.
// The local sums are taken relative to the local max (one pass over the logits); rescaling
// by exp(m_p - m) in the combine gives the same S as the literal max-then-sum order.
// Reductions inside a CTA use a fixed tree (thread-serial, warp butterfly, warps in order),
// so results are reproducible for a given shape.
#include <cuda_bf16.h>

#include <algorithm>
#include <cfloat>
#include <cmath>

#include <mutex>

#include "bounds_check.h"
#include "sbp_internal.h"

namespace sbp {

constexpr int kThreads = 256;
constexpr int kLoadsPerThread = 4;    // vectors per thread per chunk
constexpr int kMaxChunksPerCta = 16;  // a CTA walks up to this many chunks of one row

struct XentParams {
  const char* logits[SBP_MAX_K];
  const long long* labels;
  float* part_m;   // [parts][rows]
  float* part_s;
  float* part_t;
  long long rows, classes;
  long long pitch[SBP_MAX_K];   // elements between consecutive rows of shard r's logits
  int k, nsplit;
  long long span;    // elements per CTA
  long long keep_from;          // row, or CTA of the partial kernel, from which on what is read stays in L2
};

struct XentCombineParams {
  const float* part_m;
  const float* part_s;
  const float* part_t;
  float* loss[SBP_MAX_K];
  float* row_max[SBP_MAX_K];
  float* row_sum[SBP_MAX_K];
  int n_loss, n_max, n_sum;
  long long rows;
  int parts;
};

constexpr float kLog2e = 1.4426950408889634f;

__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// (m, s) <- merge with (m2, s2), where s is a sum of exp(z - m).  A piece with no elements
// carries (m = -inf, s = 0) and must not produce inf - inf.
__device__ __forceinline__ void merge(float& m, float& s, float m2, float s2) {
  const float mm = fmaxf(m, m2);
  const float a = (m == -INFINITY) ? 0.f : s * ex2((m - mm) * kLog2e);
  const float b = (m2 == -INFINITY) ? 0.f : s2 * ex2((m2 - mm) * kLog2e);
  s = a + b;
  m = mm;
}

// Loss, max and sum of a finished row, to every replica.
__device__ __forceinline__ void write_row(const XentCombineParams& p, long long row, float m, float S, float zy) {
  const float loss = logf(S) + (m - zy);       // in this order: the sum of a large m and the logarithm would be rounded to m's last place
  for (int j = 0; j < p.n_loss; ++j)
    if (SBP_GUARD(p.loss[j] + row, 4)) p.loss[j][row] = loss;
  for (int j = 0; j < p.n_max; ++j)
    if (SBP_GUARD(p.row_max[j] + row, 4)) p.row_max[j][row] = m;
  for (int j = 0; j < p.n_sum; ++j)
    if (SBP_GUARD(p.row_sum[j] + row, 4)) p.row_sum[j][row] = S;
}

// The (m, s) pairs of a warp's lanes into one, the same in all of them: the maximum first, then every sum rescaled once.
// (Merging pair by pair rescales a sum at every level, and the unit's exponentials are 5e-8 low on the average.)
__device__ __forceinline__ void merge_warp(float& m, float& s) {
  float top = m;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, off));
  s = m == -INFINITY ? 0.f : s * ex2((m - top) * kLog2e);
  m = top;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
}

// n pairs into one, in their order.
__device__ __forceinline__ void merge_all(const float* ms, const float* ss, int n, float& m, float& s) {
  m = ms[0];
  for (int w = 1; w < n; ++w) m = fmaxf(m, ms[w]);
  s = 0.f;
  for (int w = 0; w < n; ++w) s += ms[w] == -INFINITY ? 0.f : ss[w] * ex2((ms[w] - m) * kLog2e);
}

// ---- chunk policies: how one thread of a team loads, maxes and exp-sums its kLoadsPerThread vectors of 16 bytes.  z
// points at the first vector (16-byte aligned), nv counts the vectors there are.

// The logits are read twice, by the forward pass and from their end by the backward.  What the forward pass reads last, as
// much as stays in L2 beside the gradient, it reads with the usual priority, the rest as first to go; the backward's reads
// and its results are the first to go as well.  (us, forward and backward, all with the usual priority / so: fp32
// [256, 100003] over four 57.7 / 54.7, [128, 100003] 30.5 / 29.0, [256, 200000] 106.5 / 102.9, [4000, 8000] 72.7 / 71.1;
// bf16 [512, 100000] 65.8 / 63.1.  The part to keep, MB, [256, 100003]: 40 55.4, 50 54.8, 60 54.7, 70 55.1, 100 55.4; the
// priority to keep longest instead of the usual one 0.1 to 1 us slower.  Passes over the same logits; on logits just made, whose
// producer has left a part of them in L2, the two are level.)
constexpr long long kKeepNum = 7, kKeepDen = 16;      // of the device's L2 (126 MB: 55)
__device__ __forceinline__ unsigned long long l2_usual() {
  unsigned long long p;
  asm("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(p));
  return p;
}
// (made where it is used: kept in a register across the backward's loop it cost a CTA an SM, and more than it gave)
__device__ __forceinline__ unsigned long long l2_first() {
  unsigned long long p;
  asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
  return p;
}

__device__ __forceinline__ uint4 ld_logits(const void* p, unsigned long long priority) {
  uint4 r;
  asm volatile("ld.global.nc.L1::no_allocate.L2::cache_hint.v4.u32 {%0,%1,%2,%3}, [%4], %5;"
               : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w)
               : "l"(p), "l"(priority));
  return r;
}

// Two numbers in a register pair; two exponentials of (z - m) log2e, added to two sums.  The difference is exact in m, and in
// pairs it and the product cost no more than one multiply-add an element did.
__device__ __forceinline__ unsigned long long pair(float x, float y) {
  unsigned long long v;
  asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(x), "f"(y));
  return v;
}
__device__ __forceinline__ void expsum_pair(unsigned long long z, unsigned long long neg_m, float& s0, float& s1) {
  asm("add.rn.f32x2 %0, %0, %1;" : "+l"(z) : "l"(neg_m));
  asm("mul.rn.f32x2 %0, %0, %1;" : "+l"(z) : "l"(pair(kLog2e, kLog2e)));
  s0 += ex2(__uint_as_float((unsigned)z));
  s1 += ex2(__uint_as_float((unsigned)(z >> 32)));
}

// bf16, 8 elements per load; max on packed pairs, exp in fp32.
struct ChunkBF16 {
  using T = __nv_bfloat16;
  static constexpr int VEC = 8;
  uint4 raw[kLoadsPerThread];
  __device__ __forceinline__ void load(const T* z, long long nv, int tid, int team, unsigned long long priority) {
#pragma unroll
    for (int u = 0; u < kLoadsPerThread; ++u) {
      const long long v = (long long)u * team + tid;
      if (v < nv && SBP_GUARD(z + v * VEC, 16)) raw[u] = ld_logits(z + v * VEC, priority);
      else raw[u] = make_uint4(0xFF80FF80u, 0xFF80FF80u, 0xFF80FF80u, 0xFF80FF80u);   // -inf, -inf
    }
  }
  __device__ __forceinline__ float max() const {
    __nv_bfloat162 mx = *reinterpret_cast<const __nv_bfloat162*>(&raw[0].x);
#pragma unroll
    for (int u = 0; u < kLoadsPerThread; ++u) {
      const uint32_t* w = reinterpret_cast<const uint32_t*>(&raw[u]);
#pragma unroll
      for (int i = 0; i < 4; ++i) mx = __hmax2(mx, *reinterpret_cast<const __nv_bfloat162*>(&w[i]));
    }
    return fmaxf(__low2float(mx), __high2float(mx));
  }
  // sum of 2^((z - m) log2e) over the thread's elements
  __device__ __forceinline__ float expsum(float m) const {
    const unsigned long long neg = pair(-m, -m);
    float s0 = 0.f, s1 = 0.f;
#pragma unroll
    for (int u = 0; u < kLoadsPerThread; ++u) {
      const uint32_t* w = reinterpret_cast<const uint32_t*>(&raw[u]);
#pragma unroll
      for (int i = 0; i < 4; ++i) expsum_pair(pair(__uint_as_float(w[i] << 16), __uint_as_float(w[i] & 0xffff0000u)), neg, s0, s1);
    }
    return s0 + s1;
  }
};

// fp32, 4 elements per load.
struct ChunkF32 {
  using T = float;
  static constexpr int VEC = 4;
  uint4 raw[kLoadsPerThread];
  __device__ __forceinline__ void load(const T* z, long long nv, int tid, int team, unsigned long long priority) {
#pragma unroll
    for (int u = 0; u < kLoadsPerThread; ++u) {
      const long long v = (long long)u * team + tid;
      if (v < nv && SBP_GUARD(z + v * VEC, 16)) raw[u] = ld_logits(z + v * VEC, priority);
      else raw[u] = make_uint4(0xFF800000u, 0xFF800000u, 0xFF800000u, 0xFF800000u);   // -inf
    }
  }
  __device__ __forceinline__ float max() const {
    float m = -INFINITY;
#pragma unroll
    for (int u = 0; u < kLoadsPerThread; ++u) {
      const float* f = reinterpret_cast<const float*>(&raw[u]);
#pragma unroll
      for (int i = 0; i < 4; ++i) m = fmaxf(m, f[i]);
    }
    return m;
  }
  __device__ __forceinline__ float expsum(float m) const {
    const unsigned long long neg = pair(-m, -m);
    float s0 = 0.f, s1 = 0.f;
#pragma unroll
    for (int u = 0; u < kLoadsPerThread; ++u) {
      const float* f = reinterpret_cast<const float*>(&raw[u]);
      expsum_pair(pair(f[0], f[1]), neg, s0, s1);
      expsum_pair(pair(f[2], f[3]), neg, s0, s1);
    }
    return s0 + s1;
  }
};

// Elements before the first 16-byte boundary at or after z, at most n.
template <typename T>
__device__ __forceinline__ int to_boundary(const T* z, long long n) {
  const int h = (int)((0ull - reinterpret_cast<unsigned long long>(z)) & 15) / (int)sizeof(T);
  return h < n ? h : (int)n;
}

// A team's pass over the n > 0 logits at z: the running (m, s) of each of its threads, s a sum of exp(z - m).
// A row starts wherever the class count and the pitch put it: up to 15 bytes on either end of the span are taken
// element by element, one element a thread, and what lies between as aligned vectors; the loads of the next chunk
// are issued before the current one is reduced.  (Unaligned rows element by element throughout: fp32 [256, 100003]
// over four shards 33 us, backward 76; as here 25 and 35: 0.62 and 0.89 of the copy bandwidth.)
// An exponential is 2^((z - m) log2e): exact in the maximum, finite for every finite z.  (As 2^(z log2e - c), c = m log2e rounded,
// with what the rounding leaves taken out of the sum to first order, rows wholly at -1e8 had a negative sum.)
// What is carried from chunk to chunk is rescaled by the difference of the maxima: exactly 1 while the maximum stands.
template <typename Chunk>
__device__ __forceinline__ void walk_span(const typename Chunk::T* z, long long n, int tid, int team, unsigned long long priority, float& m, float& s) {
  using T = typename Chunk::T;
  constexpr int VEC = Chunk::VEC;
  const int head = to_boundary(z, n);
  const long long nv = (n - head) / VEC;
  const int tail = (int)(n - head - nv * VEC);
  const T* zv = z + head;
  const long long step = (long long)team * kLoadsPerThread;     // vectors per chunk
  Chunk cur, nxt;
  if (nv > 0) cur.load(zv, nv, tid, team, priority);
  const T* lone = tid < head ? z + tid : (tid >= 16 && tid - 16 < tail ? zv + nv * VEC + (tid - 16) : nullptr);
  if (lone && SBP_GUARD(lone, sizeof(T))) {
    const float x = static_cast<float>(*lone);
    if (x != -INFINITY) merge(m, s, x, 1.f);
  }
  for (long long off = 0; off < nv; off += step) {
    const bool more = off + step < nv;
    if (more) nxt.load(zv + (off + step) * VEC, nv - off - step, tid, team, priority);
    const float cm = cur.max();
    if (cm != -INFINITY) {                                      // not the threads of a short row that have nothing
      const float mm = fmaxf(m, cm);
      s = s * ex2((m - mm) * kLog2e) + cur.expsum(mm);          // s is 0 as long as m is -inf
      m = mm;
    }
    if (more) cur = nxt;
  }
}

// Many rows: a team of 1 << team_log2 threads takes a whole row, shard after shard, and finishes it -- no partials,
// no second kernel.  Taken from five rows an SM on (740), with the team that spreads the rows over the device
// once.  (us, partial + combine kernels / this: fp32 [4096, 1003] over two shards 24 / 8.5, bf16 [1000, 30000] over
// four 39 / 24.)  The team grows with the row, so that a thread adds up no more elements than in the partial kernel;
// rows that take more than 128 threads so are left to that kernel, which is as fast for them or faster (fp32 [2000,
// 134217] over four 254 us with teams of 64, 168 there; [3000, 30000] over two 73 either way; bf16 [2000, 100000] over
// two 92 with teams of 256, 75 there).  Relative error of the row sums at any team 0.6e-7 to 0.9e-7 rms, 3.5e-7 at most.
// log2 of the team for this many rows and classes in vectors of `vec` elements; 0: the partial kernel
static int team_for(long long rows, long long classes, int vec) {
  const long long least = 5LL * device_sms();
  if (rows < least) return 0;
  int t = rows < 2 * least ? 7 : (rows < 4 * least ? 6 : 5);
  const long long most = (long long)kMaxChunksPerCta * kLoadsPerThread * vec;
  while (t <= 7 && (classes >> t) > most) ++t;
  return t <= 7 ? t : 0;
}

template <typename Chunk>
__global__ void __launch_bounds__(kThreads) xent_rows_kernel(const __grid_constant__ XentParams p, const __grid_constant__ XentCombineParams c,
                                                            int team_log2) {
  using T = typename Chunk::T;
  const int team = 1 << team_log2, tl = threadIdx.x & (team - 1);
  const long long row = (long long)blockIdx.x * (kThreads >> team_log2) + (threadIdx.x >> team_log2);
  SBP_PDL_RELEASE();
  SBP_PDL_WAIT();
  float m = -INFINITY, s = 0.f, t = 0.f;
  if (row < p.rows) {
    const long long y = SBP_GUARD(p.labels + row, 8) ? p.labels[row] : -1;
    for (int r = 0; r < p.k; ++r) {
      long long c_start, c_len;
      split_range(p.classes, p.k, r, (int64_t*)&c_start, (int64_t*)&c_len);
      const T* z = reinterpret_cast<const T*>(p.logits[r]) + row * p.pitch[r];
      if (c_len > 0) walk_span<Chunk>(z, c_len, tl, team, row >= p.keep_from ? l2_usual() : l2_first(), m, s);
      if (tl == 0 && y >= c_start && y < c_start + c_len && SBP_GUARD(z + (y - c_start), sizeof(T))) t = static_cast<float>(z[y - c_start]);
    }
  }
  merge_warp(m, s);
  if (team > 32) {
    __shared__ float sm[kThreads / 32], ss[kThreads / 32];
    const int w0 = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) {
      sm[w0] = m;
      ss[w0] = s;
    }
    __syncthreads();
    if (tl == 0) merge_all(sm + w0, ss + w0, team / 32, m, s);
  }
  if (tl == 0 && row < p.rows) write_row(c, row, m, s, t);
}

// One CTA per (row, shard, column span).  Each thread keeps a running (m, s) over the chunks
// of its span -- the loads of the next chunk are issued before the current one is reduced --
// and the CTA merges its threads' pairs in a fixed order.
template <typename Chunk, int THREADS>
__global__ void __launch_bounds__(THREADS) xent_partial_kernel(const __grid_constant__ XentParams p) {
  using T = typename Chunk::T;
  const long long row = blockIdx.x;
  const int split = blockIdx.y;
  const int shard = blockIdx.z;
  long long c_start, c_len;
  split_range(p.classes, p.k, shard, (int64_t*)&c_start, (int64_t*)&c_len);
  const long long c0 = (long long)split * p.span;
  long long n = c_len - c0;       // elements of this CTA's span (may be <= 0 on uneven shards)
  if (n > p.span) n = p.span;
  const int part = shard * p.nsplit + split;
  const T* z = reinterpret_cast<const T*>(p.logits[shard]) + row * p.pitch[shard] + c0;
  const int tid = threadIdx.x;
  // The kernel that combines the partials may be set up while this one runs; it waits for
  // this grid to finish before it reads anything.
  SBP_PDL_RELEASE();
  SBP_PDL_WAIT();

  float m = -INFINITY, s = 0.f;
  const long long cta = blockIdx.x + (long long)gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z);
  if (n > 0) walk_span<Chunk>(z, n, tid, THREADS, cta >= p.keep_from ? l2_usual() : l2_first(), m, s);

  merge_warp(m, s);
  __shared__ float sm[THREADS / 32], ss[THREADS / 32];
  if ((tid & 31) == 0) {
    sm[tid >> 5] = m;
    ss[tid >> 5] = s;
  }
  __syncthreads();
  if (tid == 0) {
    float mm, sv;
    merge_all(sm, ss, THREADS / 32, mm, sv);
    float t = 0.f;
    const long long y = (SBP_GUARD(p.labels + row, 8) ? p.labels[row] : -1) - c_start - c0;
    if (y >= 0 && y < n && SBP_GUARD(z + y, sizeof(T))) t = static_cast<float>(z[y]);
    const long long at = (long long)part * p.rows + row;
    if (SBP_GUARD(p.part_m + at, 4)) p.part_m[at] = mm;
    if (SBP_GUARD(p.part_s + at, 4)) p.part_s[at] = sv;
    if (SBP_GUARD(p.part_t + at, 4)) p.part_t[at] = t;
  }
}

// Short rows get no more threads than there are vectors (fp32 [700, 100] over four 11.0 us with 256 threads, 6.1 with 32).
template <typename Chunk>
static void launch_partial(const XentParams& p, dim3 grid, long long widest, cudaStream_t st) {
  const long long vectors = (widest + Chunk::VEC - 1) / Chunk::VEC;
  if (vectors <= 32) launch_dependent(xent_partial_kernel<Chunk, 32>, grid, dim3(32), 0, st, p);
  else if (vectors <= 64) launch_dependent(xent_partial_kernel<Chunk, 64>, grid, dim3(64), 0, st, p);
  else if (vectors <= 128) launch_dependent(xent_partial_kernel<Chunk, 128>, grid, dim3(128), 0, st, p);
  else launch_dependent(xent_partial_kernel<Chunk, kThreads>, grid, dim3(kThreads), 0, st, p);
}

// One warp per row: lane j takes the parts j, j + 32, ... in ascending order, then the lanes
// are merged by a butterfly -- a fixed tree for a given number of parts.
constexpr int kCombineThreads = 256;

__global__ void __launch_bounds__(kCombineThreads) xent_combine_kernel(const __grid_constant__ XentCombineParams p) {
  // When launched as the programmatic dependent of the kernel that writes the partials, wait
  // here until that grid has finished and its writes are visible (a no-op otherwise).
  SBP_PDL_RELEASE();
  SBP_PDL_WAIT();
  const long long row = (long long)blockIdx.x * (kCombineThreads / 32) + (threadIdx.x >> 5);
  if (row >= p.rows) return;
  const int lane = threadIdx.x & 31;
  float m = -INFINITY, S = 0.f, zy = 0.f;
  for (int q = lane; q < p.parts; q += 32) {
    const long long at = (long long)q * p.rows + row;
    if (!SBP_GUARD(p.part_m + at, 4) || !SBP_GUARD(p.part_s + at, 4) || !SBP_GUARD(p.part_t + at, 4)) continue;
    merge(m, S, p.part_m[at], p.part_s[at]);
    zy += p.part_t[at];
  }
  merge_warp(m, S);
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) zy += __shfl_xor_sync(0xffffffffu, zy, off);
  if (lane == 0) write_row(p, row, m, S, zy);
}

// Elements of one CTA's column span, and how many spans cover the widest shard, for loads of `vec` elements.
static void tiling_for(const sbp_tensor* logits, int vec, long long* span, int* nsplit) {
  const int k = placement_k(logits);
  const long long c_max = (logits->shape[1] + k - 1) / k;
  const long long chunk = (long long)kThreads * kLoadsPerThread * vec;
  long long chunks = (c_max + chunk - 1) / chunk;
  if (chunks < 1) chunks = 1;
  const long long per_cta = chunks < kMaxChunksPerCta ? chunks : kMaxChunksPerCta;
  *span = chunk * per_cta;
  *nsplit = (int)((chunks + per_cta - 1) / per_cta);
}

static int nsplit_for(const sbp_tensor* logits, int vec) {
  long long span;
  int ns;
  tiling_for(logits, vec, &span, &ns);
  return ns;
}

static int vec_of(const sbp_tensor* logits) { return 16 / elem_size(logits->dtype); }

// The spans a call uses: those of tiling_for, or shorter ones (down to one chunk) when the rows alone do not fill the
// device four CTAs deep and the scratch has room for the partials.
static void tiling_in(const sbp_tensor* logits, size_t ws_bytes, long long* span, int* nsplit) {
  tiling_for(logits, vec_of(logits), span, nsplit);
  const int k = placement_k(logits);
  const long long rows = logits->shape[0], c_max = (logits->shape[1] + k - 1) / k;
  const long long chunk = (long long)kThreads * kLoadsPerThread * vec_of(logits);
  // (never more scratch than the size query answers or the built-in array holds, so that both entry points cut alike)
  const size_t most = std::min({ws_bytes, sbp_softmax_xent_workspace_bytes(logits), (size_t)SBP_SOFTMAX_XENT_STATIC_SCRATCH_BYTES});
  const long long room = (long long)(most / (3 * sizeof(float) * (size_t)k * (size_t)rows));
  while (*nsplit * rows * k < 4LL * device_sms() && *span > chunk) {
    const long long sp = (*span / chunk + 1) / 2 * chunk, ns = (c_max + sp - 1) / sp;
    if (ns > room) break;
    *span = sp;
    *nsplit = (int)ns;
  }
}

static int dedup(float** out, const sbp_tensor* t, int k) {
  int n = 0;
  for (int r = 0; r < k; ++r) {
    float* ptr = static_cast<float*>(t->local[r]);
    bool seen = false;
    for (int q = 0; q < n; ++q) seen = seen || out[q] == ptr;
    if (!seen) out[n++] = ptr;
  }
  return n;
}

static sbp_status check_row_vector(const sbp_tensor* t, const char* name, long long rows, int k) {
  sbp_status st = check_tensor(t, name, true);
  if (st != SBP_OK) return st;
  if (t->ndim != 1 || t->shape[0] != rows) return fail(SBP_ERR_SHAPE, "%s must be [rows]", name);
  if (t->dtype != SBP_F32) return fail(SBP_ERR_DTYPE, "%s must be F32", name);
  if (t->sbp[0].kind != SBP_BROADCAST) return fail(SBP_ERR_SIGNATURE, "%s must be B", name);
  if (placement_k(t) != k) return fail(SBP_ERR_INVALID_ARG, "%s differs in k", name);
  return SBP_OK;
}

// ---- second-level reduction for many partials per row (used after the fused classifier
// kernel, which leaves one partial per 128 classes).  Thread (tx, ty) of a 32 x 8 CTA owns row
// 32 bx + tx and walks the parts of slice `by` with stride 8 in ascending order; the 8 lanes
// of a row are then merged in lane order.  Output: one partial per (slice, row).
struct XentReduceParams {
  const float* in_m;
  const float* in_s;
  const float* in_t;
  float* out_m;
  float* out_s;
  float* out_t;
  long long rows;
  int parts, per_slice;
};

__global__ void __launch_bounds__(256) xent_reduce_parts_kernel(const __grid_constant__ XentReduceParams p) {
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const long long row = (long long)blockIdx.x * 32 + tx;
  const int lo = blockIdx.y * p.per_slice;
  const int hi = min(p.parts, lo + p.per_slice);
  // The partials come from the kernel just before this one in the stream; when launched as its
  // programmatic dependent, wait for it here (a no-op otherwise), and let the combine kernel
  // that follows be set up meanwhile.
  SBP_PDL_RELEASE();
  SBP_PDL_WAIT();
  float m = -INFINITY, s = 0.f, t = 0.f;
  if (row < p.rows) {
    // four parts (stride 8) are loaded before they are merged, in ascending order
    for (int q = lo + ty; q < hi; q += 32) {
      float pm[4], ps[4], pt[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int qq = q + 8 * j;
        const long long at = (long long)(qq < hi ? qq : q) * p.rows + row;
        const bool in_ok = SBP_GUARD(p.in_m + at, 4) && SBP_GUARD(p.in_s + at, 4) && SBP_GUARD(p.in_t + at, 4);
        pm[j] = in_ok ? p.in_m[at] : -INFINITY;
        ps[j] = in_ok ? p.in_s[at] : 0.f;
        pt[j] = in_ok ? p.in_t[at] : 0.f;
      }
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (q + 8 * j < hi) {
          merge(m, s, pm[j], ps[j]);
          t += pt[j];
        }
    }
  }
  __shared__ float sm[8][33], ss[8][33], st[8][33];
  sm[ty][tx] = m;
  ss[ty][tx] = s;
  st[ty][tx] = t;
  __syncthreads();
  if (ty == 0 && row < p.rows) {
#pragma unroll
    for (int j = 1; j < 8; ++j) {
      merge(m, s, sm[j][tx], ss[j][tx]);
      t += st[j][tx];
    }
    const long long at = (long long)blockIdx.y * p.rows + row;
    if (SBP_GUARD(p.out_m + at, 4)) p.out_m[at] = m;
    if (SBP_GUARD(p.out_s + at, 4)) p.out_s[at] = s;
    if (SBP_GUARD(p.out_t + at, 4)) p.out_t[at] = t;
  }
}

constexpr int kMaxSlices = 64;

// Enough slices for four CTAs an SM, at least two parts a thread in each; one slice per 256 parts at least.  (1024
// parts of 64 rows: 8 CTAs with 32 parts a thread before.)
static int slices_for(int parts, long long rows) {
  const long long row_ctas = (rows + 31) / 32;
  long long s = std::min((long long)parts / 16, 4LL * device_sms() / row_ctas);
  s = std::max(s, (long long)parts / 256);
  return (int)std::max(1LL, std::min(s, (long long)kMaxSlices));
}

size_t xent_finish_stage_floats(long long rows) { return 3 * (size_t)kMaxSlices * (size_t)rows; }

sbp_status check_xent_outputs(const sbp_tensor* labels, const sbp_tensor* loss, const sbp_tensor* row_max,
                              const sbp_tensor* row_sum, long long rows, int k) {
  sbp_status st = check_tensor(labels, "labels", true);
  if (st != SBP_OK) return st;
  if (labels->ndim != 1 || labels->shape[0] != rows) return fail(SBP_ERR_SHAPE, "labels must be [rows]");
  if (labels->dtype != SBP_I64) return fail(SBP_ERR_DTYPE, "labels must be I64");
  if (labels->sbp[0].kind != SBP_BROADCAST) return fail(SBP_ERR_SIGNATURE, "labels must be B");
  if (placement_k(labels) != k) return fail(SBP_ERR_INVALID_ARG, "labels differ in k");
  st = check_row_vector(loss, "loss", rows, k);
  if (st != SBP_OK) return st;
  if (row_max && (st = check_row_vector(row_max, "row_max", rows, k)) != SBP_OK) return st;
  if (row_sum && (st = check_row_vector(row_sum, "row_sum", rows, k)) != SBP_OK) return st;
  return SBP_OK;
}

// parts partials per row in part_* ([parts][rows]) -> loss / row_max / row_sum.
sbp_status launch_xent_finish(float* part_m, float* part_s, float* part_t, int parts, long long rows, float* stage,
                              sbp_tensor* loss, sbp_tensor* row_max, sbp_tensor* row_sum, int k, cudaStream_t st) {
  const int slices = slices_for(parts, rows);
  XentReduceParams r{};
  r.in_m = part_m;
  r.in_s = part_s;
  r.in_t = part_t;
  r.out_m = stage;
  r.out_s = stage + (size_t)slices * rows;
  r.out_t = stage + 2 * (size_t)slices * rows;
  r.rows = rows;
  r.parts = parts;
  r.per_slice = (parts + slices - 1) / slices;
  // Both kernels are launched as programmatic dependents of their predecessors in the stream.
  cudaLaunchAttribute pdl[1];
  pdl[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  pdl[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)((rows + 31) / 32), (unsigned)slices);
  cfg.blockDim = dim3(256);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = st;
  cfg.attrs = pdl;
  cfg.numAttrs = 1;
  SBP_BOUNDS_UPLOAD(st);
  cudaError_t e = cudaLaunchKernelEx(&cfg, xent_reduce_parts_kernel, r);
  if (e != cudaSuccess) return cuda_fail(e, "softmax reduce launch");
  XentCombineParams c{};
  c.part_m = r.out_m;
  c.part_s = r.out_s;
  c.part_t = r.out_t;
  c.rows = rows;
  c.parts = slices;
  c.n_loss = dedup(c.loss, loss, k);
  c.n_max = row_max ? dedup(c.row_max, row_max, k) : 0;
  c.n_sum = row_sum ? dedup(c.row_sum, row_sum, k) : 0;
  cfg.gridDim = dim3((unsigned)((rows + kCombineThreads / 32 - 1) / (kCombineThreads / 32)));
  cfg.blockDim = dim3(kCombineThreads);
  e = cudaLaunchKernelEx(&cfg, xent_combine_kernel, c);
  if (e != cudaSuccess) return cuda_fail(e, "softmax combine launch");
  count_launch(2);
  return SBP_OK;
}

// ---- backward of the per-row loss with respect to the logits: softmax - onehot, kept S(1).
// Element-wise given the row max and row sum of the forward pass: one read and one write of
// the logits' size.
struct XentBwdParams {
  const char* logits[SBP_MAX_K];
  char* grad[SBP_MAX_K];
  const long long* labels;
  const float* row_max;
  const float* row_sum;
  long long rows, classes;
  long long lpitch[SBP_MAX_K], gpitch[SBP_MAX_K];   // elements between consecutive rows: logits, gradient
  int k, team_log2;
};

// VEC elements of 16 bytes a thread and step where both rows stand alike modulo 16 (always, for dense tensors
// with aligned bases), the elements before and after the whole vectors one a thread; VEC = 1 otherwise.
constexpr int kBwdVecs = 4;      // vectors in flight per thread

template <typename T, int VEC>
__global__ void __launch_bounds__(kThreads) xent_backward_kernel(const __grid_constant__ XentBwdParams p) {
  const int team = 1 << p.team_log2, tid = threadIdx.x & (team - 1);      // short rows: several to a CTA
  const long long row = (long long)(gridDim.x - 1 - blockIdx.x) * (kThreads >> p.team_log2) + (threadIdx.x >> p.team_log2);
  if (row >= p.rows) return;
  const int shard = p.k - 1 - (int)blockIdx.z;
  long long c_start, c_len;
  split_range(p.classes, p.k, shard, (int64_t*)&c_start, (int64_t*)&c_len);
  const T* z = reinterpret_cast<const T*>(p.logits[shard]) + row * p.lpitch[shard];
  T* g = reinterpret_cast<T*>(p.grad[shard]) + row * p.gpitch[shard];
  SBP_PDL_RELEASE();
  SBP_PDL_WAIT();
  // softmax = 2^((z - m) log2e - log2 S): the division by the row sum is folded into the exponent, and z - m keeps it exact
  // at any maximum
  if (!SBP_GUARD(p.row_max + row, 4) || !SBP_GUARD(p.row_sum + row, 4) || !SBP_GUARD(p.labels + row, 8)) return;
  const float m = p.row_max[row], neg = -log2f(p.row_sum[row]);
  const long long y = p.labels[row] - c_start;      // label's column inside this shard, if any
  const int head = VEC > 1 ? to_boundary(z, c_len) : 0;
  const long long nv = (c_len - head) / VEC;
  const int tail = (int)(c_len - head - nv * VEC);
  struct alignas(sizeof(T) * VEC) Pack { T e[VEC]; };
  if (VEC > 1 && blockIdx.y == 0) {
    const long long at = tid < head ? tid : (tid >= 16 && tid - 16 < tail ? head + nv * VEC + (tid - 16) : -1);
    if (at >= 0 && SBP_GUARD(z + at, sizeof(T)) && SBP_GUARD(g + at, sizeof(T))) {
      float v = ex2(fmaf(static_cast<float>(z[at]) - m, kLog2e, neg));
      if (at == y) v -= 1.0f;
      g[at] = static_cast<T>(v);
    }
  }
  const T* zv = z + head;
  T* gv = g + head;
  const long long step = (long long)gridDim.y * team;
  for (long long v0 = (long long)blockIdx.y * team + tid; v0 < nv; v0 += kBwdVecs * step) {
    Pack in[kBwdVecs];
#pragma unroll
    for (int u = 0; u < kBwdVecs; ++u) {
      const long long v = v0 + u * step;
      if (v >= nv || !SBP_GUARD(zv + v * VEC, sizeof(Pack))) continue;
      if constexpr (VEC > 1) *reinterpret_cast<uint4*>(&in[u]) = ld_logits(zv + v * VEC, l2_first());
      else in[u] = *reinterpret_cast<const Pack*>(zv + v * VEC);
    }
#pragma unroll
    for (int u = 0; u < kBwdVecs; ++u) {
      const long long v = v0 + u * step;
      if (v >= nv || !SBP_GUARD(gv + v * VEC, sizeof(Pack))) continue;
      const long long rel = y - head - v * VEC;
      const int y_rel = rel >= 0 && rel < VEC ? (int)rel : -1;   // the label's place in this vector, if it is here
      Pack out;
#pragma unroll
      for (int i = 0; i < VEC; ++i) {
        float f = ex2(fmaf(static_cast<float>(in[u].e[i]) - m, kLog2e, neg));
        if (i == y_rel) f -= 1.0f;
        out.e[i] = static_cast<T>(f);
      }
      if constexpr (VEC > 1) __stcs(reinterpret_cast<uint4*>(gv + v * VEC), *reinterpret_cast<const uint4*>(&out));
      else *reinterpret_cast<Pack*>(gv + v * VEC) = out;
    }
  }
}

}  // namespace sbp

using namespace sbp;

extern "C" {

size_t sbp_softmax_xent_workspace_bytes(const sbp_tensor* logits) {
  if (check_tensor(logits, "logits", false) != SBP_OK || logits->ndim != 2) return 0;
  // room for spans of a sixteenth of a chunk's elements too: short rows are cut finer when there is room
  const int k = placement_k(logits);
  const int ns = nsplit_for(logits, 1);
  const int ns_vec = nsplit_for(logits, vec_of(logits));
  const size_t parts = (size_t)k * (size_t)(ns > ns_vec ? ns : ns_vec);
  return 3 * parts * (size_t)logits->shape[0] * sizeof(float);
}

sbp_status sbp_softmax_xent(const sbp_tensor* logits, const sbp_tensor* labels, sbp_tensor* loss,
                            sbp_tensor* row_max, sbp_tensor* row_sum, void* ws, size_t ws_bytes,
                            void* cuda_stream) {
  SBP_RANGE("sbp_softmax_xent");
  sbp_status st = check_tensor(logits, "logits", true);
  if (st != SBP_OK) return st;
  st = check_tensor(labels, "labels", true);
  if (st != SBP_OK) return st;
  if (logits->ndim != 2) return fail(SBP_ERR_SHAPE, "logits must be [rows, classes]");
  if (logits->dtype != SBP_BF16 && logits->dtype != SBP_F32) return fail(SBP_ERR_DTYPE, "logits must be BF16 or F32");
  if (!(logits->sbp[0].kind == SBP_SPLIT && logits->sbp[0].axis == 1))
    return fail(SBP_ERR_SIGNATURE, "logits must be S(1)");
  const int k = placement_k(logits);
  const long long rows = logits->shape[0], classes = logits->shape[1];
  if (labels->ndim != 1 || labels->shape[0] != rows) return fail(SBP_ERR_SHAPE, "labels must be [rows]");
  if (labels->dtype != SBP_I64) return fail(SBP_ERR_DTYPE, "labels must be I64");
  if (labels->sbp[0].kind != SBP_BROADCAST) return fail(SBP_ERR_SIGNATURE, "labels must be B");
  if (placement_k(labels) != k) return fail(SBP_ERR_INVALID_ARG, "labels differ in k");
  st = check_row_vector(loss, "loss", rows, k);
  if (st != SBP_OK) return st;
  if (row_max && (st = check_row_vector(row_max, "row_max", rows, k)) != SBP_OK) return st;
  if (row_sum && (st = check_row_vector(row_sum, "row_sum", rows, k)) != SBP_OK) return st;
  if (classes < 1) return fail(SBP_ERR_SHAPE, "softmax over zero classes");
  if (rows == 0) return SBP_OK;

  const size_t least = 3 * (size_t)k * (size_t)nsplit_for(logits, vec_of(logits)) * rows * sizeof(float);
  if (!ws || ws_bytes < least) return fail(SBP_ERR_WORKSPACE, "workspace of %zu bytes needed, %zu given", least, ws_bytes);
  if (reinterpret_cast<uintptr_t>(ws) % 4 != 0) return fail(SBP_ERR_ALIGNMENT, "workspace must be 4-byte aligned");
  long long span;
  int nsplit;
  tiling_in(logits, ws_bytes, &span, &nsplit);
  if (rows > 0x7fffffffLL || nsplit > 65535) return fail(SBP_ERR_UNSUPPORTED, "shape too large for one launch");
  const int parts = k * nsplit;

  XentParams p{};
  for (int r = 0; r < k; ++r) {
    p.logits[r] = static_cast<const char*>(logits->local[r]);
    p.pitch[r] = local_pitch(logits, r);
  }
  p.labels = static_cast<const long long*>(labels->local[0]);
  p.part_m = static_cast<float*>(ws);
  p.part_s = p.part_m + (size_t)parts * rows;
  p.part_t = p.part_s + (size_t)parts * rows;
  p.rows = rows;
  p.classes = classes;
  p.k = k;
  p.nsplit = nsplit;
  p.span = span;

  XentCombineParams c{};
  c.part_m = p.part_m;
  c.part_s = p.part_s;
  c.part_t = p.part_t;
  c.rows = rows;
  c.parts = parts;
  c.n_loss = dedup(c.loss, loss, k);
  c.n_max = row_max ? dedup(c.row_max, row_max, k) : 0;
  c.n_sum = row_sum ? dedup(c.row_sum, row_sum, k) : 0;

  cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
  SBP_BOUNDS_RESET();
  SBP_BOUNDS_TENSOR(logits);
  SBP_BOUNDS_TENSOR(labels);
  SBP_BOUNDS_TENSOR(loss);
  SBP_BOUNDS_TENSOR(row_max);
  SBP_BOUNDS_TENSOR(row_sum);
  SBP_BOUNDS_ADD(ws, 3 * (size_t)parts * rows * sizeof(float));
  SBP_BOUNDS_UPLOAD(stream);
  const int team_log2 = team_for(rows, classes, logits->dtype == SBP_BF16 ? 8 : 4);
  // the last units of the walk, rows or CTAs, whose logits make up the part to keep
  const double keep = std::min(1.0, (double)device_l2_bytes() * kKeepNum / kKeepDen / ((double)rows * classes * elem_size(logits->dtype)));
  const long long units = team_log2 > 0 ? rows : rows * parts;
  p.keep_from = units - (long long)(keep * units);
  if (team_log2 > 0) {
    const int per_cta = kThreads >> team_log2;
    const dim3 g((unsigned)((rows + per_cta - 1) / per_cta));
    if (logits->dtype == SBP_BF16) launch_dependent(xent_rows_kernel<ChunkBF16>, g, dim3(kThreads), 0, stream, p, c, team_log2);
    else launch_dependent(xent_rows_kernel<ChunkF32>, g, dim3(kThreads), 0, stream, p, c, team_log2);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "softmax launch");
    count_launch();
    return SBP_OK;
  }
  dim3 grid((unsigned)rows, (unsigned)nsplit, (unsigned)k);
  if (logits->dtype == SBP_BF16) launch_partial<ChunkBF16>(p, grid, (classes + k - 1) / k, stream);
  else launch_partial<ChunkF32>(p, grid, (classes + k - 1) / k, stream);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(e, "softmax partial launch");

  // Launched as the programmatic dependent of the partial kernel: it may be set up while that
  // kernel still runs and waits, on the device, for it to finish before reading the partials.
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)((rows + kCombineThreads / 32 - 1) / (kCombineThreads / 32)));
  cfg.blockDim = dim3(kCombineThreads);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  e = cudaLaunchKernelEx(&cfg, xent_combine_kernel, c);
  if (e != cudaSuccess) return cuda_fail(e, "softmax combine launch");
  count_launch(2);
  return SBP_OK;
}

}  // extern "C"

// ------------------------------------------------------------------ built-in scratch variant
//
// Scratch for callers that cannot hand in a workspace.  It lives in the library's image, so
// every GPU that loads the library carries these 3 MiB until the process exits.
namespace sbp {
constexpr size_t kStaticScratchBytes = SBP_SOFTMAX_XENT_STATIC_SCRATCH_BYTES;
static __device__ __align__(256) float g_xent_static_scratch[kStaticScratchBytes / sizeof(float)];
constexpr int kMaxDevices = 64;
}  // namespace sbp

extern "C" sbp_status sbp_softmax_xent_static(const sbp_tensor* logits, const sbp_tensor* labels, sbp_tensor* loss,
                                              sbp_tensor* row_max, sbp_tensor* row_sum, void* cuda_stream) {
  SBP_RANGE("sbp_softmax_xent_static");
  // Size check first, so that an oversized request is refused before anything else happens.
  sbp_status st = check_tensor(logits, "logits", true);
  if (st != SBP_OK) return st;
  if (logits->ndim != 2) return fail(SBP_ERR_SHAPE, "logits must be [rows, classes]");
  const size_t need =
      3 * (size_t)placement_k(logits) * (size_t)nsplit_for(logits, vec_of(logits)) * (size_t)logits->shape[0] * sizeof(float);
  if (need > kStaticScratchBytes)
    return fail(SBP_ERR_WORKSPACE,
                "this shape needs %zu bytes of scratch but the built-in array holds %zu; call sbp_softmax_xent "
                "with a workspace of your own instead",
                need, kStaticScratchBytes);

  // In host code the array's name is only a handle; its device address has to be looked up,
  // once per device, while that device is current.
  static float* dev_ptr[kMaxDevices] = {};
  static std::mutex mu;
  int dev = 0;
  SBP_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kMaxDevices) return fail(SBP_ERR_UNSUPPORTED, "device ordinal %d out of range", dev);
  float* scratch = nullptr;
  {
    std::lock_guard<std::mutex> lock(mu);
    if (!dev_ptr[dev]) {
      void* ptr = nullptr;
      SBP_CUDA_TRY(cudaGetSymbolAddress(&ptr, g_xent_static_scratch));
      dev_ptr[dev] = static_cast<float*>(ptr);
    }
    scratch = dev_ptr[dev];
  }
  return sbp_softmax_xent(logits, labels, loss, row_max, row_sum, scratch, kStaticScratchBytes, cuda_stream);
}

extern "C" sbp_status sbp_softmax_xent_backward(const sbp_tensor* logits, const sbp_tensor* labels,
                                                const sbp_tensor* row_max, const sbp_tensor* row_sum,
                                                sbp_tensor* grad_logits, void* cuda_stream) {
  SBP_RANGE("sbp_softmax_xent_backward");
  sbp_status st = check_tensor(logits, "logits", true);
  if (st != SBP_OK) return st;
  st = check_tensor(grad_logits, "grad_logits", true);
  if (st != SBP_OK) return st;
  if (logits->ndim != 2 || grad_logits->ndim != 2 || logits->shape[0] != grad_logits->shape[0] ||
      logits->shape[1] != grad_logits->shape[1])
    return fail(SBP_ERR_SHAPE, "logits and grad_logits must be [rows, classes] alike");
  if (logits->dtype != SBP_BF16 && logits->dtype != SBP_F32) return fail(SBP_ERR_DTYPE, "logits must be BF16 or F32");
  if (grad_logits->dtype != logits->dtype) return fail(SBP_ERR_DTYPE, "grad_logits and logits differ in dtype");
  const int k = placement_k(logits);
  if (placement_k(grad_logits) != k) return fail(SBP_ERR_INVALID_ARG, "operands differ in k");
  auto is_s1 = [](const sbp_tensor* t) { return t->sbp[0].kind == SBP_SPLIT && t->sbp[0].axis == 1; };
  if (!is_s1(logits) || !is_s1(grad_logits)) return fail(SBP_ERR_SIGNATURE, "logits and grad_logits must be S(1)");
  const long long rows = logits->shape[0], classes = logits->shape[1];
  if (!row_max || !row_sum) return fail(SBP_ERR_INVALID_ARG, "row_max and row_sum of the forward pass are required");
  st = check_xent_outputs(labels, row_max, row_max, row_sum, rows, k);
  if (st != SBP_OK) return st;
  if (rows == 0 || classes == 0) return SBP_OK;
  if (rows > 0x7fffffffLL) return fail(SBP_ERR_UNSUPPORTED, "too many rows for one launch");

  XentBwdParams p{};
  bool vec_ok = true;
  const int esz = elem_size(logits->dtype);
  for (int r = 0; r < k; ++r) {
    p.lpitch[r] = local_pitch(logits, r);
    p.gpitch[r] = local_pitch(grad_logits, r);
    // every row of the gradient stands as the logits' row does, modulo 16 bytes
    vec_ok = vec_ok && (reinterpret_cast<uintptr_t>(logits->local[r]) - reinterpret_cast<uintptr_t>(grad_logits->local[r])) % 16 == 0 &&
             ((p.lpitch[r] - p.gpitch[r]) * esz) % 16 == 0;
    p.logits[r] = static_cast<const char*>(logits->local[r]);
    p.grad[r] = static_cast<char*>(grad_logits->local[r]);
  }
  p.labels = static_cast<const long long*>(labels->local[0]);
  p.row_max = static_cast<const float*>(row_max->local[0]);
  p.row_sum = static_cast<const float*>(row_sum->local[0]);
  p.rows = rows;
  p.classes = classes;
  p.k = k;
  const int vec = vec_ok ? 16 / esz : 1;
  const long long c_max = (classes + k - 1) / k;
  long long gy = (c_max + (long long)kThreads * vec * kBwdVecs - 1) / ((long long)kThreads * vec * kBwdVecs);
  if (gy < 1) gy = 1;
  if (gy > 65535) gy = 65535;
  p.team_log2 = 5;
  while (p.team_log2 < 8 && ((long long)vec * kBwdVecs << p.team_log2) < c_max) ++p.team_log2;
  const int per_cta = kThreads >> p.team_log2;
  dim3 grid((unsigned)((rows + per_cta - 1) / per_cta), (unsigned)gy, (unsigned)k);
  cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
  SBP_BOUNDS_RESET();
  SBP_BOUNDS_TENSOR(logits);
  SBP_BOUNDS_TENSOR(labels);
  SBP_BOUNDS_TENSOR(row_max);
  SBP_BOUNDS_TENSOR(row_sum);
  SBP_BOUNDS_TENSOR(grad_logits);
  SBP_BOUNDS_UPLOAD(stream);
  if (logits->dtype == SBP_BF16) {
    if (vec > 1) launch_dependent(xent_backward_kernel<__nv_bfloat16, 8>, grid, dim3(kThreads), 0, stream, p);
    else launch_dependent(xent_backward_kernel<__nv_bfloat16, 1>, grid, dim3(kThreads), 0, stream, p);
  } else {
    if (vec > 1) launch_dependent(xent_backward_kernel<float, 4>, grid, dim3(kThreads), 0, stream, p);
    else launch_dependent(xent_backward_kernel<float, 1>, grid, dim3(kThreads), 0, stream, p);
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(e, "softmax backward launch");
  count_launch();
  return SBP_OK;
}
