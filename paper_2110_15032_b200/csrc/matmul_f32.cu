// fp32 MatMul: executes a grouped-GEMM plan (matmul_plan.h) on the FMA pipes.  (Products that fill tiles of the tensor cores
// go to matmul_f32_tc.cu.)
//
// Every element of the result is a chain of fused multiply-adds in fp32, k ascending, segments in rank order; where K is
// split over the CTAs of a cluster (below) one chain for each, the chains added in their
// order; there is no reduced-precision product.  Bound: the FMA pipe (128 lanes per SM and clock, 74
// TFLOP/s at 1.965 GHz) once a product fills the device, the latency of load -> shared memory -> first
// FMA and the launch for the small ones.
//
//   * A CTA of 256 threads owns a (16 TM) x (16 TN) tile, TM x TN elements per thread.  Multiply-adds are
//     issued as packed pairs (fma.rn.f32x2, each half an IEEE fma), which leaves half of the issue slots to
//     the shared-memory reads.
//   * Operands arrive through a kStages-deep ring of 16-deep K-slices filled with asynchronous copies: 16
//     bytes each where base, leading dimension and offsets allow, else 4 bytes each; positions past an
//     edge are zero-filled by the copy.  A slice keeps the order it has in memory -- K contiguous or M / N
//     contiguous -- so nothing is transposed on the way and both stored forms of either operand cost the
//     same.
//   * A tile whose K is long and whose device is otherwise idle is split along K over the CTAs of a
//     cluster (S = 2, 4, 8): each CTA runs its range of slices, then reads the others' partial sums of its
//     own rows from their shared memory and adds them in slice order.  No workspace, no atomics, the same
//     bits every time.
#include <cuda_runtime.h>

#include <atomic>
#include <type_traits>

#include "bounds_check.h"
#include "matmul_plan.h"
#include "sbp_internal.h"

namespace sbp {

namespace {

constexpr int kBK = 16;          // K-slice
constexpr int kStages = 4;
constexpr int kThreads = 256;
constexpr int kKPitch = kBK + 4; // floats per row of a K-contiguous slice: 16-byte aligned, and 4 (8) neighbouring
                                 // rows read at once fall into different banks

struct F32Params {
  MatmulPlan plan;
  int splits;                    // CTAs per tile (cluster size)
  int a_vec, b_vec, y_vec;       // 16-byte copies / stores are possible everywhere
  int early;                     // the small kernel lets the next one in at once
  int a_quad, b_quad;            // and every quad of an operand lies inside it as a whole or not at all
};

__device__ __forceinline__ void cp_async16(unsigned dst, const void* src, unsigned bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async4(unsigned dst, const void* src, unsigned bytes) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ unsigned long long pack2(float lo, float hi) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void unpack2(unsigned long long v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ void fma2(unsigned long long& acc, unsigned long long a, unsigned long long b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b));
}
__device__ __forceinline__ float gelu_erf(float v) { return 0.5f * v * (1.0f + erff(v * 0.70710678118654752440f)); }

template <int EXT, bool KC>
constexpr int slice_floats() {
  return KC ? EXT * kKPitch : kBK * EXT;
}

// One slice of an operand: EXT positions of its M / N index x kBK of K.  g points at position (0, 0) of
// the slice; ext / kk are how many positions / K-steps of it lie inside the operand (any may be <= 0).
// KC: K is contiguous in memory (and in shared memory: rows of kKPitch floats), else the M / N index is.
template <int EXT, bool KC>
__device__ __forceinline__ void load_slice(float* s, const float* g, long long ld, long long ext, long long kk, bool vec, int tid) {
  const unsigned base = (unsigned)__cvta_generic_to_shared(s);
  constexpr int kRows = KC ? EXT : kBK, kCols = KC ? kBK : EXT, kPitch = KC ? kKPitch : EXT;
  const long long rows = KC ? ext : kk, cols = KC ? kk : ext;
  if (vec) {
#pragma unroll
    for (int j = 0; j < kRows * kCols / 4 / kThreads; ++j) {
      const int idx = tid + j * kThreads, r = idx / (kCols / 4), c = idx % (kCols / 4) * 4;
      const long long left = r < rows ? cols - c : 0;
      int n = left >= 4 ? 4 : (left > 0 ? (int)left : 0);
      const float* src = g + (long long)r * ld + c;
      if (n > 0 && !SBP_GUARD(src, (size_t)n * 4)) n = 0;
      cp_async16(base + (unsigned)(r * kPitch + c) * 4, n > 0 ? src : g, (unsigned)n * 4);
    }
  } else {
#pragma unroll
    for (int j = 0; j < kRows * kCols / kThreads; ++j) {
      const int idx = tid + j * kThreads, r = idx / kCols, c = idx % kCols;
      const float* src = g + (long long)r * ld + c;
      const bool in = r < rows && c < cols && SBP_GUARD(src, 4);
      cp_async4(base + (unsigned)(r * kPitch + c) * 4, in ? src : g, in ? 4u : 0u);
    }
  }
}

// AT / BT: the operand is stored transposed.  A as given and B transposed are K-contiguous.
template <int TM, int TN, int AT, int BT>
__global__ void __launch_bounds__(kThreads, TM == 8 ? 2 : 3) matmul_f32_kernel(const __grid_constant__ F32Params P) {
  constexpr int BM = 16 * TM, BN = 16 * TN;
  constexpr bool AKC = !AT, BKC = BT;
  constexpr int kA = slice_floats<BM, AKC>(), kB = slice_floats<BN, BKC>();
  constexpr int KS = TM == 8 ? 2 : 4;              // K-steps whose A values a thread holds at once
  extern __shared__ __align__(16) float smem[];
  const MatmulPlan& p = P.plan;
  const int g = blockIdx.z;
  const int splits = P.splits, slice = (int)(blockIdx.x % (unsigned)splits);
  const long long M = p.m[g], N = p.n[g];
  const long long m0 = (long long)blockIdx.y * BM, n0 = (long long)(blockIdx.x / (unsigned)splits) * BN;
  if (m0 >= M || n0 >= N) return;                  // the whole cluster
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int ty = (warp >> 1) * 4 + (lane >> 3), tx = (warp & 1) * 8 + (lane & 7);
  // element (i, j) of a thread: strided over a K-contiguous slice's rows, in runs of four otherwise
  auto row_of = [&](int i) { return AKC ? i * 16 + ty : (i / 4) * 64 + ty * 4 + (i & 3); };
  auto col_of = [&](int j) { return BKC ? j * 16 + tx : (j / 4) * 64 + tx * 4 + (j & 3); };

  // this CTA's range of K-slices over all segments
  const int s_lo = p.chain ? 0 : g, s_hi = p.chain ? p.nseg : g + 1;
  long long total = 0;
  for (int s = s_lo; s < s_hi; ++s) total += (p.kseg[s] + kBK - 1) / kBK;
  const long long it0 = total * slice / splits, it1 = total * (slice + 1) / splits;
  const int iters = (int)(it1 - it0);
  int ls = s_lo;                                   // the loader's position: segment and K inside it
  long long lk = it0 * kBK;
  {
    long long skip = it0;
    while (ls < s_hi) {
      const long long n = (p.kseg[ls] + kBK - 1) / kBK;
      if (skip < n) break;
      skip -= n;
      ++ls;
    }
    lk = skip * kBK;
  }
  auto load_next = [&](int stage) {
    while (ls < s_hi && lk >= p.kseg[ls]) { ++ls; lk = 0; }      // also steps over empty segments
    const long long lda = p.lda[ls], ldb = p.ldb[ls], left = p.kseg[ls] - lk;
    const float* A = static_cast<const float*>(p.a[ls]) + (AT ? lk * lda + p.row_off[g] + m0 : (p.row_off[g] + m0) * lda + lk);
    const float* B = static_cast<const float*>(p.b[ls]) + (BT ? (p.col_off[g] + n0) * ldb + lk : lk * ldb + p.col_off[g] + n0);
    float* sa = smem + stage * (kA + kB);
    load_slice<BM, AKC>(sa, A, lda, M - m0, left, P.a_vec != 0, tid);
    load_slice<BN, BKC>(sa + kA, B, ldb, N - n0, left, P.b_vec != 0, tid);
    lk += kBK;
  };

  unsigned long long acc[TM][TN / 2];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN / 2; ++j) acc[i][j] = 0ull;

  SBP_PDL_WAIT();                                  // everything up to here overlaps the kernel before this one
#pragma unroll
  for (int st = 0; st < kStages - 1; ++st) {
    if (st < iters) load_next(st);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  int stage = 0, fill = kStages - 1;
  for (int it = 0; it < iters; ++it) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kStages - 2) : "memory");
    __syncthreads();                               // slice `it` is there, and everyone is done with the one before it
    if (it + kStages - 1 < iters) load_next(fill);
    asm volatile("cp.async.commit_group;" ::: "memory");
    const float* sa = smem + stage * (kA + kB);
    const float* sb = sa + kA;
#pragma unroll
    for (int k0 = 0; k0 < kBK; k0 += KS) {
      float a[TM][KS], b[TN][KS];
      if constexpr (AKC) {
#pragma unroll
        for (int i = 0; i < TM; ++i) {
          if constexpr (KS == 4) *reinterpret_cast<float4*>(a[i]) = *reinterpret_cast<const float4*>(sa + row_of(i) * kKPitch + k0);
          else *reinterpret_cast<float2*>(a[i]) = *reinterpret_cast<const float2*>(sa + row_of(i) * kKPitch + k0);
        }
      }
      if constexpr (BKC) {
#pragma unroll
        for (int j = 0; j < TN; ++j) {
          if constexpr (KS == 4) *reinterpret_cast<float4*>(b[j]) = *reinterpret_cast<const float4*>(sb + col_of(j) * kKPitch + k0);
          else *reinterpret_cast<float2*>(b[j]) = *reinterpret_cast<const float2*>(sb + col_of(j) * kKPitch + k0);
        }
      }
#pragma unroll
      for (int k = 0; k < KS; ++k) {
        float ak[TM], bk[TN];
#pragma unroll
        for (int i = 0; i < TM; i += 4) {
          if constexpr (AKC) { ak[i] = a[i][k]; ak[i + 1] = a[i + 1][k]; ak[i + 2] = a[i + 2][k]; ak[i + 3] = a[i + 3][k]; }
          else *reinterpret_cast<float4*>(ak + i) = *reinterpret_cast<const float4*>(sa + (k0 + k) * BM + row_of(i));
        }
#pragma unroll
        for (int j = 0; j < TN; j += 4) {
          if constexpr (BKC) { bk[j] = b[j][k]; bk[j + 1] = b[j + 1][k]; bk[j + 2] = b[j + 2][k]; bk[j + 3] = b[j + 3][k]; }
          else *reinterpret_cast<float4*>(bk + j) = *reinterpret_cast<const float4*>(sb + (k0 + k) * BN + col_of(j));
        }
        unsigned long long bp[TN / 2];
#pragma unroll
        for (int j = 0; j < TN / 2; ++j) bp[j] = pack2(bk[2 * j], bk[2 * j + 1]);
#pragma unroll
        for (int i = 0; i < TM; ++i) {
          const unsigned long long ap = pack2(ak[i], ak[i]);
#pragma unroll
          for (int j = 0; j < TN / 2; ++j) fma2(acc[i][j], ap, bp[j]);
        }
      }
    }
    stage = stage + 1 == kStages ? 0 : stage + 1;
    fill = fill + 1 == kStages ? 0 : fill + 1;
  }

  // The next kernel's CTAs are let in only now: set up earlier, they take the free slots of the SMs that
  // finish first and the next product runs unevenly (1000 x 1500 x 777 over four shards, back to back:
  // 171 us released at the start, 99 us here).
  SBP_PDL_RELEASE();

  // four neighbouring results of one row: GeLU, then the result and its replicas
  float* const y = static_cast<float*>(p.y[g]);
  const long long ldy = p.ldy[g];
  const int n_out = (g == 0 ? p.n_rep : 0) + 1;
  auto store4 = [&](long long r, long long c, const float (&v)[4], int step) {
    if (r >= M) return;
    float o[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) o[e] = p.gelu ? gelu_erf(v[e]) : v[e];
    for (int q = 0; q < n_out; ++q) {
      float* at = (q == 0 ? y : static_cast<float*>(p.y_rep[q - 1])) + r * ldy + c;
      if (step == 1 && P.y_vec && c + 3 < N) {
        if (SBP_GUARD(at, 16)) *reinterpret_cast<float4*>(at) = make_float4(o[0], o[1], o[2], o[3]);
      } else {
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (c + e * step < N && SBP_GUARD(at + e * step, 4)) at[e * step] = o[e];
      }
    }
  };

  if (splits == 1) {
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < TN; j += 4) {
        float v[4];
        unpack2(acc[i][j / 2], v[0], v[1]);
        unpack2(acc[i][j / 2 + 1], v[2], v[3]);
        store4(m0 + row_of(i), n0 + col_of(j), v, BKC ? 16 : 1);
      }
    return;
  }

  // K was split: park the partial tile, then add up the rows this CTA answers for, slice by slice.
  // (The ring holds the tile: kStages slices of (BM + BN) x 16 are at least BM x BN floats.)
  static_assert(kStages * (kA + kB) >= BM * BN, "the ring has to hold the partial tile");
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; j += 4) {
      float v[4];
      unpack2(acc[i][j / 2], v[0], v[1]);
      unpack2(acc[i][j / 2 + 1], v[2], v[3]);
      float* at = smem + row_of(i) * BN + col_of(j);
      if constexpr (BKC) {
#pragma unroll
        for (int e = 0; e < 4; ++e) at[e * 16] = v[e];
      } else {
        *reinterpret_cast<float4*>(at) = make_float4(v[0], v[1], v[2], v[3]);
      }
    }
  asm volatile("barrier.cluster.arrive.release;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
  const int rows_each = BM / splits;
  const unsigned mine = (unsigned)__cvta_generic_to_shared(smem);
  for (int idx = tid; idx < rows_each * (BN / 4); idx += kThreads) {
    const int r = slice * rows_each + idx / (BN / 4), c = idx % (BN / 4) * 4;
    if (m0 + r >= M || n0 + c >= N) continue;
    float v[4] = {0.f, 0.f, 0.f, 0.f};
    for (int q = 0; q < splits; ++q) {
      unsigned remote;
      float x0, x1, x2, x3;
      asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(mine + (unsigned)(r * BN + c) * 4), "r"(q));
      asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(x0), "=f"(x1), "=f"(x2), "=f"(x3) : "r"(remote) : "memory");
      if (q == 0) { v[0] = x0; v[1] = x1; v[2] = x2; v[3] = x3; }
      else { v[0] += x0; v[1] += x1; v[2] += x2; v[3] += x3; }
    }
    store4(m0 + r, n0 + c, v, 1);
  }
  asm volatile("barrier.cluster.arrive.release;" ::: "memory");      // nobody leaves while its tile may still be read
  asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}

template <int TM, int TN, int AT, int BT>
cudaError_t launch_form(const F32Params& P, dim3 grid, cudaStream_t st) {
  constexpr int kSmem = kStages * (slice_floats<16 * TM, !AT>() + slice_floats<16 * TN, (bool)BT>()) * 4;
  if (kSmem > 48 * 1024) {
    static std::atomic<unsigned long long> opted{0};      // one bit per device
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = 1ull << (dev & 63);
    if (dev >= 64 || !(opted.load(std::memory_order_relaxed) & bit)) {
      e = cudaFuncSetAttribute(matmul_f32_kernel<TM, TN, AT, BT>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
      if (e != cudaSuccess) return e;
      if (dev < 64) opted.fetch_or(bit, std::memory_order_relaxed);
    }
  }
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = kSmem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned)P.splits;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = P.splits > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, matmul_f32_kernel<TM, TN, AT, BT>, P);
}

template <int TM, int TN>
cudaError_t launch_stored(const F32Params& P, dim3 grid, cudaStream_t st) {
  switch ((P.plan.a_trans ? 2 : 0) | (P.plan.b_trans ? 1 : 0)) {
    case 0: return launch_form<TM, TN, 0, 0>(P, grid, st);
    case 1: return launch_form<TM, TN, 0, 1>(P, grid, st);
    case 2: return launch_form<TM, TN, 1, 0>(P, grid, st);
    default: return launch_form<TM, TN, 1, 1>(P, grid, st);
  }
}

// ------------------------------------------------------------------ small products
//
// A product of a few small tiles is latency: launch, first loads, a chain of K-slices, an exchange.  Here the eight warps of a
// CTA share a 32 x 32 tile and cut its contraction between them: a warp loads its slices into registers a slice ahead, passes
// them through shared memory of its own and multiplies 4 x 8 elements a lane; the eight partial tiles are added in
// pairs.  No cluster to be placed, no barrier but the one before the sums.
constexpr int kST = 32;                  // tile
constexpr int kSWarps = 8;              // (the sum of their tiles is written out for eight)
template <bool KC>
constexpr int small_floats() { return KC ? kST * kKPitch : kBK * kST; }

// One K-slice of an operand, 16 elements a lane.  KC: quad j of a lane is K quad (lane mod 4) of row lane / 4 + 8 j, else position
// quad (lane mod 8) of K-step lane / 8 + 4 j.  The loads are predicated instructions, so that none waits for the one before.
template <bool KC>
struct SmallSlice {
  float4 r[4];
  template <bool VEC>
  __device__ __forceinline__ void load(const float* g, long long ld, long long ext, long long kk, int lane) {
    const int row = KC ? lane >> 2 : lane >> 3, col = (KC ? lane & 3 : lane & 7) * 4;
    const long long rows = KC ? ext : kk, cols = KC ? kk : ext;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int at = row + j * (KC ? 8 : 4);
      const float* src = g + at * ld + col;
      const long long have = at < rows ? cols - col : 0;
      r[j] = make_float4(0.f, 0.f, 0.f, 0.f);
      if constexpr (VEC) {       // whole quads inside or none
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %5, 0;\n\t@p ld.global.v4.f32 {%0, %1, %2, %3}, [%4];\n\t}"
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
  __device__ __forceinline__ void store(float* s, int lane) const {
    const int row = KC ? lane >> 2 : lane >> 3, col = (KC ? lane & 3 : lane & 7) * 4;
#pragma unroll
    for (int j = 0; j < 4; ++j) *reinterpret_cast<float4*>(s + (row + j * (KC ? 8 : 4)) * (KC ? kKPitch : kST) + col) = r[j];
  }
};

template <int AT, int BT>
__global__ void __launch_bounds__(32 * kSWarps) matmul_f32_small_kernel(const __grid_constant__ F32Params P) {
  constexpr bool AKC = !AT, BKC = BT;
  constexpr int kA = small_floats<AKC>(), kB = small_floats<BKC>(), kPitch = kST + 4;
  constexpr int kFloats = kSWarps * (kA + kB) > kSWarps * kST * kPitch ? kSWarps * (kA + kB) : kSWarps * kST * kPitch;
  __shared__ __align__(16) float smem[kFloats];
  const MatmulPlan& p = P.plan;
  const int g = blockIdx.z;
  const long long M = p.m[g], N = p.n[g];
  const long long m0 = (long long)blockIdx.y * kST, n0 = (long long)blockIdx.x * kST;
  if (m0 >= M || n0 >= N) return;
  // A product of a few CTAs lets the next kernel's in at once, they find SMs of their own; one of more, only when its sums are
  // parked: earlier they delay it.  (Programs, us, at once / then: 64 x 128 x 96 x 80 on two shards, 6 and 8 CTAs, 9.2 / 10.4;
  // 1734 x 72 x 90 x 16, 110 CTAs, 17.4 / 12.1; 336 x 334 x 435 x 172 on eight 31.4 / 28.4 where it was the slices' end.)
  if (P.early) SBP_PDL_RELEASE();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, ty = lane >> 2, tx = lane & 3;
  auto row_of = [&](int i) { return AKC ? i * 8 + ty : ty * 4 + i; };
  auto col_of = [&](int j) { return BKC ? j * 4 + tx : (j / 4) * 16 + tx * 4 + (j & 3); };

  // this warp's range of K-slices over all segments
  const int s_lo = p.chain ? 0 : g, s_hi = p.chain ? p.nseg : g + 1;
  long long total = 0;
  for (int s = s_lo; s < s_hi; ++s) total += (p.kseg[s] + kBK - 1) / kBK;
  const long long it0 = total * warp / kSWarps;
  const int iters = (int)(total * (warp + 1) / kSWarps - it0);
  int ls = s_lo;
  long long lk = it0;
  while (ls < s_hi) {
    const long long n = (p.kseg[ls] + kBK - 1) / kBK;
    if (lk < n) break;
    lk -= n;
    ++ls;
  }
  lk *= kBK;
  unsigned long long acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0ull;
  float* sa = smem + warp * (kA + kB);
  float* sb = sa + kA;
  SBP_PDL_WAIT();

  auto run = [&](auto av, auto bv) {
    constexpr bool AV = decltype(av)::value, BV = decltype(bv)::value;
    SmallSlice<AKC> a;
    SmallSlice<BKC> b;
    auto load_next = [&]() {
      while (ls < s_hi && lk >= p.kseg[ls]) { ++ls; lk = 0; }      // also steps over empty segments
      const long long lda = p.lda[ls], ldb = p.ldb[ls], left = p.kseg[ls] - lk;
      a.template load<AV>(static_cast<const float*>(p.a[ls]) + (AT ? lk * lda + p.row_off[g] + m0 : (p.row_off[g] + m0) * lda + lk), lda, M - m0, left, lane);
      b.template load<BV>(static_cast<const float*>(p.b[ls]) + (BT ? (p.col_off[g] + n0) * ldb + lk : lk * ldb + p.col_off[g] + n0), ldb, N - n0, left, lane);
      lk += kBK;
    };
    if (iters > 0) load_next();
    for (int it = 0; it < iters; ++it) {
      a.store(sa, lane);
      b.store(sb, lane);
      __syncwarp();
      if (it + 1 < iters) load_next();
#pragma unroll
      for (int k0 = 0; k0 < kBK; k0 += 4) {
        float x[4][4], w[8][4];
        if constexpr (AKC) {
#pragma unroll
          for (int i = 0; i < 4; ++i) *reinterpret_cast<float4*>(x[i]) = *reinterpret_cast<const float4*>(sa + row_of(i) * kKPitch + k0);
        }
        if constexpr (BKC) {
#pragma unroll
          for (int j = 0; j < 8; ++j) *reinterpret_cast<float4*>(w[j]) = *reinterpret_cast<const float4*>(sb + col_of(j) * kKPitch + k0);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          float ak[4], bk[8];
          if constexpr (AKC) {
#pragma unroll
            for (int i = 0; i < 4; ++i) ak[i] = x[i][k];
          } else {
            *reinterpret_cast<float4*>(ak) = *reinterpret_cast<const float4*>(sa + (k0 + k) * kST + row_of(0));
          }
#pragma unroll
          for (int j = 0; j < 8; j += 4) {
            if constexpr (BKC) { bk[j] = w[j][k]; bk[j + 1] = w[j + 1][k]; bk[j + 2] = w[j + 2][k]; bk[j + 3] = w[j + 3][k]; }
            else *reinterpret_cast<float4*>(bk + j) = *reinterpret_cast<const float4*>(sb + (k0 + k) * kST + col_of(j));
          }
          unsigned long long bp[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) bp[j] = pack2(bk[2 * j], bk[2 * j + 1]);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const unsigned long long ap = pack2(ak[i], ak[i]);
#pragma unroll
            for (int j = 0; j < 4; ++j) fma2(acc[i][j], ap, bp[j]);
          }
        }
      }
      __syncwarp();              // the slice has been read
    }
  };
  if (P.a_quad && P.b_quad) run(std::true_type{}, std::true_type{});
  else if (P.a_quad) run(std::true_type{}, std::false_type{});
  else if (P.b_quad) run(std::false_type{}, std::true_type{});
  else run(std::false_type{}, std::false_type{});

  __syncthreads();               // every warp is done with its slices
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 8; j += 4) {
      float v[4];
      unpack2(acc[i][j / 2], v[0], v[1]);
      unpack2(acc[i][j / 2 + 1], v[2], v[3]);
      float* at = smem + (warp * kST + row_of(i)) * kPitch + col_of(j);
      if constexpr (BKC) {
#pragma unroll
        for (int e = 0; e < 4; ++e) at[e * 4] = v[e];
      } else {
        *reinterpret_cast<float4*>(at) = make_float4(v[0], v[1], v[2], v[3]);
      }
    }
  __syncthreads();
  if (!P.early) SBP_PDL_RELEASE();
  const int r = tid >> 3, c = (tid & 7) * 4;
  if (m0 + r >= M || n0 + c >= N) return;
  // Added in pairs, the pairs in pairs: three roundings of sums as large as a half, a quarter and all of the result, where one after
  // the other makes seven.  (Error against fp64, operands of one sign, 87 x 66 x 334: 5.5e-8 one after the other, 4.8e-8 in pairs, 5.0e-8 the tiled kernel.)
  float v[4], x[kSWarps][4];
#pragma unroll
  for (int w = 0; w < kSWarps; ++w) *reinterpret_cast<float4*>(x[w]) = *reinterpret_cast<const float4*>(smem + (w * kST + r) * kPitch + c);
#pragma unroll
  for (int e = 0; e < 4; ++e)
    v[e] = ((x[0][e] + x[1][e]) + (x[2][e] + x[3][e])) + ((x[4][e] + x[5][e]) + (x[6][e] + x[7][e]));
  if (p.gelu) {
#pragma unroll
    for (int e = 0; e < 4; ++e) v[e] = gelu_erf(v[e]);
  }
  const int n_out = (g == 0 ? p.n_rep : 0) + 1;
  for (int q = 0; q < n_out; ++q) {
    float* at = static_cast<float*>(q == 0 ? p.y[g] : p.y_rep[q - 1]) + (m0 + r) * p.ldy[g] + n0 + c;
    if (P.y_vec && n0 + c + 3 < N) {
      if (SBP_GUARD(at, 16)) *reinterpret_cast<float4*>(at) = make_float4(v[0], v[1], v[2], v[3]);
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (n0 + c + e < N && SBP_GUARD(at + e, 4)) at[e] = v[e];
    }
  }
}

cudaError_t launch_small(const F32Params& P, dim3 grid, cudaStream_t st) {
  switch ((P.plan.a_trans ? 2 : 0) | (P.plan.b_trans ? 1 : 0)) {
    case 0: return launch_dependent(matmul_f32_small_kernel<0, 0>, grid, dim3(32 * kSWarps), 0, st, P);
    case 1: return launch_dependent(matmul_f32_small_kernel<0, 1>, grid, dim3(32 * kSWarps), 0, st, P);
    case 2: return launch_dependent(matmul_f32_small_kernel<1, 0>, grid, dim3(32 * kSWarps), 0, st, P);
    default: return launch_dependent(matmul_f32_small_kernel<1, 1>, grid, dim3(32 * kSWarps), 0, st, P);
  }
}

bool aligned16(const void* p) { return reinterpret_cast<uintptr_t>(p) % 16 == 0; }

}  // namespace

// Test and measurement override of the choice below, and the launches of each kernel: [0] tiled, [1] small, [2] tensor cores.
static std::atomic<int> g_f32_form{SBP_F32_FORM_AUTO};
static std::atomic<unsigned long long> g_f32_launches[3];

void f32_set_form(int form) { g_f32_form.store(form, std::memory_order_relaxed); }
void f32_form_stats(unsigned long long out[3]) {
  for (int i = 0; i < 3; ++i) out[i] = g_f32_launches[i].load(std::memory_order_relaxed);
}
static void count_f32_launch(int form) {
  g_f32_launches[form - 1].fetch_add(1, std::memory_order_relaxed);
  count_launch();
}

// Defined in matmul_f32_tc.cu: the same product from bf16 parts on the tensor cores.
double f32_tc_cost(const MatmulPlan& plan, double limit, int* nb, int* splits);
sbp_status launch_matmul_f32_tc(const MatmulPlan& plan, int nb, int splits, cudaStream_t st);

sbp_status launch_matmul_f32(const MatmulPlan& plan, cudaStream_t st) {
  F32Params P;
  P.plan = plan;
  P.a_vec = P.b_vec = P.y_vec = 1;
  bool whole_k = true, whole_m = true, whole_n = true;
  long long iters = 0, mmax = 0, nmax = 0;
  for (int s = 0; s < plan.nseg; ++s) {
    if (!plan.chain && s >= plan.ngroups) continue;
    if (!aligned16(plan.a[s]) || plan.lda[s] % 4 != 0) P.a_vec = 0;
    if (!aligned16(plan.b[s]) || plan.ldb[s] % 4 != 0) P.b_vec = 0;
    if (plan.kseg[s] % 4 != 0) whole_k = false;
    const long long n = (plan.kseg[s] + kBK - 1) / kBK;
    iters = plan.chain ? iters + n : (n > iters ? n : iters);
  }
  for (int g = 0; g < plan.ngroups; ++g) {
    mmax = plan.m[g] > mmax ? plan.m[g] : mmax;
    nmax = plan.n[g] > nmax ? plan.n[g] : nmax;
    if (plan.m[g] % 4 != 0) whole_m = false;
    if (plan.n[g] % 4 != 0) whole_n = false;
    if (plan.a_trans && plan.row_off[g] % 4 != 0) P.a_vec = 0;
    if (!plan.b_trans && plan.col_off[g] % 4 != 0) P.b_vec = 0;
    if (!aligned16(plan.y[g]) || plan.ldy[g] % 4 != 0) P.y_vec = 0;
  }
  for (int q = 0; q < plan.n_rep; ++q)
    if (!aligned16(plan.y_rep[q])) P.y_vec = 0;
  P.a_quad = P.a_vec && (plan.a_trans ? whole_m : whole_k);
  P.b_quad = P.b_vec && (plan.b_trans ? whole_k : whole_n);
  if (mmax == 0 || nmax == 0) return SBP_OK;
  if (iters > 0x7fffffffLL) return fail(SBP_ERR_UNSUPPORTED, "contraction too long for one launch");

  // Which tile and how many CTAs per tile: the smallest estimated time, in clocks.  Measured per K-slice
  // of 16 (2048 clocks of the FMA pipe for a 128 x 128 tile, 512 for 64 x 64): the large tile takes 3590
  // clocks alone on its SM and 3170 each once two share one; the small one 1500 alone, 1230 each for two,
  // 1075 each from three.  A round of CTAs costs about 4000 clocks of launch and pipeline fill, a split
  // its exchange through distributed shared memory.  (us, this rule / the other choices: 1000 x 1500 x 777
  // on four shards 92 / 98-189, 700 x 2000 x 700 81 / 88-232, 100 x 2000 x 100 16 / 28-226.)
  const int sms = device_sms(), form = g_f32_form.load(std::memory_order_relaxed);
  int best_t = 0, best_s = 1;
  double best = 1e300, best_per_sm = 0;
  for (int t = 0; t < 2; ++t) {
    const int b = t == 0 ? 128 : 64;
    long long tiles = 0;
    for (int g = 0; g < plan.ngroups; ++g) tiles += ((plan.m[g] + b - 1) / b) * ((plan.n[g] + b - 1) / b);
    if ((mmax + b - 1) / b > 65535) continue;
    for (int s = 1; s <= 8; s *= 2) {
      if (s > 1 && iters < s) break;
      const double per_sm = (double)((tiles * s + sms - 1) / sms), resident = t == 0 ? 2 : 3;
      const double it = (double)((iters + s - 1) / s);
      const double each = t == 0 ? (per_sm > 1 ? 3170 : 3590) : (per_sm > 2 ? 1075 : (per_sm > 1 ? 1230 : 1500));
      const double exchange = s == 1 ? 0 : (t == 0 ? 4000 : 1000 + 450 * s);
      const double rounds = (double)(long long)((per_sm + resident - 1) / resident);
      const double cost = it * per_sm * each + rounds * (4000 + exchange);
      if (cost < best) { best = cost; best_per_sm = per_sm; best_t = t; best_s = s; }
    }
  }
  // Alone and in a row this kernel takes 0.5 us and a us for 1950 of those clocks (1680 where CTAs share an SM), 5 more with the
  // large tile, 6 % more off the 16-byte rule (rms 13 %).  Another kernel is taken only where it beats less than that, since
  // between kernels of another kind it loses part of what it gains alone: the small one against best / 1640, or 1.6 + best / 3125
  // where every CTA has an SM of its own, the tensor cores against best / 1750.  (1600 drawn products, alone and after a boxing op
  // of their operand: one of what these lines pick is over 4 % slower than this kernel, by 10 %; on the geometric mean it is 9 %
  // off the best of the three.  By the prices as they are it would be 4 % off, and 27 to 60 of the picks slower than this kernel, by up to 46 %.)
  //
  // The small kernel: 2.2 us and 1.25 a slice of a warp's, 0.45 more for an operand that comes element by element, CTAs that
  // share an SM 0.6 each, from seven on 1.6 us each (they no longer run at once: 1155 x 124 x 416 on three, ten an SM, 20.7 us, 17.2
  // here).  (us, this kernel / the small one: 64 x 96 x 80 on two shards 4.9 / 3.4, 40 x 98 x 640 5.0 / 3.4, 215 x 89 x 113 on
  // eight 5.2 / 3.8, 1031 x 325 x 228 on three 17.4 / 10.4, 722 x 258 x 99 on two 8.1 / 9.1, 32 x 512 x 32 6.3 / 7.2, 90 x 789 x 85
  // 10.0 / 12.4: a long contraction wants the cluster.  From four slices a warp on the switch has to win by a fifth, and with one
  // slice and CTAs that share an SM by 2.5 us: in a program of 133 x 620 x 622 x 187 on three the small kernel alone took
  // 9.4, this one 13.0, the program 26.4 and 24.9; one of 185 x 112 x 1082 x 100 on four took 29.9 with the small kernel's 272 CTAs
  // first, 27.2 without.)
  double beat_us = best_per_sm > 1 ? best / 1640 : 1.6 + best / 3125;
  const long long small_x = (nmax + kST - 1) / kST, small_y = (mmax + kST - 1) / kST;
  bool small = false;
  if (small_x <= 0x7fffffffLL && small_y <= 65535) {
    long long tiles = 0;
    for (int g = 0; g < plan.ngroups; ++g) tiles += ((plan.m[g] + kST - 1) / kST) * ((plan.n[g] + kST - 1) / kST);
    const double per_sm = (double)((tiles + sms - 1) / sms);
    const double slices = (double)((iters + kSWarps - 1) / kSWarps);
    double cost = 2.2 + slices * (1.25 + (P.a_quad ? 0 : 0.45) + (P.b_quad ? 0 : 0.45)) * (0.4 + 0.6 * per_sm);
    if (per_sm >= 7 && cost < 2.2 + 1.6 * slices * per_sm) cost = 2.2 + 1.6 * slices * per_sm;
    const bool wins = slices == 1 && per_sm > 1 ? cost + 2.5 < beat_us : cost < (slices > 3 ? 0.8 : 0.95) * beat_us;
    if (form == SBP_F32_FORM_AUTO ? wins : form == SBP_F32_FORM_SMALL) {
      small = true;
      P.early = 8 * tiles <= sms;
      beat_us = cost;
    }
  }
  // The tensor cores take it where their estimate (us) and 4 are below best / 1750, and the small kernel's estimate: alone the other kernel
  // wins earlier, but between kernels of another kind each of its launches waits some 5 us for whole SMs.  (us, this kernel / the
  // other, alone: 69 x 270 x 1639 on four shards 14.3 / 13.7, 187 x 1092 x 339 on four 17.9 / 14.6, 1170 x 256 x 808 on three 30 / 17,
  // 1000 x 1500 x 777 on four 92 / 38, 2048 x 2048 x 2048 422 / 153; programs of 116 x 1047 x 387 x 16 on three 24.8 / 27.3, 58 x 79 x
  // 1132 x 1272 on eight 28.4 / 30.7, 1809 x 26 x 1014 x 51 on three 59 / 53.)
  if (form == SBP_F32_FORM_AUTO ? best > 11000 : form == SBP_F32_FORM_TENSOR) {
    int nb = 0, splits = 1;
    const double limit = form != SBP_F32_FORM_AUTO ? 1e300 : (small && beat_us < best / 1750 ? beat_us : best / 1750) - 4;
    const double tc = f32_tc_cost(plan, limit, &nb, &splits);
    if (tc >= 0 && tc < limit) {
      const sbp_status status = launch_matmul_f32_tc(plan, nb, splits, st);
      if (status == SBP_OK) count_f32_launch(SBP_F32_FORM_TENSOR);
      return status;
    }
  }
  if (small) {
    SBP_BOUNDS_UPLOAD(st);
    const cudaError_t e = launch_small(P, dim3((unsigned)small_x, (unsigned)small_y, (unsigned)plan.ngroups), st);
    if (e != cudaSuccess) return cuda_fail(e, "matmul launch");
    count_f32_launch(SBP_F32_FORM_SMALL);
    return SBP_OK;
  }
  if (best == 1e300) return fail(SBP_ERR_UNSUPPORTED, "matrix too large for the FMA kernel");
  const int b = best_t == 0 ? 128 : 64;
  P.splits = best_s;
  const long long gx = (nmax + b - 1) / b * best_s;
  if (gx > 0x7fffffffLL) return fail(SBP_ERR_UNSUPPORTED, "matrix too large for the FMA kernel");
  const dim3 grid((unsigned)gx, (unsigned)((mmax + b - 1) / b), (unsigned)plan.ngroups);
  SBP_BOUNDS_UPLOAD(st);
  const cudaError_t e = best_t == 0 ? launch_stored<8, 8>(P, grid, st) : launch_stored<4, 4>(P, grid, st);
  if (e != cudaSuccess) return cuda_fail(e, "matmul launch");
  count_f32_launch(SBP_F32_FORM_TILED);
  return SBP_OK;
}

}  // namespace sbp
