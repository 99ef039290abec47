// Logits -> (argmax id, confidence) per position: the inputs of the token
// decisions (Sec. 2 confidence-based sampling; Sec. 5 serial denoising
// commits the position with the highest peak probability).
//   m = max_v l_v, id = the lowest v with l_v = m,
//   conf = max_v softmax(l)_v = 1 / sum_v exp(l_v - m).
// A row is cut into `split` pieces, one CTA each (a thread-block cluster when
// split > 1). Pieces of at most 4096 vectors of 8 logits are kept in
// registers: every thread loads its vectors at once and folds them in one pass.
// Longer pieces stream: in a CTA one producer warp
// streams the piece through a ring of 16 KB stages with bulk copies (TMA
// engine) and eight warps fold each 8-logit vector into a running (max, sum
// of exp(l - max), argmax): the vector max comes first, so the rare rescale
// happens once per vector, then one exp per logit. The partial states merge
// by the log-sum-exp rule (ties: the lower index) across the warps, the CTA
// and, through distributed shared memory, the cluster. NaN logits never win
// the argmax and make the sum NaN; a row with nothing above -inf gets id 0
// and confidence 0.
#include <limits.h>

#include <type_traits>

#include "logits_rows.cuh"
#include "nld_internal.cuh"

namespace nld {
namespace {

constexpr int kLgConsumerWarps = 8;
constexpr int kLgThreads = 32 * (kLgConsumerWarps + 1);  // + the producer warp
constexpr int kLgStages = 4;
constexpr int kLgStageVecs = 1024;                       // 16-byte vectors (8 logits): 16 KB a stage
constexpr int kLgRingBytes = kLgStages * kLgStageVecs * 16;
constexpr int kLgSmemBytes = kLgRingBytes + 2 * kLgStages * 8 + 4 * 8 * 3 + 16 + 128;  // + alignment slack

// Merge (m2, s2, i2) into (m, s, i): the max, the sums rescaled to it, and
// the argmax (the lower index when the maxima are equal). A state whose max
// is still -inf has sum 0, or NaN if it met a NaN logit; it enters the merge
// as sum * 0, which keeps the NaN.
__device__ __forceinline__ void lg_merge(float& m, float& s, int& i, float m2, float s2, int i2) {
  const float mm = fmaxf(m, m2);
  i = m > m2 ? i : (m2 > m ? i2 : min(i, i2));
  const float a = m == -INFINITY ? s * 0.f : s * ex2((m - mm) * kLog2e);
  const float b = m2 == -INFINITY ? s2 * 0.f : s2 * ex2((m2 - mm) * kLog2e);
  m = mm;
  s = a + b;
}

// Fold x[0..n) (logits e0 .. e0+n-1, in index order) into (m, s, i).
template <int N>
__device__ __forceinline__ void lg_fold(const float (&x)[N], int e0, float& m, float& s, int& i) {
  float vm = x[0];
#pragma unroll
  for (int j = 1; j < N; ++j) vm = fmaxf(vm, x[j]);
  if (vm > m) {  // a new running max (NaN never is)
    s = m == -INFINITY ? s * 0.f : s * ex2((m - vm) * kLog2e);
    m = vm;
    int first = N - 1;
#pragma unroll
    for (int j = N - 1; j >= 0; --j)
      if (x[j] == vm) first = j;
    i = e0 + first;
  }
  if (m != -INFINITY) {
#pragma unroll
    for (int j = 0; j < N; ++j) s += ex2((x[j] - m) * kLog2e);  // a NaN logit makes s NaN
  } else {
#pragma unroll
    for (int j = 0; j < N; ++j)
      if (isnan(x[j])) s = NAN;  // nothing finite yet: the NaN must still reach the sum
  }
}

__global__ void __launch_bounds__(kLgThreads)
    logits_argmax_kernel(const __nv_bfloat16* __restrict__ logits, int vocab, long ld, int split,
                         int32_t* __restrict__ ids, float* __restrict__ conf, unsigned int* err) {
  extern __shared__ uint8_t lg_smem_raw[];
  uint8_t* ring = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(lg_smem_raw) + 127) & ~uintptr_t(127));
  uint64_t* full = reinterpret_cast<uint64_t*>(ring + kLgRingBytes);
  uint64_t* empty = full + kLgStages;
  float* red = reinterpret_cast<float*>(empty + kLgStages);  // [consumer warp][m, s, i]
  float* part = red + 3 * kLgConsumerWarps;                   // this CTA's merged state, for the cluster

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int piece = static_cast<int>(blockIdx.x % split);
  const long row = static_cast<long>(blockIdx.x / split);
  const int nvec = vocab >> 3, tail = vocab & 7;
  const int per = (nvec + split - 1) / split;
  const int v0 = min(nvec, piece * per), v1 = min(nvec, v0 + per);
  const int nst = (v1 - v0 + kLgStageVecs - 1) / kLgStageVecs;

  if (threadIdx.x == 0) {
    for (int st = 0; st < kLgStages; ++st) {
      mbar_init(&full[st], 1);
      mbar_init(&empty[st], kLgConsumerWarps);
    }
    fence_mbar_init();
  }
  __syncthreads();
  grid_launch_dependents();  // dependents launch early; they wait on this grid themselves
  grid_dependency_wait();    // the logits come from the previous kernel
  const uint8_t* grow = reinterpret_cast<const uint8_t*>(logits + row * ld);

  float m = -INFINITY, s = 0.f;
  int idx = 0;
  if (warp == kLgConsumerWarps) {
    // ---- producer: one lane issues the stages of this piece ----
    if (lane == 0) {
      int issued = 0;
      bool ok = true;
      for (int k = 0; k < nst; ++k) {
        const int st = k % kLgStages;
        if (k >= kLgStages && !mbar_wait(&empty[st], ((k / kLgStages) - 1) & 1, err)) {
          ok = false;
          break;
        }
        const uint32_t bytes = static_cast<uint32_t>(min(kLgStageVecs, v1 - v0 - k * kLgStageVecs)) * 16u;
        mbar_arrive_expect_tx(&full[st], bytes);
        bulk_load(ring + st * kLgStageVecs * 16, grow + static_cast<long>(v0 + k * kLgStageVecs) * 16, bytes,
                  &full[st]);
        issued = k + 1;
      }
      if (!ok) {
        // Gave up on a timeout: let the copies in flight land before exit (bounded).
        for (int k = max(0, issued - kLgStages); k < issued; ++k)
          mbar_wait(&full[k % kLgStages], (k / kLgStages) & 1, err);
      }
    }
  } else {
    // ---- consumers: thread t folds vectors t, t+256, ... of each stage ----
    const int t = threadIdx.x;
    for (int k = 0; k < nst; ++k) {
      const int st = k % kLgStages;
      if (!__all_sync(0xffffffffu, mbar_wait(&full[st], (k / kLgStages) & 1, err))) break;
      const int nv = min(kLgStageVecs, v1 - v0 - k * kLgStageVecs);
      const uint4* sv = reinterpret_cast<const uint4*>(ring + st * kLgStageVecs * 16);
      const int ebase = (v0 + k * kLgStageVecs) * 8;
      for (int j = t; j < nv; j += 32 * kLgConsumerWarps) {
        const uint4 w = sv[j];
        float x[8];
        unpack_bf16(w.x, x[0], x[1]);
        unpack_bf16(w.y, x[2], x[3]);
        unpack_bf16(w.z, x[4], x[5]);
        unpack_bf16(w.w, x[6], x[7]);
        lg_fold(x, ebase + j * 8, m, s, idx);
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&empty[st]);
    }
    if (piece == split - 1 && t < tail) {  // the last vocab % 8 logits, after every vector
      const uint16_t bits = reinterpret_cast<const uint16_t*>(grow)[nvec * 8 + t];
      const float x[1] = {__uint_as_float(static_cast<uint32_t>(bits) << 16)};
      lg_fold(x, nvec * 8 + t, m, s, idx);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      const float m2 = __shfl_xor_sync(0xffffffffu, m, off);
      const float s2 = __shfl_xor_sync(0xffffffffu, s, off);
      const int i2 = __shfl_xor_sync(0xffffffffu, idx, off);
      lg_merge(m, s, idx, m2, s2, i2);
    }
    if (lane == 0) {
      red[3 * warp] = m;
      red[3 * warp + 1] = s;
      red[3 * warp + 2] = __int_as_float(idx);
    }
  }
  __syncthreads();
  if (warp == 0) {
    m = lane < kLgConsumerWarps ? red[3 * lane] : -INFINITY;
    s = lane < kLgConsumerWarps ? red[3 * lane + 1] : 0.f;
    idx = lane < kLgConsumerWarps ? __float_as_int(red[3 * lane + 2]) : 0;
#pragma unroll
    for (int off = 4; off > 0; off >>= 1) {
      const float m2 = __shfl_xor_sync(0xffffffffu, m, off);
      const float s2 = __shfl_xor_sync(0xffffffffu, s, off);
      const int i2 = __shfl_xor_sync(0xffffffffu, idx, off);
      lg_merge(m, s, idx, m2, s2, i2);
    }
    if (lane == 0) {
      if (split == 1) {
        ids[row] = idx;
        conf[row] = m == -INFINITY ? 0.f : 1.f / s;
      } else {
        part[0] = m;
        part[1] = s;
        part[2] = __int_as_float(idx);
      }
    }
  }
  if (split > 1) {
    // Merge the pieces of the row: rank 0 reads every CTA's state through
    // distributed shared memory; the second barrier keeps the peers' shared
    // memory alive until it has.
    cluster_sync();
    if (cluster_ctarank() == 0 && warp == 0) {
      const uint32_t pa = smem_u32(part);
      m = -INFINITY;
      s = 0.f;
      idx = 0;
      if (lane < split) {
        m = ld_dsmem_f32(dsmem_addr(pa, lane));
        s = ld_dsmem_f32(dsmem_addr(pa + 4, lane));
        idx = __float_as_int(ld_dsmem_f32(dsmem_addr(pa + 8, lane)));
      }
#pragma unroll
      for (int off = 4; off > 0; off >>= 1) {
        const float m2 = __shfl_xor_sync(0xffffffffu, m, off);
        const float s2 = __shfl_xor_sync(0xffffffffu, s, off);
        const int i2 = __shfl_xor_sync(0xffffffffu, idx, off);
        lg_merge(m, s, idx, m2, s2, i2);
      }
      if (lane == 0) {
        ids[row] = idx;
        conf[row] = m == -INFINITY ? 0.f : 1.f / s;
      }
    }
    cluster_sync();
  }
}

// Pieces that fit in a CTA's registers (at most THREADS * VECS 8-logit
// vectors): no ring. Every thread loads all its vectors at once (one memory
// round trip); the logits' max is taken on packed bf16 pairs, then one exp
// per logit against the warp's max; the index of the max is searched only by
// the warps that hold the CTA's. The pieces of a row push their states into
// rank 0's shared memory with a remote store and a release arrival on rank
// 0's mbarrier, and rank 0 merges them, so no peer waits for another. Same
// rules as logits_argmax_kernel (ties to the lower index; NaN never wins and
// makes the sum NaN; nothing above -inf: id 0, conf 0).
// Bound: few rows, the chain load - exps - three merges; many rows,
// instruction issue (53% of the cycles at 512 rows x 131072, 7.3 instructions a
// logit) and CTAs
// that hold their slots through the merges, at 16 rows x 131072 3.6 us (a
// per-logit max and index search: 4.6), at 512 rows 25.9 us = 5.2 TB/s (the
// streaming kernel, one CTA a row: 34.7, its 512 CTAs being 1.1 waves), at
// 1024 rows 47 us = 5.7 TB/s (55). Measured and left out: clusters that stay
// and prefetch the next row's vectors (32 us at 512 rows: one chain per row),
// clusters that stream several rows through a ring (28.7 us), the exponent as
// one FMA against an integer reference (28.6 us: paired subtract and multiply
// take fewer issue slots).
constexpr int kLsMaxVecs = 8;  // vectors a thread holds in flight

__device__ __forceinline__ void cluster_arrive_relaxed() {
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void st_dsmem_f32(uint32_t addr, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}
__device__ __forceinline__ void mbar_arrive_remote_release(uint32_t addr) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(addr) : "memory");
}
// Wait (bounded) with acquire at cluster scope, for arrivals made by peers.
__device__ __forceinline__ bool mbar_wait_cluster(uint64_t* bar, uint32_t parity, unsigned int* err) {
  const uint64_t t0 = global_timer_ns();
  for (uint32_t it = 0;; ++it) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    if (ok) return true;
    if ((it & 255u) == 255u && global_timer_ns() - t0 > kWaitLimitNs) {
      atomicOr(err, NLD_DEVERR_WAIT_TIMEOUT);
      return false;
    }
  }
}

// Warp max of values that are never NaN.
__device__ __forceinline__ float warp_max(float x) {
  const int b = __float_as_int(x);
  const int k = __reduce_max_sync(0xffffffffu, b ^ ((b >> 31) & 0x7fffffff));  // signed order of the floats
  return __int_as_float(k ^ ((k >> 31) & 0x7fffffff));
}

// Merge the (m, s, i) states of a warp's lanes: the max, the sums rescaled to
// it, the lowest index holding it; every lane returns the merged state. m is
// never NaN; a state whose m is -inf has s 0, or NaN if it met a NaN logit.
__device__ __forceinline__ void lg_warp_merge(float& m, float& s, int& i) {
  const float mm = warp_max(m);
  if (m != -INFINITY) s *= ex2((m - mm) * kLog2e);
  i = static_cast<int>(__reduce_min_sync(0xffffffffu, static_cast<unsigned>(m == mm ? i : INT_MAX)));
  m = mm;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
}

// 8 logits of a vector as packed bf16 pairs: their max, per half.
__device__ __forceinline__ uint32_t bf16x2_max(uint32_t a, uint32_t b) {
  const __nv_bfloat162 r =
      __hmax2(*reinterpret_cast<const __nv_bfloat162*>(&a), *reinterpret_cast<const __nv_bfloat162*>(&b));
  return *reinterpret_cast<const uint32_t*>(&r);  // a NaN operand gives the other one
}
__device__ __forceinline__ uint32_t vec_max(uint4 w) { return bf16x2_max(bf16x2_max(w.x, w.y), bf16x2_max(w.z, w.w)); }

// acc += exp(x - m) over the 8 logits of w, m finite: a pair of logits takes
// two widenings, a paired subtract, multiply and add and two exponentials (4
// cycles of the MUFU pipe per warp instruction here).
__device__ __forceinline__ void add_exps(uint4 w, float m, float2& acc) {
  const uint32_t q[4] = {w.x, w.y, w.z, w.w};
  const float2 nm = make_float2(-m, -m), l2 = make_float2(kLog2e, kLog2e);
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    float2 x;
    unpack_bf16(q[j], x.x, x.y);
    x = mul2(add2(x, nm), l2);
    acc = add2(acc, make_float2(ex2(x.x), ex2(x.y)));
  }
}

// Position (from the first vector's start) of the first logit equal to m
// among vectors w (their per-half maxima in vm), vector j starting at j*STRIDE;
// some logit is m.
template <int STRIDE, int VECS>
__device__ __forceinline__ int first_of_max(const uint4 (&w)[VECS], const uint32_t (&vm)[VECS], float m) {
  int jb = 0;
  uint4 wb = w[0];
  float lo, hi;
#pragma unroll
  for (int j = VECS - 1; j >= 0; --j) {
    unpack_bf16(vm[j], lo, hi);
    if (lo == m || hi == m) {
      jb = j;
      wb = w[j];
    }
  }
  const uint32_t q[4] = {wb.x, wb.y, wb.z, wb.w};
  int e = 0;
#pragma unroll
  for (int j = 3; j >= 0; --j) {
    unpack_bf16(q[j], lo, hi);
    if (hi == m) e = 2 * j + 1;
    if (lo == m) e = 2 * j;
  }
  return jb * STRIDE + e;
}

template <int THREADS, int VECS, bool TAIL>
__global__ void __launch_bounds__(THREADS, 1024 / THREADS)
    logits_argmax_small_kernel(const __nv_bfloat16* __restrict__ logits, int vocab, long ld, int log2_split, int per,
                               int32_t* __restrict__ ids, float* __restrict__ conf, unsigned int* err) {
  constexpr int kW = THREADS / 32;
  __shared__ float red_m[kW], red_s[kW];
  __shared__ int first;          // the lowest index holding this CTA's max
  __shared__ float parts[8][3];  // rank 0: the pieces' (m, s, id)
  __shared__ __align__(8) uint64_t arrived;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, t = threadIdx.x;
  const int split = 1 << log2_split;
  const int piece = static_cast<int>(blockIdx.x) & (split - 1);
  const long row = static_cast<long>(blockIdx.x >> log2_split);
  const int nvec = (vocab + 7) >> 3;
  const int v0 = min(nvec, piece * per), v1 = min(nvec, v0 + per);
  if (t == 0) {
    first = INT_MAX;
    if (split > 1) {
      mbar_init(&arrived, static_cast<uint32_t>(split));
      fence_mbar_init();
    }
  }
  if (split > 1) cluster_arrive_relaxed();  // rank 0's barrier is ready once every CTA has arrived (waited below)
  grid_launch_dependents();                 // dependents launch early; they wait on this grid themselves
  grid_dependency_wait();                   // the logits come from the previous kernel
  const uint4* grow = reinterpret_cast<const uint4*>(logits + row * ld);
  uint4 w[VECS];
  load_logit_vecs<THREADS>(grow, v0, v1, t, vocab, w);
  if constexpr (TAIL) load_logit_tail<THREADS>(grow, v0, v1, t, vocab, w);
  // the max of this thread's logits (NaN is passed over), then of the warp's
  uint32_t vm[VECS];
  uint32_t pm = kNegInf2;
#pragma unroll
  for (int j = 0; j < VECS; ++j) {
    vm[j] = vec_max(w[j]);
    pm = bf16x2_max(pm, vm[j]);
  }
  float lo, hi;
  unpack_bf16(pm, lo, hi);
  const float mt = fmaxf(lo, hi);
  const float mw = warp_max(mt);
  // one exp per logit against the warp's max, so the lanes' sums just add
  float2 acc[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
  const float mref = mw == -INFINITY ? 0.f : mw;
#pragma unroll
  for (int j = 0; j < VECS; ++j) add_exps(w[j], mref, acc[j & 1]);
  float s = (acc[0].x + acc[0].y) + (acc[1].x + acc[1].y);
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
  if (lane == 0) {
    red_m[warp] = mw;
    red_s[warp] = s;
  }
  __syncthreads();
  // the CTA's max; its first index is searched only by the warps that hold it
  const float ml = lane < kW ? red_m[lane] : -INFINITY;
  const float m = warp_max(ml);
  if (mt == m && m != -INFINITY)
    atomicMin(&first, (v0 + t) * 8 + first_of_max<THREADS * 8>(w, vm, m));
  if (warp == 0) {
    s = lane < kW ? red_s[lane] : 0.f;
    if (ml != -INFINITY) s *= ex2((ml - m) * kLog2e);  // a warp without finite logits has sum 0 or NaN
#pragma unroll
    for (int off = kW / 2; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
  }
  __syncthreads();
  int idx = m == -INFINITY ? 0 : first;
  if (split == 1) {
    if (t == 0) {
      ids[row] = idx;
      conf[row] = m == -INFINITY ? 0.f : 1.f / s;
    }
    return;
  }
  cluster_wait();
  if (t == 0) {
    const uint32_t slot = dsmem_addr(smem_u32(&parts[piece][0]), 0);
    st_dsmem_f32(slot, m);
    st_dsmem_f32(slot + 4, s);
    st_dsmem_f32(slot + 8, __int_as_float(idx));
    mbar_arrive_remote_release(dsmem_addr(smem_u32(&arrived), 0));
  }
  if (piece == 0 && warp == 0) {
    bool ok = true;
    if (lane == 0) ok = mbar_wait_cluster(&arrived, 0, err);
    ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
    float mr = -INFINITY;
    s = 0.f;
    idx = 0;
    if (ok && lane < split) {
      mr = parts[lane][0];
      s = parts[lane][1];
      idx = __float_as_int(parts[lane][2]);
    }
    lg_warp_merge(mr, s, idx);
    if (lane == 0 && ok) {
      ids[row] = idx;
      conf[row] = mr == -INFINITY ? 0.f : 1.f / s;
    }
  }
}

// ---------------------------------------------------------------------------
// AR-diffusion ensemble verifier (appendix, verification with the ensemble):
// p = lambda softmax(ar) + (1 - lambda) softmax(diff); id = lowest argmax,
// conf = max p. Two passes over the row pair in one launch: the pieces of a
// row pair first fold both rows into (max, sum), merge them across the
// cluster (distributed shared memory), then re-read their pieces (now in L2)
// to evaluate p and keep its lowest-index maximum.
// ---------------------------------------------------------------------------

constexpr int kEnThreads = 256;

// (p, i) merge: the larger p, the lower index on ties.
__device__ __forceinline__ void en_merge(float& p, int& i, float p2, int i2) {
  if (p2 > p || (p2 == p && i2 < i)) {
    p = p2;
    i = i2;
  }
}

__global__ void __launch_bounds__(kEnThreads)
    ensemble_argmax_kernel(const __nv_bfloat16* __restrict__ ar, const __nv_bfloat16* __restrict__ diff, int vocab,
                           long ld, int split, float lambda, int32_t* __restrict__ ids, float* __restrict__ conf) {
  __shared__ float red[kEnThreads / 32][6];
  __shared__ float tot[4];  // rank 0: m_a, s_a, m_b, s_b of the row pair
  __shared__ float best[2];  // this CTA's (p, index)
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, t = threadIdx.x;
  const int piece = static_cast<int>(blockIdx.x % split);
  const long row = static_cast<long>(blockIdx.x / split);
  const int nvec = vocab >> 3, tail = vocab & 7;
  const int per = (nvec + split - 1) / split;
  const int v0 = min(nvec, piece * per), v1 = min(nvec, v0 + per);
  const bool has_tail = piece == split - 1 && t < tail;
  grid_launch_dependents();
  grid_dependency_wait();  // the logits come from earlier kernels
  const uint4* ra = reinterpret_cast<const uint4*>(ar + row * ld);
  const uint4* rb = reinterpret_cast<const uint4*>(diff + row * ld);
  const uint16_t* ta = reinterpret_cast<const uint16_t*>(ar + row * ld) + nvec * 8;
  const uint16_t* tb = reinterpret_cast<const uint16_t*>(diff + row * ld) + nvec * 8;

  // ---- pass 1: (max, sum) of each row over this piece ----
  float ma = -INFINITY, sa = 0.f, mb = -INFINITY, sb = 0.f;
  int ia = 0, ib = 0;
  for (int v = v0 + t; v < v1; v += kEnThreads) {
    const uint4 wa = __ldg(ra + v), wb = __ldg(rb + v);
    float xa[8], xb[8];
    unpack_bf16(wa.x, xa[0], xa[1]); unpack_bf16(wa.y, xa[2], xa[3]);
    unpack_bf16(wa.z, xa[4], xa[5]); unpack_bf16(wa.w, xa[6], xa[7]);
    unpack_bf16(wb.x, xb[0], xb[1]); unpack_bf16(wb.y, xb[2], xb[3]);
    unpack_bf16(wb.z, xb[4], xb[5]); unpack_bf16(wb.w, xb[6], xb[7]);
    lg_fold(xa, v * 8, ma, sa, ia);
    lg_fold(xb, v * 8, mb, sb, ib);
  }
  if (has_tail) {
    const float xa[1] = {__uint_as_float(static_cast<uint32_t>(ta[t]) << 16)};
    const float xb[1] = {__uint_as_float(static_cast<uint32_t>(tb[t]) << 16)};
    lg_fold(xa, nvec * 8 + t, ma, sa, ia);
    lg_fold(xb, nvec * 8 + t, mb, sb, ib);
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    lg_merge(ma, sa, ia, __shfl_xor_sync(0xffffffffu, ma, off), __shfl_xor_sync(0xffffffffu, sa, off),
             __shfl_xor_sync(0xffffffffu, ia, off));
    lg_merge(mb, sb, ib, __shfl_xor_sync(0xffffffffu, mb, off), __shfl_xor_sync(0xffffffffu, sb, off),
             __shfl_xor_sync(0xffffffffu, ib, off));
  }
  if (lane == 0) {
    red[warp][0] = ma; red[warp][1] = sa; red[warp][2] = mb; red[warp][3] = sb;
  }
  __syncthreads();
  if (warp == 0) {
    ma = lane < kEnThreads / 32 ? red[lane][0] : -INFINITY;
    sa = lane < kEnThreads / 32 ? red[lane][1] : 0.f;
    mb = lane < kEnThreads / 32 ? red[lane][2] : -INFINITY;
    sb = lane < kEnThreads / 32 ? red[lane][3] : 0.f;
#pragma unroll
    for (int off = 4; off > 0; off >>= 1) {
      lg_merge(ma, sa, ia, __shfl_xor_sync(0xffffffffu, ma, off), __shfl_xor_sync(0xffffffffu, sa, off), 0);
      lg_merge(mb, sb, ib, __shfl_xor_sync(0xffffffffu, mb, off), __shfl_xor_sync(0xffffffffu, sb, off), 0);
    }
    if (lane == 0) {
      tot[0] = ma; tot[1] = sa; tot[2] = mb; tot[3] = sb;
    }
  }
  if (split > 1) {
    cluster_sync();  // every piece's (max, sum) is in its shared memory
    if (cluster_ctarank() == 0 && warp == 0) {
      const uint32_t base = smem_u32(tot);
      ma = -INFINITY; sa = 0.f; mb = -INFINITY; sb = 0.f;
      if (lane < split) {
        ma = ld_dsmem_f32(dsmem_addr(base, lane));
        sa = ld_dsmem_f32(dsmem_addr(base + 4, lane));
        mb = ld_dsmem_f32(dsmem_addr(base + 8, lane));
        sb = ld_dsmem_f32(dsmem_addr(base + 12, lane));
      }
#pragma unroll
      for (int off = 4; off > 0; off >>= 1) {
        lg_merge(ma, sa, ia, __shfl_xor_sync(0xffffffffu, ma, off), __shfl_xor_sync(0xffffffffu, sa, off), 0);
        lg_merge(mb, sb, ib, __shfl_xor_sync(0xffffffffu, mb, off), __shfl_xor_sync(0xffffffffu, sb, off), 0);
      }
    }
    cluster_sync();  // every rank has read the pieces' states before rank 0 overwrites its own
    if (cluster_ctarank() == 0 && threadIdx.x == 0) {
      tot[0] = ma; tot[1] = sa; tot[2] = mb; tot[3] = sb;
    }
    cluster_sync();  // the row pair's totals are in rank 0's shared memory
    const uint32_t base0 = dsmem_addr(smem_u32(tot), 0);
    ma = ld_dsmem_f32(base0);
    sa = ld_dsmem_f32(base0 + 4);
    mb = ld_dsmem_f32(base0 + 8);
    sb = ld_dsmem_f32(base0 + 12);
  } else {
    __syncthreads();
    ma = tot[0]; sa = tot[1]; mb = tot[2]; sb = tot[3];
  }
  // An empty distribution (max -inf) gets weight 0 and a stand-in max of 0,
  // so its terms are exp(-inf) * 0 = 0.
  const float ca = ma == -INFINITY ? 0.f : lambda / sa;
  const float cb = mb == -INFINITY ? 0.f : (1.f - lambda) / sb;
  const float ma2 = (ma == -INFINITY ? 0.f : ma) * kLog2e;
  const float mb2 = (mb == -INFINITY ? 0.f : mb) * kLog2e;

  // ---- pass 2: p over this piece (re-read, now in L2), lowest-index max ----
  float pbest = -1.f;
  int ibest = 0;
  for (int v = v0 + t; v < v1; v += kEnThreads) {
    const uint4 wa = __ldg(ra + v), wb = __ldg(rb + v);
    float xa[8], xb[8];
    unpack_bf16(wa.x, xa[0], xa[1]); unpack_bf16(wa.y, xa[2], xa[3]);
    unpack_bf16(wa.z, xa[4], xa[5]); unpack_bf16(wa.w, xa[6], xa[7]);
    unpack_bf16(wb.x, xb[0], xb[1]); unpack_bf16(wb.y, xb[2], xb[3]);
    unpack_bf16(wb.z, xb[4], xb[5]); unpack_bf16(wb.w, xb[6], xb[7]);
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const float p = ca * ex2(fmaf(xa[j], kLog2e, -ma2)) + cb * ex2(fmaf(xb[j], kLog2e, -mb2));
      if (p > pbest) {
        pbest = p;
        ibest = v * 8 + j;
      }
    }
  }
  if (has_tail) {
    const float a = __uint_as_float(static_cast<uint32_t>(ta[t]) << 16);
    const float b = __uint_as_float(static_cast<uint32_t>(tb[t]) << 16);
    const float p = ca * ex2(fmaf(a, kLog2e, -ma2)) + cb * ex2(fmaf(b, kLog2e, -mb2));
    if (p > pbest) {
      pbest = p;
      ibest = nvec * 8 + t;
    }
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1)
    en_merge(pbest, ibest, __shfl_xor_sync(0xffffffffu, pbest, off), __shfl_xor_sync(0xffffffffu, ibest, off));
  if (lane == 0) {
    red[warp][4] = pbest;
    red[warp][5] = __int_as_float(ibest);
  }
  __syncthreads();
  if (warp == 0) {
    pbest = lane < kEnThreads / 32 ? red[lane][4] : -1.f;
    ibest = lane < kEnThreads / 32 ? __float_as_int(red[lane][5]) : 0;
#pragma unroll
    for (int off = 4; off > 0; off >>= 1)
      en_merge(pbest, ibest, __shfl_xor_sync(0xffffffffu, pbest, off), __shfl_xor_sync(0xffffffffu, ibest, off));
    if (lane == 0) {
      best[0] = pbest;
      best[1] = __int_as_float(ibest);
    }
  }
  if (split > 1) {
    cluster_sync();
    if (cluster_ctarank() == 0 && warp == 0) {
      const uint32_t base = smem_u32(best);
      pbest = -1.f;
      ibest = 0;
      if (lane < split) {
        pbest = ld_dsmem_f32(dsmem_addr(base, lane));
        ibest = __float_as_int(ld_dsmem_f32(dsmem_addr(base + 4, lane)));
      }
#pragma unroll
      for (int off = 4; off > 0; off >>= 1)
        en_merge(pbest, ibest, __shfl_xor_sync(0xffffffffu, pbest, off), __shfl_xor_sync(0xffffffffu, ibest, off));
      if (lane == 0) {
        ids[row] = ibest;
        conf[row] = pbest;
      }
    }
    cluster_sync();  // the peers keep their shared memory until rank 0 has read it
  } else if (threadIdx.x == 0) {
    ids[row] = ibest;
    conf[row] = pbest;
  }
}

// The same for pieces that fit in a CTA's registers (both rows' vectors of a
// thread, VECS each): the logits are read once. Pass 1 as in
// logits_argmax_small_kernel; each piece pushes its (max, sum) pairs to every
// CTA of the cluster (remote stores, release arrivals), so the totals take
// one hop; pass 2 evaluates p only where it can be the maximum. With
// ca = lambda / sum_a, cb = (1 - lambda) / sum_b, the largest p is at least
// c = max(ca, cb), its value at that row's own maximum, so a vector whose
// terms ca exp(a - max_a) and cb exp(b - max_b) all lie below 0.49 c cannot
// hold it: two compares of a vector's maxima decide.
// Bound by the chain load - sums - exchange - best, during which a CTA holds
// its registers (ncu at 160 row pairs: 43% of issue cycles, waits at CTA
// barriers first): 160 x 100003 25.1 us (reading both rows twice, with two
// exponentials a logit each time: 54.6, both with the logits in L2), 16 x 131072
// 5.8 us (12.7), 512 x 131072 72 us (132).
template <int THREADS, int VECS, bool TAIL>
__global__ void __launch_bounds__(THREADS, VECS <= 4 ? 1024 / THREADS : 1)
    ensemble_argmax_small_kernel(const __nv_bfloat16* __restrict__ ar, const __nv_bfloat16* __restrict__ diff,
                                 int vocab, long ld, int log2_split, int per, float lambda, int32_t* __restrict__ ids,
                                 float* __restrict__ conf, unsigned int* err) {
  constexpr int kW = THREADS / 32;
  __shared__ float red[kW][4];       // the warps' m_a, s_a, m_b, s_b, then their (p, index)
  __shared__ float totals[8][4];     // the pieces' m_a, s_a, m_b, s_b
  __shared__ float whole[4];         // the row pair's
  __shared__ float best[8][2];       // rank 0: the pieces' (p, index)
  __shared__ __align__(8) uint64_t have_totals, have_best;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, t = threadIdx.x;
  const int split = 1 << log2_split;
  const int piece = static_cast<int>(blockIdx.x) & (split - 1);
  const long row = static_cast<long>(blockIdx.x >> log2_split);
  const int nvec = (vocab + 7) >> 3;
  const int v0 = min(nvec, piece * per), v1 = min(nvec, v0 + per);
  if (split > 1) {
    if (t == 0) {
      mbar_init(&have_totals, static_cast<uint32_t>(split));
      mbar_init(&have_best, static_cast<uint32_t>(split));
      fence_mbar_init();
    }
    cluster_arrive_relaxed();  // the barriers are ready once every CTA has arrived (waited below)
  }
  grid_launch_dependents();
  grid_dependency_wait();  // the logits come from earlier kernels
  uint4 wa[VECS], wb[VECS];
  const uint4* ga = reinterpret_cast<const uint4*>(ar + row * ld);
  const uint4* gb = reinterpret_cast<const uint4*>(diff + row * ld);
  load_logit_vecs<THREADS>(ga, v0, v1, t, vocab, wa);
  load_logit_vecs<THREADS>(gb, v0, v1, t, vocab, wb);

  // ---- pass 1: (max, sum) of each row over this piece ----
  auto fold = [&](const uint4* row_vecs, uint4(&w)[VECS], float& m, float& s) {
    if constexpr (TAIL) load_logit_tail<THREADS>(row_vecs, v0, v1, t, vocab, w);
    uint32_t pm = kNegInf2;
#pragma unroll
    for (int j = 0; j < VECS; ++j) pm = bf16x2_max(pm, vec_max(w[j]));
    float lo, hi;
    unpack_bf16(pm, lo, hi);
    m = warp_max(fmaxf(lo, hi));
    s = 0.f;
    // A warp past the piece has no sum to take. The branch also keeps the second
    // row's maxima behind the first row's exponentials (512 x 262144: 180 us
    // without it, 172 with).
    if (m == -INFINITY && v0 + warp * 32 >= v1) return;
    float2 acc[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
    const float mref = m == -INFINITY ? 0.f : m;
#pragma unroll
    for (int j = 0; j < VECS; ++j) add_exps(w[j], mref, acc[j & 1]);
    s = (acc[0].x + acc[0].y) + (acc[1].x + acc[1].y);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
  };
  // the lanes' states of one row merged: the max, and the sum rescaled to it
  auto merge = [](float& m, float& s) {
    const float mm = warp_max(m);
    if (m != -INFINITY) s *= ex2((m - mm) * kLog2e);
    m = mm;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
  };
  float ma, sa, mb, sb;
  fold(ga, wa, ma, sa);
  fold(gb, wb, mb, sb);
  if (lane == 0) {
    red[warp][0] = ma; red[warp][1] = sa; red[warp][2] = mb; red[warp][3] = sb;
  }
  __syncthreads();
  bool ok = true;
  if (split > 1) cluster_wait();
  if (warp == 0) {
    ma = lane < kW ? red[lane][0] : -INFINITY;
    sa = lane < kW ? red[lane][1] : 0.f;
    mb = lane < kW ? red[lane][2] : -INFINITY;
    sb = lane < kW ? red[lane][3] : 0.f;
    merge(ma, sa);
    merge(mb, sb);
    if (split > 1) {
      if (lane < split) {  // to every CTA of the cluster
        const uint32_t slot = dsmem_addr(smem_u32(&totals[piece][0]), lane);
        st_dsmem_f32(slot, ma);
        st_dsmem_f32(slot + 4, sa);
        st_dsmem_f32(slot + 8, mb);
        st_dsmem_f32(slot + 12, sb);
        mbar_arrive_remote_release(dsmem_addr(smem_u32(&have_totals), lane));
      }
      __syncwarp();
      if (lane == 0) ok = mbar_wait_cluster(&have_totals, 0, err);
      ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
      ma = -INFINITY; sa = 0.f; mb = -INFINITY; sb = 0.f;
      if (ok && lane < split) {
        ma = totals[lane][0]; sa = totals[lane][1]; mb = totals[lane][2]; sb = totals[lane][3];
      }
      merge(ma, sa);
      merge(mb, sb);
    }
    if (lane == 0) {
      whole[0] = ma; whole[1] = sa; whole[2] = mb; whole[3] = sb;
    }
  }
  __syncthreads();
  ma = whole[0]; sa = whole[1]; mb = whole[2]; sb = whole[3];
  // An empty distribution (max -inf) gets weight 0 and a stand-in max of 0,
  // so its terms are exp(-inf) * 0 = 0.
  const float ca = ma == -INFINITY ? 0.f : lambda / sa;
  const float cb = mb == -INFINITY ? 0.f : (1.f - lambda) / sb;
  ma = ma == -INFINITY ? 0.f : ma;
  mb = mb == -INFINITY ? 0.f : mb;

  // ---- pass 2: the lowest-index maximum of p over this piece ----
  const float c = 0.49f * fmaxf(ca, cb);
  const float da = lg2(c / ca) * kLn2, db = lg2(c / cb) * kLn2;  // NaN when both rows are empty: every vector is taken
  float pbest = -1.f;
  int ibest = 0;
  unsigned take = 0;
#pragma unroll
  for (int j = 0; j < VECS; ++j) {
    float lo, hi;
    unpack_bf16(vec_max(wa[j]), lo, hi);
    const float xa = fmaxf(lo, hi);
    unpack_bf16(vec_max(wb[j]), lo, hi);
    const float xb = fmaxf(lo, hi);
    if (!(xa - ma < da && xb - mb < db)) take |= 1u << j;
  }
#pragma unroll 1
  for (; take != 0; take &= take - 1) {  // few vectors, in index order
    const int jt = __ffs(take) - 1;
    uint4 va = wa[0], vb = wb[0];
#pragma unroll
    for (int j = 1; j < VECS; ++j)
      if (j == jt) {
        va = wa[j];
        vb = wb[j];
      }
    const uint32_t qa[4] = {va.x, va.y, va.z, va.w}, qb[4] = {vb.x, vb.y, vb.z, vb.w};
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const uint32_t ba = qa[e >> 1], bb = qb[e >> 1];
      const float a = __uint_as_float((e & 1) ? ba & 0xFFFF0000u : ba << 16);
      const float b = __uint_as_float((e & 1) ? bb & 0xFFFF0000u : bb << 16);
      const float p = ca * ex2((a - ma) * kLog2e) + cb * ex2((b - mb) * kLog2e);
      if (p > pbest) {
        pbest = p;
        ibest = (v0 + t + jt * THREADS) * 8 + e;
      }
    }
  }
  // the lanes' best: the largest p, its lowest index
  auto best_of = [](float& p, int& i) {
    const float pp = warp_max(p);
    i = static_cast<int>(__reduce_min_sync(0xffffffffu, static_cast<unsigned>(p == pp ? i : INT_MAX)));
    p = pp;
  };
  best_of(pbest, ibest);
  if (lane == 0) {
    red[warp][0] = pbest;
    red[warp][1] = __int_as_float(ibest);
  }
  __syncthreads();
  if (warp != 0) return;
  pbest = lane < kW ? red[lane][0] : -1.f;
  ibest = lane < kW ? __float_as_int(red[lane][1]) : 0;
  best_of(pbest, ibest);
  if (split > 1) {
    if (lane == 0) {
      const uint32_t slot = dsmem_addr(smem_u32(&best[piece][0]), 0);
      st_dsmem_f32(slot, pbest);
      st_dsmem_f32(slot + 4, __int_as_float(ibest));
      mbar_arrive_remote_release(dsmem_addr(smem_u32(&have_best), 0));
    }
    if (piece != 0) return;
    __syncwarp();
    bool got = true;
    if (lane == 0) got = mbar_wait_cluster(&have_best, 0, err);
    ok = ok && __shfl_sync(0xffffffffu, got ? 1 : 0, 0) != 0;
    pbest = -1.f;
    ibest = 0;
    if (ok && lane < split) {
      pbest = best[lane][0];
      ibest = __float_as_int(best[lane][1]);
    }
    best_of(pbest, ibest);
  }
  if (lane == 0 && ok) {
    ids[row] = ibest;
    conf[row] = pbest;
  }
}

}  // namespace

namespace {
// launch(THREADS, VECS) with the fewest vectors a thread that hold a piece:
// slots past the piece are filler whose exponentials cost as much as a logit's
// (1000 rows x 1000: 125 vectors in 2048 slots 12.4 us, in 256 slots 7.8; 1000
// x 40000: 1250 in 2048 48.0 us, in 1280 43.8). A test of each slot instead
// costs full pieces 3 to 6%.
template <int THREADS, int VECS, int MAX, typename Launch>
cudaError_t with_vecs(long piece_vecs, Launch launch) {
  if constexpr (VECS < MAX) {
    if (piece_vecs > THREADS * VECS) return with_vecs<THREADS, VECS + 1, MAX>(piece_vecs, launch);
  }
  return launch(std::integral_constant<int, THREADS>{}, std::integral_constant<int, VECS>{});
}
}  // namespace

int logits_split_vectors() { return kLgStageVecs; }
int logits_piece_limit() { return 512 * kLsMaxVecs; }

cudaError_t launch_ensemble_argmax(const __nv_bfloat16* ar, const __nv_bfloat16* diff, int rows, int vocab, long ld,
                                   int split, float lambda, int32_t* ids, float* conf, unsigned int* err,
                                   cudaStream_t stream) {
  const bool stream_rows = split == 0;  // whole rows, read twice, whatever their length
  if (stream_rows) split = 1;
  const dim3 grid(static_cast<unsigned>(static_cast<long>(rows) * split));
  const long piece_vecs = ((static_cast<long>(vocab) + 7) / 8 + split - 1) / split;
  const int log2_split = __builtin_ctz(static_cast<unsigned>(split)), per = static_cast<int>(piece_vecs);
  auto in_registers = [&](auto threads, auto vecs) {
    constexpr int kT = decltype(threads)::value, kV = decltype(vecs)::value;
    auto* kernel = vocab % 8 ? ensemble_argmax_small_kernel<kT, kV, true> : ensemble_argmax_small_kernel<kT, kV, false>;
    return launch_kernel_cluster(kernel, grid, dim3(kT), 0, stream, split, ar, diff,
                                 vocab, ld, log2_split, per, lambda, ids, conf, err);
  };
  if (stream_rows)
    return launch_kernel_cluster(ensemble_argmax_kernel, grid, dim3(kEnThreads), 0, stream, split, ar, diff, vocab, ld,
                                 split, lambda, ids, conf);
  if (piece_vecs <= 256 * 4) return with_vecs<256, 1, 4>(piece_vecs, in_registers);
  if (piece_vecs <= 512 * kLsMaxVecs) return with_vecs<512, 3, kLsMaxVecs>(piece_vecs, in_registers);
  return launch_kernel_cluster(ensemble_argmax_kernel, grid, dim3(kEnThreads), 0, stream, split, ar, diff, vocab, ld,
                               split, lambda, ids, conf);
}

cudaError_t launch_logits_argmax(const __nv_bfloat16* logits, int rows, int vocab, long ld, int split, int32_t* ids,
                                 float* conf, unsigned int* err, cudaStream_t stream) {
  static int configured[64] = {0};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (!__atomic_load_n(&configured[dev], __ATOMIC_ACQUIRE)) {
    e = cudaFuncSetAttribute(logits_argmax_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kLgSmemBytes);
    if (e != cudaSuccess) return e;
    __atomic_store_n(&configured[dev], 1, __ATOMIC_RELEASE);
  }
  const dim3 grid(static_cast<unsigned>(static_cast<long>(rows) * split));
  const long piece_vecs = ((static_cast<long>(vocab) + 7) / 8 + split - 1) / split;
  const int log2_split = __builtin_ctz(static_cast<unsigned>(split));
  auto in_registers = [&](auto threads, auto vecs) {
    constexpr int kT = decltype(threads)::value, kV = decltype(vecs)::value;
    auto* kernel = vocab % 8 ? logits_argmax_small_kernel<kT, kV, true> : logits_argmax_small_kernel<kT, kV, false>;
    return launch_kernel_cluster(kernel, grid, dim3(kT), 0, stream, split, logits, vocab, ld,
                                 log2_split, static_cast<int>(piece_vecs), ids, conf, err);
  };
  if (piece_vecs <= 256L * kLsMaxVecs) return with_vecs<256, 1, kLsMaxVecs>(piece_vecs, in_registers);
  if (piece_vecs <= 512L * kLsMaxVecs) return with_vecs<512, 5, kLsMaxVecs>(piece_vecs, in_registers);
  return launch_kernel_cluster(logits_argmax_kernel, grid, dim3(kLgThreads), kLgSmemBytes, stream, split, logits,
                               vocab, ld, split, ids, conf, err);
}

}  // namespace nld
