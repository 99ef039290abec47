// Split-KV combine: merge per-split softmax-normalised partial outputs (bf16)
// and their log-sum-exps (fp32) into the full attention result.
//   m = max_s lse_s, c_s = exp(lse_s - m), out = sum_s c_s o_s / sum_s c_s,
//   lse = m + ln sum_s c_s.
// One warp per output row (b, h, i); each lane owns D/32 consecutive dims, so
// every partial row is read as one coalesced 128/256-byte segment; lane j
// holds the lse of splits j, j+32, ... Partials of splits without keys
// (lse = -inf) are never used. The weights and sums are fp32.
// Bound: the chain after the dependency wait. One memory round trip (lse and
// partial rows together), one reduction for the max, then the weights go round
// by shuffles in groups of eight splits, every lane summing them on the way. A
// pass with its combine: one sequence, 8B heads, 4096 tokens (17 splits) 10.3 ->
// 9.7 us, 16 / 4 heads, 1000 tokens (16 splits) 7.5 -> 6.6, against ten
// dependent shuffles for max and sum, all 32 shuffles at any split count and
// 64-bit row divisions after the wait.
#include <type_traits>

#include "nld_internal.cuh"

namespace nld {
namespace {

// Warp max of values that are never NaN: one reduction on keys in float order.
__device__ __forceinline__ float warp_max(float x) {
  const uint32_t b = __float_as_uint(x);
  const uint32_t k = __reduce_max_sync(0xffffffffu, (b >> 31) ? ~b : b | 0x80000000u);
  return __uint_as_float((k >> 31) ? k & 0x7fffffffu : ~k);
}

// Row `row` of R = B*Hq*bl rows (partial row order [B, Hq, bl]), row orow of the
// output [B, bl, Hq]; o_part [S, R, D] bf16, lse_part [S, R] (natural log).
// Warp-collective.
template <int D, int kRound>
__device__ __forceinline__ void merge_split_row(const __nv_bfloat16* __restrict__ o_part,
                                                const float* __restrict__ lse_part,
                                                int S, long R, long row, long orow,
                                                __nv_bfloat16* __restrict__ out, float* __restrict__ lse) {
  constexpr int V = D / 32;  // dims per lane (2 or 4)
  const int lane = threadIdx.x & 31;

  // One memory round trip per kRound splits: each lane loads its share of the
  // partial rows at the same time as the lse values.
  constexpr int kMaxPerLane = kMaxSplits / 32;
  const long split_stride = R * static_cast<long>(D);
  const __nv_bfloat16* base = o_part + row * D + lane * V;
  float ls[kMaxPerLane];
#pragma unroll
  for (int u = 0; u < kMaxPerLane; ++u) {
    const int s = lane + 32 * u;
    ls[u] = s < S ? __ldg(lse_part + static_cast<long>(s) * R + row) : -INFINITY;
  }
  uint32_t x[kRound][V / 2];  // bf16 pairs
  auto load_round = [&](int s0) {
#pragma unroll
    for (int u = 0; u < kRound; ++u) {
      const int s = s0 + u;
      if (s < S) {
        const __nv_bfloat16* op = base + s * split_stride;
        if constexpr (V == 4) {
          const uint2 t = __ldg(reinterpret_cast<const uint2*>(op));
          x[u][0] = t.x;
          x[u][1] = t.y;
        } else {
          x[u][0] = __ldg(reinterpret_cast<const unsigned int*>(op));
        }
      }
    }
  };
  load_round(0);
  float m = -INFINITY;
#pragma unroll
  for (int u = 0; u < kMaxPerLane; ++u) m = fmaxf(m, ls[u]);
  m = warp_max(m);

  float acc[V];
#pragma unroll
  for (int v = 0; v < V; ++v) acc[v] = 0.f;
  float csum = 0.f;
  if (m != -INFINITY) {
    const float m2 = m * kLog2e;
    float w[kMaxPerLane];  // weight of split lane + 32u; 0 for empty splits
#pragma unroll
    for (int u = 0; u < kMaxPerLane; ++u) {
      w[u] = ls[u] == -INFINITY ? 0.f : ex2(fmaf(ls[u], kLog2e, -m2));
    }
    for (int s0 = 0; s0 < S; s0 += kRound) {
      if (s0 > 0) load_round(s0);
      const int blk = s0 >> 5;  // warp-uniform
      const float wsrc = blk == 0 ? w[0] : blk == 1 ? w[1] : blk == 2 ? w[2] : w[3];
#pragma unroll
      for (int u8 = 0; u8 < kRound; u8 += 8) {
        if (s0 + u8 >= S) break;  // warp-uniform
#pragma unroll
        for (int u = u8; u < u8 + 8; ++u) {
          const float wu = __shfl_sync(0xffffffffu, wsrc, (s0 & 31) + u);  // 0 past S
          csum += wu;                                         // every lane takes the whole sum
          if (wu > 0.f) {
#pragma unroll
            for (int v = 0; v < V / 2; ++v) {
              float lo, hi;
              unpack_bf16(x[u][v], lo, hi);
              acc[2 * v] = fmaf(wu, lo, acc[2 * v]);
              acc[2 * v + 1] = fmaf(wu, hi, acc[2 * v + 1]);
            }
          }
        }
      }
    }
  }
  const float inv = csum > 0.f ? 1.f / csum : 0.f;
  __nv_bfloat16* o = out + orow * D + lane * V;
#pragma unroll
  for (int v = 0; v < V; v += 2)
    *reinterpret_cast<uint32_t*>(o + v) = pack_bf16(acc[v] * inv, acc[v + 1] * inv);
  if (lse != nullptr && lane == 0)
    lse[row] = csum > 0.f ? fmaf(lg2(csum), kLn2, m) : -INFINITY;
}


constexpr int kCombineWarps = 8;

template <int D, int kRound>
__global__ void __launch_bounds__(kCombineWarps * 32)
    combine_kernel(const __nv_bfloat16* __restrict__ o_part, const float* __restrict__ lse_part, int S, int B, int Hq,
                   int bl, __nv_bfloat16* __restrict__ out, float* __restrict__ lse) {
  grid_launch_dependents();  // dependents launch early; they wait on this grid themselves
  // The output row by 32-bit divisions, before the dependency wait (64-bit ones
  // behind it cost 0.2 us). R < 2^32: the partial rows alone are 128 R bytes.
  const long row = static_cast<long>(blockIdx.x) * kCombineWarps + (threadIdx.x >> 5);
  const long R = static_cast<long>(B) * Hq * bl;
  const uint32_t bh = static_cast<uint32_t>(row) / static_cast<uint32_t>(bl);
  const uint32_t i = static_cast<uint32_t>(row) - bh * static_cast<uint32_t>(bl);
  const uint32_t b = bh / static_cast<uint32_t>(Hq), h = bh - b * static_cast<uint32_t>(Hq);
  const long orow = (static_cast<long>(b) * bl + i) * Hq + h;
  grid_dependency_wait();
  if (row >= R) return;
  merge_split_row<D, kRound>(o_part, lse_part, S, R, row, orow, out, lse);
}

// The combine is bound by the rate at which an SM pulls partial rows from L2,
// so its CTAs should sit on as many SMs as possible, but the scheduler packs
// them. A dynamic shared-memory request (used for nothing) allows each SM no
// more CTAs than an even spread puts there, up to four, 1/(n+1) of an SM and a
// little each (measured at 17 partials x 512 rows, one CTA a SM: 3.0 -> 2.8 us;
// two to four a SM with rounds of 8 or 16 splits, whose registers leave room for
// them: 5 slots x 6144 rows, pass with its combine 47.6 -> 45.8 us, 9 x 2560
// 17.8 -> 17.4; without the spread the smaller kernels pack, 9 x 1280 12.1 ->
// 12.8). Larger grids launch without it.
constexpr int kMaxSpread = 4;
constexpr int spread_bytes(int per_sm) { return 227 * 1024 / (per_sm + 1) + 1024; }

template <int D, int kRound>
cudaError_t configure_combine(int dev) {
  static int configured[64] = {0};
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (!__atomic_load_n(&configured[dev], __ATOMIC_ACQUIRE)) {
    cudaError_t e =
        cudaFuncSetAttribute(combine_kernel<D, kRound>, cudaFuncAttributeMaxDynamicSharedMemorySize, spread_bytes(1));
    if (e != cudaSuccess) return e;
    __atomic_store_n(&configured[dev], 1, __ATOMIC_RELEASE);
  }
  return cudaSuccess;
}

template <int D, int kRound>
cudaError_t launch_combine_d(const __nv_bfloat16* o_part, const float* lse_part, int S, int B, int Hq, int bl,
                             __nv_bfloat16* out, float* lse, int sm_count, cudaStream_t stream) {
  const long R = static_cast<long>(B) * Hq * bl;
  const unsigned blocks = static_cast<unsigned>((R + kCombineWarps - 1) / kCombineWarps);
  size_t smem = 0;
  const int per_sm = static_cast<int>((blocks + sm_count - 1) / sm_count);
  if (per_sm <= kMaxSpread) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if ((e = configure_combine<D, kRound>(dev)) != cudaSuccess) return e;
    smem = spread_bytes(per_sm);
  }
  return launch_kernel(combine_kernel<D, kRound>, dim3(blocks), dim3(kCombineWarps * 32), smem, stream, o_part, lse_part, S,
                       B, Hq, bl, out, lse);
}

}  // namespace

cudaError_t launch_combine(const __nv_bfloat16* o_part, const float* lse_part, int S, int B, int Hq, int bl, int D,
                           __nv_bfloat16* out, float* lse, int sm_count, cudaStream_t stream) {
  auto go = [&](auto d) {
    constexpr int kD = decltype(d)::value;
    const long rows = static_cast<long>(B) * Hq * bl;
    const long blocks = (rows + kCombineWarps - 1) / kCombineWarps;
    if (S <= 8) return launch_combine_d<kD, 8>(o_part, lse_part, S, B, Hq, bl, out, lse, sm_count, stream);
    if (S <= 16 || blocks > 2l * sm_count)
      return launch_combine_d<kD, 16>(o_part, lse_part, S, B, Hq, bl, out, lse, sm_count, stream);
    return launch_combine_d<kD, 32>(o_part, lse_part, S, B, Hq, bl, out, lse, sm_count, stream);
  };
  return D == 128 ? go(std::integral_constant<int, 128>{}) : go(std::integral_constant<int, 64>{});
}

}  // namespace nld
