// Loads of a logits row's 16-byte vectors into a thread's registers, for the
// kernels that keep a piece of a row there. Nothing past `vocab` is read: the
// last row of a caller's buffer may end with its last logit. Plain index
// arithmetic around __ldg, so that a host compiler can run it as well.
#pragma once

#include <stdint.h>

namespace nld {

constexpr uint32_t kNegInf2 = 0xFF80FF80u;  // two bf16 -inf

// Row vectors v0 + t + j*THREADS < v1 into w, all loads in flight; -inf past
// v1 and past the vocabulary. The thread that holds a last vector the
// vocabulary does not fill loads its vocab % 8 logits one by one (the branch
// is on indices alone, so it waits for no load).
template <int THREADS, int VECS>
__device__ __forceinline__ void load_logit_vecs(const uint4* row, int v0, int v1, int t, int vocab, uint4 (&w)[VECS]) {
  const int nfull = vocab >> 3;
  const int end = v1 < nfull ? v1 : nfull;
#pragma unroll
  for (int j = 0; j < VECS; ++j) {
    const int v = v0 + t + j * THREADS;
    w[j] = v < end ? __ldg(row + v) : make_uint4(kNegInf2, kNegInf2, kNegInf2, kNegInf2);
  }
  if (v1 > nfull && v0 < v1 && (v1 - 1 - v0 - t) % THREADS == 0) {
    const unsigned short* tail = reinterpret_cast<const unsigned short*>(row + nfull);
    uint32_t q[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int left = vocab - nfull * 8 - 2 * e;  // logits from the pair's first on
      const uint32_t lo = left > 0 ? __ldg(tail + 2 * e) : kNegInf2 & 0xFFFFu;
      const uint32_t hi = left > 1 ? __ldg(tail + 2 * e + 1) : kNegInf2 & 0xFFFFu;
      q[e] = lo | hi << 16;
    }
#pragma unroll
    for (int j = 0; j < VECS; ++j)
      if (v0 + t + j * THREADS == nfull) w[j] = make_uint4(q[0], q[1], q[2], q[3]);
  }
}

}  // namespace nld
