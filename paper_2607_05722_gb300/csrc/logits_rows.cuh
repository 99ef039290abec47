// Loads of a logits row's 16-byte vectors into a thread's registers, for the
// kernels that keep a piece of a row there. Nothing past `vocab` is read: the
// last row of a caller's buffer may end with its last logit. Plain index
// arithmetic around __ldg, so that a host compiler can run it as well.
#pragma once

#include <stdint.h>

namespace nld {

constexpr uint32_t kNegInf2 = 0xFF80FF80u;  // two bf16 -inf

// Row vectors v0 + t + j*THREADS < v1 that the vocabulary fills into w, all
// loads in flight; -inf elsewhere.
template <int THREADS, int VECS>
__device__ __forceinline__ void load_logit_vecs(const uint4* row, int v0, int v1, int t, int vocab, uint4 (&w)[VECS]) {
  const int nfull = vocab >> 3;
  const int end = v1 < nfull ? v1 : nfull;
#pragma unroll
  for (int j = 0; j < VECS; ++j) {
    const int v = v0 + t + j * THREADS;
    w[j] = v < end ? __ldg(row + v) : make_uint4(kNegInf2, kNegInf2, kNegInf2, kNegInf2);
  }
}

// The last vector of a row where the vocabulary does not fill it: the thread
// that holds it loads its vocab % 8 logits, four, two and one at a time, and
// leaves -inf past them. Apart from the loads above, behind the last of them:
// the values meet in one register here, so a warp that gets here waits.
template <int THREADS, int VECS>
__device__ __forceinline__ void load_logit_tail(const uint4* row, int v0, int v1, int t, int vocab, uint4 (&w)[VECS]) {
  const int nfull = vocab >> 3, tail = vocab & 7;
  if (v0 < v1 && v1 > nfull && (v1 - 1 - v0 - t) % THREADS == 0) {
    const uint32_t* p = reinterpret_cast<const uint32_t*>(row + nfull);
    uint4 q = make_uint4(kNegInf2, kNegInf2, kNegInf2, kNegInf2);
    uint32_t pair = kNegInf2, one = kNegInf2;
    if (tail & 4) {
      const uint2 four = __ldg(reinterpret_cast<const uint2*>(p));
      q.x = four.x;
      q.y = four.y;
      p += 2;
    }
    if (tail & 2) pair = __ldg(p++);
    if (tail & 1) one = __ldg(reinterpret_cast<const unsigned short*>(p)) | (kNegInf2 & 0xFFFF0000u);
    const uint32_t first = (tail & 2) ? pair : one, second = (tail & 2) ? one : kNegInf2;
    if (tail & 4) {
      q.z = first;
      q.w = second;
    } else {
      q.x = first;
      q.y = second;
    }
#pragma unroll
    for (int j = 0; j < VECS; ++j)
      if (v0 + t + j * THREADS == nfull) w[j] = q;
  }
}

}  // namespace nld
