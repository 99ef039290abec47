"""What the register logits kernels read of a row, on the host: their load
routine (csrc/logits_rows.cuh) compiled by the C++ compiler, with an __ldg
that records every address, over all threads and pieces of a row."""
import shutil
import subprocess

import pytest

from paper_2607_05722_gb300 import build as B

HARNESS = r"""
#include <stdint.h>
#include <stdio.h>
#include <stdlib.h>
#include <vector>
#define __device__
#define __forceinline__ inline
struct alignas(8) uint2 { uint32_t x, y; };
struct alignas(16) uint4 { uint32_t x, y, z, w; };
static uint4 make_uint4(uint32_t x, uint32_t y, uint32_t z, uint32_t w) { return uint4{x, y, z, w}; }
static std::vector<int> reads;  // per 16-bit entry of the row
static const char* base;
static long bad;                // reads past the last entry
template <typename T> static T __ldg(const T* p) {
  const long e = ((const char*)p - base) / 2;
  for (long i = e; i < e + (long)(sizeof(T) / 2); ++i) {
    if (i < 0 || i >= (long)reads.size()) ++bad; else ++reads[i];
  }
  return *p;
}
#include "logits_rows.cuh"
template <int THREADS, int VECS> static int check(int vocab, int split) {
  const int nvec = (vocab + 7) / 8, per = (nvec + split - 1) / split;
  if (per > THREADS * VECS) return 0;
  std::vector<uint4> row(nvec + 1);  // room behind the row, so that a read past it can be counted
  uint16_t* x = (uint16_t*)row.data();
  for (int i = 0; i < nvec * 8 + 8; ++i) x[i] = i < vocab ? (uint16_t)(i * 7 + 3) : 0x7F7F;  // behind it: the largest bf16
  base = (const char*)x;
  reads.assign(vocab, 0);
  bad = 0;
  int wrong = 0;
  for (int piece = 0; piece < split; ++piece) {
    const int v0 = nvec < piece * per ? nvec : piece * per, v1 = nvec < v0 + per ? nvec : v0 + per;
    for (int t = 0; t < THREADS; ++t) {
      uint4 w[VECS];
      nld::load_logit_vecs<THREADS>(row.data(), v0, v1, t, vocab, w);
      nld::load_logit_tail<THREADS>(row.data(), v0, v1, t, vocab, w);
      for (int j = 0; j < VECS; ++j)
        for (int e = 0; e < 8; ++e) {
          const long v = v0 + t + (long)j * THREADS, i = v * 8 + e;
          const uint16_t want = v < v1 && i < vocab ? x[i] : 0xFF80;
          wrong += ((const uint16_t*)&w[j])[e] != want;
        }
    }
  }
  for (int n : reads) wrong += n != 1;
  if (bad || wrong) printf("vocab %d split %d threads %d vecs %d: %ld reads past the row, %d wrong\n", vocab, split, THREADS, VECS, bad, wrong);
  return bad || wrong;
}
int main() {
  int n = 0;
  const int vocabs[] = {1, 2, 3, 4, 5, 6, 7, 8, 9, 15, 16, 2047, 2048, 2050, 8191, 8193, 16383, 16384, 16385, 32766, 32769, 50257};
  for (int vocab : vocabs)
    for (int split = 1; split <= 8; split *= 2)
      n += check<256, 8>(vocab, split) + check<512, 8>(vocab, split) + check<256, 4>(vocab, split) + check<512, 4>(vocab, split);
  return n != 0;
}
"""


def test_register_kernels_read_the_vocabulary_and_no_more(tmp_path):
    """Every logit of a row is read once, entries past `vocab` never: a buffer
    may end with its last row's last logit."""
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "reads.cpp", tmp_path / "reads"
    src.write_text(HARNESS)
    subprocess.run([cxx, "-std=c++17", "-O1", "-w", "-fno-strict-aliasing", "-I", B.CSRC, str(src), "-o", str(exe)],
                   check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
