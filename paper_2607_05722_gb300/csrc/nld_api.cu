// C ABI of libnld (include/nld.h): host-side argument checks, KV split choice,
// TMA descriptor encoding and kernel launches. Nothing here allocates device
// memory or synchronises, except nld_device_error().
#include <climits>
#include <math.h>
#include <stdio.h>
#include <stdlib.h>

#include <mutex>

#include "nld_internal.cuh"

namespace {

using nld::AttnArgs;

// Error word the kernels OR their NLD_DEVERR_* bits into, and the count of
// running-max rescales (a diagnostic).
__device__ unsigned int g_device_error;
__device__ unsigned long long g_rescale_count;

constexpr int kMaxDevices = 64;
unsigned int* g_err_ptr[kMaxDevices];
unsigned long long* g_rescale_ptr[kMaxDevices];
int g_sm_count[kMaxDevices];
std::mutex g_mu;

bool aligned(const void* p, size_t a) { return p != nullptr && (reinterpret_cast<uintptr_t>(p) % a) == 0; }

// Per-device state: addresses of the error word and the rescale counter and
// the SM count, looked up once.
nld_status_t device_state(unsigned int** err, int* sms, unsigned long long** rescales = nullptr) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return NLD_ERR_CUDA;
  std::lock_guard<std::mutex> lock(g_mu);
  if (g_err_ptr[dev] == nullptr) {
    void* p = nullptr;
    void* c = nullptr;
    if (cudaGetSymbolAddress(&p, g_device_error) != cudaSuccess) return NLD_ERR_CUDA;
    if (cudaGetSymbolAddress(&c, g_rescale_count) != cudaSuccess) return NLD_ERR_CUDA;
    int n = 0;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return NLD_ERR_CUDA;
    g_sm_count[dev] = n;
    g_rescale_ptr[dev] = static_cast<unsigned long long*>(c);
    g_err_ptr[dev] = static_cast<unsigned int*>(p);
  }
  if (err) *err = g_err_ptr[dev];
  if (sms) *sms = g_sm_count[dev];
  if (rescales) *rescales = g_rescale_ptr[dev];
  return NLD_OK;
}

bool is_pow2(int x) { return x > 0 && (x & (x - 1)) == 0; }

nld_status_t check_params(const nld_attn_params_t* p, int block_len) {
  if (p == nullptr) return NLD_ERR_INVALID_ARG;
  if (p->batch < 1 || p->num_q_heads < 1 || p->num_kv_heads < 1 || p->num_pages < 1 ||
      p->max_pages_per_seq < 1 || p->num_splits < 0 || p->softmax_scale < 0.f || !isfinite(p->softmax_scale))
    return NLD_ERR_INVALID_ARG;
  if (p->num_q_heads % p->num_kv_heads != 0) return NLD_ERR_INVALID_ARG;
  if (p->flags & ~(NLD_ATTN_PREFIX_READY | NLD_ATTN_NO_CLUSTER))
    return NLD_ERR_INVALID_ARG;
  if (block_len < 1 || block_len > nld::kMaxBlock) return NLD_ERR_INVALID_ARG;
  if (p->num_splits > nld::kMaxSplits) return NLD_ERR_INVALID_ARG;
  if (!is_pow2(p->page_size) || p->page_size < 16 || p->page_size > 256) return NLD_ERR_INVALID_ARG;
  if (p->batch > 65535 || p->num_kv_heads > 65535) return NLD_ERR_UNSUPPORTED;
  if (p->head_dim != 64 && p->head_dim != 128) return NLD_ERR_UNSUPPORTED;
  if ((p->num_q_heads / p->num_kv_heads) * block_len > nld::kMaxRows) return NLD_ERR_UNSUPPORTED;
  // logical token positions must fit in int
  if (static_cast<long long>(p->max_pages_per_seq) * p->page_size > (1ll << 30)) return NLD_ERR_UNSUPPORTED;
  if (static_cast<long long>(p->max_pages_per_seq) * p->page_size < block_len) return NLD_ERR_INVALID_ARG;
  return NLD_OK;
}

// Split plan: S splits of `chunk` tokens (a multiple of 16) over the longest
// possible sequence, max_pages_per_seq * page_size tokens. Splits past a
// shorter sequence's end do no work. With num_splits = 0 the count is
// chosen so that (splits x sequences x KV heads) covers the SMs once.
// On the tcgen05 kernel the splits of a (sequence, KV head) can run as one
// thread-block cluster that merges its results on chip and writes the final
// output, so no workspace and no combine launch are needed. An automatic plan
// takes floor(SMs / units) splits (one wave) and, when that is 2..8, uses one
// cluster of as many CTAs per unit as are resident for all units at once. An
// explicit split count of 2, 4 or 8 uses one cluster; a larger count divisible
// by 8, 4 or 2 uses clusters of that size, leaving one partial per cluster for
// the combine.
constexpr long long kMaxAutoChunk = 2048;  // tokens per piece in an automatic plan (1 MiB of K+V at D=128)

struct SplitPlan {
  int splits;    // CTAs along the KV range per (sequence, KV head)
  int chunk;     // tokens per split
  int csize;     // cluster size (1 = none)
  int partials;  // splits / csize
};

// Longest split that sits in the ring whole at both head sizes (6 tiles at
// head_dim 128).
constexpr long long kPairedChunk = 384;

// A piece of 129..256 rows runs as two CTAs of half the block slots each where
// all of those fit in one wave: the pair reads every tile twice, but a half's
// chain is shorter (1.15 us per 128 tokens against 1.67 with two M tiles, Q by
// TMA, half the rows to store). Automatic plans cut pieces for that up to this
// length, and else twice as many for one CTA each. Halves / two M tiles, us:
// one sequence, 8 KV heads, 160 rows 6880 tokens 14.7 / 16.1, 18400 26.4 / 27.1,
// 27616 35.7 / 34.9; 256 rows 18400 27.4 / 29.8, 36832 45.5 / 45.8; head_dim 64,
// 2272 9.3 / 9.7, 4576 12.0 / 11.1. Several sequences of a range the longest
// may not fill: the line lies lower (two of 2000..8000, 224 rows, 26.4 / 24.4;
// two of 4064, 256 rows, 17.5 / 20.6).
long long halves_chunk(const nld_attn_params_t* p, int rows) {
  if (p->head_dim == 64) return 384;
  return (p->batch == 1 ? 12ll : 6ll) * rows;
}

// Unsplit units of 129..256 rows, fewer than SMs, take cluster pairs of half
// sequences above this many tokens (10 sequences of 100..9000 tokens 71 us, whole
// or as halves 86; head_dim 64, 16 of 512..4096 48, 54), below that whole
// sequences and block-slot halves mixed, and whole sequences alone below
// kMixedMinTokens (the ranking is 1 us).
long long pair_tokens(const nld_attn_params_t* p) { return p->head_dim == 64 ? 2048 : 4352; }
constexpr long long kMixedMinTokens = 512;

// Several sequences share a launch whose pieces the kernel may balance over
// the SMs, knowing their lengths.
bool can_balance(const nld_attn_params_t* p) {
  return p->num_splits == 0 && p->batch > 1 && p->batch <= nld::kMaxBalanced;
}

// The plan for `sms` SMs; `clusters_resident(cs)` says how many clusters of
// cs CTAs can be resident at once (0: none considered).
template <typename ClustersResident>
void plan_splits_for(const nld_attn_params_t* p, int block_len, int sms, ClustersResident clusters_resident,
                     SplitPlan* out) {
  const long long max_tokens = static_cast<long long>(p->max_pages_per_seq) * p->page_size;
  const int rows = (p->num_q_heads / p->num_kv_heads) * block_len;
  const long long units = static_cast<long long>(p->batch) * p->num_kv_heads;  // CTAs per split
  const bool tc = nld::tc_supports(rows, p->head_dim);
  // 129..256 rows of an even block length stay unsplit (and never take the
  // cluster plans below) from half as many units on: their split partials are
  // bf16, and plans of that many units have always merged in fp32.
  const bool wide_even = rows > 128 && block_len % 2 == 0;
  const long long unsplit_units = wide_even ? 2 * units : units;
  const bool clusters = tc && !wide_even && !(p->flags & NLD_ATTN_NO_CLUSTER);
  const bool automatic = p->num_splits == 0;
  int want = p->num_splits;
  int csize = 1;
  if (automatic) {
    // Fill the SMs once; when the (sequence, KV head) units fit in one wave,
    // also cut long ranges into pieces of at most kMaxAutoChunk tokens: with
    // ragged lengths (not known on the host) the longest sequence would
    // otherwise set the time; pieces past a shorter sequence's end exit at
    // once. With more units than SMs the hardware scheduler balances them.
    const long long by_chunk = (max_tokens + kMaxAutoChunk - 1) / kMaxAutoChunk;
    long long s = sms / unsplit_units;
    const bool halves = wide_even && s > 1 && max_tokens <= s * halves_chunk(p, rows);
    if (unsplit_units < sms && !halves) {  // a single wave: the longest range would set the time
      // at most one slot more than two waves of CTAs have (balanced pieces use
      // no more, and the combine reads every slot). Pieces that are not balanced
      // need more waves to even out while there are few units: 48 units of
      // 512..32768 tokens 92 us in 2.5 waves, 83 in 4; one sequence of 98304
      // tokens, 8 units, 95 in 2.05 waves, 89 in 2.5; 128 units 177 in 3.4 waves,
      // 192 in 4.2. They get them as far as the library's own scratch holds
      // the partials, so that a call that uses it is not refused for it.
      long long by_waves = (2 * sms + units - 1) / units + 1;
      if (!can_balance(p) && 2 * units <= sms) {
        const long long in_scratch = static_cast<long long>(nld::kStaticScratchBytes - 256) /
                                     (units * rows * (p->head_dim * 2 + 4));
        const long long four = (4 * sms + units - 1) / units;
        const long long more = four < in_scratch ? four : in_scratch;
        if (more > by_waves) by_waves = more;
      }
      if (s < by_chunk) s = by_chunk < by_waves ? by_chunk : by_waves;
      // More pieces where they run as one CTA each, not as block-slot halves.
      if (s > 1 && s < sms / units) s = sms / units;
    }
    const long long by_tiles = (max_tokens + nld::kTileTok - 1) / nld::kTileTok;  // >= one tile per split
    if (s > by_tiles) s = by_tiles;
    if (s > nld::kMaxSplits) s = nld::kMaxSplits;
    if (s < 1) s = 1;
    want = static_cast<int>(s);
    if (clusters && want >= 2 && want <= 8) {
      // The largest cluster resident for every unit at once, not below the
      // power of two under `want` (a third of the SMs idle costs more than the
      // combine): 8B heads, 3 sequences of 4000 tokens as clusters of 5 15.6 us,
      // of 4 16.4; 5 of 3000 of 3 17.1, of 2 20.4. Sizes between the powers of
      // two only for pieces of two score products or more (28 units of 912
      // tokens: 5 pieces 10.5 us, 4 pieces 10.1).
      const int floor2 = want >= 8 ? 8 : want >= 4 ? 4 : 2;
      int cs = want;
      if (rows <= 128) {
        while (cs >= floor2 && (units > clusters_resident(cs) || (!is_pow2(cs) && max_tokens < 256 * cs))) --cs;
      } else {
        // With two M tiles a piece's time goes by its products of 128 tokens:
        // the fewest CTAs with the fewest products (20 units of 721 tokens, 168
        // rows, 6 pieces of one product 13.4 us, 4 of one and a half 14.7).
        const auto products = [&](int n) { return (max_tokens + 128ll * n - 1) / (128ll * n); };
        while (cs >= floor2 && units > clusters_resident(cs)) --cs;
        for (int n = cs - 1; n >= floor2; --n)
          if (products(n) <= products(cs)) cs = n;
      }
      if (cs >= floor2) {
        want = cs;
        csize = cs;
      }
    }
    // Unsplit long units of 129..256 rows that fit in one wave: each runs as a
    // cluster of two CTAs that take half of its sequence, longest first, and
    // merge on chip in fp32, so that ragged lengths fill the SMs (14B heads, 16
    // sequences of 8192..16384 tokens: one CTA each 230 us, pairs 197). With
    // up to 128 rows, whole sequences measured faster (24 sequences of 64 rows,
    // 192 units: 60 us against 64; 32 of 32 rows, 256 units: 96 against 111).
    if (want == 1 && rows > 128 && units < sms && unsplit_units >= sms && p->batch > 1 && p->batch <= 1024 &&
        max_tokens > pair_tokens(p) && !(p->flags & NLD_ATTN_NO_CLUSTER) && 2 * clusters_resident(2) >= sms - 1) {
      want = 2;
      csize = 2;
    }
  } else if (clusters && want >= 2) {
    for (int cs = 8; cs >= 2; cs >>= 1)
      if (want % cs == 0) {
        csize = cs;
        break;
      }
  }
  long long chunk = (max_tokens + want - 1) / want;
  chunk = (chunk + nld::kGroupTok - 1) / nld::kGroupTok * nld::kGroupTok;
  if (automatic && csize == 1 && tc && chunk <= kPairedChunk) {
    // Short splits take whole products (128 tokens) when that keeps at least
    // 85% of the splits: no half-filled product or tile in every CTA (8B shape: 19 splits of 224 tokens become
    // 17 of 256, measured faster).
    const long long c2 = (chunk + 2 * nld::kTileTok - 1) / (2 * nld::kTileTok) * (2 * nld::kTileTok);
    const long long s2 = (max_tokens + c2 - 1) / c2;
    if (s2 * 100 >= static_cast<long long>(want) * 85) chunk = c2;
  } else if (automatic && tc && (csize == 1 || chunk > kPairedChunk)) {
    // Streaming splits end on a whole tile when that keeps their number.
    const long long c1 = (chunk + nld::kTileTok - 1) / nld::kTileTok * nld::kTileTok;
    if ((max_tokens + c1 - 1) / c1 == (max_tokens + chunk - 1) / chunk) chunk = c1;
  }
  long long splits = (max_tokens + chunk - 1) / chunk;
  splits = (splits + csize - 1) / csize * csize;  // trailing empty splits complete a cluster
  out->chunk = static_cast<int>(chunk);
  out->splits = static_cast<int>(splits);
  out->csize = csize;
  out->partials = static_cast<int>(splits / csize);
}

nld_status_t plan_splits(const nld_attn_params_t* p, int block_len, SplitPlan* out) {
  int sms = 0;
  if (p->num_splits == 0) {
    nld_status_t st = device_state(nullptr, &sms);
    if (st != NLD_OK) return st;
  }
  const int rows = (p->num_q_heads / p->num_kv_heads) * block_len;
  plan_splits_for(
      p, block_len, sms, [&](int cs) { return static_cast<long long>(nld::tc_max_active_clusters(cs, p->head_dim, rows)); },
      out);
  return NLD_OK;
}

// What a call launches: its plan, and how the CTAs take the pieces.
struct Route {
  SplitPlan plan;
  int nh;             // CTAs per piece (2: block-slot halves)
  int halved;         // > 0: unsplit sequences, that many as block-slot halves, the longest
  bool longest_first; // CTAs take the sequences by length; cluster pairs each half of their own
  int balanced_ctas;  // > 0: pieces balanced on the device over that many CTAs
};

Route route_for(const nld_attn_params_t* p, int block_len, bool table_mask, int sms, const SplitPlan& plan) {
  const int rows = (p->num_q_heads / p->num_kv_heads) * block_len;
  const long long units = static_cast<long long>(p->batch) * p->num_kv_heads;
  const long long max_tokens = static_cast<long long>(p->max_pages_per_seq) * p->page_size;
  const long long ctas = units * plan.splits;
  const bool automatic = p->num_splits == 0;
  Route r;
  r.plan = plan;
  r.nh = rows > 128 && block_len % 2 == 0 && plan.csize == 1 && 2 * ctas <= sms ? 2 : 1;
  // Longest sequences first when one split each leaves several waves: the last
  // wave then holds the short sequences. With a table mask only ranges above
  // 2048 tokens, since the ranking takes about 1 us of a CTA's start (31
  // sequences of 277..555 tokens: 31.4 us ordered, 30.8 in grid order). And
  // where the plan made cluster pairs of unsplit units of 129..256 rows, whose
  // CTAs take half of their own sequence each. Pairs of fewer rows come from a
  // plan of two pieces, which fills one wave and keeps its pieces (76 units of
  // 1024 tokens, 32 rows, 12.8 us, as own halves 14.0).
  // Whole sequences and block-slot halves mixed in one wave, where the longest
  // sequence sets the time and there are SMs left for the halves of a fifth of
  // them (18 sequences of 100..2000 tokens, one of which could be: 34.5 us all
  // whole, 37.0).
  const long long spare = (sms - units) / p->num_kv_heads;  // sequences that can run as halves
  const bool mixed = plan.splits == 1 && rows > 128 && block_len % 2 == 0 && r.nh == 1 && 5 * spare >= p->batch && p->batch > 1 &&
                     p->batch <= 1024 && max_tokens >= kMixedMinTokens;
  r.halved = !mixed ? 0 : spare < p->batch ? static_cast<int>(spare) : p->batch;
  const bool waves = plan.splits == 1 && units > sms && (!table_mask || max_tokens > kMaxAutoChunk);
  const bool pairs = automatic && rows > 128 && plan.csize == 2 && plan.splits == 2 && 2 * units >= sms;
  r.longest_first = (waves || pairs) && p->batch > 1 && p->batch <= 1024;
  // Balanced pieces: a plan of several streaming pieces a sequence, none of
  // them in clusters, more slots than SMs. The launch has CTAs for two waves,
  // or one per slot. Measured against the plan's own pieces (8B heads, 32 rows):
  // 8 sequences of 512..8192 tokens 43.4 -> 38.6 us, 8 of 4096 39.8 -> 32.4, 18
  // of 8192 115 -> 103; 14B heads, 4 of 4096..16384 77 -> 59. A CTA learns its
  // piece about 2 us later, so a single wave keeps the plan's pieces, and so
  // does a plan of at most three that fill their last wave to 90% (12 of 4096:
  // 46.5 us against 50.5).
  r.balanced_ctas = 0;
  if (can_balance(p) && plan.csize == 1 && plan.splits > 1 && plan.chunk > kPairedChunk &&
      !nld::tc_row_copies(rows, p->head_dim, plan.chunk)) {
    const long long in_waves = (ctas + sms - 1) / sms;
    if (ctas > sms && units <= 2 * sms && !(plan.splits <= 3 && 10 * ctas >= 9 * in_waves * sms))
      r.balanced_ctas = static_cast<int>(ctas < 2 * sms ? ctas : 2 * sms);
  }
  return r;
}

size_t align256(size_t x) { return (x + 255) & ~size_t(255); }

size_t partial_o_bytes(const nld_attn_params_t* p, int block_len, int splits) {
  return static_cast<size_t>(splits) * p->batch * p->num_q_heads * block_len * p->head_dim * sizeof(__nv_bfloat16);
}
size_t partial_lse_bytes(const nld_attn_params_t* p, int block_len, int splits) {
  return static_cast<size_t>(splits) * p->batch * p->num_q_heads * block_len * sizeof(float);
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(f);
  });
  return fn;
}

// Tokens of a K/V box: as many as a page holds, up to a tile, and as the
// pieces' starts (multiples of `chunk` with more than one split) allow without
// a box crossing a page: 16, 32 or 64. Short pieces are bound by latency, not
// by TMA issue, and the zeroing of V rows past a sequence's end, up to a box
// less one row, is part of it: 16.
int box_tokens(const nld_attn_params_t* p, const SplitPlan& plan) {
  if (plan.chunk <= kPairedChunk) return 16;
  int n = p->page_size < nld::kTileTok ? p->page_size : nld::kTileTok;
  while (plan.splits > 1 && plan.chunk % n != 0) n /= 2;  // chunk is a multiple of 16
  return n;
}

// 5-D map over a page pool [num_pages, Hkv, P, D], innermost first: 64 dims,
// 8 tokens, the 64-dim column blocks, the 8-token groups of a page, (page, KV
// head). A box is all dims of box_tok tokens of one (page, KV head), in shared
// memory as [8-token group][column block][8 rows of 128 bytes] with the
// 128-byte swizzle: 8-token groups a fixed stride apart, as the MMA operands
// want them, also over the boxes and tiles that follow one another. Boxes past
// num_pages read as zeros.
nld_status_t encode_pool_map(CUtensorMap* map, const void* base, const nld_attn_params_t* p, int num_pages,
                             int box_tok) {
  EncodeTiledFn fn = encode_fn();
  if (fn == nullptr) return NLD_ERR_CUDA;
  const cuuint64_t planes = static_cast<cuuint64_t>(num_pages) * p->num_kv_heads;
  const cuuint64_t D = static_cast<cuuint64_t>(p->head_dim);
  const cuuint64_t P = static_cast<cuuint64_t>(p->page_size);
  cuuint64_t dims[5] = {64, 8, D / 64, P / 8, planes};
  cuuint64_t strides[4] = {D * 2, 128, D * 2 * 8, D * 2 * P};
  cuuint32_t box[5] = {64, 8, static_cast<cuuint32_t>(D / 64), static_cast<cuuint32_t>(box_tok / 8), 1};
  cuuint32_t estr[5] = {1, 1, 1, 1, 1};
  CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void*>(base), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? NLD_OK : NLD_ERR_CUDA;
}

// Map over a [B, bl, Hq, D] bf16 block (queries or output) whose box is one
// CTA's R = G * bl rows of 64 dims (G heads x bl slots), 128-byte swizzle.
nld_status_t encode_block_map(CUtensorMap* map, const void* base, const nld::AttnArgs& a, int D) {
  EncodeTiledFn fn = encode_fn();
  if (fn == nullptr) return NLD_ERR_CUDA;
  cuuint32_t estr[3] = {1, 1, 1};
  cuuint64_t dims[3] = {static_cast<cuuint64_t>(D), static_cast<cuuint64_t>(a.Hq), static_cast<cuuint64_t>(a.B) * a.bl};
  cuuint64_t strides[2] = {static_cast<cuuint64_t>(D) * 2, static_cast<cuuint64_t>(D) * 2 * a.Hq};
  cuuint32_t box[3] = {64, static_cast<cuuint32_t>(a.G), static_cast<cuuint32_t>(a.bl_c)};
  CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_NONE,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? NLD_OK : NLD_ERR_CUDA;
}

// Map for the tiled output stores of one CTA's R = G * bl rows, 128-byte
// swizzle, rows in packed order (block slot major), box 64 dims x G heads x
// bl slots, bf16. Final output [B, bl, Hq, D]. Split partials [partials * B,
// Hq, bl, D]: the map walks dims, heads (stride bl * D), block slots (stride
// D), then (partial, sequence).
nld_status_t encode_out_map(CUtensorMap* map, const nld::AttnArgs& a, int D) {
  if (a.o_part == nullptr) return encode_block_map(map, a.out, a, D);
  EncodeTiledFn fn = encode_fn();
  if (fn == nullptr) return NLD_ERR_CUDA;
  const long long units = static_cast<long long>(a.num_partials) * a.B;
  if (units > INT_MAX) return NLD_ERR_UNSUPPORTED;  // coordinates are int
  const cuuint64_t row = static_cast<cuuint64_t>(D) * 2;
  cuuint32_t estr[4] = {1, 1, 1, 1};
  cuuint64_t dims[4] = {static_cast<cuuint64_t>(D), static_cast<cuuint64_t>(a.Hq), static_cast<cuuint64_t>(a.bl),
                        static_cast<cuuint64_t>(units)};
  cuuint64_t strides[3] = {row * a.bl, row, row * a.bl * a.Hq};
  cuuint32_t box[4] = {64, static_cast<cuuint32_t>(a.G), static_cast<cuuint32_t>(a.bl_c), 1};
  CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, a.o_part, dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_NONE,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? NLD_OK : NLD_ERR_CUDA;
}

// Pieces (CTAs of one cluster, 1..8) per row of the logits kernels. With fewer
// rows than SMs: enough to fill the SMs once, of at least 1024 vectors of 8
// logits each. Then as many as bring a piece down to `fit` vectors, where 8
// pieces can be kept in registers at all; a row that one CTA can keep (4096
// vectors) is cut no further once its pieces fill the SMs (1000 rows x 20000: 4
// pieces 24.6 us, whole 19.1; as ensemble 31.4 and 21.4). Times here and below:
// a pass of two reductions with their decisions, or of one ensemble.
int logits_pieces(int rows, long nvec, int sms, int fit) {
  int split = 1;
  if (rows < sms) {
    const int by_sms = sms / rows;
    const long by_len = nvec / nld::logits_split_vectors();
    const long want = by_sms < by_len ? by_sms : by_len;
    while (split * 2 <= want && split * 2 <= 8) split *= 2;
  }
  const long whole = nld::logits_piece_limit();
  if (nvec <= 8 * whole)
    while (split < 8 && nvec > static_cast<long>(split) * fit && (nvec > whole || 2L * split * rows <= sms)) split *= 2;
  return split;
}

// The pieces' CTAs each pay a chain of merges, so with many rows the streaming
// kernel, one CTA a row, is ahead where pieces are short for their CTA: at 1000
// rows x 150000 (8 pieces of 2344 vectors) 128 us against 168, at 3000 x 80000
// (1250) 200 against 215, at 1000 x 72001 (1126) 75 against 78; at 512 x 200001
// (3126) both 102, and 200 x 150000 is 45 us in pieces, 51 streamed.
int logits_split(int rows, int vocab, int sms) {
  const long nvec = (static_cast<long>(vocab) + 7) / 8;
  const int split = logits_pieces(rows, nvec, sms, 2048);
  const long per = (nvec + split - 1) / split;
  if (split == 8 && rows >= 2 * sms && per > 2048 && per < 3200) return 1;
  if (split == 8 && ((rows >= 12 * sms && per < 1408) || (rows >= 6 * sms && per < 1200))) return 1;
  return split;
}

// 0: the streaming kernel. It reads a row pair twice, and is still ahead of
// pieces at many rows: with pieces over 2048 vectors, one CTA an SM, at 400 rows
// x 150000 (2344 vectors) 109 us against 118, 512 x 200001 (3126) 155 against
// 169, 1000 x 262144 (4096) 305 against 332, and behind at 304 x 170000 (111
// against 103), 512 x 262144 (195 against 172); below that where a CTA's slots
// are not nearly full: 1000 rows x 40000 (625 of 768) 54 us against 60, 1000 x
// 100003 (1563 of 2048) 125 against 142, 700 x 100003 106 against 99, and 512 x
// 72001 (1126 of 1536) 61 against 68, 512 x 80000 (1250) 66 each; whole rows
// in one CTA at 3000 x 16392 (2049 of 2560) 58 against 66, 1000 x 16392 23
// against 21.
int ensemble_split(int rows, int vocab, int sms) {
  const long nvec = (static_cast<long>(vocab) + 7) / 8;
  const int split = logits_pieces(rows, nvec, sms, 1024);
  const long per = (nvec + split - 1) / split;
  if (rows < 2 * sms) return split;
  if (per > 2048) {
    if (split == 1) return rows >= 12 * sms && per < 2400 ? 0 : 1;
    return rows >= 6 * sms || per < (rows >= 3 * sms ? 3584 : 2600) ? 0 : split;
  }
  if (split > 1 && rows >= 3 * sms && per > 1024 && per < 1200) return 0;
  const int threads = per <= 1024 ? 256 : 512;
  const long slots = (per + threads - 1) / threads * threads;
  return split > 1 && rows >= 6 * sms && 16 * per < 15 * slots ? 0 : split;
}

}  // namespace

namespace nld {
bool pdl_enabled() {
  static const bool on = [] {
    const char* v = getenv("NLD_DISABLE_PDL");
    return !(v != nullptr && v[0] == '1');
  }();
  return on;
}
}  // namespace nld

extern "C" {

const char* nld_status_string(nld_status_t s) {
  switch (s) {
    case NLD_OK: return "NLD_OK";
    case NLD_ERR_INVALID_ARG: return "NLD_ERR_INVALID_ARG";
    case NLD_ERR_UNSUPPORTED: return "NLD_ERR_UNSUPPORTED";
    case NLD_ERR_WORKSPACE: return "NLD_ERR_WORKSPACE";
    case NLD_ERR_CUDA: return "NLD_ERR_CUDA";
  }
  return "NLD_ERR_UNKNOWN";
}

int nld_block_attn_plan(const nld_attn_params_t* params, int block_len, int sm_count, int32_t plan[4]) {
  if (plan == nullptr || sm_count < 1) return -1;
  if (check_params(params, block_len) != NLD_OK) return -1;
  SplitPlan sp;
  plan_splits_for(params, block_len, sm_count, [](int) { return 0LL; }, &sp);
  plan[0] = sp.splits;
  plan[1] = sp.chunk;
  plan[2] = sp.csize;
  plan[3] = sp.partials;
  return 0;
}

int nld_block_attn_route(const nld_attn_params_t* params, int block_len, int table_mask, int sm_count,
                         const int32_t* resident, int32_t route[8]) {
  if (route == nullptr || (resident != nullptr && sm_count < 1)) return -1;
  if (check_params(params, block_len) != NLD_OK) return -1;
  SplitPlan plan;
  if (resident != nullptr) {
    plan_splits_for(params, block_len, sm_count, [&](int cs) { return static_cast<long long>(resident[cs]); }, &plan);
  } else if (plan_splits(params, block_len, &plan) != NLD_OK || device_state(nullptr, &sm_count) != NLD_OK) {
    return -1;
  }
  const Route r = route_for(params, block_len, table_mask != 0, sm_count, plan);
  const long long ctas = (static_cast<long long>(plan.splits) * params->batch * r.nh + r.halved) * params->num_kv_heads;
  route[0] = plan.splits;
  route[1] = plan.chunk;
  route[2] = plan.csize;
  route[3] = plan.partials;
  route[4] = r.nh;
  route[5] = r.halved > 0 ? 3 : r.balanced_ctas > 0 ? 2 : r.longest_first ? 1 : 0;
  route[6] = r.balanced_ctas > 0 ? r.balanced_ctas : ctas > INT_MAX ? INT_MAX : static_cast<int32_t>(ctas);
  route[7] = box_tokens(params, plan);
  return 0;
}

int nld_block_attn_num_splits(const nld_attn_params_t* params, int block_len) {
  if (check_params(params, block_len) != NLD_OK) return -1;
  SplitPlan plan;
  if (plan_splits(params, block_len, &plan) != NLD_OK) return -1;
  return plan.partials;
}

int nld_block_attn_kernels(const nld_attn_params_t* params, int block_len) {
  if (check_params(params, block_len) != NLD_OK) return -1;
  SplitPlan plan;
  if (plan_splits(params, block_len, &plan) != NLD_OK) return -1;
  return plan.partials <= 1 ? 1 : 2;
}

size_t nld_block_attn_workspace_size(const nld_attn_params_t* params, int block_len) {
  if (check_params(params, block_len) != NLD_OK) return static_cast<size_t>(-1);
  SplitPlan plan;
  if (plan_splits(params, block_len, &plan) != NLD_OK) return static_cast<size_t>(-1);
  if (plan.partials == 1) return 0;
  return align256(partial_o_bytes(params, block_len, plan.partials)) +
         partial_lse_bytes(params, block_len, plan.partials);
}

}  // extern "C"

namespace {

nld_status_t block_attn_impl(const nld_attn_params_t* params, const void* q_block, const void* k_pages,
                             const void* v_pages, const int32_t* page_table, const int32_t* prefix_lens,
                             int block_len, int mode, const uint32_t* block_mask, void* out, float* lse,
                             void* workspace, size_t workspace_bytes, bool run_combine, cudaStream_t stream) {
  nld_status_t st = check_params(params, block_len);
  if (st != NLD_OK) return st;
  if (mode != NLD_MODE_DIFFUSION && mode != NLD_MODE_VERIFY && mode != nld::kModeBlockMask)
    return NLD_ERR_INVALID_ARG;
  if (mode == nld::kModeBlockMask && !aligned(block_mask, 4)) return NLD_ERR_INVALID_ARG;
  if (!aligned(q_block, 16) || !aligned(k_pages, 16) || !aligned(v_pages, 16) || !aligned(out, 16) ||
      !aligned(page_table, 4) || !aligned(prefix_lens, 4))
    return NLD_ERR_INVALID_ARG;
  if (lse != nullptr && !aligned(lse, 4)) return NLD_ERR_INVALID_ARG;
  SplitPlan plan;
  st = plan_splits(params, block_len, &plan);
  if (st != NLD_OK) return st;
  size_t o_bytes = 0;
  if (plan.partials > 1) {
    o_bytes = align256(partial_o_bytes(params, block_len, plan.partials));
    const size_t need = o_bytes + partial_lse_bytes(params, block_len, plan.partials);
    if (workspace == nullptr || workspace_bytes < need) return NLD_ERR_WORKSPACE;
    if (!aligned(workspace, 16)) return NLD_ERR_INVALID_ARG;
  }
  unsigned int* err = nullptr;
  unsigned long long* rescales = nullptr;
  int sms = 0;
  st = device_state(&err, &sms, &rescales);
  if (st != NLD_OK) return st;
  const Route route = route_for(params, block_len, mode == nld::kModeBlockMask, sms, plan);

  nld::TmaMaps maps;
  const int box_tok = box_tokens(params, plan);
  // (page, KV head) coordinates are int, the page past the pool among them; a
  // pool of more planes than that would take over 4 TB.
  const int max_pool = INT_MAX / params->num_kv_heads - 1;
  const int num_pages = params->num_pages < max_pool ? params->num_pages : max_pool;
  if ((st = encode_pool_map(&maps.k, k_pages, params, num_pages, box_tok)) != NLD_OK) return st;
  if ((st = encode_pool_map(&maps.v, v_pages, params, num_pages, box_tok)) != NLD_OK) return st;

  const int G = params->num_q_heads / params->num_kv_heads;
  const float scale = params->softmax_scale > 0.f ? params->softmax_scale : 1.0f / sqrtf((float)params->head_dim);
  AttnArgs a{};
  a.q = static_cast<const __nv_bfloat16*>(q_block);
  a.page_table = page_table;
  a.prefix_lens = prefix_lens;
  a.out = static_cast<__nv_bfloat16*>(out);
  a.lse = lse;
  a.err = err;
  a.rescales = rescales;
  a.B = params->batch;
  a.Hq = params->num_q_heads;
  a.Hkv = params->num_kv_heads;
  a.G = G;
  a.bl = block_len;
  a.nh = route.nh;
  a.bl_c = block_len / a.nh;
  a.R = G * a.bl_c;
  a.page_size = params->page_size;
  a.log2_page = __builtin_ctz(static_cast<unsigned>(params->page_size));
  a.num_pages = num_pages;
  a.max_pages = params->max_pages_per_seq;
  a.box_tok = box_tok;
  a.num_splits = plan.splits;
  a.chunk = plan.chunk;
  a.csize = plan.csize;
  a.num_partials = plan.partials;
  a.mode = mode;
  a.block_mask = mode == nld::kModeBlockMask ? block_mask : nullptr;
  a.scale_log2 = scale * nld::kLog2e;
  a.prefix_ready = (params->flags & NLD_ATTN_PREFIX_READY) ? 1 : 0;
  a.order_by_length = route.longest_first ? 1 : 0;
  a.balanced_ctas = route.balanced_ctas;
  a.halved = route.halved;
  a.sms = sms;
  if (plan.partials > 1) {
    a.o_part = static_cast<__nv_bfloat16*>(workspace);
    a.lse_part = reinterpret_cast<float*>(static_cast<char*>(workspace) + o_bytes);
  }
  if ((st = encode_out_map(&maps.o, a, params->head_dim)) != NLD_OK) return st;
  if ((st = encode_block_map(&maps.q, q_block, a, params->head_dim)) != NLD_OK) return st;
  if (route.halved > 0) {
    AttnArgs half = a;
    half.nh = 2;
    half.bl_c = block_len / 2;
    half.R = G * half.bl_c;
    nld::TmaMaps half_maps = maps;
    if ((st = encode_out_map(&half_maps.o, half, params->head_dim)) != NLD_OK) return st;
    if ((st = encode_block_map(&half_maps.q, q_block, half, params->head_dim)) != NLD_OK) return st;
    if (nld::launch_block_attn_tc_mixed(a, maps, half, half_maps, params->head_dim, stream) != cudaSuccess)
      return NLD_ERR_CUDA;
  } else if (nld::launch_block_attn_tc(a, maps, params->head_dim, stream) != cudaSuccess) {
    return NLD_ERR_CUDA;
  }
  if (plan.partials > 1 && run_combine) {
    if (nld::launch_combine(a.o_part, a.lse_part, plan.partials, a.B, a.Hq, block_len, params->head_dim, a.out, lse,
                            sms, stream) != cudaSuccess)
      return NLD_ERR_CUDA;
  }
  return NLD_OK;
}

}  // namespace

extern "C" {

nld_status_t nld_block_attn(const nld_attn_params_t* params, const void* q_block, const void* k_pages,
                            const void* v_pages, const int32_t* page_table, const int32_t* prefix_lens,
                            int block_len, nld_mode_t mode, void* out, float* lse, void* workspace,
                            size_t workspace_bytes, cudaStream_t stream) {
  return block_attn_impl(params, q_block, k_pages, v_pages, page_table, prefix_lens, block_len, mode, nullptr, out,
                         lse, workspace, workspace_bytes, true, stream);
}

nld_status_t nld_block_attn_masked(const nld_attn_params_t* params, const void* q_block, const void* k_pages,
                                   const void* v_pages, const int32_t* page_table, const int32_t* prefix_lens,
                                   int block_len, const uint32_t* block_mask, void* out, float* lse, void* workspace,
                                   size_t workspace_bytes, cudaStream_t stream) {
  return block_attn_impl(params, q_block, k_pages, v_pages, page_table, prefix_lens, block_len, nld::kModeBlockMask,
                         block_mask, out, lse, workspace, workspace_bytes, true, stream);
}

int nld_quadss_block_mask(int k, uint32_t* masks) {
  // Slot order (Eq. quad_input): the AR token, then for each of the k
  // speculative tokens that token followed by its k masks. The chain (AR
  // and speculative tokens) is causal and sees no mask; the masks of a
  // speculative token see the chain up to it and their own k masks.
  const int n = 1 + k + k * k;
  if (k < 1 || n > nld::kMaxBlock || masks == nullptr) return -1;
  uint32_t chain = 1u;  // chain slots seen so far (the AR token, slot 0)
  masks[0] = chain;
  for (int g = 0; g < k; ++g) {
    const int spec = 1 + g * (k + 1);
    chain |= 1u << spec;
    masks[spec] = chain;
    const uint32_t group = ((1u << k) - 1u) << (spec + 1);  // this token's k masks
    for (int r = 1; r <= k; ++r) masks[spec + r] = chain | group;
  }
  return n;
}

nld_status_t nld_block_attn_partials(const nld_attn_params_t* params, const void* q_block, const void* k_pages,
                                     const void* v_pages, const int32_t* page_table, const int32_t* prefix_lens,
                                     int block_len, nld_mode_t mode, void* out, float* lse, void* workspace,
                                     size_t workspace_bytes, cudaStream_t stream) {
  return block_attn_impl(params, q_block, k_pages, v_pages, page_table, prefix_lens, block_len, mode, nullptr, out,
                         lse, workspace, workspace_bytes, false, stream);
}

nld_status_t nld_split_kv_combine(const void* o_part, const float* lse_part, int num_splits, int batch,
                                  int num_q_heads, int block_len, int head_dim, void* out, float* lse,
                                  cudaStream_t stream) {
  if (num_splits < 1 || num_splits > nld::kMaxSplits || batch < 1 || num_q_heads < 1 || block_len < 1 ||
      block_len > nld::kMaxBlock)
    return NLD_ERR_INVALID_ARG;
  if (head_dim != 64 && head_dim != 128) return NLD_ERR_UNSUPPORTED;
  if (!aligned(o_part, 16) || !aligned(lse_part, 4) || !aligned(out, 16)) return NLD_ERR_INVALID_ARG;
  if (lse != nullptr && !aligned(lse, 4)) return NLD_ERR_INVALID_ARG;
  int sms = 0;
  const nld_status_t st = device_state(nullptr, &sms);
  if (st != NLD_OK) return st;
  if (nld::launch_combine(static_cast<const __nv_bfloat16*>(o_part), lse_part, num_splits, batch, num_q_heads,
                          block_len, head_dim, static_cast<__nv_bfloat16*>(out), lse, sms, stream) != cudaSuccess)
    return NLD_ERR_CUDA;
  return NLD_OK;
}

nld_status_t nld_accept(const int32_t* draft_ids, const int32_t* verify_ids, int batch, int n,
                        int32_t* accepted_len, cudaStream_t stream) {
  if (batch < 1 || n < 1 || n > nld::kMaxBlock) return NLD_ERR_INVALID_ARG;
  if (!aligned(draft_ids, 4) || !aligned(verify_ids, 4) || !aligned(accepted_len, 4)) return NLD_ERR_INVALID_ARG;
  return nld::launch_accept(draft_ids, verify_ids, batch, n, accepted_len, stream) == cudaSuccess ? NLD_OK
                                                                                                   : NLD_ERR_CUDA;
}

nld_status_t nld_unmask(const float* confidences, int batch, int n, int k, int32_t* positions,
                        int32_t* num_selected, cudaStream_t stream) {
  if (batch < 1 || n < 1 || n > nld::kMaxBlock || k < 1 || k > n) return NLD_ERR_INVALID_ARG;
  if (!aligned(confidences, 4) || !aligned(positions, 4)) return NLD_ERR_INVALID_ARG;
  if (num_selected != nullptr && !aligned(num_selected, 4)) return NLD_ERR_INVALID_ARG;
  return nld::launch_unmask(confidences, batch, n, k, positions, num_selected, stream) == cudaSuccess
             ? NLD_OK
             : NLD_ERR_CUDA;
}

nld_status_t nld_unmask_threshold(const float* confidences, int batch, int n, float threshold, int32_t* positions,
                                  int32_t* num_selected, cudaStream_t stream) {
  if (batch < 1 || n < 1 || n > nld::kMaxBlock) return NLD_ERR_INVALID_ARG;
  if (!aligned(confidences, 4) || !aligned(positions, 4)) return NLD_ERR_INVALID_ARG;
  if (num_selected != nullptr && !aligned(num_selected, 4)) return NLD_ERR_INVALID_ARG;
  return nld::launch_unmask_threshold(confidences, batch, n, threshold, positions, num_selected, stream) ==
                 cudaSuccess
             ? NLD_OK
             : NLD_ERR_CUDA;
}

nld_status_t nld_greedy_accept(const int32_t* pred_ids, const int32_t* target_ids, const float* confidences,
                               int batch, int n, int32_t* positions, int32_t* num_selected, cudaStream_t stream) {
  if (batch < 1 || n < 1 || n > nld::kMaxBlock) return NLD_ERR_INVALID_ARG;
  if (!aligned(pred_ids, 4) || !aligned(target_ids, 4) || !aligned(confidences, 4) || !aligned(positions, 4))
    return NLD_ERR_INVALID_ARG;
  if (num_selected != nullptr && !aligned(num_selected, 4)) return NLD_ERR_INVALID_ARG;
  return nld::launch_greedy_accept(pred_ids, target_ids, confidences, batch, n, positions, num_selected, stream) ==
                 cudaSuccess
             ? NLD_OK
             : NLD_ERR_CUDA;
}

nld_status_t nld_logits_argmax(const void* logits, int rows, int vocab, int ld, int32_t* ids, float* conf,
                               cudaStream_t stream) {
  if (rows < 1 || vocab < 1 || ld < vocab || ld % 8 != 0) return NLD_ERR_INVALID_ARG;
  if (!aligned(logits, 16) || !aligned(ids, 4) || !aligned(conf, 4)) return NLD_ERR_INVALID_ARG;
  unsigned int* err = nullptr;
  int sms = 0;
  nld_status_t st = device_state(&err, &sms);
  if (st != NLD_OK) return st;
  const int split = logits_split(rows, vocab, sms);
  return nld::launch_logits_argmax(static_cast<const __nv_bfloat16*>(logits), rows, vocab, ld, split, ids, conf, err,
                                   stream) == cudaSuccess
             ? NLD_OK
             : NLD_ERR_CUDA;
}

nld_status_t nld_logits_ensemble_argmax(const void* ar_logits, const void* diff_logits, int rows, int vocab, int ld,
                                        float lambda, int32_t* ids, float* conf, cudaStream_t stream) {
  if (rows < 1 || vocab < 1 || ld < vocab || ld % 8 != 0) return NLD_ERR_INVALID_ARG;
  if (!(lambda >= 0.f && lambda <= 1.f)) return NLD_ERR_INVALID_ARG;  // also rejects NaN
  if (!aligned(ar_logits, 16) || !aligned(diff_logits, 16) || !aligned(ids, 4) || !aligned(conf, 4))
    return NLD_ERR_INVALID_ARG;
  unsigned int* err = nullptr;
  int sms = 0;
  nld_status_t st = device_state(&err, &sms);
  if (st != NLD_OK) return st;
  const int split = ensemble_split(rows, vocab, sms);
  return nld::launch_ensemble_argmax(static_cast<const __nv_bfloat16*>(ar_logits),
                                     static_cast<const __nv_bfloat16*>(diff_logits), rows, vocab, ld, split, lambda,
                                     ids, conf, err, stream) == cudaSuccess
             ? NLD_OK
             : NLD_ERR_CUDA;
}

nld_status_t nld_kv_commit(const nld_attn_params_t* params, const void* k_new, const void* v_new,
                           const int32_t* counts, const int32_t* page_table, int32_t* prefix_lens, int block_len,
                           int advance, void* k_pages, void* v_pages, cudaStream_t stream) {
  nld_status_t st = check_params(params, block_len);
  if (st != NLD_OK) return st;
  if (!aligned(k_new, 16) || !aligned(v_new, 16) || !aligned(k_pages, 16) || !aligned(v_pages, 16) ||
      !aligned(page_table, 4) || !aligned(prefix_lens, 4))
    return NLD_ERR_INVALID_ARG;
  if (counts != nullptr && !aligned(counts, 4)) return NLD_ERR_INVALID_ARG;
  unsigned int* err = nullptr;
  if ((st = device_state(&err, nullptr)) != NLD_OK) return st;
  return nld::launch_kv_commit(static_cast<const __nv_bfloat16*>(k_new), static_cast<const __nv_bfloat16*>(v_new),
                               counts, page_table, prefix_lens, static_cast<__nv_bfloat16*>(k_pages),
                               static_cast<__nv_bfloat16*>(v_pages), params->batch, params->num_kv_heads,
                               params->head_dim, params->page_size, params->num_pages, params->max_pages_per_seq,
                               block_len, advance != 0, err, stream) == cudaSuccess
             ? NLD_OK
             : NLD_ERR_CUDA;
}

nld_status_t nld_check_wait_timeout(uint64_t limit_ns, cudaStream_t stream) {
  if (limit_ns == 0 || limit_ns > nld::kWaitLimitNs) return NLD_ERR_INVALID_ARG;
  unsigned int* err = nullptr;
  nld_status_t st = device_state(&err, nullptr);
  if (st != NLD_OK) return st;
  return nld::launch_wait_timeout_check(limit_ns, err, stream) == cudaSuccess ? NLD_OK : NLD_ERR_CUDA;
}

nld_status_t nld_device_error(uint32_t* bits, int clear) {
  if (bits == nullptr) return NLD_ERR_INVALID_ARG;
  unsigned int* err = nullptr;
  nld_status_t st = device_state(&err, nullptr);
  if (st != NLD_OK) return st;
  unsigned int v = 0;
  if (cudaMemcpy(&v, err, sizeof v, cudaMemcpyDeviceToHost) != cudaSuccess) return NLD_ERR_CUDA;
  *bits = v;
  if (clear) {
    const unsigned int zero = 0;
    if (cudaMemcpy(err, &zero, sizeof zero, cudaMemcpyHostToDevice) != cudaSuccess) return NLD_ERR_CUDA;
  }
  return NLD_OK;
}

nld_status_t nld_rescale_count(uint64_t* count, int clear) {
  if (count == nullptr) return NLD_ERR_INVALID_ARG;
  unsigned long long* c = nullptr;
  nld_status_t st = device_state(nullptr, nullptr, &c);
  if (st != NLD_OK) return st;
  unsigned long long v = 0;
  if (cudaMemcpy(&v, c, sizeof v, cudaMemcpyDeviceToHost) != cudaSuccess) return NLD_ERR_CUDA;
  *count = static_cast<uint64_t>(v);
  if (clear) {
    const unsigned long long zero = 0;
    if (cudaMemcpy(c, &zero, sizeof zero, cudaMemcpyHostToDevice) != cudaSuccess) return NLD_ERR_CUDA;
  }
  return NLD_OK;
}

}  // extern "C"
