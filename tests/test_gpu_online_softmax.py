"""The online softmax when a row's running maximum jumps mid-stream.

Block attention (Sec. 2.2 attention pattern; Sec. 3 Modes 2 and 3) is a
softmax over arbitrary score magnitudes. The kernels keep each row's running
maximum lazily: the output accumulated in tensor memory is rescaled only when
a later tile raises the maximum by more than 2^8 (base 2). N(0,1) inputs never
get there, so these inputs are built to:

  - "sink" keys: every query row gets a large component along dimension 0
    and a few runs of keys get a large dimension-0 value, so a row's scores
    jump by tens of base-2 units at those keys: a run of 128 keys starting on
    a 64-token tile boundary in mid-prefix, a 16-key run late in the prefix
    and the last block slot (seen only by the last row in the verify pass).
    A second, milder strength puts the jump near 2^10, where the keys before
    the sinks still carry a few percent of the weight;
  - queries scaled by 8 under softmax_scale 0.5: scores spread over hundreds
    of base-2 units, so the running maximum grows several times per split.

Every case runs both passes and is compared on every row with the fp64
oracle. The sink cases use the bars of the other attention tests (max-abs
1e-2, rel-L2 5e-3, lse 2e-3). The scaled-query case makes each row nearly
one-hot, so its outputs sit close to single V values of magnitude up to ~4.5,
where one bf16 half-ulp is 2^-8 |o| (0.0156 at |o| >= 4): the bf16 output
format alone can exceed a flat 1e-2 there. Its max-abs bar is the bound of
the two bf16 roundings on the path (round to nearest, unit roundoff 2^-8):
the output, 2^-8 |o_ref|, and P before the PV product, 2^-8 sum_t p_t |v_t|
<= 2^-8 max |V|, plus 1e-4 for the fp32 sums; rel-L2 and lse keep their bars.
The device's rescale counter
(nld_rescale_count) shows the rescale path ran: with one split per (sequence,
KV head), and with explicit split counts, every call must rescale.
"""
import dataclasses

import numpy as np
import pytest
import torch

from gpu_helpers import DeviceCase, compare_attn, oracle_full
from paper_2607_05722_gb300 import nld
from paper_2607_05722_gb300 import workloads as W

pytestmark = pytest.mark.gpu

DIFF, VER = W.MODE_DIFFUSION, W.MODE_VERIFY


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2607_05722_gb300 import build
    build.build()
    nld.lib()
    nld.nld_device_error(clear=True)
    yield
    assert nld.nld_device_error(clear=True) == 0, "a kernel flagged a device error"


# name, B, Hq, Hkv, D, P, bl, prefix lengths; packed rows G*bl and the pieces
# set the kernel: two softmax groups for up to 128 rows, of 33..64 only in pieces
# longer than the ring (shorter: two row copies, in a test of their own below);
# more rows as block-slot halves on that kernel where the block length is even
# and the wave holds them, with two M tiles where it is odd
SHAPES = [
    ("rows32_cg2_d64", 1, 4, 1, 64, 16, 8, [700]),
    ("rows64_rep2_d128", 1, 32, 8, 128, 16, 16, [1500]),
    ("rows96_rep1_d128", 2, 6, 2, 128, 16, 32, [900, 400]),
    ("rows160_mt2_d128", 1, 10, 2, 128, 16, 32, [1200]),
    ("rows180_mt2_d64", 1, 6, 1, 64, 32, 30, [800]),
    ("rows145_odd_mt2_d128", 1, 10, 2, 128, 16, 29, [1200]),
    ("rows248_odd_mt2_d64", 1, 8, 1, 64, 32, 31, [800]),
    ("rows248_odd_mt2_d128", 1, 8, 1, 128, 32, 31, [800]),
]

BF16_8 = np.uint16(0x4100)  # 8.0


def _bf16(x):
    return W.f32_to_bf16_bits(np.float32(x).reshape(1))[0]


def with_sinks(case, strength):
    """Copy of `case` with dimension 0 of every query row set to 8 and
    dimension 0 of the sink keys (all KV heads) set to `strength`."""
    kv = case.kv
    k_bits = kv.k_bits.copy()
    qd, qv = case.q_draft_bits.copy(), case.q_verify_bits.copy()
    qd[..., 0] = BF16_8
    qv[..., 0] = BF16_8
    h = _bf16(strength)
    for b in range(case.batch):
        L = int(kv.prefix_lens[b])
        mid = (L // 2) // 64 * 64
        sinks = list(range(mid, min(mid + 128, L))) + list(range(max(L - 40, 0), max(L - 24, 0)))
        sinks.append(L + case.block_len - 1)  # the last block slot
        for t in sinks:
            page, slot = kv.page_table[b, t // kv.page_size], t % kv.page_size
            k_bits[page, :, slot, 0] = h
    return dataclasses.replace(case, q_draft_bits=qd, q_verify_bits=qv,
                               kv=dataclasses.replace(kv, k_bits=k_bits))


def with_scaled_queries(case, factor, scale):
    qd = W.f32_to_bf16_bits(W.bf16_bits_to_f32(case.q_draft_bits) * np.float32(factor))
    qv = W.f32_to_bf16_bits(W.bf16_bits_to_f32(case.q_verify_bits) * np.float32(factor))
    return dataclasses.replace(case, q_draft_bits=qd, q_verify_bits=qv, scale=scale)


def _case(spec, seed):
    name, B, Hq, Hkv, D, P, bl, prefix = spec
    return W.make_block_attn_case(name, B, Hq, Hkv, D, block_len=bl, page_size=P, prefix_lens=prefix, seed=seed)


def rounding_bound(case, o_ref):
    """Elementwise bound of the bf16 roundings of P and of the output."""
    vmax = float(np.max(np.abs(W.bf16_bits_to_f32(case.kv.v_bits))))
    return 2.0 ** -8 * (np.abs(o_ref) + vmax) + 1e-4


def _check_runs(orc, case, splits_list, softmax_scale=0.0, must_rescale=(1, 3), derived_bound=False):
    dc = DeviceCase(case)
    for mode in (DIFF, VER):
        ro, rl = oracle_full(orc, case, mode)
        bound = rounding_bound(case, ro) if derived_bound else None
        for S in splits_list:
            nld.nld_rescale_count(clear=True)
            out, lse = dc.run(mode, num_splits=S, softmax_scale=softmax_scale)
            torch.cuda.synchronize()
            n = nld.nld_rescale_count(clear=True)
            what = f"{case.name} mode={mode} S={S} rescales={n}"
            if bound is None:
                compare_attn(out, lse, ro, rl, what)
            else:
                err = np.abs(out.float().cpu().numpy().astype(np.float64) - ro)
                assert np.all(err <= bound), f"{what}: max excess {float(np.max(err - bound)):.3e}"
                compare_attn(out, lse, ro, rl, what, max_abs=float(np.max(bound)))
            if S in must_rescale:
                assert n > 0, f"{case.name} mode={mode} S={S}: the rescale path did not run"


@pytest.mark.parametrize("spec", SHAPES, ids=[s[0] for s in SHAPES])
@pytest.mark.parametrize("strength", [32.0, 14.0], ids=["strong", "mild"])
def test_sink_keys_rescale(orc, spec, strength):
    """Runs of sink keys mid-prefix (tile-aligned), late in the prefix and in
    the last block slot; one split, three splits and the automatic plan."""
    case = with_sinks(_case(spec, seed=sum(spec[7]) + 41), strength)
    _check_runs(orc, case, (1, 3, 0))


@pytest.mark.parametrize("spec", [SHAPES[i] for i in (0, 1, 3, 5, 6)], ids=[SHAPES[i][0] for i in (0, 1, 3, 5, 6)])
def test_sink_keys_cluster_merges(orc, spec):
    """Explicit split counts that run as thread-block clusters: CTAs whose
    log-sum-exps differ by far more than 2^8 merge through shared memory.
    With 4 or 8 pieces a split can be a single softmax step (no step after
    the first to rescale), so only the 2-piece plan must rescale."""
    case = with_sinks(_case(spec, seed=sum(spec[7]) + 43), 32.0)
    _check_runs(orc, case, (2, 4, 8), must_rescale=(2,))


@pytest.mark.parametrize("D,splits", [(128, 5), (64, 4)])
@pytest.mark.parametrize("strength", [32.0, 14.0], ids=["strong", "mild"])
def test_row_copies_rescale(orc, D, splits, strength):
    """33..64 rows in pieces that sit in the ring whole (at most 384 tokens at
    head_dim 128, 512 at 64): the kernel with two copies of each row, whose
    copies hold maxima of their own. A piece holds several products, so that the
    sink run falls behind the first."""
    case = with_sinks(_case(("rows64", 1, 8, 2, D, 16, 16, [1500]), seed=5), strength)
    dc = DeviceCase(case)
    assert nld.nld_block_attn_route(dc.params(splits), 16)["chunk"] <= (384 if D == 128 else 512)
    _check_runs(orc, case, (splits,), must_rescale=(splits,))


@pytest.mark.parametrize("spec", [s for s in SHAPES if "odd" in s[0]], ids=[s[0] for s in SHAPES if "odd" in s[0]])
def test_odd_blocks_run_on_two_tiles(spec):
    """What the shapes above named odd are for: one CTA with two M tiles."""
    dc = DeviceCase(_case(spec, seed=1))
    for splits in (0, 1, 2, 3, 4, 8):
        route = nld.nld_block_attn_route(dc.params(splits), spec[6])
        assert route["halves"] == 1 and route["order"] == 0


@pytest.mark.parametrize("spec", SHAPES, ids=[s[0] for s in SHAPES])
def test_scaled_queries_custom_scale(orc, spec):
    """Queries times 8 and softmax_scale 0.5 (not the 1/sqrt(D) default):
    scores spread over hundreds of base-2 units."""
    case = with_scaled_queries(_case(spec, seed=sum(spec[7]) + 47), 8.0, 0.5)
    _check_runs(orc, case, (1, 3, 0), softmax_scale=0.5, derived_bound=True)


def test_rescale_counter_counts_only_rescales(orc):
    """The counter is a diagnostic: the same call on the same inputs gives the
    same output whether or not the counter was cleared, and a row set whose
    scores are all equal (identical keys) never rescales."""
    spec = SHAPES[1]
    case = _case(spec, seed=3)
    kv = case.kv
    k_same = np.broadcast_to(kv.k_bits[:1, :, :1, :], kv.k_bits.shape).copy()
    flat = dataclasses.replace(case, kv=dataclasses.replace(kv, k_bits=k_same))
    dc = DeviceCase(flat)
    nld.nld_rescale_count(clear=True)
    o1, l1 = dc.run(VER, 1)
    torch.cuda.synchronize()
    assert nld.nld_rescale_count(clear=True) == 0
    o2, l2 = dc.run(VER, 1)
    assert torch.equal(o1, o2) and torch.equal(l1, l2)
    ro, rl = oracle_full(orc, flat, VER)
    compare_attn(o1, l1, ro, rl, "identical keys")
