"""Whole-sequence forward attention under the event-factorized mask (Sec. 3.4, Fig. 3)
through the C ABI, against the fp64 oracle.  Same bar as the decode path: max-abs <= 1e-2,
relative-L2 <= 2e-3, LSE within 1e-3."""
import math

import numpy as np
import pytest
import torch

import oracle
from late_writer import late_store
from paper_2607_02963_gb300 import binding as B
from paper_2607_02963_gb300 import synth

pytestmark = pytest.mark.gpu

MAX_ABS, REL_L2, LSE_ABS = 1e-2, 2e-3, 1e-3


@pytest.fixture(scope="module", autouse=True)
def _cuda(padlib):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.init()


def _dev(bits):
    return torch.from_numpy(np.ascontiguousarray(bits).view(np.int16)).view(torch.bfloat16).cuda()


def _run(prefix, lens, h_q, h_kv, D, seed, out_dtype=0, heads=None, sigma=None, flags=0):
    qb, kb, vb = synth.prefill_inputs(seed, prefix, lens, h_q, h_kv, D, k_scale_sigma=sigma)
    N = qb.shape[0]
    prob = B.make_problem(h_q, h_kv, D, 16, 1.0 / math.sqrt(D), out_dtype=out_dtype, flags=flags)
    out = torch.empty((N, h_q, D), dtype=torch.float32 if out_dtype == 0 else torch.bfloat16, device="cuda")
    lse = torch.empty((N, h_q), dtype=torch.float32, device="cuda")
    B.pad_prefill_attn(prob, prefix, lens, _dev(qb), _dev(kb), _dev(vb), out, lse)
    torch.cuda.synchronize()
    B.pad_prefill_status()
    ro, rl = oracle.prefill_attention(oracle.bf16_to_f64(qb), oracle.bf16_to_f64(kb), oracle.bf16_to_f64(vb),
                                      prefix, lens, 1.0 / math.sqrt(D), heads=heads)
    go, gl = out.float().cpu().numpy(), lse.cpu().numpy()
    hs = list(range(h_q)) if heads is None else heads
    go, gl, ro, rl = go[:, hs], gl[:, hs], ro[:, hs], rl[:, hs]
    assert np.all(np.isfinite(go))
    err = np.abs(go - ro)
    assert err.max() <= MAX_ABS, err.max()
    assert np.linalg.norm(go - ro) / np.linalg.norm(ro) <= REL_L2 + (2.0 ** -9 if out_dtype else 0)
    assert np.abs(gl - rl).max() <= LSE_ABS


@pytest.mark.parametrize("prefix,lens", [
    (300, [5, 0, 70, 1, 129]),      # ragged branches, one empty, tiles straddling branches
    (257, []),                      # no branches: plain causal attention
    (0, [40, 90]),                  # no shared prefix
    (64, [64, 64]),                 # every boundary on a tile edge
    (1000, [42] * 13),              # the paper's average: 13 events of ~42 caption tokens
])
@pytest.mark.parametrize("flags", [0, B.FLAG_PREFIX_MMA])
def test_prefill_matches_oracle_d128(prefix, lens, flags):
    """head_dim 128 on the tensor-core kernel (default) and on the warp-level kernel."""
    _run(prefix, lens, 28, 4, 128, seed=prefix + len(lens), flags=flags)


def test_prefill_d64_and_bf16_output():
    _run(200, [3, 17, 66], 8, 2, 64, seed=5)
    _run(200, [3, 17, 66], 8, 2, 64, seed=6, out_dtype=1)


def test_prefill_long_prefix_sampled_heads():
    """An 8k-token prefix with 13 branches (outlier K channels); two heads checked."""
    _run(8192, [42] * 13, 28, 4, 128, seed=7, heads=[0, 27], sigma=0.5)


def test_prefill_tc_group_sizes_and_bf16():
    """Other GQA groups on the tensor-core kernel (128 / G tokens per CTA), bf16 output."""
    _run(500, [30, 2, 77], 8, 2, 128, seed=8)            # G = 4: 32 tokens per CTA
    _run(500, [30, 2, 77], 16, 1, 128, seed=9)           # G = 16: 8 tokens per CTA
    _run(500, [30, 2, 77], 28, 4, 128, seed=10, out_dtype=1)


@pytest.mark.parametrize("D,h_q,h_kv,prefix,lens", [
    (64, 14, 2, 36, [1]),                 # one query tile (36 tokens at G = 7) and one token over
    (64, 14, 2, 127, [1, 127, 2]),        # key tiles one short of full, a branch across a tile edge
    (64, 4, 1, 129, []),                  # a key tile of one token; tail slot with no rows
    (64, 16, 1, 0, [1]),                  # one token in all
    (64, 3, 3, 300, [60, 0, 200]),        # G = 1: 128 tokens per slot
    (128, 3, 3, 300, [60, 0, 200]),
    (128, 28, 4, 18, [17, 19, 36]),       # branches that begin and end inside a slot
    (128, 32, 2, 640, [128] * 3),         # G = 16: 8 tokens per slot
])
@pytest.mark.parametrize("out_dtype", [0, 1])
def test_prefill_tc_edges(D, h_q, h_kv, prefix, lens, out_dtype):
    """Tile, slot and branch edges of the tensor-core kernel at both head sizes."""
    _run(prefix, lens, h_q, h_kv, D, seed=prefix + D, out_dtype=out_dtype)


@pytest.mark.parametrize("D", [64, 128])
def test_prefill_warp_level_kernel_still_forced(D):
    _run(200, [3, 17, 66], 8, 2, D, seed=D, flags=B.FLAG_PREFIX_MMA)


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("at", [100, 130, 230, 255, 600])
def test_prefill_growing_maximum(D, at):
    """Scores that outgrow the running maximum by far more than 2^8 at one key, in the first or
    the last part of a tile, so that O, l and the part's P are redone there.  The bar stays
    the usual one: P's rounding (2^-9 per weight) enters as it does elsewhere."""
    prefix, lens, h_q, h_kv = 700, [40, 50], 14, 2
    qb, kb, vb = synth.prefill_inputs(at, prefix, lens, h_q, h_kv, D)
    q, k = oracle.bf16_to_f64(qb), oracle.bf16_to_f64(kb)
    q[:, :, 0] = 4.0                      # exact in bf16
    k[:, :, 0] = 0.0
    k[at, :, 0] = 32.0                    # score +128 / sqrt(D): 16 at D 64, 11.3 at D 128 (nats)
    qb, kb = synth.f32_to_bf16_bits(q.astype(np.float32)), synth.f32_to_bf16_bits(k.astype(np.float32))
    N = qb.shape[0]
    out = torch.empty((N, h_q, D), device="cuda")
    lse = torch.empty((N, h_q), device="cuda")
    B.pad_prefill_attn(B.make_problem(h_q, h_kv, D, 16, 1.0 / math.sqrt(D)), prefix, lens, _dev(qb), _dev(kb),
                       _dev(vb), out, lse)
    torch.cuda.synchronize()
    B.pad_prefill_status()
    ro, rl = oracle.prefill_attention(oracle.bf16_to_f64(qb), oracle.bf16_to_f64(kb), oracle.bf16_to_f64(vb),
                                      prefix, lens, 1.0 / math.sqrt(D))
    go = out.cpu().numpy()
    assert np.abs(go - ro).max() <= MAX_ABS
    assert np.linalg.norm(go - ro) / np.linalg.norm(ro) <= REL_L2
    assert np.abs(lse.cpu().numpy() - rl).max() <= LSE_ABS


@pytest.mark.parametrize("D,h_q,h_kv,prefix,lens", [
    # one slot of queries, its key tiles shared out: one tile, two, an odd and an even number of them
    (128, 28, 4, 100, [3]), (128, 28, 4, 120, [40]), (128, 16, 1, 300, [5, 0, 130]), (64, 14, 2, 400, [1, 20]),
    # enough kv-heads for two waves of those: two slots of queries, the last one empty or full
    (128, 64, 32, 640, [30, 34]), (128, 64, 32, 690, [14, 0, 65]), (64, 64, 32, 700, [3]),
])
def test_prefill_slots(D, h_q, h_kv, prefix, lens):
    """fp32 against the oracle; bf16 output is the same result rounded to nearest even."""
    _run(prefix, lens, h_q, h_kv, D, seed=31)
    q, k, v = (_dev(x) for x in synth.prefill_inputs(31, prefix, lens, h_q, h_kv, D))
    outs = []
    for dt in (torch.float32, torch.bfloat16):
        out, lse = torch.empty(q.shape, dtype=dt, device="cuda"), torch.empty(q.shape[:2], device="cuda")
        prob = B.make_problem(h_q, h_kv, D, 16, 1.0 / math.sqrt(D), out_dtype=int(dt == torch.bfloat16))
        B.pad_prefill_attn(prob, prefix, lens, q, k, v, out, lse)
        outs.append(out)
    torch.cuda.synchronize()
    assert torch.equal(outs[0].bfloat16(), outs[1])


@pytest.mark.parametrize("D,h_q,h_kv,prefix,lens", [
    (64, 14, 2, 300, [200, 90, 130]),     # key tiles shared out of one query group
    (128, 28, 4, 300, [200, 90, 130]),
    (64, 64, 32, 700, [140, 100, 200]),   # two query groups
    (128, 64, 32, 700, [140, 100, 200]),
])
@pytest.mark.parametrize("flags", [0, B.FLAG_PREFIX_MMA])
def test_prefill_branch_does_not_reach_the_others(D, h_q, h_kv, prefix, lens, flags):
    """A branch of NaN and infinite K and V leaves the prefix and the other branches as they are, beside the
    query tile that it shares with its neighbours (at most two groups of 128 / G tokens, or 64 on the
    warp-level kernel)."""
    q, k, v = (_dev(x) for x in synth.prefill_inputs(5, prefix, lens, h_q, h_kv, D))
    prob = B.make_problem(h_q, h_kv, D, 16, 1.0 / math.sqrt(D), flags=flags)
    lo = prefix
    res = []
    for bad in (False, True):
        if bad:
            k[lo:lo + lens[0]] = float("nan")
            v[lo:lo + lens[0]] = float("inf")
            v[lo:lo + lens[0]:2] = float("nan")
        out, lse = torch.empty(q.shape, device="cuda"), torch.empty(q.shape[:2], device="cuda")
        B.pad_prefill_attn(prob, prefix, lens, q, k, v, out, lse)
        torch.cuda.synchronize()
        B.pad_prefill_status()
        res.append((out, lse))
    share = 64 if flags else 2 * (128 // (h_q // h_kv))
    keep = torch.ones(q.shape[0], dtype=torch.bool, device="cuda")
    keep[max(0, lo - share):lo + lens[0] + share] = False
    assert int(keep.sum()) > 100 and bool(keep[-1])
    for a, b in zip(*res):
        assert torch.equal(a[keep], b[keep])


@pytest.mark.parametrize("D,h_q,h_kv,prefix,lens", [
    # a few CTAs over one wave of 152 SMs: the first tokens in pairs beside the rest, from one token group
    # in pairs to nearly half; all prefix, all branches and both among the pairs
    (128, 32, 8, 600, [10]), (128, 32, 8, 500, [40, 0, 80, 40]), (128, 28, 4, 700, [40] * 4),
    (128, 32, 8, 0, [200, 150, 300, 33]), (64, 32, 8, 560, [7] * 9), (128, 8, 8, 2300, [140, 1]),
])
@pytest.mark.parametrize("out_dtype", [0, 1])
def test_prefill_two_grids(D, h_q, h_kv, prefix, lens, out_dtype):
    """Behind a grid that stores the inputs long after it has released its dependents, and ahead of one that
    reads the result at once: both grids of the call keep stream order.  (fp32 against the oracle; the bf16
    output is that result rounded.)"""
    if out_dtype == 0:
        _run(prefix, lens, h_q, h_kv, D, seed=prefix + len(lens))
    true = [_dev(x) for x in synth.prefill_inputs(prefix + len(lens), prefix, lens, h_q, h_kv, D)]
    prob = B.make_problem(h_q, h_kv, D, 16, 1.0 / math.sqrt(D), out_dtype=out_dtype)
    side, res = torch.cuda.Stream(), []
    if out_dtype:
        out32 = torch.empty(true[0].shape, device="cuda")
        B.pad_prefill_attn(B.make_problem(h_q, h_kv, D, 16, 1.0 / math.sqrt(D)), prefix, lens, *true, out32)
    for late in (False, True):
        q, k, v = (torch.full_like(t, 2.0) if late else t.clone() for t in true)
        out = torch.full(q.shape, float("nan"), dtype=torch.bfloat16 if out_dtype else torch.float32, device="cuda")
        lse = torch.full(q.shape[:2], float("nan"), device="cuda")
        torch.cuda.synchronize()
        with torch.cuda.stream(side):
            if late:
                late_store(list(zip((q, k, v), true)), side)
            B.pad_prefill_attn(prob, prefix, lens, q, k, v, out, lse)
            res.append((out.clone(), lse.clone()))
        torch.cuda.synchronize()
        B.pad_prefill_status(side)
    for a, b in zip(*res):
        assert torch.equal(a, b) and bool(torch.isfinite(a).all())
    assert not out_dtype or torch.equal(res[0][0], out32.bfloat16())
