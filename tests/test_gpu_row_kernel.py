"""The streaming row kernel (every row call here goes through it) and the entropy mean at the edges of their splits, against the fp64
oracle (tolerances of `_compare`)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2505_18573_b200 import inputs
from _compare import ATOL, assert_close, assert_tokens
from _routes import Streaming

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(scope="module")
def e3():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2505_18573_b200 import binding
    binding.lib()
    return Streaming(binding)


def _check(e3, logits, temps, samplers=(0, 1), mask=None, workspace=None):
    rows, V = logits.shape
    z, t = inputs.to_oracle_array(logits), temps.cpu().numpy()
    for sampler in samplers:
        tok, lp, en = e3.e3_sample(logits, temps, 3, 1 << 34, 5, sampler, workspace=workspace)[:3]
        ref = oracle.sample(z, t, 3, 1 << 34, 5, sampler)
        tok = tok.cpu().numpy()
        assert_tokens(f"V{V}r{rows}s{sampler}", tok, ref, sampler)
        same = tok == ref.tok
        assert_close("ent", en.cpu().numpy(), ref.ent, ATOL[logits.dtype])
        assert_close("logp", lp.cpu().numpy()[same], ref.logp[same], ATOL[logits.dtype])
    targets = inputs.uniform_targets(rows, V, seed=3, device=DEV)
    lp, en = e3.e3_token_logp_entropy(logits, targets, mask=mask, temps=temps, workspace=workspace)[:2]
    rlp, ren, _ = oracle.token_logp_entropy(z, targets.cpu().numpy(), mask=None if mask is None else mask.cpu().numpy(), temps=t)
    assert_close("train.logp", lp.cpu().numpy(), rlp, ATOL[logits.dtype])
    assert_close("train.ent", en.cpu().numpy(), ren, ATOL[logits.dtype])


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("rows, V", [
    (5, 1024), (37, 2049), (149, 6145),   # one tile a row, a tile and an entry, three tiles and an entry
    (17, 101000), (100, 101000),          # one strip per warp of 1 and of a few tiles
    (290, 101000), (600, 33333),          # ... of a few tiles more, most warps busy; rows that begin anywhere
    (700, 65001)])                        # more than one strip per warp
def test_strip_lengths(e3, dtype, rows, V):
    logits = inputs.zipf_gaussian_logits(rows, V, seed=rows, dtype=dtype, device=DEV)
    _check(e3, logits, inputs.uniform_temps(rows, seed=V, device=DEV))


@pytest.mark.parametrize("dtype, rows, V", [(torch.bfloat16, 1790, 18001),   # one strip in a hundred more than warps, a short one
                                            (torch.float32, 300, 252000)])   # one strip per warp of more tiles than bf16 has
def test_strips_of_the_statistics(e3, dtype, rows, V):
    logits = inputs.zipf_gaussian_logits(rows, V, seed=rows, dtype=dtype, device=DEV)
    _check(e3, logits, inputs.uniform_temps(rows, seed=V, device=DEV), samplers=())


@pytest.mark.parametrize("sampler, dtype, rows, V", [
    (None, torch.bfloat16, 9000, 70001), (None, torch.bfloat16, 600, 1200001),  # runs of 305 strips, rows of 5 and 74 of 8 tiles
    (None, torch.bfloat16, 300, 2200001), (1, torch.float32, 250, 1300001),     # ... of 270, rows of two segments
    (1, torch.bfloat16, 9000, 70001), (0, torch.bfloat16, 20000, 70001),        # ... of 305, of 271 with rows of two strips of 25
    (1, torch.bfloat16, 2500, 70001), (1, torch.bfloat16, 4000, 70001), (1, torch.float32, 400, 300001),  # shorter runs than the ring
    (1, torch.float32, 200, 700001), (0, torch.bfloat16, 16000, 70001)])
def test_runs_longer_than_the_ring(e3, sampler, dtype, rows, V):
    """More strips in a block's run than the 256 it keeps records of (and nearly as many), rows that begin anywhere: the same as in
    batches of a few rows, where no warp takes a second strip."""
    g = torch.Generator(device=DEV); g.manual_seed(rows)
    logits = torch.empty((rows, V), dtype=dtype, device=DEV)
    for lo in range(0, rows, 500):
        logits[lo:lo + 500] = torch.randn((min(500, rows - lo), V), generator=g, device=DEV) * 2.5
    temps, targets = inputs.uniform_temps(rows, seed=V, device=DEV), inputs.uniform_targets(rows, V, seed=3, device=DEV)

    def call(lo, hi):
        if sampler is None:
            return e3.e3_token_logp_entropy(logits[lo:hi], targets[lo:hi], temps=temps[lo:hi])
        return e3.e3_sample(logits[lo:hi], temps[lo:hi], 7, 8, lo, sampler)
    got = call(0, rows)
    step = max(1, min(rows, 40 * 70001 // V))
    parts = [torch.cat(t) for t in zip(*(call(lo, min(lo + step, rows)) for lo in range(0, rows, step)))]
    if sampler is not None:
        assert torch.equal(got[0], parts[0])
    for a, b in zip(got[-2:], parts[-2:]):  # logp and ent: fp32 sums in another order
        assert_close("small batches", a.cpu().numpy(), b.cpu().numpy(), 2e-5)
    some = torch.arange(0, rows, max(1, rows // 9), device=DEV)
    p = torch.log_softmax(logits[some].double() / temps[some, None].double(), 1)
    assert_close("ent", got[-1][some].cpu().numpy(), -(p.exp() * p).sum(1).cpu().numpy(), ATOL[torch.float32])
    at = (targets if sampler is None else got[0])[some].long()
    assert_close("logp", got[-2][some].cpu().numpy(), p.gather(1, at[:, None])[:, 0].cpu().numpy(), ATOL[torch.float32])


@pytest.mark.parametrize("dtype, V", [(torch.bfloat16, 260001), (torch.bfloat16, 270001), (torch.float32, 300001)])
def test_whole_rows_of_several_segments(e3, dtype, V):
    """Without room for cut rows a block takes whole rows: more strips than half a ring of records, than a whole one."""
    logits = inputs.zipf_gaussian_logits(3, V, seed=V, dtype=dtype, device=DEV)
    tiny = torch.zeros(64, dtype=torch.uint8, device=DEV)
    _check(e3, logits, inputs.uniform_temps(3, seed=1, device=DEV), samplers=(0,), workspace=tiny)


@pytest.mark.parametrize("rows, V", [(140, 400001),    # 25 strips of 16 tiles a row
                                     (148, 1080001)])  # 132 strips of 8 tiles a row, which a block holds whole
def test_blocked_sampler_rows_longer_than_its_half_ring(e3, rows, V):
    """Long rows, also of several segments, in a run that still fits the ring."""
    logits = inputs.zipf_gaussian_logits(rows, V, seed=9, dtype=torch.float32, device=DEV)
    _check(e3, logits, inputs.uniform_temps(rows, seed=2, device=DEV), samplers=(1,))


@pytest.mark.parametrize("dtype, rows, V", [(torch.float32, 148, 600000), (torch.bfloat16, 300, 700001)])
def test_same_bits_with_entries_ruled_out(e3, dtype, rows, V):
    """Logits of -inf here and there: the sums of a strip do not depend on which warp took it or what that warp summed before."""
    g = torch.Generator(device=DEV); g.manual_seed(1)
    logits = torch.randn((rows, V), generator=g, device=DEV).to(dtype)
    logits.view(-1)[torch.randint(0, rows * V, (rows * 25,), generator=g, device=DEV)] = float("-inf")
    temps, targets = torch.full((rows,), 0.9, device=DEV), torch.zeros(rows, dtype=torch.int32, device=DEV)
    calls = (lambda: e3.e3_token_logp_entropy(logits, targets, temps=temps, want_gap=True),
             lambda: e3.e3_sample(logits, temps, 1, 2), lambda: e3.e3_sample(logits, temps, 1, 2, sampler=e3.E3_SAMPLER_BLOCK))
    for call in calls:
        first = call()
        for _ in range(12):
            assert all(torch.equal(a, b) for a, b in zip(first, call()))


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_entries_ruled_out(e3, dtype):
    """-inf logits in whole tiles, in parts of them, with a logit far above the others, with a NaN or a +inf (the row reads NaN)."""
    V, rows = 41003, 12
    g = torch.Generator(device=DEV); g.manual_seed(6)
    z = torch.randn((rows, V), generator=g, device=DEV)
    drop = torch.rand((rows, V), generator=g, device=DEV) < 0.1
    z[0][drop[0]] = float("-inf")
    z[1, V // 2:] = float("-inf"); z[2, :V // 2] = float("-inf")
    z[3, :] = float("-inf"); z[3, 7777] = 0.5
    z[4][~drop[4]] = float("-inf")
    z[5][drop[5]] = float("-inf"); z[5, 30000] = 60.0
    z[6][drop[6]] = float("-inf"); z[6, 12345] = float("nan")
    z[7][drop[7]] = float("-inf"); z[7, 12345] = float("inf")
    z[8, 4096:8192] = float("-inf"); z[8, 5000] = float("nan")
    z[9, 4096:8192] = float("-inf"); z[9, 5000] = float("inf")
    z[10, 100:] = float("-inf")
    z[11, 20000] = -3.0e38
    _check(e3, z.to(dtype), inputs.uniform_temps(rows, seed=4, device=DEV))


@pytest.mark.parametrize("shift, rows", [(0, 1), (1, 15), (3, 16), (7, 17), (15, 500), (5, 12300)])
def test_masks_that_begin_anywhere(e3, shift, rows):
    g = torch.Generator(device="cpu").manual_seed(rows)
    mask = (torch.rand(rows + shift, generator=g) < 0.6).to(torch.uint8).to(DEV)[shift:]
    logits = inputs.zipf_gaussian_logits(rows, 2500, seed=rows, dtype=torch.bfloat16, device=DEV)
    _check(e3, logits, inputs.uniform_temps(rows, seed=3, device=DEV), samplers=(), mask=mask)


@pytest.mark.parametrize("std, temp", [(0.05, 1.0), (1.0, 1.0), (1.0, 3.0), (2.5, 1.0)])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_token_sampler_on_flat_rows(e3, dtype, std, temp):
    """Rows with many logits close to the largest, on both sides of the rule that passes over them for the first bound."""
    g = torch.Generator(device=DEV); g.manual_seed(4)
    logits = (torch.randn((65, 20000), generator=g, device=DEV) * std).to(dtype)
    _check(e3, logits, torch.full((65,), temp, device=DEV), samplers=(0,))


@pytest.mark.parametrize("n", [1, 1023, 32767, 32768, 32769, 65537, 262143, 262144, 262145, 300001])
def test_mean_at_the_edges_of_a_cluster(e3, n):
    g = torch.Generator(device="cpu").manual_seed(n)
    ent = (torch.rand(n, generator=g) * 10).to(DEV)
    mask = (torch.rand(n + 1, generator=g) < 0.7).to(torch.uint8).to(DEV)[1:]
    for m in (mask, None):
        out = e3.e3_masked_mean_entropy(ent, m)
        mean, count = oracle.masked_mean_entropy(ent.cpu().numpy(), None if m is None else m.cpu().numpy())
        assert float(out[1]) == count and float(out[0]) == pytest.approx(mean, rel=1e-12)
