"""The row kernel of short calls at the edges of its parts, against the fp64 oracle and against the streaming kernel."""
import numpy as np
import pytest
import torch

import oracle
from paper_2505_18573_b200 import inputs
from _compare import ATOL, assert_close, assert_tokens
from _routes import Streaming, short

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(scope="module")
def e3():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2505_18573_b200 import binding
    binding.lib()
    return binding


def _check(e3, logits, temps, mask=None):
    rows, V = logits.shape
    z, t = inputs.to_oracle_array(logits), temps.cpu().numpy()
    atol = ATOL[logits.dtype]
    assert any(short(e3, rows, V, logits.dtype, sampler) for sampler in (-1, 0, 1)) or (V == 212993 and logits.dtype == torch.float32)
    for sampler in (0, 1):
        tok, lp, en, gap = e3.e3_sample(logits, temps, 3, 1 << 34, 5, sampler, want_gap=True)
        ref = oracle.sample(z, t, 3, 1 << 34, 5, sampler)
        tok = tok.cpu().numpy()
        assert_tokens(f"V{V}r{rows}s{sampler}", tok, ref, sampler)
        same = tok == ref.tok
        assert_close("ent", en.cpu().numpy(), ref.ent, atol)
        assert_close("logp", lp.cpu().numpy()[same], ref.logp[same], atol)
        assert_close("gap", gap.cpu().numpy(), oracle.row_gap(z, t), atol)
    targets = inputs.uniform_targets(rows, V, seed=3, device=DEV)
    m = None if mask is None else mask.cpu().numpy()
    lp, en = e3.e3_token_logp_entropy(logits, targets, mask=mask, temps=temps)
    rlp, ren, _ = oracle.token_logp_entropy(z, targets.cpu().numpy(), mask=m, temps=t)
    assert_close("train.logp", lp.cpu().numpy(), rlp, atol)
    assert_close("train.ent", en.cpu().numpy(), ren, atol)


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("rows, V", [
    (3, 4095), (3, 4096), (3, 4097), (2, 65537),           # one part, two, sixteen: a last part of a few entries or of none
    (40, 16640), (40, 16641), (12, 70001),                 # parts of 256-thread blocks, of 512-thread ones; rows that begin anywhere
    (200, 26624), (200, 53248), (7, 212992), (1, 425984),  # the longest parts
    (7, 212993),                                           # ... one entry more than those of fp32 hold
    (500, 17408), (300, 35841),                            # three and four blocks of 256 threads per SM
    (900, 26001)])                                         # sampler 0: a block a row, more than two waves of them
def test_parts(e3, dtype, rows, V):
    logits = inputs.zipf_gaussian_logits(rows, V, seed=rows, dtype=dtype, device=DEV)
    _check(e3, logits, inputs.uniform_temps(rows, seed=V, device=DEV))


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("rows, V", [(301, 20001), (2000, 17001), (1300, 26100)])  # four waves, up to seven of a block a row
def test_mask(e3, dtype, rows, V):
    logits = inputs.zipf_gaussian_logits(rows, V, seed=1, dtype=dtype, device=DEV)
    mask = (torch.rand(rows, generator=torch.Generator().manual_seed(2)) < 0.5).to(torch.uint8).to(DEV)
    logits[mask == 0] = float("nan")  # (these are not looked at)
    temps, targets = inputs.uniform_temps(rows, seed=3, device=DEV), inputs.uniform_targets(rows, V, seed=4, device=DEV)
    assert short(e3, rows, V, dtype, masked=True)
    total = torch.zeros(2, dtype=torch.float64, device=DEV)
    lp, en = e3.e3_token_logp_entropy(logits, targets, mask=mask, temps=temps, out_sum=total)
    rlp, ren, _ = oracle.token_logp_entropy(inputs.to_oracle_array(logits), targets.cpu().numpy(), mask=mask.cpu().numpy(), temps=temps.cpu().numpy())
    assert_close("logp", lp.cpu().numpy(), rlp, ATOL[dtype])
    assert_close("ent", en.cpu().numpy(), ren, ATOL[dtype])
    assert float(total[1]) == int(mask.sum()) and float(total[0]) == pytest.approx(float(en.double().sum()), rel=1e-12)


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("std", [0.0, 0.02, 3.0, 40.0])
def test_few_entries_and_flat_rows(e3, dtype, std):
    """No entry with coarse byte 255 at all, or every entry above the gate."""
    g = torch.Generator(device=DEV); g.manual_seed(7)
    for V in (1, 15, 17, 100, 257, 1000, 5000):
        _check(e3, (torch.randn((9, V), generator=g, device=DEV) * std).to(dtype), torch.full((9,), 0.7, device=DEV))


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("V, first", [(41000, 0), (41003, 0), (41000, 1)])
def test_same_as_the_streaming_kernel(e3, dtype, V, first):
    """A batch through the streaming kernel and the same rows a few at a time: entries ruled out, NaN, infinities, greedy rows, temperatures
    that cannot be used, rows of any alignment."""
    rows, unit = 1040, 13
    g = torch.Generator(device=DEV); g.manual_seed(V)
    z = torch.randn((unit, V + first), generator=g, device=DEV) * 2.5
    drop = torch.rand((unit, V + first), generator=g, device=DEV) < 0.1
    ninf = float("-inf")
    z[0][drop[0]] = ninf
    z[1, V // 2:] = ninf
    z[2, :V // 2] = ninf
    z[3, :] = ninf; z[3, 7777] = 0.5
    z[4, :] = ninf
    z[5][drop[5]] = ninf; z[5, 30000] = 60.0
    z[6, 12345] = float("nan")
    z[7][drop[7]] = ninf; z[7, 40990] = float("inf")
    z[8, 20000] = -3.0e38
    z[9] = z[9].round()  # (ties)
    logits = z.to(dtype).repeat(rows // unit, 1)[:, first:]
    temps = inputs.uniform_temps(rows, seed=5, device=DEV)
    temps[10::unit] = 0.0
    temps[11::2 * unit] = -1.0
    temps[12::unit] = 1e-3
    temps[9::2 * unit] = 0.0
    targets = inputs.uniform_targets(rows, V, seed=6, device=DEV)
    targets[::17] = V  # (not a token: no log-probability)

    def call(which, lo, hi):
        way = Streaming(e3) if hi - lo == rows else e3
        assert way is not e3 or short(e3, hi - lo, V, dtype, -1 if which is None else which)
        if which is None:
            return way.e3_token_logp_entropy(logits[lo:hi], targets[lo:hi], temps=temps[lo:hi], want_gap=True)
        return way.e3_sample(logits[lo:hi], temps[lo:hi], 11, 12, lo, which, want_gap=True)
    for which in (None, 0, 1, e3.E3_SAMPLER_TOKEN_AUDIT):
        got = [t.cpu().numpy() for t in call(which, 0, rows)]
        parts = [call(which, lo, lo + 40) for lo in range(0, rows, 40)]
        few = [torch.cat(t).cpu().numpy() for t in zip(*parts)]
        if which is not None:
            assert np.array_equal(got[0], few[0])
            got, few = got[1:], few[1:]
        for a, b in zip(got, few):
            assert np.array_equal(np.isnan(a), np.isnan(b))
            ok = ~np.isnan(a)
            assert_close("values", a[ok], b[ok], 2e-5)


@pytest.mark.parametrize("sampler", [None, 0, 1])
def test_graph_replay_on_cut_rows_of_the_streaming_kernel(e3, sampler):
    rows, V = 330, 151936
    data = [inputs.zipf_gaussian_logits(rows, V, seed=80 + i, dtype=torch.bfloat16, device=DEV) for i in range(2)]
    logits, temps = data[0].clone(), inputs.uniform_temps(rows, seed=84, device=DEV)
    targets = inputs.uniform_targets(rows, V, seed=85, device=DEV)

    assert not short(e3, rows, V, torch.bfloat16, -1 if sampler is None else sampler)

    def run(stream=None):
        if sampler is None:
            return e3.e3_token_logp_entropy(logits, targets, temps=temps, stream=stream)
        return e3.e3_sample(logits, temps, 3, 4, 0, sampler, stream=stream)
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        run(side)
    side.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        out = run(side)
    for i in (1, 0, 1):
        logits.copy_(data[i])
        graph.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(out, run()))


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_temperatures_that_cannot_be_used_between_others(e3, dtype):
    """Several waves of blocks of which every other one has nothing to sum: its copies land before its memory goes to the next one."""
    rows, V = 1100, 20001 if dtype == torch.float32 else 40001
    logits = inputs.zipf_gaussian_logits(rows, V, seed=2, dtype=dtype, device=DEV)
    temps = inputs.uniform_temps(rows, seed=3, device=DEV)
    for k, bad in enumerate((-1.0, float("nan"), float("inf"))):
        temps[2 * k::6] = bad
    assert short(e3, rows, V, dtype, 0) and short(e3, rows, V, dtype, masked=True)
    z, t = inputs.to_oracle_array(logits), temps.cpu().numpy()
    ref = oracle.sample(z, t, 3, 4, 0, 0)
    targets = inputs.uniform_targets(rows, V, seed=3, device=DEV)
    mask = torch.ones(rows, dtype=torch.uint8, device=DEV)
    rlp, ren, _ = oracle.token_logp_entropy(z, targets.cpu().numpy(), temps=t)
    for _ in range(5):
        tok, lp, en = e3.e3_sample(logits, temps, 3, 4)
        assert_tokens("tok", tok.cpu().numpy(), ref)
        assert_close("ent", en.cpu().numpy(), ref.ent, ATOL[dtype])
        lp, en = e3.e3_token_logp_entropy(logits, targets, mask=mask, temps=temps)
        assert_close("train.logp", lp.cpu().numpy(), rlp, ATOL[dtype])
        assert_close("train.ent", en.cpu().numpy(), ren, ATOL[dtype])


@pytest.mark.parametrize("rows, V, row", [(6, 151936, 2), (6, 151936, 5), (1, 151936, 0), (100, 20001, 99)])  # 8, 16 and 2 parts a row
@pytest.mark.parametrize("sampler", [None, 0, 1])
def test_a_part_that_is_never_handed_over(e3, sampler, rows, V, row):
    """The wait for it runs out: the row reads NaN, the status word says so, the other rows and the next call are as ever."""
    assert short(e3, rows, V, torch.bfloat16, -1 if sampler is None else sampler) > 1
    logits = inputs.zipf_gaussian_logits(rows, V, seed=5, dtype=torch.bfloat16, device=DEV)
    temps, targets = inputs.uniform_temps(rows, seed=6, device=DEV), inputs.uniform_targets(rows, V, seed=7, device=DEV)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)

    def run():
        if sampler is None:
            return e3.e3_token_logp_entropy(logits, targets, temps=temps, status=status)
        return e3.e3_sample(logits, temps, 3, 4, 0, sampler, status=status)
    want = run()
    assert int(status[0]) == 0
    e3.e3_test_arm_stall(-2 - row, 5_000_000)  # 5 ms instead of two seconds
    got = run()
    assert int(status[0]) == e3.E3_STATUS_TIMEOUT
    others = torch.arange(rows, device=DEV) != row
    for g, w in zip(got, want):
        assert torch.equal(g[others], w[others])
        assert int(g[row]) == -1 if g.dtype == torch.int32 else bool(torch.isnan(g[row]))
    status.zero_()
    assert all(torch.equal(a, b) for a, b in zip(run(), want)) and int(status[0]) == 0
