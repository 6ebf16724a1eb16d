"""Rows in which runs of logits are a large negative number (a fill value in place of -inf), against the fp64 oracle: in the kernel of
short calls and in the streaming kernel."""
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


def _rows(V, dtype):
    """Runs of the lengths that a warp, a tile or a block of either kernel looks at, at the start, inside and at the end of a row; padding
    with a large logit beside it; rows of the fill value alone, and of all of it but one entry."""
    g = torch.Generator().manual_seed(V)
    z = []
    for fill in (-1e9, -1e10, -1e30, torch.finfo(dtype).min):
        def row(*spans):
            z.append(torch.randn(V, generator=g) * 2.5)
            for lo, hi in spans:
                z[-1][lo:hi] = fill
            return z[-1]
        for n in (512, 1024, 2048, 8192):
            row((0, n)), row((V - n, V)), row((V // 2 - 5, V // 2 - 5 + n))
        row((100, V)), row((0, V - 100))
        row((0, V // 2))[V - 7] = 1e4
        row((0, V))[V // 3] = 1.5
        row((0, V))
        row((0, V))[V // 3] = 1e9
        row((512, 7000), (8000, V))[3] = 50.0
    return torch.stack(z).to(dtype)


@pytest.mark.parametrize("kernel", ["short", "streaming"])
@pytest.mark.parametrize("V", [20480, 20001, 2000])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_runs_of_a_fill_value(e3, dtype, V, kernel):
    logits = (_rows(V, dtype) if V > 16384 else _rows(20001, dtype)[:, 18001:].contiguous()).to(DEV)
    rows, atol = len(logits), ATOL[dtype]
    if kernel == "streaming":
        e3 = Streaming(e3)
    else:
        assert all(short(e3, rows, V, dtype, sampler) for sampler in (-1, 0, 1, 2))
    for tau in (1.0, 0.61, 0.87, 1.37):
        temps = torch.full((rows,), tau, device=DEV)
        z, t = inputs.to_oracle_array(logits), temps.cpu().numpy()
        gap = oracle.row_gap(z, t)
        for sampler in (0, 1, e3.E3_SAMPLER_TOKEN_AUDIT):
            tok, lp, en, gp = e3.e3_sample(logits, temps, 3, 9, 5, sampler, want_gap=True)
            ref = oracle.sample(z, t, 3, 9, 5, sampler % 2)
            tok = tok.cpu().numpy()
            assert_tokens(f"tau{tau}s{sampler}", tok, ref, sampler)
            same = tok == ref.tok
            assert_close("ent", en.cpu().numpy(), ref.ent, atol)
            assert_close("logp", lp.cpu().numpy()[same], ref.logp[same], atol)
            assert_close("gap", gp.cpu().numpy(), gap, atol)
        targets = logits.float().argmax(1).to(torch.int32)
        lp, en, gp = e3.e3_token_logp_entropy(logits, targets, temps=temps, want_gap=True)
        rlp, ren, _ = oracle.token_logp_entropy(z, targets.cpu().numpy(), temps=t)
        assert_close("train.logp", lp.cpu().numpy(), rlp, atol)
        assert_close("train.ent", en.cpu().numpy(), ren, atol)
        assert_close("train.gap", gp.cpu().numpy(), gap, atol)
        # entries of the fill value as targets: the division by tau and the product with its reciprocal round once each
        targets = logits.float().argmin(1).to(torch.int32)
        lp, _ = e3.e3_token_logp_entropy(logits, targets, temps=temps)
        rlp = oracle.token_logp_entropy(z, targets.cpu().numpy(), temps=t)[0]
        ok = np.abs(rlp) < 3e38
        assert_close("fill.logp", lp.cpu().numpy()[ok] / np.maximum(1, np.abs(rlp[ok])), rlp[ok] / np.maximum(1, np.abs(rlp[ok])), atol)
