"""Performance cases: the work a reinforcement-learning program has this library do, through the public binding.

One step of such a program samples tokens for every running rollout (`e3_sample`), later takes the log-probabilities and
entropies of the response tokens (`e3_token_logp_entropy`), turns rewards into advantages and the entropies into a batch mean
(`e3_group_advantage`, `e3_masked_mean_entropy`), evaluates the objective (`e3_grpo_objective`) and goes back to the logits
(`e3_token_logp_entropy_backward`).  `listed()` holds sizes of each of these calls, `draw()` gives more from the same ranges.
"""
import math

import torch

from paper_2505_18573_b200 import binding as e3

DEVICE = "cuda"
DTYPES = {"fp32": torch.float32, "bf16": torch.bfloat16}
ESIZE = {"fp32": 4, "bf16": 2}
SAMPLERS = {"token": e3.E3_SAMPLER_TOKEN, "block": e3.E3_SAMPLER_BLOCK}
CHUNK = 1 << 28  # logits made at a time


def _sample(rows, vocab, dtype, sampler, like="text"):
    return {"call": "sample", "rows": rows, "vocab": vocab, "dtype": dtype, "sampler": sampler, "like": like}


def _train(seqs, tokens, min_len, vocab, dtype, gap=False, row_temps=False):
    return {"call": "train", "seqs": seqs, "tokens": tokens, "min_len": min_len, "vocab": vocab, "dtype": dtype, "gap": gap,
            "row_temps": row_temps}


def _backward(seqs, tokens, min_len, vocab, dtype, entropy_grad):
    return {"call": "backward", "seqs": seqs, "tokens": tokens, "min_len": min_len, "vocab": vocab, "dtype": dtype,
            "entropy_grad": entropy_grad}


def _objective(seqs, tokens, min_len):
    return {"call": "objective", "seqs": seqs, "tokens": tokens, "min_len": min_len}


def _statistics(seqs, tokens, min_len):
    return {"call": "statistics", "seqs": seqs, "tokens": tokens, "min_len": min_len}


def listed():
    return [
        # one decode step of a small run: 8 prompts x 8 rollouts, a 32,000-entry vocabulary in fp32; launch latency counts
        dict(_sample(64, 32000, "fp32", "block"), name="sample block small"),
        # the tail of a rollout, when only one prompt's group of 8 is still decoding; the default sampler
        dict(_sample(8, 151936, "bf16", "token"), name="sample token few rows"),
        # one decode step of the headline batch: 64 prompts x 8 rollouts, both samplers
        dict(_sample(512, 151936, "bf16", "block"), name="sample block rollout"),
        dict(_sample(512, 151936, "bf16", "token"), name="sample token rollout"),
        # one decode step under the dynamic budget: 256 prompts sharing 4,096 rollouts
        dict(_sample(4096, 151936, "bf16", "block"), name="sample block budget"),
        # peaked and flat rows side by side at widely different temperatures, the widest vocabulary, fp32
        dict(_sample(1024, 256000, "fp32", "token", "stress"), name="sample token stress"),
        # training forward over four responses of up to 2,048 tokens with the batch entropy
        dict(_train(4, 2048, 256, 151936, "bf16"), name="train forward"),
        # training forward with a vocabulary whose rows start at any address, one temperature per row and the gap statistic
        dict(_train(3, 231, 64, 33333, "bf16", True, True), name="train forward odd vocab"),
        # backward of a 2,048-token chunk for the policy gradient alone
        dict(_backward(1, 2048, 1500, 151936, "bf16", False), name="backward chunk"),
        # backward with an entropy bonus, fp32, odd vocabulary
        dict(_backward(3, 100, 30, 33333, "fp32", True), name="backward odd vocab"),
        # the objective of one batch: 512 responses of up to 2,048 tokens
        dict(_objective(512, 2048, 256), name="objective batch"),
        # advantages of 512 rollouts in ragged groups, then the mean entropy of 64 responses: a few hundred kilobytes in all
        dict(_statistics(64, 2048, 256), name="batch statistics"),
    ]


# Largest sizes of each call (logits, or tokens where there are none): no drawn case is larger than the listed ones.
MOST = {"sample": 4096 * 151936, "token": 1024 * 256000, "train": 6144 * 151936, "backward": 2048 * 151936,
        "objective": 512 * 2048, "statistics": 512 * 2048}


def draw(rng):
    def spread(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def a_vocab():  # padded to a multiple of 64 as most are, or whatever the tokenizer has
        v = spread(8000, 256000)
        return v // 64 * 64 if rng.random() < 0.5 else v

    def lengths(most):  # responses and their longest length; a batch of a few short ones up to the listed batches
        tokens = spread(min(16, most), min(2048, most))
        seqs = spread(1, max(1, min(512, most // tokens)))
        return seqs, tokens, max(1, tokens // rng.randint(2, 8))

    call = rng.choice(("sample", "sample", "sample", "train", "train", "backward", "backward", "objective", "statistics"))
    dtype = rng.choice(("bf16", "bf16", "fp32"))
    if call == "sample":
        sampler, vocab = rng.choice(("block", "token")), a_vocab()
        most = MOST["token" if sampler == "token" else "sample"] * 2 // (1 if sampler == "token" else ESIZE[dtype])
        return _sample(spread(1, min(4096, max(1, most // 2 // vocab))), vocab, dtype, sampler, rng.choice(("text", "text", "text", "stress")))
    if call == "train":
        vocab = a_vocab()
        return _train(*lengths(MOST["train"] * 2 // ESIZE[dtype] // vocab), vocab, dtype, rng.random() < 0.3, rng.random() < 0.5)
    if call == "backward":
        vocab = a_vocab()
        return _backward(*lengths(MOST["backward"] * 2 // ESIZE[dtype] // vocab), vocab, dtype, rng.random() < 0.5)
    return (_objective if call == "objective" else _statistics)(*lengths(MOST[call]))


# ------------------------------------------------------------------------------------------------------------------- inputs
def _generator(seed):
    g = torch.Generator(device=DEVICE)
    g.manual_seed(seed)
    return g


def _logits(g, rows, vocab, dtype, like="text"):
    """Rows as a language model gives them: a Gaussian body and a Zipf-like bias over a random ranking ("text"), or in turn
    one entry far above the rest and nearly equal entries ("stress")."""
    out = torch.empty((rows, vocab), dtype=DTYPES[dtype], device=DEVICE)
    step = max(2, CHUNK // vocab // 2 * 2)
    for lo in range(0, rows, step):
        n = min(step, rows - lo)
        z = torch.randn((n, vocab), generator=g, device=DEVICE)
        if like == "text":
            rank = torch.rand((n, vocab), generator=g, device=DEVICE).mul_(vocab)
            z.mul_(3.0).sub_(rank.log1p_().mul_(1.2))
        else:
            z[1::2] *= 0.1
            hot = torch.randint(0, vocab, (len(z[0::2]), 1), generator=g, device=DEVICE)
            z[0::2].scatter_(1, hot, z[0::2].amax(1, keepdim=True) + 25.0)
        out[lo:lo + n] = z
    return out


def _uniform(g, n, lo, hi):
    return torch.rand(n, generator=g, device=DEVICE) * (hi - lo) + lo


def _lengths(case):
    """Response lengths of a batch, evenly spread between the shortest and the longest: a list."""
    n, lo, hi = case["seqs"], case["min_len"], case["tokens"]
    return [hi] if n == 1 and lo == hi else [lo + (hi - lo) * (2 * i + 1) // (2 * n) for i in range(n)]


def _mask(g, case):
    """uint8 [seqs, tokens]: the first L tokens of every response count, the lengths in a random order."""
    lens = torch.tensor(_lengths(case), device=DEVICE)[torch.randperm(case["seqs"], generator=g, device=DEVICE)]
    return (torch.arange(case["tokens"], device=DEVICE) < lens[:, None]).to(torch.uint8)


def _groups(g, n):
    """Offsets of ragged groups of n rollouts: sizes evenly spread from 2 to 32 in a random order, the last one takes the rest."""
    k = max(1, n // 17)
    sizes = torch.tensor([2 + 30 * (2 * i + 1) // (2 * k) for i in range(k)], device=DEVICE)[torch.randperm(k, generator=g, device=DEVICE)]
    ends = torch.cumsum(sizes, 0)
    ends[-1] = n
    return torch.cat([ends.new_zeros(1), ends])


def _rollouts(case):
    return 8 * case["seqs"]  # rewards of a batch whose responses are looked at in eight micro-batches


def prepare(case, seed):
    g = _generator(seed)
    call = case["call"]
    s = {"case": case, "seed": seed}
    if call == "sample":
        s["logits"] = _logits(g, case["rows"], case["vocab"], case["dtype"], case["like"])
        u = _uniform(g, case["rows"], 0.0, 1.0)
        s["temps"] = u * 0.8 + 0.6 if case["like"] == "text" else torch.exp(u * math.log(20.0) + math.log(0.1))
    elif call in ("train", "backward"):
        rows = case["seqs"] * case["tokens"]
        s["logits"] = _logits(g, rows, case["vocab"], case["dtype"])
        s["targets"] = torch.randint(0, case["vocab"], (rows,), generator=g, device=DEVICE, dtype=torch.int32)
        s["mask"] = _mask(g, case).reshape(-1)
        if call == "train":
            s["temps"] = _uniform(g, rows, 0.6, 1.4) if case["row_temps"] else None
            s["sum"] = torch.zeros(2, dtype=torch.float64, device=DEVICE)
        else:
            s["logp"], s["ent"] = e3.e3_token_logp_entropy(s["logits"], s["targets"], mask=s["mask"], temp_scalar=0.9)
            s["g_logp"] = torch.randn(rows, generator=g, device=DEVICE)
            s["g_ent"] = 0.01 * torch.randn(rows, generator=g, device=DEVICE) if case["entropy_grad"] else None
            s["out"] = torch.empty_like(s["logits"])
    elif call == "objective":
        shape = (case["seqs"], case["tokens"])
        s["mask"] = _mask(g, case)
        s["logp_old"] = -torch.empty(shape, device=DEVICE).exponential_(1.0, generator=g)
        s["logp"] = s["logp_old"] + 0.15 * torch.randn(shape, generator=g, device=DEVICE)
        s["offsets"] = _groups(g, case["seqs"])
        s["adv"] = torch.randn(case["seqs"], generator=g, device=DEVICE)
    else:
        s["rewards"] = (_uniform(g, _rollouts(case), 0.0, 1.0) < 0.5).to(torch.float32)
        s["offsets"] = _groups(g, _rollouts(case))
        s["ent"] = torch.empty(case["seqs"] * case["tokens"], device=DEVICE).exponential_(1.0, generator=g)
        s["mask"] = _mask(g, case).reshape(-1)
    return s


# --------------------------------------------------------------------------------------------------------------- what is run
def run(s):
    case = s["case"]
    call = case["call"]
    if call == "sample":
        return e3.e3_sample(s["logits"], s["temps"], s["seed"], 17, 0, SAMPLERS[case["sampler"]])
    if call == "train":
        got = e3.e3_token_logp_entropy(s["logits"], s["targets"], mask=s["mask"], temps=s["temps"], temp_scalar=0.9,
                                       want_gap=case["gap"], out_sum=s["sum"])
        return got, s["sum"]
    if call == "backward":
        return e3.e3_token_logp_entropy_backward(s["logits"], s["targets"], s["logp"], s["ent"], s["g_logp"], s["g_ent"],
                                                 mask=s["mask"], temp_scalar=0.9, out=s["out"])
    if call == "objective":
        return e3.e3_grpo_objective(s["logp"], s["logp_old"], s["adv"], s["offsets"], mask=s["mask"])
    return e3.e3_group_advantage(s["rewards"], s["offsets"]), e3.e3_masked_mean_entropy(s["ent"], s["mask"])


def work(case):
    call = case["call"]
    if call == "sample":
        rows, v = case["rows"], case["vocab"]
        # per logit: scale, exponential, two sums; the token, its log-probability and the entropy come back
        return {"bytes": rows * v * ESIZE[case["dtype"]] + rows * (4 + 12), "flops": 5.0 * rows * v}
    live, tokens = sum(_lengths(case)), case["seqs"] * case["tokens"]
    if call == "train":
        return {"bytes": live * (case["vocab"] * ESIZE[case["dtype"]] + 4) + tokens * (9 + 4 * case["gap"] + 4 * case["row_temps"]) + 16,
                "flops": 5.0 * live * case["vocab"]}
    if call == "backward":  # rows outside the mask are only written
        return {"bytes": (live + tokens) * case["vocab"] * ESIZE[case["dtype"]] + live * (16 + 4 * case["entropy_grad"]) + tokens,
                "flops": 6.0 * live * case["vocab"]}
    if call == "objective":
        return {"bytes": live * 8 + tokens * 5 + case["seqs"] * 4 + 16, "flops": 10.0 * live}
    return {"bytes": live * 4 + tokens + _rollouts(case) * 8 + 16, "flops": 1.0 * live + 6.0 * _rollouts(case)}


def tolerance(case):
    if case["call"] == "backward" and case["dtype"] == "bf16":
        return {"rel": 5e-3}  # gradients are stored with eight significant bits: half a unit is 2^-9 of the value
    # sums, logarithms and gradients in fp32 (or wider) of values given exactly; tokens, flags and counts are the same
    return {"rel": 1e-5, "differ": 0.0}
