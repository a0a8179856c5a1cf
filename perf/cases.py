"""The work a program that uses this library gives it: draft-verify rounds over the range of batch sizes, vocabularies,
draft lengths, logit types and options that the public entry points take.

A pass is one round as a serving loop runs it: ``verify`` on the logits at hand, then ``select`` for the drafters of the
next round (a context), one ``verify_host`` call (host buffers) or one ``verify_noalloc`` call (no context).  The bandits
are in the middle of their run, every sequence with statistics of its own; the inputs are the seeded synthetic logits of
``paper_2604_05417_b200.workloads``.
"""
import math

import numpy as np
import torch

from paper_2604_05417_b200 import binding as M
from paper_2604_05417_b200.workloads import RoundGenerator, Workload

SIZE = {"bf16": 2, "fp32": 4}

# Fields of a case
#   entry    "context": verify + select;  "host": verify_host;  "noalloc": verify_noalloc
#   B, N, k, V, T (0: greedy), dtype, bandit, reward ("bd" | "be")
#   table    the N drafters' logits and tokens through the pointer table (the kernels pick by arm); else gathered
#   ragged   per-sequence draft lengths, uniform in 1 .. k
#   diag     the per-position diagnostics are asked for as well
#   order    where the likely tokens sit in the vocabulary
DEFAULTS = dict(entry="context", N=4, T=1.0, dtype="bf16", bandit="ucb", reward="bd", table=True, ragged=False, diag=False,
                order="rank")


def _case(name, **kw):
    case = dict(DEFAULTS, **kw)
    if name:
        case["name"] = name
    return case


def listed():
    return [
        # one chat session on a small model: the smallest call, all latency
        _case("one_sequence", B=1, N=3, k=4, V=32000),
        # a handful of sessions on a model with a large vocabulary: far fewer rows than the chip has multiprocessors
        _case("few_sequences", B=4, k=8, V=152064, T=0.7, diag=True),
        # a mid-size batch whose best drafter moves (the discounted policy)
        _case("moving_batch", B=64, N=5, k=5, V=32000, bandit="ducb"),
        # a large serving batch over several tasks, tempered sampling
        _case("task_batch", B=256, N=8, k=7, V=128256, T=0.7),
        # greedy decoding of a large batch on the largest configured vocabulary
        _case("greedy_batch", B=512, k=8, V=152064, T=0.0),
        # fp32 logits, the largest batch, draft rows gathered by the caller
        _case("fp32_batch", B=1024, N=8, k=5, V=128256, dtype="fp32", table=False),
        # a vocabulary that is no multiple of anything: most rows start off a 16-byte boundary
        _case("odd_vocabulary", B=96, N=3, k=5, V=50257, T=0.9, bandit="exp3", diag=True),
        # fp32 logits on an odd vocabulary, a few sequences, the block-efficiency reward
        _case("odd_fp32", B=8, N=2, k=3, V=32001, T=0.8, dtype="fp32", bandit="petc", reward="be", table=False),
        # sequences that drafted different lengths, the sliding-window policy, greedy
        _case("ragged_batch", B=192, k=8, V=50264, T=0.0, bandit="swucb", ragged=True),
        # deep drafts on a very large vocabulary in no frequency order, with diagnostics
        _case("deep_drafts", B=40, N=2, k=16, V=262144, T=0.6, diag=True, order="shuffled"),
        # logits that a framework on the host hands over (pinned buffers, blocking call)
        _case("host_buffers", B=40, k=5, V=32000, T=0.8, entry="host", table=False),
        # a caller that may not allocate, greedy
        _case("no_allocation", B=16, N=1, k=5, V=32000, T=0.0, entry="noalloc", table=False),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    while True:
        entry = rng.choice(["context"] * 8 + ["host", "noalloc"])
        V = _log_uniform(rng, 4000, 262144)
        if rng.random() < 0.7:
            V -= V % 8       # most vocabularies are padded
        case = _case(None, entry=entry, B=_log_uniform(rng, 1, 1024), N=rng.randint(2, 8), k=rng.randint(1, 16), V=V,
                     T=rng.choice([0.0, 0.7, round(rng.uniform(0.5, 1.0), 2)]), dtype=rng.choice(["bf16", "bf16", "fp32"]),
                     bandit=rng.choice(["ucb", "ucb", "ducb", "swucb", "exp3", "rand"]),
                     reward=rng.choice(["bd", "bd", "bd", "be"]), table=entry == "context" and rng.random() < 0.6,
                     ragged=entry == "context" and rng.random() < 0.2, diag=entry == "context" and rng.random() < 0.2,
                     order=rng.choice(["rank", "rank", "shuffled", "reversed"]))
        logits = case["B"] * (2 * case["k"] + 1) * case["V"] * SIZE[case["dtype"]]
        held = logits * (case["N"] + 1) // 2 if case["table"] else logits
        if logits <= (100e6 if entry == "host" else 2.6e9) and held <= 8e9:
            return case


def _workload(case):
    N = case["N"]
    return Workload(name="case", B=case["B"], N=N, k=case["k"], V=case["V"], rounds=1, temperature=case["T"], dtype=case["dtype"],
                    bandit=case["bandit"], sigmas=tuple(float(s) for s in np.linspace(0.3, 3.0, N)) if N > 1 else (0.8,),
                    schedule="task", zipf=(0.9, 1.1, 1.25, 1.4), order=case["order"])


def _running_bandits(msd, case, rng):
    """State of bandits in the middle of their run: counts, rewards around each sequence's own levels, the current arms."""
    if case["bandit"] == "petc":
        return      # its exploration schedule starts with the query
    B, N, tau = case["B"], case["N"], msd.cfg.window
    parts = M.parse_state(msd.state_export(), B, N, tau)
    level = rng.uniform(0.1, 0.9, size=(B, N))
    count = rng.integers(1, 30, size=(B, N)).astype(np.float64)
    parts["arm"] = rng.integers(0, N, size=B).astype(np.int32)
    if case["bandit"] == "ucb":
        parts["t"] = count.sum(axis=1).astype(np.int32)
        parts["stat_a"], parts["stat_b"] = level, count
    elif case["bandit"] == "ducb":
        parts["t"] = (count.sum(axis=1) + N).astype(np.int32)
        count = count * 0.4
        parts["stat_a"], parts["stat_b"] = level * count, count
    elif case["bandit"] == "exp3":
        parts["t"] = count.sum(axis=1).astype(np.int32)
        parts["stat_a"] = level / level.max(axis=1, keepdims=True)
    else:
        parts["t"] = np.full(B, 3 * tau, dtype=np.int32)
        if case["bandit"] == "swucb":
            parts["win_arm"] = rng.integers(0, N, size=(B, tau)).astype(np.int32)
            parts["win_reward"] = np.clip(np.take_along_axis(level, parts["win_arm"], axis=1) +
                                          rng.normal(0.0, 0.05, size=(B, tau)), 0.0, 1.0)
    msd.state_import(M.pack_state(parts))


def prepare(case, seed):
    dev = torch.device("cuda", torch.cuda.current_device())
    wl, rng = _workload(case), np.random.default_rng(seed)
    gen = RoundGenerator(wl, device=dev, seed=seed)
    B, k, N = wl.B, wl.k, wl.N
    s = dict(case, seed=seed + 12345, reward_kind=M.REWARD_BE if case["reward"] == "be" else M.REWARD_BD, round=7)
    if case["table"]:
        rd = gen.table_round(0)
        s["drafts"], s["tokens"] = rd["drafts"], rd["tokens"].contiguous()
        s["pointers"] = M.pointer_table(rd["drafts"])
    else:
        rd = gen.gathered_round(0, rng.integers(0, N, size=B))
        s["draft"], s["tokens"] = rd["draft"], rd["tokens"]
    s["target"] = rd["target"]

    # the integer results share one buffer, so that one copy takes them to the host
    host = dict(pin_memory=True) if case["entry"] == "host" else dict(device=dev)
    s["ints"] = torch.zeros((3, B), dtype=torch.int32, **host)      # accepted lengths, next tokens, next arms
    s["reward_out"] = torch.zeros(B, dtype=torch.float32, **host)
    if case["entry"] == "noalloc":
        s["status"] = torch.zeros(1, dtype=torch.int32, device=dev)
        return s
    s["msd"] = M.MetaSD(B, N, k, wl.V, dtype=wl.dtype, bandit=wl.bandit, reward=s["reward_kind"], device=dev.index,
                        host_staging=case["entry"] == "host")
    _running_bandits(s["msd"], case, rng)
    if case["entry"] == "host":
        for name in ("target", "draft", "tokens"):
            s[name] = s[name].cpu().pin_memory()
        return s
    if case["ragged"]:
        s["lengths"] = torch.from_numpy(rng.integers(1, k + 1, size=B).astype(np.int32)).to(dev)
        s["msd"].set_draft_lengths(s["lengths"])
    s["out"] = M.VerifyResult(s["ints"][0], s["ints"][1], s["reward_out"])
    if case["diag"]:
        s["out"].diag = torch.zeros((B, k, 5), dtype=torch.float32, device=dev)
    return s


def run(s):
    if s["entry"] == "noalloc":
        M.verify_noalloc(s["target"], s["draft"], s["tokens"], s["T"], s["seed"], s["round"], s["ints"][0], s["ints"][1],
                         s["reward_out"], status=s["status"], reward_kind=s["reward_kind"])
        s["round"] += 1
        return s["ints"], s["reward_out"], s["status"]
    if s["entry"] == "host":
        s["msd"].verify_host(s["target"], s["draft"], s["tokens"], s["T"], s["seed"], s["ints"][0], s["ints"][1],
                             s["reward_out"], arm_next=s["ints"][2])
        return s["ints"], s["reward_out"]
    if s["table"]:
        s["msd"].verify(s["target"], None, s["tokens"], s["T"], s["seed"], drafter_table=s["pointers"],
                        token_arm_stride=s["B"] * s["k"], out=s["out"], want_diag=s["diag"])
    else:
        s["msd"].verify(s["target"], s["draft"], s["tokens"], s["T"], s["seed"], out=s["out"], want_diag=s["diag"])
    s["msd"].select(out=s["ints"][2])
    if s["diag"]:
        return s["ints"], s["reward_out"], s["out"].diag
    return s["ints"], s["reward_out"]


def work(case):
    B, k, V = case["B"], case["k"], case["V"]
    rows = B * (2 * k + 1)
    if case["ragged"]:
        rows = B * (k + 2)      # the mean length of 1 .. k is (k + 1) / 2
    pairs = (rows - B) // 2
    # every row: scale and shift, exponential, sum (4 operations a logit); every pair of rows: the smaller of the two
    # probabilities and its sum (4 a token)
    flops = 4.0 * rows * V + 4.0 * pairs * V
    small = B * (4 * k + 12) + B * case["N"] * 32 + (B * k * 20 if case["diag"] else 0)
    return {"bytes": float(rows * V * SIZE[case["dtype"]] + small), "flops": flops}


def tolerance(case):
    # rewards and probabilities: fp32 sums of V terms with 2^-22 exponentials.  Against float64 on the same inputs they were
    # seen off by at most 1.6e-6 (2-norm) and 2.6e-6 (largest difference); four times that is allowed.
    # Sampled tokens: a draw that lands within rounding of an edge between two tokens may take either.
    return {"rel": 6e-6, "max": 1e-5, "differ": 0.0 if case["T"] == 0.0 else 0.01}
