"""A sequence's results do not depend on what else is in its batch: one large launch against launches of a few of its
sequences, which take other shapes of the row-statistics kernel, bit for bit in every output.  Of an odd vocabulary a
sequence's rows also start at other offsets from a 16-byte boundary in another batch."""
import numpy as np
import pytest
import torch

from paper_2604_05417_b200 import binding as M
from paper_2604_05417_b200.workloads import RoundGenerator, Workload

pytestmark = pytest.mark.gpu


# 1200 (3000) row pairs and bonus rows in one launch
BATCHES = [("bf16", 4096, 400), ("bf16", 4101, 400), ("bf16", 20001, 400), ("bf16", 32000, 400),
           ("bf16", 50257, 400), ("bf16", 50264, 400), ("bf16", 80008, 400), ("bf16", 100003, 400),
           ("bf16", 131072, 400), ("fp32", 4096, 400), ("fp32", 4099, 400), ("fp32", 32000, 400),
           ("fp32", 32001, 400), ("fp32", 64008, 400), ("fp32", 64009, 400), ("fp32", 110000, 400),
           ("fp32", 64003, 1000)]
# every shape of the hinted kernel, against launches by the staged one: bf16 512/6/1 and 256/6/2, fp32 256/6/2, 256/6/4 and 1024/6/1 (128/6/8:
# V = 110000 above); and short fp32 rows, whose shape the hinted kernel is not built in
LONG_LAUNCHES = [("bf16", 152064, 400), ("fp32", 20400, 400), ("fp32", 48000, 400), ("fp32", 80000, 400), ("fp32", 80000, 1000)]
PARTS = [(0, 1), (1, 13), (13, 60), (60, 200), (200, 400)]


@pytest.mark.parametrize("dtype,V,B", BATCHES)
def test_results_do_not_depend_on_the_batch(dtype, V, B):
    """All sequences in one launch; 3, 36, 141, 420 and 600 row pairs and bonus rows in launches of their own."""
    k, N = 2, 2
    wl = Workload("t", B=B, N=N, k=k, V=V, rounds=1, temperature=0.9, dtype=dtype, bandit="ucb", sigmas=(0.4, 1.5))
    rd = RoundGenerator(wl, device=torch.device("cuda", 0), seed=V % 89).table_round(0)
    drafts, tokens = rd["drafts"], rd["tokens"]

    def play(first, last):
        msd = M.MetaSD(last - first, N, k, V, dtype=dtype, sequence_base=first)
        part = [d[first:last].clone() for d in drafts]
        table = M.pointer_table(part)
        target, toks = rd["target"][first:last].clone(), tokens[:, first:last].contiguous()
        out = []
        for t in range(2):
            res = msd.verify(target, None, toks, 0.9, 31, drafter_table=table, token_arm_stride=(last - first) * k, want_diag=True)
            out += [res.accepted_len, res.next_token, res.reward, res.diag, msd.select()]
        torch.cuda.synchronize()
        state = M.parse_state(msd.state_export(), last - first, N, msd.cfg.window)
        msd.close()
        return out + [torch.from_numpy(np.array(state[n])) for n in ("stat_a", "stat_b")]

    whole = play(0, B)
    for first, last in PARTS:
        for x, y in zip(whole, play(first, last)):
            assert torch.equal(x[first:last], y)


@pytest.mark.parametrize("dtype,V,B", LONG_LAUNCHES)
def test_results_do_not_depend_on_the_kernel_of_long_launches(dtype, V, B):
    """More row pairs in flight than L2 holds, which the hinted kernel takes, against launches of few by the staged one (which kernel
    takes which: test_row_shapes_cpu.py)."""
    test_results_do_not_depend_on_the_batch(dtype, V, B)


@pytest.mark.parametrize("dtype,V,few", [("bf16", 152064, 80), ("fp32", 128256, 40)])
@pytest.mark.parametrize("octave", [0, 4])
def test_rows_whose_sums_are_a_power_of_two_times_the_square_root_of_two_apart(dtype, V, few, octave):
    """Where log2(sum_a / sum_b) lies half way between two whole numbers, both row-statistics kernels must take the same one: the
    rounding of the draft row's exponents follows it.  400 rows whose ratio, 1.4142135 (1 + d) 2^octave with d in -3e-7 .. 3e-7,
    meets every fp32 number there; 800 row pairs and bonus rows in a launch, and `few` sequences at a time."""
    B, T = 400, 0.9
    dev = torch.device("cuda", 0)
    rng = np.random.default_rng(4)
    low = -rng.integers(39, 512, size=20000 >> octave) / 64.0
    low = torch.from_numpy(low).to(torch.bfloat16 if dtype == "bf16" else torch.float32)
    S = float(torch.exp2(low.double() * float(np.float32(1.4426950408889634 / T))).sum())
    ones = np.arange(20000 >> octave, 45000 >> octave)
    pairs = []
    for d in np.linspace(-3e-7, 3e-7, B):
        want = 1.41421354 * 2 ** octave * (1.0 + d)
        n = np.rint(want * (ones + S))
        i = int(np.argmin(np.abs(n / (ones + S) / want - 1.0)))
        pairs.append((int(n[i]), int(ones[i])))
    target = torch.full((B, 2, V), float("-inf"), dtype=low.dtype, device=dev)
    draft = torch.full((B, 1, V), float("-inf"), dtype=low.dtype, device=dev)
    for b, (n, m) in enumerate(pairs):
        target[b, :, :n] = 0.0
        draft[b, 0, 75000:75000 + m] = 0.0
    draft[:, 0, :low.numel()] = low.to(dev)
    tokens = torch.zeros((B, 1), dtype=torch.int32, device=dev)

    def play(first, last):
        msd = M.MetaSD(last - first, 1, 1, V, dtype=dtype, sequence_base=first)
        res = msd.verify(target[first:last], draft[first:last], tokens[first:last], T, 31, want_diag=True)
        torch.cuda.synchronize()
        assert msd.last_status() == 0
        reward = torch.from_numpy(np.array(M.parse_state(msd.state_export(), last - first, 1, msd.cfg.window)["stat_a"]))   # fp64
        msd.close()
        return [res.accepted_len, res.next_token, res.diag, reward]

    whole = play(0, B)
    differ = torch.zeros(B, dtype=torch.bool)
    for first in range(0, B, few):
        for x, y in zip(whole, play(first, first + few)):
            differ[first:first + few] |= (x[first:first + few].cpu() != y.cpu()).reshape(few, -1).any(1)
    assert int(differ.sum()) == 0


PINNED = [(512, 6, 1), (512, 4, 1), (1024, 6, 1), (1024, 4, 1), (768, 4, 1), (384, 4, 1), (512, 4, 3), (512, 4, 2), (768, 4, 2)]


@pytest.mark.parametrize("dtype,V,B,shape", [("bf16", 152064, 400, None), ("bf16", 262144, 100, None), ("fp32", 80000, 1000, None)] +
                         [(dtype, V, 7, shape) for shape in PINNED for dtype, V in (("bf16", 50264), ("fp32", 33000))])
def test_results_do_not_depend_on_l2_policies(dtype, V, B, shape):
    """keep_permille < 0: aligned rows of long launches and of pinned shapes by the staged kernel, which has no policies, instead of
    the hinted one.  Bit for bit."""
    k, N = 2, 2
    wl = Workload("t", B=B, N=N, k=k, V=V, rounds=1, temperature=0.9, dtype=dtype, bandit="ucb", sigmas=(0.4, 1.5))
    rd = RoundGenerator(wl, device=torch.device("cuda", 0), seed=V % 89).table_round(0)
    table = M.pointer_table(rd["drafts"])
    tuning = {} if shape is None else dict(row_kernel=M.ROWS_STAGED, row_threads=shape[0], row_stages=shape[1], row_cluster=shape[2])
    results = []
    for keep in (0, -1):
        msd = M.MetaSD(B, N, k, V, dtype=dtype, keep_permille=keep, **tuning)
        out = []
        for T in (0.9, 0.0):
            res = msd.verify(rd["target"], None, rd["tokens"], T, 31, drafter_table=table, token_arm_stride=B * k, want_diag=True)
            out += [res.accepted_len, res.next_token, res.reward, res.diag, msd.select()]
        assert msd.last_status() == 0
        out.append(torch.from_numpy(np.array(M.parse_state(msd.state_export(), B, N, msd.cfg.window)["stat_a"])))
        msd.close()
        results.append(out)
    for x, y in zip(*results):
        assert torch.equal(x, y)
