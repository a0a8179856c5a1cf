"""A sequence's results do not depend on what else is in its batch: one large launch against launches of a few of its
sequences, which take other shapes of the row-statistics kernel, bit for bit in every output.  Of an odd vocabulary a
sequence's rows also start at other offsets from a 16-byte boundary in another batch."""
import numpy as np
import pytest
import torch

from paper_2604_05417_b200 import binding as M
from paper_2604_05417_b200.workloads import RoundGenerator, Workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,V,B", [("bf16", 4096, 400), ("bf16", 4101, 400), ("bf16", 20001, 400), ("bf16", 32000, 400),
                                       ("bf16", 50257, 400), ("bf16", 50264, 400), ("bf16", 80008, 400), ("bf16", 100003, 400),
                                       ("bf16", 131072, 400), ("fp32", 4096, 400), ("fp32", 4099, 400), ("fp32", 32000, 400),
                                       ("fp32", 32001, 400), ("fp32", 64008, 400), ("fp32", 64009, 400), ("fp32", 110000, 400),
                                       ("fp32", 64003, 1000)])
def test_results_do_not_depend_on_the_batch(dtype, V, B):
    """1200 (3000) row pairs and bonus rows in one launch; 3, 36, 141, 420 and 600 of them in launches of their own."""
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
    for first, last in [(0, 1), (1, 13), (13, 60), (60, 200), (200, 400)]:
        for x, y in zip(whole, play(first, last)):
            assert torch.equal(x[first:last], y)


@pytest.mark.parametrize("dtype,V", [("bf16", 80008), ("bf16", 152064), ("fp32", 20400)])
def test_results_do_not_depend_on_the_kernel_of_long_launches(dtype, V):
    """1200 row pairs and bonus rows, more than L2 holds, which the kernel with L2 policies takes where it has their shape (fp32,
    V = 20400: it has not); 141 of them by the other."""
    test_results_do_not_depend_on_the_batch(dtype, V, 400)
