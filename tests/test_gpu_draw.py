"""The draw's searches at the edges: parts of one vector, parts that need a second level, a residual with next to no mass
(walked over the whole row), rows reported on as a whole, and the sliding window's length around a warp."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2604_05417_b200 import binding as M
from paper_2604_05417_b200.workloads import RoundGenerator, Workload

pytestmark = pytest.mark.gpu


def workload(**kw):
    d = dict(name="t", B=12, N=2, k=3, V=4096, rounds=4, temperature=1.0, dtype="bf16", bandit="ucb", sigmas=(0.5, 2.0), order="shuffled")
    d.update(kw)
    return Workload(**d)


@pytest.mark.parametrize("kernel", [M.ROWS_AUTO, M.ROWS_PLAIN])
@pytest.mark.parametrize("dtype,V", [("bf16", 24), ("bf16", 4104), ("bf16", 300000), ("bf16", 300001), ("fp32", 70003), ("fp32", 33)])
def test_parts_of_every_length(dtype, V, kernel):
    """300000 tokens in one part per row are 147 vectors a thread (two levels); in parts of their own at most five."""
    from _harness import run_lockstep
    c = run_lockstep(workload(V=V, dtype=dtype, temperature=0.7), rounds=4, seed=V % 67, path=M.PATH_STREAMING, row_kernel=kernel)
    assert c["rounds"] == 4 and c["status"] == 0


@pytest.mark.parametrize("V", [2008, 2003])
def test_a_residual_with_next_to_no_mass_is_drawn_from_token_by_token(V):
    """Drafters so close that sum max(0, p - q) is below a thousandth.  p and q are fp32: each is off by at most a few
    2^-22 of itself, so a cumulative weight is off by 1e-6 of the row's mass at most -- the bound used here, in place of a
    bound relative to the residual, which is 1e3 times smaller than the row."""
    B, k = 600, 8
    wl = workload(B=B, k=k, V=V, sigmas=(0.0008,), N=1, dtype="fp32")
    gen = RoundGenerator(wl, device=torch.device("cuda", 0), seed=4)
    gpu = M.MetaSD(B, 1, k, V, dtype="fp32")
    drawn = 0
    for t in range(12):
        rd = gen.gathered_round(t, np.zeros(B, dtype=np.int64))
        res = gpu.verify(rd["target"], rd["draft"], rd["tokens"], 1.0, 11)
        n_acc, tok = res.accepted_len.cpu().numpy(), res.next_token.cpu().numpy()
        for b in np.nonzero(n_acc < k)[0]:
            j = int(n_acc[b])
            p, q = (O.softmax(rd[n][b, j].double().cpu().numpy(), 1.0)[0] for n in ("target", "draft"))
            w = np.maximum(p - q, 0.0)
            if w.sum() > 1e-3:
                continue
            cdf = np.cumsum(w)
            at = O.round_uniforms(11, int(b), t, j)[1] * cdf[-1]
            assert cdf[tok[b]] + 1e-6 > at and cdf[tok[b]] - w[tok[b]] < at + 1e-6
            drawn += 1
    gpu.close()
    assert drawn > 5


@pytest.mark.parametrize("window", [1, 2, 31, 32, 33, 64, 65])
def test_sliding_windows_around_a_warp(window):
    from _harness import run_lockstep
    wl = workload(B=6, N=3, k=2, V=512, sigmas=(0.3, 1.0, 2.5)).scaled(tau=window)
    c = run_lockstep(wl, rounds=70, bandit="swucb", table_mode=True, path=M.PATH_STREAMING)
    assert c["rounds"] == 70 and c["near_tie_arm"] == 0
