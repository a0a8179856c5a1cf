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


@pytest.mark.parametrize("sigma", [0.15, 0.03])
def test_draws_from_small_residuals_are_those_of_the_whole_row(sigma):
    """Good drafters: residuals of a thousandth to a sixteenth of the row's mass, whose parts are differences of numbers up
    to 1e3 times larger.  A token taken from the parts alone was up to 9e-8 of the row's mass away from its interval of the
    float64 CDF; a walk over the row, which takes the differences token by token, each off by 2^-25 of the heaviest token at
    most, stays within 2^-24 of it."""
    B, k, V, dev = 256, 4, 32000, torch.device("cuda", 0)
    wl = workload(B=B, N=1, k=k, V=V, sigmas=(sigma,), order="rank")
    acc, tok = (torch.zeros(B, dtype=torch.int32, device=dev) for _ in range(2))
    reward = torch.zeros(B, device=dev)
    draws = 0
    for s in range(4):
        rd = RoundGenerator(wl, device=dev, seed=100 + s).gathered_round(0, np.zeros(B, dtype=np.int64))
        p, q = torch.softmax(rd["target"].double(), -1), torch.softmax(rd["draft"].double(), -1)
        cdf = (p[:, :k] - q).clamp_min(0).cumsum(-1)
        for i in range(100):
            assert M.verify_noalloc(rd["target"], rd["draft"], rd["tokens"], 1.0, 7 + i, i, acc, tok, reward) == M.OK
            n = acc.cpu().numpy()
            u = torch.tensor([O.round_uniforms(7 + i, b, i, int(n[b]))[1] for b in range(B)], dtype=torch.float64, device=dev)
            row = cdf[torch.arange(B, device=dev), acc.long().clamp_max(k - 1)]
            band = (acc < k) & (row[:, -1] > 1e-3) & (row[:, -1] < 1 / 16)
            at, end = u * row[:, -1], row.gather(1, tok.long()[:, None])[:, 0]
            front = torch.where(tok > 0, row.gather(1, (tok.long() - 1).clamp_min(0)[:, None])[:, 0], torch.zeros_like(end))
            off = torch.maximum(front - at, at - end)[band]
            assert off.numel() == 0 or float(off.max()) < 2.0 ** -24
            draws += int(band.sum())
    assert draws > 2000


@pytest.mark.parametrize("window", [1, 2, 31, 32, 33, 64, 65])
def test_sliding_windows_around_a_warp(window):
    from _harness import run_lockstep
    wl = workload(B=6, N=3, k=2, V=512, sigmas=(0.3, 1.0, 2.5)).scaled(tau=window)
    c = run_lockstep(wl, rounds=70, bandit="swucb", table_mode=True, path=M.PATH_STREAMING)
    assert c["rounds"] == 70 and c["near_tie_arm"] == 0


@pytest.mark.parametrize("dtype,V", [("bf16", 131072), ("bf16", 131080), ("bf16", 151937), ("fp32", 131072), ("fp32", 131076), ("fp32", 140001)])
def test_draws_on_both_sides_of_long_parts(dtype, V):
    """Parts of up to 16 KB, which 256 threads walk, and longer ones, which 512 do where every sequence has an SM."""
    from _harness import run_lockstep
    wl = workload(B=4, N=2, k=2, V=V, sigmas=(0.4, 1.5)).scaled(dtype=dtype, temperature=0.8, order="shuffled")
    c = run_lockstep(wl, rounds=4, seed=V % 83, path=M.PATH_STREAMING)
    assert c["rounds"] == 4 and c["status"] == 0
