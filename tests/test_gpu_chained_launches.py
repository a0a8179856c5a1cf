"""Rounds issued back to back: the library's kernels are set up while the ones before them drain, so every buffer they share
or that the caller refills in stream order must still be read after it was written.  Compared bit for bit with the same
rounds issued one at a time with a synchronisation after every call."""
import numpy as np
import pytest
import torch

from paper_2604_05417_b200 import binding as M
from paper_2604_05417_b200.workloads import RoundGenerator, Workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,V,k", [(1, 32000, 4), (4, 100000, 8), (64, 32000, 5), (200, 20008, 3), (96, 30003, 5)])
@pytest.mark.parametrize("T", [0.0, 0.9])
def test_rounds_back_to_back_equal_rounds_one_at_a_time(B, V, k, T):
    wl = Workload("t", B=B, N=3, k=k, V=V, rounds=6, temperature=T, dtype="bf16", bandit="ducb", sigmas=(0.3, 1.0, 2.5))
    dev = torch.device("cuda", 0)
    gen = RoundGenerator(wl, device=dev, seed=B)
    rounds = [gen.table_round(t) for t in range(3)]

    def play(wait):
        msd = [M.MetaSD(B, 3, k, V, bandit="ducb"), M.MetaSD(B, 3, k, V, bandit="swucb", window=3)]   # two contexts take turns
        lengths = torch.full((B,), k, dtype=torch.int32, device=dev)
        msd[1].set_draft_lengths(lengths)
        target, tokens = rounds[0]["target"].clone(), rounds[0]["tokens"].clone()
        drafts = [d.clone() for d in rounds[0]["drafts"]]
        table = M.pointer_table(drafts)
        torch.cuda.synchronize()
        seen = []
        for t in range(6):
            target.copy_(rounds[t % 3]["target"]); tokens.copy_(rounds[t % 3]["tokens"])
            for dst, src in zip(drafts, rounds[t % 3]["drafts"]):
                dst.copy_(src)
            lengths.fill_(1 + t % k)
            for i, m in enumerate(msd):
                for _ in range(2):          # the second round follows the first without a select between them
                    res = m.verify(target, None, tokens, T, 5 + t, drafter_table=table, token_arm_stride=B * k)
                    if wait:
                        torch.cuda.synchronize()
                    seen += [res.accepted_len.clone(), res.next_token.clone(), res.reward.clone()]
                seen.append(m.select())
                if wait:
                    torch.cuda.synchronize()
        torch.cuda.synchronize()
        state = [m.state_export() for m in msd]
        for m in msd:
            m.close()
        return seen, state

    one, state_one = play(True)
    many, state_many = play(False)
    assert all(torch.equal(x, y) for x, y in zip(one, many))
    assert state_one == state_many


def test_no_allocation_calls_back_to_back():
    B, k, V = 24, 4, 16000
    wl = Workload("t", B=B, N=1, k=k, V=V, rounds=1, temperature=1.0, dtype="bf16", bandit="ucb", sigmas=(1.0,))
    rd = RoundGenerator(wl, device=torch.device("cuda", 0), seed=3).gathered_round(0, np.zeros(B, dtype=np.int64))
    bad = rd["tokens"].clone()
    bad[0, 0] = V + 7                                                  # sets a status bit in every other call only

    def call(i):
        out = [torch.zeros(B, dtype=torch.int32, device="cuda"), torch.zeros(B, dtype=torch.int32, device="cuda"),
               torch.zeros(B, device="cuda"), torch.full((1,), 77, dtype=torch.int32, device="cuda")]
        assert M.verify_noalloc(rd["target"], rd["draft"], bad if i & 1 else rd["tokens"], 1.0, 9, i, *out[:3], status=out[3]) == M.OK
        return out

    one = []
    for i in range(8):
        one.append(call(i))
        torch.cuda.synchronize()
    many = [call(i) for i in range(8)]
    torch.cuda.synchronize()
    for i, (x, y) in enumerate(zip(one, many)):
        assert all(torch.equal(p, q) for p, q in zip(x, y))
        assert int(x[3]) == (M.STATUS_TOKEN_OOR if i & 1 else 0)


@pytest.mark.parametrize("B,V,k,bandit", [(10, 152064, 3, "swucb"), (7, 100003, 4, "ucb"), (3, 300000, 2, "exp3")])
@pytest.mark.parametrize("T", [0.0, 0.8])
def test_host_buffers_give_the_device_calls_round(B, V, k, bandit, T):
    """Results that the kernels write to host memory: outputs, next arms and bandit state of the device call, bit for bit."""
    wl = Workload("t", B=B, N=2, k=k, V=V, rounds=3, temperature=T, dtype="bf16", bandit="ucb", sigmas=(0.4, 2.0))
    gen = RoundGenerator(wl, device=torch.device("cuda", 0), seed=V % 71)
    a = M.MetaSD(B + 2, 2, k + 1, V, bandit=bandit, window=4, sequence_base=5)
    b = M.MetaSD(B + 2, 2, k + 1, V, bandit=bandit, window=4, sequence_base=5, host_staging=True)
    lengths = torch.tensor([1 + i % k for i in range(B + 2)], dtype=torch.int32, device="cuda")
    for t in range(3):
        rd = gen.gathered_round(t, np.zeros(B, dtype=np.int64))
        for m in (a, b):
            m.set_draft_lengths(lengths if t == 1 else None)
        ra = a.verify(rd["target"], rd["draft"], rd["tokens"], T, 3)
        host = [rd[n].cpu().pin_memory() for n in ("target", "draft", "tokens")]
        acc, tok, nxt = (torch.zeros(B, dtype=torch.int32) for _ in range(3))
        rew = torch.zeros(B)
        b.verify_host(*host, T, 3, acc, tok, rew, nxt)
        assert torch.equal(ra.accepted_len.cpu(), acc) and torch.equal(ra.next_token.cpu(), tok) and torch.equal(ra.reward.cpu(), rew)
        assert torch.equal(a.select(B).cpu(), nxt)
    assert a.state_export() == b.state_export()
    a.close(); b.close()
