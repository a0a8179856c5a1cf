"""Row-statistics kernels at the edges of their tiles: lengths around whole trips and whole groups of trips per warp, and
masked stretches that leave a warp without a finite logit.  Oracle: the float64 CPU implementation.  The 1e-5 bound on
every probability is the lock-step harness's (2^-22 exponentials, fp32 sums of at most a few hundred terms per lane)."""
import numpy as np
import pytest
import torch

from paper_2604_05417_b200 import binding as M
from paper_2604_05417_b200.workloads import RoundGenerator, Workload

pytestmark = pytest.mark.gpu

# Launches of a few rows are the staged kernel's.  Long launches are the hinted kernel's (csrc/metasd_hinted.cu), which has a text of its
# own: these are the shapes it takes the largest ones in, and pinned it takes aligned rows of any launch.
KERNELS = ["auto", "pinned"]
PINNED = {"bf16": dict(row_kernel=M.ROWS_STAGED, row_threads=512, row_stages=6), "fp32": dict(row_kernel=M.ROWS_STAGED, row_threads=1024, row_stages=6)}


def shape(kernel, dtype):
    return PINNED[dtype] if kernel == "pinned" else {}


def workload(**kw):
    d = dict(name="t", B=3, N=2, k=2, V=1024, rounds=2, temperature=1.0, dtype="bf16", bandit="ucb", sigmas=(0.5, 2.0))
    d.update(kw)
    return Workload(**d)


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("V", [8, 248, 256, 264, 4088, 4096, 4104, 6 * 4096, 6 * 4096 + 8, 11 * 4096, 12 * 4096 - 8, 12 * 4096 + 264])
@pytest.mark.parametrize("kernel", KERNELS)
def test_row_lengths_at_the_edges_of_trips_and_groups(dtype, V, kernel):
    from _harness import run_lockstep
    c = run_lockstep(workload(V=V, dtype=dtype), rounds=3, seed=V % 83, path=M.PATH_STREAMING, **shape(kernel, dtype))
    assert c["rounds"] == 3 and c["status"] == 0


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("shift", [0.0, 120.0, -120.0])
@pytest.mark.parametrize("kernel", KERNELS)
def test_masked_stretches_cover_whole_warps(dtype, shift, kernel):
    """Target and / or draft logits of whole ranges of the vocabulary are -inf, the draft row on another scale."""
    from _harness import make_pair, compare_round
    V = 3 * 4096 + 40
    wl = workload(V=V, dtype=dtype, B=6)
    rd = RoundGenerator(wl, device=torch.device("cuda", 0), seed=9).gathered_round(0, np.zeros(6, dtype=np.int64))
    target, draft = rd["target"].clone(), (rd["draft"].float() + shift).to(rd["draft"].dtype)
    ninf = float("-inf")
    target[0, :, : V // 2] = ninf
    target[1, :, V // 2:] = ninf
    draft[1, :, : V // 4] = ninf
    target[2, :, :-3] = ninf
    draft[3, :, : V - 9] = ninf
    target[4, :, 3:] = ninf
    draft[4, :, : V // 3] = ninf
    gpu, orc = make_pair(wl, path=M.PATH_STREAMING, **shape(kernel, dtype))
    try:
        res = gpu.verify(target, draft, rd["tokens"], 1.0, 3, want_diag=True)
        out = orc.verify(target, draft, rd["tokens"].cpu().numpy(), 1.0, 3)
        compare_round(res, out, target, draft, 1.0, 1.0, {})
        assert gpu.last_status() & M.STATUS_NONFINITE == 0
    finally:
        gpu.close()


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("V", [3 * 4096 + 40, 3 * 4096 + 41])
@pytest.mark.parametrize("T", [1.0, 2.0])
@pytest.mark.parametrize("kernel", KERNELS)
def test_masks_of_the_types_lowest_value(dtype, V, T, kernel):
    """Masks written as torch.finfo(dtype).min (and as -1e38) over stretches that hold the first trips of some warps: they
    weigh nothing, as -inf does, although their product with log2(e) / T leaves the range of fp32."""
    from _harness import make_pair, compare_round
    wl = workload(V=V, dtype=dtype, B=6, temperature=T)
    rd = RoundGenerator(wl, device=torch.device("cuda", 0), seed=9).gathered_round(0, np.zeros(6, dtype=np.int64))
    target, draft = rd["target"].clone(), rd["draft"].clone()
    low = torch.finfo(target.dtype).min
    target[0, :, : V // 2] = low
    target[1, :, V // 2:] = low
    draft[1, :, : V // 4] = low
    target[2, :, :-3] = low
    draft[3, :, : V - 9] = low
    target[4, :, 3:] = -1e38
    draft[4, :, : V // 3] = low
    gpu, orc = make_pair(wl, path=M.PATH_STREAMING, **shape(kernel, dtype))
    try:
        res = gpu.verify(target, draft, rd["tokens"], T, 3, want_diag=True)
        out = orc.verify(target, draft, rd["tokens"].cpu().numpy(), T, 3)
        compare_round(res, out, target, draft, T, 1.0, {})
        assert gpu.last_status() & M.STATUS_NONFINITE == 0
    finally:
        gpu.close()


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("V", [4096, 4099])
@pytest.mark.parametrize("kernel", KERNELS)
def test_draft_sums_next_to_the_end_of_the_fp32_range(dtype, V, kernel):
    """Draft rows whose sum, relative to the target row's maximum (0 here), is 2^99 .. 2^128: 2^127.6 is a finite fp32
    number, and its inverse's whole exponent, 128, is not one that an fp32 power of two can have."""
    from _harness import make_pair, compare_round
    wl = workload(V=V, dtype=dtype, B=8, N=1, k=2)
    dev = torch.device("cuda", 0)
    target = torch.full((8, 3, V), -30.0, dtype=torch.float32, device=dev)
    target[:, :, 0] = 0.0
    draft = torch.full((8, 2, V), -30.0, dtype=torch.float32, device=dev)
    for b, (low, high) in enumerate([(68.0, 68.5), (69.0, 69.5), (70.0, 70.0), (87.0, 87.0), (87.5, 87.5), (87.5, 88.0), (88.0, 87.5),
                                     (88.5, 88.5)]):
        draft[b, :, 0], draft[b, :, 5] = low, high
    target, draft = (x.to({"bf16": torch.bfloat16, "fp32": torch.float32}[dtype]) for x in (target, draft))
    tokens = torch.zeros((8, 2), dtype=torch.int32, device=dev)
    gpu, orc = make_pair(wl, path=M.PATH_STREAMING, **shape(kernel, dtype))
    try:
        res = gpu.verify(target, draft, tokens, 1.0, 3, want_diag=True)
        out = orc.verify(target, draft, tokens.cpu().numpy(), 1.0, 3)
        compare_round(res, out, target, draft, 1.0, 1.0, {})
        assert gpu.last_status() == 0
    finally:
        gpu.close()


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("V", [1, 2, 7, 9, 250, 255, 257, 4085, 4095, 4097, 6 * 4096 + 3, 12 * 4096 - 1, 50257])
def test_rows_off_a_16_byte_boundary(dtype, V):
    """Odd vocabularies: every row starts at an offset of its own, target and draft rows at different ones."""
    from _harness import run_lockstep
    c = run_lockstep(workload(V=V, dtype=dtype, k=3), rounds=3, seed=V % 83, path=M.PATH_STREAMING)
    assert c["rounds"] == 3 and c["status"] == 0


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("V", [40, 8200, 33003])
def test_tensors_that_start_anywhere(dtype, V):
    """Target, and each drafter's tensor, as views that start 0 .. 9 logits into a buffer; what surrounds them is NaN."""
    from _harness import make_pair, compare_round, gather_by_arm
    wl = workload(V=V, dtype=dtype, B=4, N=3, k=3, sigmas=(0.4, 1.0, 2.5))
    dev = torch.device("cuda", 0)
    gen = RoundGenerator(wl, device=dev, seed=5)

    def moved(t, off):
        back = torch.full((t.numel() + 32,), float("nan"), dtype=t.dtype, device=dev)
        view = back[off:off + t.numel()].view(t.shape)
        view.copy_(t)
        return view

    gpu, orc = make_pair(wl, path=M.PATH_STREAMING)
    try:
        for t in range(4):
            arm = orc.select()
            assert np.array_equal(gpu.select().cpu().numpy(), arm)
            rd = gen.table_round(t)
            target = moved(rd["target"], 1 + 2 * t)
            drafts = [moved(d, (3 * i + t) % 10) for i, d in enumerate(rd["drafts"])]
            res = gpu.verify(target, None, rd["tokens"], 1.0, 7, drafter_table=M.pointer_table(drafts),
                             token_arm_stride=wl.B * wl.k, want_diag=True)
            draft, tokens = gather_by_arm(rd["drafts"], rd["tokens"], arm, dev)
            out = orc.verify(rd["target"], draft, tokens.cpu().numpy(), 1.0, 7)
            compare_round(res, out, rd["target"], draft, 1.0, 1.0, {})
            assert gpu.last_status() == 0
    finally:
        gpu.close()


@pytest.mark.parametrize("dtype,V,B,k", [
    ("bf16", 65536, 1, 2), ("bf16", 65543, 6, 2), ("bf16", 33000, 12, 2), ("bf16", 17001, 49, 2),        # few rows, split over CTAs
    ("bf16", 4104, 60, 2), ("bf16", 4101, 60, 2), ("bf16", 17008, 60, 2), ("bf16", 17003, 60, 2),        # short rows
    ("bf16", 50008, 60, 2), ("bf16", 50011, 60, 2), ("bf16", 100003, 60, 2),                             # a few waves of long rows
    ("bf16", 50008, 340, 2), ("bf16", 50003, 340, 2), ("bf16", 80008, 340, 2),                           # many of them
    ("fp32", 16384, 1, 2), ("fp32", 49155, 12, 2), ("fp32", 8192, 60, 2), ("fp32", 9001, 60, 2), ("fp32", 64008, 60, 2),
    ("fp32", 64009, 170, 2)])
def test_every_shape_that_a_launch_size_selects(dtype, V, B, k):
    """The row-statistics shape follows the row length, the number of rows and their alignment: one launch of each."""
    from _harness import run_lockstep
    c = run_lockstep(workload(V=V, dtype=dtype, B=B, k=k, temperature=0.9), rounds=2, seed=V % 83, path=M.PATH_STREAMING)
    assert c["rounds"] == 2 and c["status"] == 0


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("kernel", [M.ROWS_AUTO, M.ROWS_PLAIN, M.ROWS_BULK, "pinned"])
def test_alignment_of_rows_that_hardly_overlap(dtype, kernel):
    """Target and draft mass in different halves of the vocabulary: the alignment 1 - d_TV is a small sum of positive terms,
    each a 2^-22 exponential of an fp32 exponent of up to 130 (off by 2^-18 at most) over an fp32 normaliser, never a
    difference: 1e-5 of itself."""
    B, V = 12, 8200
    wl = workload(V=V, dtype=dtype, B=B, N=1, k=1)
    rd = RoundGenerator(wl, device=torch.device("cuda", 0), seed=2).gathered_round(0, np.zeros(B, dtype=np.int64))
    gap = torch.linspace(2.0, 60.0, B, device="cuda").view(B, 1, 1)
    target, draft = rd["target"].float(), rd["draft"].float()
    target[..., V // 2:] -= gap
    draft[..., : V // 2] -= gap
    target, draft = target.to(rd["target"].dtype), draft.to(rd["draft"].dtype)
    gpu = M.MetaSD(B, 1, 1, V, dtype=dtype, path=M.PATH_STREAMING, **(shape(kernel, dtype) or dict(row_kernel=kernel)))
    try:
        res = gpu.verify(target, draft, rd["tokens"], 1.0, 3, want_diag=True)
        p, q = (torch.softmax(x[:, 0].double(), -1) for x in (target, draft))
        want = torch.minimum(p, q).sum(-1)
        assert float(want.min()) < 1e-20 and float(res.reward.min()) > 0 and float(res.diag_fields()[2].max()) <= 1.0
        torch.testing.assert_close(res.reward.double(), want, rtol=1e-5, atol=0)
    finally:
        gpu.close()


@pytest.mark.parametrize("dtype,V", [("bf16", 65536), ("bf16", 65544), ("bf16", 65519), ("bf16", 65553), ("fp32", 12288), ("fp32", 12292),
                                     ("fp32", 24576), ("fp32", 24580), ("fp32", 32765), ("fp32", 32771)])
@pytest.mark.parametrize("temperature", [0.0, 0.7])
def test_ranges_on_both_sides_of_the_rolled_form(dtype, V, temperature):
    """Ranges of 16 (fp32: 12) trips a warp, which go through rolled loops alone, and of one more."""
    from _harness import run_lockstep
    c = run_lockstep(workload(V=V, dtype=dtype, temperature=temperature), rounds=3, seed=V % 83, path=M.PATH_STREAMING)
    assert c["rounds"] == 3 and c["status"] == 0
