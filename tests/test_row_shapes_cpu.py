"""The rules that pick a row-statistics kernel and its shape (csrc/metasd_shapes.h) against the tables of what is built, on the
host: the header compiled by itself, every row length and launch size of a wide range put through it."""
import ctypes as C
import os
import subprocess

import pytest

from paper_2604_05417_b200 import binding as M

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SMS = 148

SHIM = r"""
#include "metasd_shapes.h"
using namespace metasd;

// Which form of which kernel takes a launch, as launch_staged_t() decides; form 0: aligned, groups; 1: aligned, compact; 2: shifted,
// groups; 3: shifted, compact; 4: the hinted kernel.  Returns whether it is built.
extern "C" int route(int dtype, int vocab, long long units, int n_sm, int aligned, int policies, int *threads, int *stages, int *cluster, int *form)
{
    const long long bytes = row_bytes(dtype, vocab);
    const StagedShape s = staged_shape(dtype, bytes, units, aligned, n_sm);
    *threads = s.threads; *stages = s.stages; *cluster = s.cluster;
    if (s.threads / 32 * s.cluster != row_warps(dtype, bytes)) return 0;
    if (aligned && hinted_takes(policies, false, dtype, bytes, units, s, n_sm)) {
        *form = 4;      // of the staged kernel's forms, the aligned one in groups alone splits logarithms as the hinted kernel does
        return hinted_built(dtype, s.threads, s.stages, s.cluster) && !compact_form(dtype, vocab, true, s);
    }
    const int f = *form = (aligned ? 0 : 2) + compact_form(dtype, vocab, aligned, s);
#define X(T, D, MINB, BL, CL, AG, AC, SG, SC) \
    if (s.threads == T && s.stages == D && s.cluster == CL) return f == 0 ? AG : f == 1 ? AC : f == 2 ? SG : SC;
    if (dtype == METASD_BF16) { METASD_STAGED_BF16_SHAPES(X) }
    else { METASD_STAGED_FP32_SHAPES(X) }
#undef X
    return 0;
}

extern "C" int pinned_takes(int policies) { return hinted_takes(policies, true, METASD_BF16, 2048, 2, StagedShape{384, 4, 1}, 148); }
"""


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    d = tmp_path_factory.mktemp("shapes")
    (d / "shim.cpp").write_text(SHIM)
    subprocess.check_call([os.environ.get("CXX", "g++"), "-O1", "-Wall", "-std=c++17", "-shared", "-fPIC", "-I", os.path.join(ROOT, "include"),
                           "-I", os.path.join(ROOT, "paper_2604_05417_b200", "csrc"), str(d / "shim.cpp"), "-o", str(d / "shim.so")])
    return C.CDLL(str(d / "shim.so"))


def route(rules, dtype, V, units, aligned=None, policies=True):
    """(threads, stages, CTAs per row, form) of a launch, and whether that is built."""
    t, s, c, f = (C.c_int() for _ in range(4))
    aligned = V % (8 if dtype == M.BF16 else 4) == 0 if aligned is None else aligned
    built = rules.route(dtype, V, C.c_longlong(units), SMS, int(aligned), int(policies), C.byref(t), C.byref(s), C.byref(c), C.byref(f))
    return (t.value, s.value, c.value, f.value), built


@pytest.mark.parametrize("dtype", [M.BF16, M.FP32])
def test_every_shape_and_form_that_a_launch_may_pick_is_built(rules, dtype):
    lengths = sorted({max(1, round(1.09 ** i) * 8 + d) for i in range(140) for d in (0, 1, 4)})
    units = sorted({max(2, round(1.15 ** i) + d) for i in range(87) for d in (0, 1)})
    taken = set()
    for V in lengths:
        for u in units:
            for aligned in ((True, False) if V % 8 == 0 else (False,)):     # a tensor may start off a boundary whatever its rows' length
                how, built = route(rules, dtype, V, u, aligned)
                assert built, (V, u, aligned, how)
                taken.add(how)
                if how[3] == 4:      # without policies: the same shape by the staged kernel
                    plain, built = route(rules, dtype, V, u, aligned, policies=False)
                    assert built and plain == how[:3] + (0,), (V, u, plain)
    assert len(taken) > 12


def test_the_batch_tests_reach_every_shape_of_the_hinted_kernel(rules):
    """Which launches of tests/test_gpu_batch_invariance.py are the hinted kernel's; each of its shapes meets the staged kernel's."""
    import test_gpu_batch_invariance as T
    met = set()
    for dtype, V, B in T.BATCHES + T.LONG_LAUNCHES:
        code = M.DTYPES[dtype]
        hows = [route(rules, code, V, 3 * n)[0] for n in [B] + [last - first for first, last in T.PARTS]]
        assert hows[1][3] != 4                      # a sequence on its own: the staged kernel
        met |= {(dtype,) + how[:3] for how in hows if how[3] == 4}
        if (dtype, V, B) in T.LONG_LAUNCHES:
            assert (hows[0][3] == 4) == (V != 20400)
    assert met == {("bf16", 512, 6, 1), ("bf16", 256, 6, 2), ("fp32", 256, 6, 2), ("fp32", 256, 6, 4), ("fp32", 1024, 6, 1), ("fp32", 128, 6, 8)}
    # and so do both sides of the test of square roots of two
    for code, V, few in ((M.BF16, 152064, 80), (M.FP32, 128256, 40)):
        assert route(rules, code, V, 800)[0][3] == 4 and route(rules, code, V, 2 * few)[0][3] == 0


@pytest.mark.parametrize("dtype,V,units,how", [
    # policies pay from 154 MB in flight on in the shape of the longest bf16 launches
    (M.BF16, 128256, 2048, (512, 6, 1, 0)), (M.BF16, 131192, 2870, (512, 6, 1, 4)), (M.BF16, 133512, 3892, (512, 6, 1, 4)),
    # many fp32 rows: in one CTA each where they are aligned, else in two
    (M.FP32, 32000, 4000, (512, 6, 1, 0)), (M.FP32, 32001, 4000, (256, 6, 2, 3)), (M.FP32, 35911, 2100, (256, 6, 2, 2))])
def test_launches_either_side_of_a_line(rules, dtype, V, units, how):
    """Kernel and shape where both sides of a rule's line were measured (the figures stand at the rules)."""
    assert route(rules, dtype, V, units)[0] == how


def test_a_configuration_without_policies_keeps_every_launch_off_the_hinted_kernel(rules):
    assert (rules.pinned_takes(1), rules.pinned_takes(0)) == (1, 0)
    for dtype, V, units in [(M.BF16, 152064, 4608), (M.FP32, 128256, 6144), (M.BF16, 262144, 680)]:
        assert route(rules, dtype, V, units)[0][3] == 4 and route(rules, dtype, V, units, policies=False)[0][3] == 0
