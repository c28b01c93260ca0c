"""Bounded waits of the sliced far field (csrc/split_tc.cu).  With one poll per mbarrier wait the
pipeline gives up at its first wait: every role runs out without waiting, the teardown waits
(with the clock bound) for the copies and products issued, tensor memory is freed and the
plan reports LFMM_ETIMEOUT; its next evaluation is bit-identical to one made before.  Lists (M2M,
M2L, L2L) and a uniform tree of two levels, whose far field is this kernel's alone (no
cooperative kernel and no grid barrier), both precisions.
"""
import numpy as np
import pytest

import oracle
from paper_1105_3505_gb300 import build, workloads

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def lfmm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    from paper_1105_3505_gb300 import lfmm as m
    m.load()
    return m


@pytest.mark.parametrize("precision", ["df", "fp64"])
@pytest.mark.parametrize("tree", ["pruned", "uniform"])
def test_one_poll_times_out_and_recovers(lfmm, precision, tree):
    prec = {"df": lfmm.LFMM_DF, "fp64": lfmm.LFMM_FP64}[precision]
    if tree == "pruned":
        prob = workloads.uniform_box(12000, 9000, 700, seed=4)
        o = lfmm.make_opts(prec, 16, 8, tree=lfmm.LFMM_TREE_PRUNED, max_leaf_side=16)
    else:
        prob = workloads.uniform_box(400, 400, 64, seed=64)
        o = lfmm.make_opts(prec, 16, 64, tree=lfmm.LFMM_TREE_UNIFORM, tc_min_level=2, max_leaf_side=16)
    idx = np.arange(0, prob.tgt.shape[0], 40)
    ref = oracle.lattice_sum(prob.src, prob.f, prob.tgt[idx])
    with lfmm.Plan(prob.src, prob.tgt, opts=o) as pl:
        if tree == "uniform":
            assert pl.info()["L"] == 2
        u0 = pl.eval(prob.f)
        pl.status()
        assert np.abs(u0[idx] - ref).max() <= 1e-10 * np.abs(ref).max()
        lfmm.lfmm_plan_set_wait_budget(pl.handle, 1)
        lfmm.lfmm_profile_enable(True)
        lfmm.lfmm_profile_read(reset=True)
        try:
            pl.eval(prob.f)
            prof = lfmm.lfmm_profile_read(reset=True)
        finally:
            lfmm.lfmm_profile_enable(False)
        assert prof["m2l_tc"][1] > 0
        with pytest.raises(lfmm.LfmmError) as ei:
            pl.status()
        assert ei.value.status == lfmm.LFMM_ETIMEOUT
        lfmm.lfmm_plan_set_wait_budget(pl.handle, 0)
        for _ in range(2):
            u1 = pl.eval(prob.f)
            pl.status()
            assert np.array_equal(u0, u1)
