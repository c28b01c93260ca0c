"""Operators of the model boxes on the device (csrc/skeleton.cpp): the sliced ones are built for
plans that use them only, beside the others or later, and plans that came before keep theirs.

The first plan of a configuration pays for its operators, so a plan that keeps the tensor
cores out must not pay for slices: device memory taken by its creation is held against the
size of its own operators (the expansion arrays come from the pool, which a plan of the same
shape has filled before).
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


def _free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


@pytest.mark.parametrize("precision", ["df", "fp64"])
def test_slices_only_where_used(lfmm, precision):
    prec = {"df": lfmm.LFMM_DF, "fp64": lfmm.LFMM_FP64}[precision]
    prob = workloads.uniform_box(3000, 2000, 8000, seed=9)
    idx = np.arange(0, 2000, 40)
    ref = oracle.lattice_sum(prob.src, prob.f, prob.tgt[idx])

    def plan(proxies, tc, side=32):
        return lfmm.Plan(prob.src, prob.tgt, opts=lfmm.make_opts(prec, 16, proxies_per_edge=proxies, tc_min_level=tc,
                                                                 tree=lfmm.LFMM_TREE_PRUNED, max_leaf_side=side))

    plan(60, 0).close()  # fills the pool, loads the kernels
    before = _free()
    with plan(52, 31) as kept:
        levels = kept.info()["L"] - 1
        taken = before - _free()
        # T_ofs, the table, per level 48 matrices of 64 x 64; a few MB of the allocator's granules
        own = 8 * (1024 * 64 + 127 * 144 + levels * 48 * 64 * 64)
        assert levels >= 6 and taken <= own + (6 << 20) < own + levels * 48 * 6 * 8192, (taken, own)
        u = [kept.eval(prob.f)]
        with plan(52, 0) as later:  # the slices come now
            u.append(later.eval(prob.f))
        u.append(kept.eval(prob.f))
    with plan(44, 0) as first:  # with the others
        u.append(first.eval(prob.f))
        with plan(44, 31) as beside:
            u.append(beside.eval(prob.f))
    for v in u:
        assert np.abs(v[idx] - ref).max() <= 1e-10 * np.abs(ref).max()
    assert np.array_equal(u[0], u[2])


@pytest.mark.parametrize("precision", ["df", "fp64"])
def test_deeper_trees_replace_the_image(lfmm, precision):
    """Three depths on one cache entry: sliced, deeper without slices, deeper still sliced, the
    first plan kept through all of them."""
    prec = {"df": lfmm.LFMM_DF, "fp64": lfmm.LFMM_FP64}[precision]
    plans, probs = [], []
    for side, tc in ((300, 0), (1500, 31), (6000, 0), (300, 0)):
        prob = workloads.uniform_box(2000, 1000, side, seed=side + tc)
        o = lfmm.make_opts(prec, 16, 8, proxies_per_edge=56, tc_min_level=tc, tree=lfmm.LFMM_TREE_PRUNED,
                           max_leaf_side=16)
        plans.append(lfmm.Plan(prob.src, prob.tgt, opts=o))
        probs.append(prob)
    for pl, prob in [*zip(plans, probs)] * 2:
        ref = oracle.lattice_sum(prob.src, prob.f, prob.tgt[::20])
        assert np.abs(pl.eval(prob.f)[::20] - ref).max() <= 1e-10 * np.abs(ref).max()
    for pl in plans:
        pl.status()
        pl.close()


def test_tiles_grow_with_the_plans(lfmm):
    """Mixed plans of one cache entry that use more and more of the tensor-core tiles: none, some
    levels of the uniform form, lists, all levels; the earlier ones are evaluated again after."""
    prob = workloads.uniform_box(9000, 7000, 1024, seed=77)
    ref = oracle.lattice_sum(prob.src, prob.f, prob.tgt[::70])
    plans = []
    for tc, tree in ((31, lfmm.LFMM_TREE_UNIFORM), (6, lfmm.LFMM_TREE_UNIFORM), (0, lfmm.LFMM_TREE_PRUNED),
                     (4, lfmm.LFMM_TREE_UNIFORM), (2, lfmm.LFMM_TREE_UNIFORM)):
        o = lfmm.make_opts(lfmm.LFMM_MIXED, 8, 64, proxies_per_edge=48, tc_min_level=tc, tree=tree, max_leaf_side=16)
        plans.append(lfmm.Plan(prob.src, prob.tgt, opts=o))
    assert plans[0].info()["L"] == 6 and plans[2].info()["n_boxes"] > 4000
    for pl in plans * 2:
        assert np.abs(pl.eval(prob.f)[::70] - ref).max() <= 1e-6 * np.abs(ref).max()
    for pl in plans:
        pl.status()
        pl.close()
