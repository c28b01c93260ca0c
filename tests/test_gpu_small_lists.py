"""Pruned trees and forests of little work (csrc/forest.cu), where other forms of a kernel run than
on large ones: P2M with several operator rows in flight where the leaves do not fill the
chip, the near field with more registers a thread where there is no far field, and its lanes
per target by the sources that a target has.

Bars: those of the paths everywhere in these tests (1e-6 of the largest value mixed at p = 8,
1e-10 float-float and binary64 at p = 16; problems of one leaf have no far field and are held
to 1e-6 and 1e-12 of sum |f|, the largest |phi| there being below 1).
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


@pytest.mark.parametrize("p", [8, 16])
@pytest.mark.parametrize("copies", [1, 700])  # 8 leaves; 5,600, more than a leaf per quarter warp of one wave
@pytest.mark.parametrize("counts", [(1, 2, 7, 8, 9, 15, 16, 17), (31, 32, 33, 60, 61, 63, 64, 0)])
def test_sources_per_leaf_mixed(lfmm, p, copies, counts):
    """Leaves of every remainder of the rounds of 16 sources, in a forest of copies."""
    rng = np.random.default_rng(sum(counts))
    src, tgt = [], []
    for c, n in enumerate(counts):  # leaves of side 16, three empty ones between
        at = lambda k: np.array([64 * c, 48 * (c % 5)]) + np.stack(np.divmod(rng.permutation(256)[:k], 16), 1)
        src.append(at(n))
        tgt.append(at(5))
    src, tgt = np.concatenate(src).astype(np.int32), np.concatenate(tgt).astype(np.int32)
    f = workloads.zero_sum(rng.standard_normal(len(src)))
    o = lfmm.make_opts(lfmm.LFMM_MIXED, p, 64, max_leaf_side=16)
    S, T = (np.ascontiguousarray(np.tile(a, (copies, 1))) for a in (src, tgt))
    so, to = (np.arange(copies + 1, dtype=np.int64) * len(a) for a in (src, tgt))
    with lfmm.Forest(S, so, T, to, opts=o) as fo:
        u = fo.eval(np.tile(f, copies)).reshape(copies, -1)
        fo.status()
    ref = oracle.lattice_sum(src, f, tgt)
    assert np.abs(u - ref).max() <= 1e-6 * np.abs(ref).max()


@pytest.mark.parametrize("precision", ["mixed", "df", "fp64"])
@pytest.mark.parametrize("parts", [False, True])
def test_problems_of_one_leaf(lfmm, precision, parts):
    """No far field: the near field alone writes the result, or the parts."""
    prec, p, tol = {"mixed": (lfmm.LFMM_MIXED, 8, 1e-6), "df": (lfmm.LFMM_DF, 16, 1e-12),
                    "fp64": (lfmm.LFMM_FP64, 16, 1e-12)}[precision]
    rng = np.random.default_rng(5)
    n = [1, 2, 3, 31, 32, 33, 64, 5] * 40
    m = [64, 1, 33, 32, 31, 5, 2, 64] * 40
    src = [workloads.distinct_in_box(rng, k, 20, -7, 11) for k in n]
    tgt = [workloads.distinct_in_box(rng, k, 20, -7, 11) for k in m]
    f = [rng.standard_normal(k) for k in n]
    so, to = (np.concatenate([[0], np.cumsum(k)]).astype(np.int64) for k in (n, m))
    S, T = (np.ascontiguousarray(np.concatenate(a).astype(np.int32)) for a in (src, tgt))
    with lfmm.Forest(S, so, T, to, opts=lfmm.make_opts(prec, p, 64)) as fo:
        assert fo.info()["L"] == 0
        if parts:
            u, far = fo.eval_parts(np.concatenate(f))
            assert not far.any()
        else:
            u = fo.eval(np.concatenate(f))
        fo.status()
    for i in range(len(n)):
        ref = oracle.lattice_sum(src[i], f[i], tgt[i])
        assert np.abs(u[to[i]:to[i + 1]] - ref).max() <= tol * np.abs(f[i]).sum()


@pytest.mark.parametrize("path", ["mixed", "df"])
def test_sparse_tree_in_few_blocks(lfmm, path):
    """Leaves of one or two points in a large box: a block of the near field takes several strips.
    Eager, recorded and serial evaluations run the same kernels."""
    prec, p, tol = (lfmm.LFMM_MIXED, 8, 1e-6) if path == "mixed" else (lfmm.LFMM_DF, 16, 1e-10)
    prob = workloads.uniform_box(9000, 5000, 3300, seed=2)
    idx = np.arange(0, 5000, 25)
    ref = oracle.lattice_sum(prob.src, prob.f, prob.tgt[idx])
    with lfmm.Plan(prob.src, prob.tgt, opts=lfmm.make_opts(prec, p, tree=lfmm.LFMM_TREE_PRUNED)) as pl:
        assert pl.info()["leaf_side"] == 32 and pl.info()["max_leaf_src"] < 12
        u = pl.eval(prob.f)
        for kw in ({"graph": True}, {"serial": True}):
            pl.set_flags(**kw)
            assert np.array_equal(pl.eval(prob.f), u)
        pl.status()
    assert np.abs(u[idx] - ref).max() <= tol * np.abs(ref).max()


@pytest.mark.parametrize("precision", ["df", "fp64"])
@pytest.mark.parametrize("side", [16, 80])  # one leaf; three by three
def test_lanes_per_target(lfmm, precision, side):
    """Every count of sources at which a target gets more lanes, few and many targets."""
    prec = {"df": lfmm.LFMM_DF, "fp64": lfmm.LFMM_FP64}[precision]
    rng = np.random.default_rng(side)
    n = [1, 7, 8, 15, 16, 17, 31, 32, 33, 63, 64, 65, 127, 128, 129, 200] * 2
    m = [3] * 16 + [150] * 16
    src = [workloads.distinct_in_box(rng, k, side) for k in n]
    tgt = [workloads.distinct_in_box(rng, k, side) for k in m]
    f = [workloads.zero_sum(rng.standard_normal(k)) if k > 1 else np.ones(1) for k in n]
    so, to = (np.concatenate([[0], np.cumsum(k)]).astype(np.int64) for k in (n, m))
    S, T = (np.ascontiguousarray(np.concatenate(a).astype(np.int32)) for a in (src, tgt))
    with lfmm.Forest(S, so, T, to, opts=lfmm.make_opts(prec, 16, 200)) as fo:
        u = fo.eval(np.concatenate(f))
        fo.status()
    for i in range(len(n)):
        ref = oracle.lattice_sum(src[i], f[i], tgt[i])
        tol = 1e-12 if side <= 32 else 1e-10
        assert np.abs(u[to[i]:to[i + 1]] - ref).max() <= tol * np.abs(f[i]).sum()
