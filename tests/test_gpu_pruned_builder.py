"""Pruned trees whose boxes come from bit grids and those that keep sorted keys
(csrc/forest_tree.cu) against the oracle: the same cloud alone, with one point far away
(the levels between are too large for grids), on the edges of 32-cell grid words, and as
one problem of a forest beside problems of one leaf and of two levels.

Bars: those of the paths everywhere in these tests (1e-6 of the largest value mixed at
p = 8, 1e-10 float-float at p = 16); a missing or doubled link changes values by far more.
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


def _check(u, prob_src, f, tgt, tol):
    ref = oracle.lattice_sum(prob_src, f, tgt)
    assert np.abs(u - ref).max() <= tol * np.abs(ref).max()


@pytest.mark.parametrize("path", ["mixed", "df"])
@pytest.mark.parametrize("n,side,far,leaf", [
    (600, 150, 0, 8),          # a few words
    (2500, 512, 0, 16),        # every row of a class is whole words
    (2500, 1 << 9, 1 << 16, 8),   # one point far away: sorted keys
    (1500, 3000, 0, 4),        # sparse: most words empty
])
def test_pruned_tree_forms(lfmm, path, n, side, far, leaf):
    prec, p, tol = (lfmm.LFMM_MIXED, 8, 1e-6) if path == "mixed" else (lfmm.LFMM_DF, 16, 1e-10)
    prob = workloads.uniform_box(n, n // 3, side, seed=n + side)
    src = prob.src.copy()
    if far:
        src[0] = (far, far - 3)
    o = lfmm.make_opts(prec, p, leaf, tree=lfmm.LFMM_TREE_PRUNED)
    for tgt in (prob.tgt, src):
        with lfmm.Plan(src, np.ascontiguousarray(tgt), opts=o) as pl:
            u = pl.eval(prob.f)
            pl.status()
        _check(u, src, prob.f, tgt, tol)


@pytest.mark.parametrize("path", ["mixed", "df"])
def test_forest_of_unlike_problems(lfmm, path):
    prec, p, tol = (lfmm.LFMM_MIXED, 8, 1e-6) if path == "mixed" else (lfmm.LFMM_DF, 16, 1e-10)
    rng = np.random.default_rng(3)
    sizes, sides = [5, 900, 40, 1300, 3, 700], [6, 130, 40, 500, 3, 33]
    src = [workloads.distinct_in_box(rng, n, s) for n, s in zip(sizes, sides)]
    f = [workloads.zero_sum(rng.standard_normal(n)) for n in sizes]
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    s = np.ascontiguousarray(np.concatenate(src))
    with lfmm.Forest(s, off, s, off, opts=lfmm.make_opts(prec, p, 16)) as fo:
        u = fo.eval(np.concatenate(f))
        fo.status()
    for i in (1, 3, 5):
        _check(u[off[i]:off[i + 1]], src[i], f[i], src[i], tol)
    for i in (0, 2, 4):
        ref = oracle.lattice_sum(src[i], f[i], src[i])
        assert np.abs(u[off[i]:off[i + 1]] - ref).max() <= tol * max(np.abs(ref).max(), np.abs(f[i]).sum())
