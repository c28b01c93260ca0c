"""The sliced tensor-core far field of the binary64-accurate paths (csrc/split_tc.cu).

Sizes at the edges of its work items (fewer boxes than one 128-box tile, one box more
than a tile, one level only, the deepest chain), each storage form and both precisions,
against the oracle and against the same plan with the tensor cores kept out
(tc_min_level > 30).

Tolerance: both forms carry about 2^-47 per translation; an entry of u is a sum over at
most ~10 levels of 27 x 64 terms, and binary64-accurate plans are held to 1e-10 of the
largest value everywhere in these tests, so 1e-10 against the oracle; between the two
forms 2^-47 x sqrt(10 x 27 x 64) x (cancellation of the far field, at most 1e2 here)
= 9e-11 at p = 16, where truncation is the same on both sides.
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
@pytest.mark.parametrize("n,side,leaf,tree,tc", [
    (40, 64, 8, "pruned", 0),        # few boxes, two levels
    (3000, 600, 24, "pruned", 0),    # classes of one tile and a bit
    (2000, 20000, 4, "pruned", 0),   # sparse and deep: most interaction lists are short
    (9000, 400, 16, "uniform", 2),   # uniform storage, every level sliced
    (40000, 900, 16, "uniform", 0),  # more tiles than SMs: no split along the offsets
])
def test_sliced_far_field(lfmm, precision, n, side, leaf, tree, tc):
    prec = {"df": lfmm.LFMM_DF, "fp64": lfmm.LFMM_FP64}[precision]
    store = {"pruned": lfmm.LFMM_TREE_PRUNED, "uniform": lfmm.LFMM_TREE_UNIFORM}[tree]
    prob = workloads.uniform_box(n, n // 2 + 1, side, seed=n)
    out = []
    for level in (tc, 31):
        o = lfmm.make_opts(prec, 16, leaf, tree=store, tc_min_level=level)
        with lfmm.Plan(prob.src, prob.tgt, opts=o) as pl:
            out.append(pl.eval(prob.f))
            pl.status()
    idx = np.arange(0, prob.tgt.shape[0], max(1, prob.tgt.shape[0] // 700))
    ref = oracle.lattice_sum(prob.src, prob.f, prob.tgt[idx])
    scale = np.abs(ref).max()
    assert np.abs(out[0][idx] - ref).max() <= 1e-10 * scale
    assert np.abs(out[0] - out[1]).max() <= 9e-11 * scale


@pytest.mark.parametrize("precision", ["df", "fp64"])
def test_sliced_far_field_scales(lfmm, precision):
    """Charges of very different sizes in different regions (slices are scaled row by
    row), very large and very small ones, and a NaN, which reaches every far target."""
    prec = {"df": lfmm.LFMM_DF, "fp64": lfmm.LFMM_FP64}[precision]
    prob = workloads.uniform_box(4000, 4000, 1000, seed=5)
    o = lfmm.make_opts(prec, 16, 16, tree=lfmm.LFMM_TREE_PRUNED)
    idx = np.arange(0, 4000, 8)
    big = 1e200 if precision == "fp64" else 1e25
    with lfmm.Plan(prob.src, prob.tgt, opts=o) as pl:
        f = prob.f * np.where(prob.src[:, 0] < 500, 1.0, 1e-9)
        f = workloads.zero_sum(f)
        ref = oracle.lattice_sum(prob.src, f, prob.tgt[idx])
        u = pl.eval(f)
        assert np.abs(u[idx] - ref).max() <= 1e-10 * np.abs(ref).max()
        for c in (big, 1.0 / big) if precision == "fp64" else (big,):
            v = pl.eval(f * c)
            assert np.abs(v / c - u).max() <= 1e-10 * np.abs(ref).max()
        f[7] = np.nan
        far = np.abs(prob.tgt - prob.src[7]).max(1) > 200
        assert far.any() and np.isnan(pl.eval(f)[far]).all()
        f[7] = 0.0
        assert np.isfinite(pl.eval(f)).all()
