"""The uniform tensor-core M2L in scaled fp16 halves (csrc/m2l_tc.cu, TMA form): the rows'
power-of-two scaling over very different charges, at every level's smallest tiles (levels
from 2 on: class grids of 2 x 2 boxes), both padded lengths and ring depths, against the
oracle.

Bar: the mixed path's 1e-6 of the largest value.  The halves carry 22 bits of each row's
largest entry and an absolute 2^-40 below that, so charges scaled by 1e-7 in half of the
box change nothing above 1e-6 of the sum, and a common factor of 1e25 or 1e-25 (exact up
to rounding) must not change the result by more than the factor.
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
@pytest.mark.parametrize("stages", [0, 2, 4])
def test_scaled_halves(lfmm, p, stages):
    prob = workloads.uniform_box(6000, 4000, 256, seed=17)
    o = lfmm.make_opts(lfmm.LFMM_MIXED, p, 32, tc_min_level=2, tree=lfmm.LFMM_TREE_UNIFORM, m2l_stages=stages)
    f = workloads.zero_sum(prob.f * np.where(prob.src[:, 0] < 128, 1.0, 1e-7))
    idx = np.arange(0, 4000, 5)
    ref = oracle.lattice_sum(prob.src, f, prob.tgt[idx])
    scale = np.abs(ref).max()
    with lfmm.Plan(prob.src, prob.tgt, opts=o) as pl:
        assert pl.info()["L"] >= 4
        u = pl.eval(f)
        assert np.abs(u[idx] - ref).max() <= 1e-6 * scale
        for c in (1e25, 1e-25):
            assert np.abs(pl.eval(f * c) / c - u).max() <= 1e-6 * scale
        f[3] = np.nan
        far = np.abs(prob.tgt - prob.src[3]).max(1) > 100
        assert far.any() and np.isnan(pl.eval(f)[far]).all()
