"""Rounding of the near field on lists, 8-byte types (csrc/forest.cu): full leaves of 200
sources, so that a lane adds about 900 terms, the large ones first.  Small terms that follow
a large sum each leave most of themselves in the sum's low word: gathered there for a whole
row they outgrow its 24 bits.

Tolerance, in units of S = sum |phi - phi0| |f| over a target's near sources and with
e = 2^-48 (float-float) or 2^-53: terms are added four by four to at least two lanes' partial
sums, N = n / 8 + 12 additions one after the other at most, each within 3 e of a partial sum.
Their errors are independent, so that they add up to more than 6 x 3 e sqrt(N) S with a
probability below 2 exp(-18) (Hoeffding).  Four terms' products, table words and charges add
at most 16 e S.  The charge channel (phi0 times the near charge, in float pairs of its own)
adds 12 e |phi0| sum |f|.
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


def _points(rng):
    """4 x 4 leaves of side 16, 200 points in each."""
    one = [workloads.distinct_in_box(rng, 200, 16, 16 * x, 16 * y) for y in range(4) for x in range(4)]
    return np.ascontiguousarray(np.concatenate(one).astype(np.int32))


@pytest.mark.parametrize("precision", ["df", "fp64"])
@pytest.mark.parametrize("large", [1.0, 2.0 ** 17, 2.0 ** 20])
def test_near_sums_keep_their_bits(lfmm, precision, large):
    prec, e = {"df": (lfmm.LFMM_DF, 2.0 ** -48), "fp64": (lfmm.LFMM_FP64, 2.0 ** -53)}[precision]
    rng = np.random.default_rng(11)
    src = _points(rng)
    f = rng.uniform(0.5, 1.0, len(src))
    f[:400] *= large  # the two leaves at the left of the lowest row: first in the order of the sums
    o = lfmm.make_opts(prec, 16, 200, tree=lfmm.LFMM_TREE_PRUNED, max_leaf_side=16)
    with lfmm.Plan(src, src, opts=o) as pl:
        info = pl.info()
        assert (info["L"], info["leaf_side"], info["max_leaf_src"]) == (2, 16, 200)
        un, _ = pl.eval_parts(f)
    ref = oracle.near_sum(src, f, src, info["x0"], info["y0"], 16)
    phi0 = abs(oracle.phi(np.array([[16, 0]]))[0])
    leaf = (src - [info["x0"], info["y0"]]) // 16
    n = np.array([(np.abs(leaf - a).max(1) <= 1).sum() for a in leaf])
    big = np.array([(f * (np.abs(leaf - a).max(1) <= 1)).sum() for a in leaf])
    # S: |phi - phi0| term by term, one block of targets at a time
    S = np.empty(len(src))
    for i in range(0, len(src), 400):
        d = src[i:i + 400, None] - src[None]
        near = np.abs(leaf[i:i + 400, None] - leaf[None]).max(2) <= 1
        p = np.abs(oracle.phi(d.reshape(-1, 2)).reshape(near.shape) + phi0)  # phi(16, 0) < 0
        S[i:i + 400] = (p * near) @ f
    tol = e * ((18 * np.sqrt(n / 8 + 12) + 16) * S + 12 * phi0 * big)
    worst = (np.abs(un - ref) / tol).max()
    assert worst <= 1.0, worst
