"""P2M of the binary64-accurate paths on lists, four warps per leaf (csrc/forest.cu): leaves
of every remainder of the split (fewer sources than warps, one more than a round of 32 per
warp, a full leaf), an odd number of leaves, and leaves without sources.

Tolerance: binary64-accurate plans at p = 16 are held to 1e-10 of the largest value, by
truncation; the sums here differ from one chain per leaf by rounding only.
"""
import numpy as np
import pytest

import oracle
from paper_1105_3505_gb300 import build

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
@pytest.mark.parametrize("counts", [
    (1, 2, 3, 4, 5, 7, 8, 9),
    (31, 32, 33, 127, 128, 129, 130),
    (192, 1, 227, 0, 64),  # 227: the fullest leaf that list storage takes
])
def test_sources_per_leaf(lfmm, precision, counts):
    rng = np.random.default_rng(sum(counts))
    src, tgt = [], []
    for c, n in enumerate(counts):  # leaves of side 16, three empty ones between
        at = lambda k: np.array([64 * c, 48 * (c % 5)]) + np.stack(np.divmod(rng.permutation(256)[:k], 16), 1)
        src.append(at(n))
        tgt.append(at(5))
    src, tgt = np.concatenate(src).astype(np.int32), np.concatenate(tgt).astype(np.int32)
    f = rng.standard_normal(len(src))
    prec = {"df": lfmm.LFMM_DF, "fp64": lfmm.LFMM_FP64}[precision]
    o = lfmm.make_opts(prec, 16, 256, tree=lfmm.LFMM_TREE_PRUNED, max_leaf_side=16)
    with lfmm.Plan(src, tgt, opts=o) as pl:
        u = pl.eval(f)
        pl.status()
    ref = oracle.lattice_sum(src, f, tgt)
    assert np.abs(u - ref).max() <= 1e-10 * np.abs(ref).max()
