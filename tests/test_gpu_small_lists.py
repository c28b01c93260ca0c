"""P2M of pruned trees and forests on the mixed path (csrc/forest.cu): several operator rows in
flight where the leaves do not fill the chip, one where they do.

Bar: that of the path everywhere in these tests, 1e-6 of the largest value at p = 8 and 16.
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
