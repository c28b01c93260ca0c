"""Rows of very different sizes in one launch of the tensor-core translations, and the digits of the
binary64 form.

The problems of a forest do not act on one another but share every launch, tile and
work item of the translations, so each one's result has to be as accurate, relative to its
own largest value, as if its charges alone were there: expansions that were scaled with the
whole level would lose the small problems altogether.

Several vectors on a uniform plan likewise share the launches of the scaled fp16 M2L: powers
of two scale through every step exactly, so vectors that differ by them give the same bits.

Binary64 in slices against the CUDA cores (tc_min_level > 30): truncation is the same on both
sides and each translation is within 2^-52 of its largest term, so 2^-52 x sqrt(10 x 27 x 64)
x (cancellation of the far field, at most 1e2 here) = 2.9e-12 of the largest value between
them: 30 times below what float-float is held to.
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


@pytest.mark.parametrize("precision,p", [("mixed", 8), ("mixed", 16), ("df", 16), ("fp64", 16)])
def test_problems_of_unlike_size(lfmm, precision, p):
    prec, tol = {"mixed": (lfmm.LFMM_MIXED, 1e-6), "df": (lfmm.LFMM_DF, 1e-10), "fp64": (lfmm.LFMM_FP64, 1e-10)}[precision]
    rng = np.random.default_rng(8)
    scales = [1.0, 1e-3, 1e-7, 1e-9, 1e-12, 1e6]
    n = [900, 1100, 700, 1000, 1300, 800]
    src = [workloads.distinct_in_box(rng, k, 130) for k in n]
    f = [workloads.zero_sum(rng.standard_normal(k)) * c for k, c in zip(n, scales)]
    copies = 6  # levels of more than 1,024 boxes: the list form of the mixed path runs there too
    off = np.concatenate([[0], np.cumsum(n * copies)]).astype(np.int64)
    S = np.ascontiguousarray(np.concatenate(src * copies).astype(np.int32))
    with lfmm.Forest(S, off, S, off, opts=lfmm.make_opts(prec, p, 16)) as fo:
        assert fo.info()["n_boxes"] > 4000
        u = fo.eval(np.concatenate(f * copies))
        fo.status()
    for i in range(len(off) - 1):
        k = i % len(n)
        ref = oracle.lattice_sum(src[k], f[k], src[k])
        assert np.abs(u[off[i]:off[i + 1]] - ref).max() <= tol * np.abs(ref).max(), (i, scales[k])


@pytest.mark.parametrize("p", [8, 16])
def test_vectors_scaled_by_powers_of_two(lfmm, p):
    prob = workloads.uniform_box(20000, 9000, 512, seed=3)
    o = lfmm.make_opts(lfmm.LFMM_MIXED, p, 32, tree=lfmm.LFMM_TREE_UNIFORM, tc_min_level=2)
    powers = [0, -40, 33, -71]
    with lfmm.Plan(prob.src, prob.tgt, opts=o) as pl:
        U = pl.eval_multi(np.stack([np.ldexp(prob.f, e) for e in powers]))
    for e, u in zip(powers, U):
        assert np.array_equal(np.ldexp(u, -e), U[0])


@pytest.mark.parametrize("n,side,leaf,tree,tc", [
    (40, 64, 8, "pruned", 0),
    (3000, 600, 24, "pruned", 0),
    (2000, 20000, 4, "pruned", 0),
    (9000, 400, 16, "uniform", 2),
])
def test_binary64_digits(lfmm, n, side, leaf, tree, tc):
    store = {"pruned": lfmm.LFMM_TREE_PRUNED, "uniform": lfmm.LFMM_TREE_UNIFORM}[tree]
    prob = workloads.uniform_box(n, n // 2 + 1, side, seed=n)
    out = []
    for level in (tc, 31):
        o = lfmm.make_opts(lfmm.LFMM_FP64, 16, leaf, tree=store, tc_min_level=level)
        with lfmm.Plan(prob.src, prob.tgt, opts=o) as pl:
            out.append(pl.eval(prob.f))
            pl.status()
    assert np.abs(out[0] - out[1]).max() <= 2.9e-12 * np.abs(out[1]).max()
