"""Device memory of plans whose far field runs in sliced products (csrc/split_tc.cu): what such a
plan holds is its own buffers and the work space, byte for byte, not also the partial sums
of the kernels that it does not launch; the shape without allocation reports the same; and
a device without room for the work space gets a plan that does without it.
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
    torch.cuda.init()
    return m


def _expected_bytes(info, chunks):
    """Uniform plan, both point sets read in place: buckets, sorted points, charges, expansions,
    near and far parts, the sliced rows and the chunks' sums."""
    L, ns, nt, boxes = info["L"], info["n_src"], info["n_tgt"], info["n_boxes"]
    leaves, words = 4 ** L, {2: 2, 0: 3}[info["precision"]]  # floats per sum
    inner = boxes - leaves
    up = lambda n: (n + 255) // 256 * 256
    work = sum(map(up, (boxes * 768, inner * 768, 4 * boxes, 4 * inner, chunks * boxes * 64 * words * 4,
                        chunks * boxes * 4, chunks * boxes * 8)))
    return (2 * (leaves + 1) * 4 + (2 * (ns + nt) + nt) * 4 + 8 * ns + 2 * boxes * 64 * 8 + 2 * boxes * 8
            + 2 * nt * 8 + 16 + work)


@pytest.mark.parametrize("precision", ["df", "fp64"])
@pytest.mark.parametrize("split,tc,side", [(9, 0, 1024), (1, 0, 1024), (5, 2, 256)])
def test_sliced_plan_holds_its_own_buffers(lfmm, precision, split, tc, side):
    prec = {"df": lfmm.LFMM_DF, "fp64": lfmm.LFMM_FP64}[precision]
    prob = workloads.uniform_box(side * side // 40, side * side // 50, side, seed=side)
    dev = torch.device("cuda:0")
    s, t, f = (torch.from_numpy(a).to(dev) for a in (prob.src, prob.tgt, prob.f))
    o = lfmm.make_opts(prec, 16, 32, tree=lfmm.LFMM_TREE_UNIFORM, tc_min_level=tc, max_leaf_side=16, m2l_split=split)
    shape = lfmm.lfmm_plan_shape_noalloc(s, s.shape[0], t, t.shape[0], o)
    with lfmm.Plan(s, t, opts=o) as pl:
        info = pl.info()
        assert info["leaf_side"] == 16 and info["L"] == {1024: 6, 256: 4}[side]
        assert info["device_bytes"] == shape["device_bytes"] == _expected_bytes(info, split)
        u = pl.eval(f)
        assert pl.info()["device_bytes"] == info["device_bytes"]
        # several vectors: their own charges, expansions and parts, and nothing else
        U = pl.eval_multi(f.repeat(3, 1))
        grown = pl.info()["device_bytes"] - info["device_bytes"]
        boxes, ns, nt = info["n_boxes"], info["n_src"], info["n_tgt"]
        assert grown == 3 * (8 * ns + 2 * boxes * 64 * 8 + 2 * boxes * 8 + 2 * nt * 8)
        assert torch.equal(U[0], u) and torch.equal(U[2], u)


@pytest.mark.parametrize("precision", ["df", "fp64"])
@pytest.mark.parametrize("tree", ["uniform", "pruned"])
def test_no_room_for_the_work_space(lfmm, precision, tree):
    """The n-th allocation fails for n = 1, 2, ...: the plan's creation reports LFMM_ENOMEM or, where
    it was the work space, gives a smaller plan with the same results to rounding."""
    prec = {"df": lfmm.LFMM_DF, "fp64": lfmm.LFMM_FP64}[precision]
    store = {"uniform": lfmm.LFMM_TREE_UNIFORM, "pruned": lfmm.LFMM_TREE_PRUNED}[tree]
    prob = workloads.uniform_box(9000, 7000, 512, seed=5)
    o = lfmm.make_opts(prec, 16, 32, tree=store, tc_min_level=2, max_leaf_side=16)
    idx = np.arange(0, 7000, 70)
    ref = oracle.lattice_sum(prob.src, prob.f, prob.tgt[idx])
    with lfmm.Plan(prob.src, prob.tgt, opts=o) as pl:
        full = pl.info()["device_bytes"]
        u = pl.eval(prob.f)
    torch.cuda.synchronize()
    base = lfmm.lfmm_pool_used_bytes()
    without = []
    for n in range(1, 200):
        lfmm.lfmm_fault_inject_alloc(n)
        try:
            pl = lfmm.Plan(prob.src, prob.tgt, opts=o)
        except lfmm.LfmmError as e:
            assert e.status == lfmm.LFMM_ENOMEM
            continue
        finally:
            lfmm.lfmm_fault_inject_alloc(0)
        with pl:
            size = pl.info()["device_bytes"]
            v = pl.eval(prob.f)
            V = pl.eval_multi(np.stack([prob.f, 2 * prob.f]))
            pl.status()
        assert np.abs(v[idx] - ref).max() <= 1e-10 * np.abs(ref).max()
        assert np.abs(V[0] - v).max() <= 1e-13 * np.abs(v).max() and np.abs(V[1] - 2 * v).max() <= 1e-12 * np.abs(v).max()
        assert np.abs(v - u).max() <= 9e-11 * np.abs(ref).max()
        if size == full:
            break
        without.append((n, size))
    assert len(without) == 1 and without[0][1] < full
    torch.cuda.synchronize()
    assert lfmm.lfmm_pool_used_bytes() == base
