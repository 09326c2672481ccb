"""New block lists of refinement and merging: offsets from totals of groups of 8
positions, families merged in a permuted order, one variable or four per block.

Forests of trees of different sizes (list lengths with every remainder by 8, a
tree that starts and ends inside a group) against one oracle per tree, FP64 bit
for bit through refine-all and the merging rounds that follow; and lists beyond
the length that one CTA scans, against the canonical order of a uniform tree.
"""
import numpy as np
import pytest

from tests import treegen
from tests.test_gpu_parity import cfg2d, mr  # noqa: F401

pytestmark = pytest.mark.gpu


def tree_cfg(dim, Bs, nvar, k):
    if nvar == 4:
        return dict(dim=dim, Bs=Bs, nvar=4, Jmin=1, Jmax=4, eps=1e-3, norm_kind=1, rhs="ns",
                    rhs_params=(1.4, 1e-3, 0.71), x0=(0.0, -0.5, 0.0), ic="mixing",
                    ic_params=(0.03 + 0.01 * k, 0.5, 0.3, 1.4, 1e-3) + (0.5, -0.3) * 4 + (0.1, 2.0) * 4)
    return cfg2d(dim=dim, Bs=Bs, Jmin=1, Jmax=4, eps=10.0 ** (-2 - k % 3), rhs_params=(1.0, 0.5, 0.0),
                 ic_params=(0.3 + 0.1 * k, 0.6, 0.4, 0.04 + 0.01 * k))


@pytest.mark.parametrize("dim,Bs,nvar,levels", [(2, 17, 1, (3, 1, 2, 3, 1)), (2, 33, 1, (2, 1, 3)),
                                                (2, 17, 4, (1, 3, 2)), (2, 33, 4, (2, 1)), (3, 17, 1, (1, 2, 1))])
def test_refine_and_merge_forest_bit_exact(mr, oracle_mod, dim, Bs, nvar, levels):  # noqa: F811
    cfgs = [tree_cfg(dim, Bs, nvar, k) for k in range(len(levels))]
    keys = ("Jmin", "Jmax", "eps", "ic", "ic_params", "rhs_params") + (("x0",) if nvar == 4 else ())
    g = mr.Forest(dim=dim, Bs=Bs, nvar=nvar, precision="fp64", rhs=cfgs[0]["rhs"], capacity=4096,
                  norm_kind=cfgs[0].get("norm_kind", 0), trees=[{q: c[q] for q in keys} for c in cfgs])
    os_, lv, cr, fl, tr = [], [], [], [], []
    for k, J in enumerate(levels):
        o = oracle_mod.Oracle(cfgs[k])
        leaves = sorted(treegen.uniform_tree(dim, J)) if k % 2 == 0 else sorted(
            treegen.random_graded_tree(dim, 1, max(J, 2), 2, k))
        lvl, crd = treegen.as_arrays(leaves)
        o.set_blocks(lvl, crd, np.zeros((len(lvl), nvar) + (Bs,) * dim))
        o.set_ic()
        b = o.blocks()
        os_.append(o)
        lv.append(b["level"]); cr.append(b["coords"]); fl.append(b["fields"]); tr.append(np.full(o.n, k))
    g.set_blocks(np.concatenate(lv), np.concatenate(cr), np.concatenate(fl), tree=np.concatenate(tr))
    merged = 0
    for mode in ("refine_all", "coarsen"):
        g.adapt(mode)
        for k, o in enumerate(os_):
            n0 = o.n
            o.refine(0) if mode == "refine_all" else o.coarsen_until_stable()
            merged += n0 > o.n
            ob = o.blocks()
            info, f = g.get_blocks(k)
            assert np.array_equal(info["level"], ob["level"])
            assert np.array_equal(info["coords"].astype(np.int64), ob["coords"])
            assert np.array_equal(f, ob["fields"])
            assert o.errors == 0
    assert merged


def test_lists_beyond_one_scan(mr):  # noqa: F811
    g = mr.Forest(dim=2, precision="fp32", capacity=340_000,
                  trees=[dict(Jmin=8, Jmax=9, eps=1e-3, ic="none")])
    lvl, crd = treegen.as_arrays(sorted(treegen.uniform_tree(2, 8)))
    g.set_blocks(lvl, crd, np.ones((len(lvl), 1, 17, 17)))
    coarse, _ = g.get_blocks(fields=False)
    g.adapt("refine_all")
    fine, _ = g.get_blocks(fields=False)
    assert len(fine) == 4 * len(lvl) and (fine["level"] == 9).all()
    assert (np.diff(fine["hilbert_key"].astype(np.int64)) > 0).all()
    assert len(np.unique(fine["coords"][:, :2].astype(np.int64) @ (1, 512))) == len(fine)
    g.adapt("coarsen")
    back, f = g.get_blocks()
    assert np.array_equal(back["level"], coarse["level"]) and np.array_equal(back["coords"], coarse["coords"])
    assert (f == 1.0).all()


@pytest.mark.parametrize("dim,Bs", [(2, 17), (2, 33), (3, 17)])
def test_plans_stand_while_the_tree_does(mr, oracle_mod, dim, Bs):  # noqa: F811
    # eps = 0: no family merges and the finest level cannot refine, so the stage plans
    # of the first step serve the next ones; then another tree takes their place, twice
    c = cfg2d(dim=dim, Bs=Bs, Jmin=1, Jmax=2, eps=0.0, ic="none", rhs_params=(0.9, -0.7, 0.4))
    o = oracle_mod.Oracle(c)
    g = mr.Forest(dim=dim, Bs=Bs, precision="fp64", rhs="adv", capacity=512,
                  trees=[{q: c[q] for q in ("Jmin", "Jmax", "eps", "ic", "rhs_params")}])
    dt = 0.1 / ((Bs - 1) * 4)
    uniform = sorted(treegen.uniform_tree(dim, 2))
    for k, leaves in enumerate((uniform, treegen.random_graded_tree(dim, 1, 2, 1, 3), uniform)):
        lvl, crd = treegen.as_arrays(leaves)
        f = np.random.default_rng(20 + k).standard_normal((len(lvl), 1) + (Bs,) * dim)
        o.set_blocks(lvl, crd, f)
        g.set_blocks(lvl, crd, f)
        for s in range(2):
            o.step(s * dt, dt)
            g.step(s * dt, dt)
            ob = o.blocks()
            info, got = g.get_blocks()
            assert np.array_equal(info["coords"].astype(np.int64), ob["coords"])
            assert np.array_equal(got, ob["fields"])


def test_long_list_without_changes(mr):  # noqa: F811
    # 65536 blocks: the scan finds that every block stays and writes no offsets
    g = mr.Forest(dim=2, precision="fp32", capacity=66_000, trees=[dict(Jmin=8, Jmax=8, eps=1e-3, ic="none")])
    lvl, crd = treegen.as_arrays(sorted(treegen.uniform_tree(2, 8)))
    g.set_blocks(lvl, crd, np.ones((len(lvl), 1, 17, 17)))
    before, _ = g.get_blocks(fields=False)
    for s in range(2):
        g.step(0.0, 1e-5)
    after, f = g.get_blocks()
    assert np.array_equal(before["hilbert_key"], after["hilbert_key"]) and (f == 1.0).all()
