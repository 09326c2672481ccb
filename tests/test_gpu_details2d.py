"""2D details per (block, variable) and refinement per (mother, variable) against
the oracle: 17^2 (a warp per item) and 33^2 (a CTA per item) blocks of one and four
variables, uniform grids (level 1: a block's neighbours on both sides are the
same block) and random adaptive trees, random nodal values.  Flags, block norms
and refined fields bit for bit in FP64; the certified FP32 evaluation (FP32 fields,
FP64 decisions) gives the flags of the FP64 evaluation of the same values, at a
threshold set to the median detail, so that about half of the blocks lie on each side.
"""
import numpy as np
import pytest

from tests import treegen
from tests.test_gpu_parity import assert_same_tree, make_pair, mr  # noqa: F401

pytestmark = pytest.mark.gpu

TREES = {"level1": lambda: sorted(treegen.uniform_tree(2, 1)), "level3": lambda: sorted(treegen.uniform_tree(2, 3)),
         "random": lambda: sorted(treegen.random_graded_tree(2, 1, 4, 6, 9))}


def config(Bs, nvar, eps):
    c = dict(dim=2, Bs=Bs, nvar=nvar, Jmin=1, Jmax=4, eps=eps, rhs="ns" if nvar == 4 else "adv",
             rhs_params=(1.4, 1e-3, 0.71) if nvar == 4 else (1.0, 0.5, 0.0), ic="none", norm_kind=int(nvar == 4))
    return c


@pytest.mark.parametrize("name", sorted(TREES))
@pytest.mark.parametrize("nvar", [1, 4])
@pytest.mark.parametrize("Bs", [17, 33])
def test_details_and_refinement_bit_exact(mr, oracle_mod, Bs, nvar, name):  # noqa: F811
    lvl, crd = treegen.as_arrays(TREES[name]())
    f = np.random.default_rng(3).standard_normal((len(lvl), nvar, Bs, Bs))
    f *= np.random.default_rng(4).uniform(0.1, 1.0, (len(lvl), 1, 1, 1))
    o, g = make_pair(mr, oracle_mod, config(Bs, nvar, 1.0))
    o.set_blocks(lvl, crd, f)
    g.set_blocks(lvl, crd, f)
    o.details()
    o.flags(0)
    g.adapt("flags_only")
    ob = o.blocks()
    gf, gm = g.get_flags()
    assert np.array_equal(gf, ob["flag"])
    assert np.array_equal(gm, ob["mdet"])
    o.refine(0)
    g.adapt("refine_all")
    ob, gfl = assert_same_tree(o, g)
    assert np.array_equal(gfl, ob["fields"])
    assert o.errors == 0


@pytest.mark.parametrize("name", sorted(TREES))
@pytest.mark.parametrize("Bs", [17, 33])
def test_certified_decisions(mr, oracle_mod, Bs, name):  # noqa: F811
    lvl, crd = treegen.as_arrays(TREES[name]())
    f = np.random.default_rng(5).standard_normal((len(lvl), 1, Bs, Bs))
    f *= np.random.default_rng(6).uniform(0.1, 1.0, (len(lvl), 1, 1, 1))
    f = f.astype(np.float32).astype(np.float64)
    o, _ = make_pair(mr, oracle_mod, config(Bs, 1, 1.0))
    o.set_blocks(lvl, crd, f)
    o.details()
    o.flags(0)
    eps = float(np.median(o.blocks()["mdet"]))  # one block's detail is the threshold itself (odd counts)
    o, g = make_pair(mr, oracle_mod, config(Bs, 1, eps), precision="fp32", detail_fp64=True)
    o.set_blocks(lvl, crd, f)
    g.set_blocks(lvl, crd, f)
    o.details()
    o.flags(0)
    g.adapt("flags_only")
    assert np.array_equal(g.get_flags()[0], o.blocks()["flag"])


@pytest.mark.parametrize("scale", [1.0, 2.0 ** -1020, 2.0 ** -1060, 2.0 ** 1000])
def test_prediction_at_the_ends_of_fp64(mr, oracle_mod, scale):  # noqa: F811
    # the prediction's division by 16 next to and below the smallest normal number
    lvl, crd = treegen.as_arrays(TREES["random"]())
    f = np.random.default_rng(8).standard_normal((len(lvl), 1, 17, 17)) * scale
    o, g = make_pair(mr, oracle_mod, config(17, 1, 1.0))
    o.set_blocks(lvl, crd, f)
    g.set_blocks(lvl, crd, f)
    o.details()  # synchronises the redundant copies, as the library's details do
    o.flags(0)
    g.adapt("flags_only")
    assert np.array_equal(g.get_flags()[1], o.blocks()["mdet"])
    o.refine(0)
    g.adapt("refine_all")
    ob, gfl = assert_same_tree(o, g)
    assert np.array_equal(gfl, ob["fields"])
