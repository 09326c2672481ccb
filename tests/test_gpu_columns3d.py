"""3D advection kernels per z-column (RK stage, refinement, details) against the
oracle on uniform and random adaptive trees with random nodal values, so that
no ghost, block-edge or predicted node agrees by accident.

Trees: level 1 (every neighbour of a block is the same block on both sides),
level 2, and two adaptive ones (levels 1-2 and 2-3: finer, equal and coarser
neighbours across faces, edges and corners).  FP64: bit for bit.  FP32 stages:
one RK4 step at CFL 0.1 amplifies the rounding of each of its four stages
(a few u = 2^-24 of the values, difference weights of size <= 1.5 / dx) by less
than 1, which leaves some tens of u: relative L2 within 1e-5.
"""
import numpy as np
import pytest

from tests import treegen
from tests.test_gpu_parity import assert_same_tree, cfg2d, make_pair, mr  # noqa: F401

pytestmark = pytest.mark.gpu

TREES = {"level1": lambda: sorted(treegen.uniform_tree(3, 1)), "level2": lambda: sorted(treegen.uniform_tree(3, 2)),
         "levels12": lambda: treegen.random_graded_tree(3, 1, 3, 3, 2),
         "levels23": lambda: treegen.random_graded_tree(3, 1, 3, 3, 4)}


def load(mr, oracle_mod, name, precision, detail_fp64=False):  # noqa: F811
    lvl, crd = treegen.as_arrays(TREES[name]())
    fields = np.random.default_rng(11).standard_normal((len(lvl), 1, 17, 17, 17)).astype(np.float32).astype(np.float64)
    o, g = make_pair(mr, oracle_mod, cfg2d(dim=3, Jmin=1, Jmax=3, ic="none", rhs_params=(0.9, -0.7, 0.4)), precision,
                     detail_fp64=detail_fp64)
    o.set_blocks(lvl, crd, fields)
    g.set_blocks(lvl, crd, fields)
    return o, g, 0.1 / (16 * (1 << int(lvl.max())))


@pytest.mark.parametrize("name", sorted(TREES))
def test_stage_refine_and_details_bit_exact(mr, oracle_mod, name):  # noqa: F811
    o, g, dt = load(mr, oracle_mod, name, "fp64")
    o.rk4(0.0, dt)
    g.rk_step(0.0, dt)
    ob, f = assert_same_tree(o, g)
    assert np.array_equal(f, ob["fields"])
    o.details()
    o.flags(0)
    g.adapt("flags_only")
    ob = o.blocks()
    gf, gm = g.get_flags()
    assert np.array_equal(gf, ob["flag"])
    assert np.array_equal(gm, ob["mdet"])
    o.refine(0)
    g.adapt("refine_all")
    ob, f = assert_same_tree(o, g)
    assert np.array_equal(f, ob["fields"])
    assert o.errors == 0


@pytest.mark.parametrize("precision", ["fp32", "fp32_acc64"])
@pytest.mark.parametrize("name", sorted(TREES))
def test_fp32_stages_within_rounding(mr, oracle_mod, name, precision):  # noqa: F811
    o, g, dt = load(mr, oracle_mod, name, precision)
    o.rk4(0.0, dt)
    g.rk_step(0.0, dt)
    ob, f = assert_same_tree(o, g)
    assert np.linalg.norm(f - ob["fields"]) <= 1e-5 * np.linalg.norm(ob["fields"])
