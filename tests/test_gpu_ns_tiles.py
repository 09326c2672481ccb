"""Navier-Stokes stages (flux and skew-symmetric form) and the shock filter on
node-major tiles against the oracle, at the trees where a tile can go wrong:
level 1 (a block's neighbours on both sides are the same block) and a random
adaptive tree (finer, equal and coarser neighbours), for both block sizes.

FP64: bit for bit.  FP32 stages: one RK4 step at CFL 0.1 of values of size 1 to 3
amplifies the rounding of its four stages (a few u = 2^-24 of the values) by less
than 1, which leaves some tens of u: relative L2 within 1e-5.
"""
import numpy as np
import pytest

from tests import treegen
from tests.test_gpu_ns_skew import dsl_cfg, dsl_dt, make, mr  # noqa: F401
from tests.test_gpu_parity import assert_same_tree

pytestmark = pytest.mark.gpu

TREES = {"level1": lambda: sorted(treegen.uniform_tree(2, 1)),
         "random": lambda: sorted(treegen.random_graded_tree(2, 1, 3, 5, 3))}


def load(mr, oracle_mod, form, Bs, name, precision):  # noqa: F811
    c = dsl_cfg(form, Bs=Bs, Jmin=1, Jmax=3)
    o, g = make(mr, oracle_mod, c, precision)
    lvl, crd = treegen.as_arrays(TREES[name]())
    o.set_blocks(lvl, crd, np.zeros((len(lvl), 4, Bs, Bs)))
    o.set_ic()
    b = o.blocks()
    f = b["fields"].astype(np.float32).astype(np.float64)
    o.set_blocks(b["level"], b["coords"], f)
    g.set_blocks(b["level"], b["coords"], f)
    return o, g, 0.2 * dsl_dt(c)


@pytest.mark.parametrize("name", sorted(TREES))
@pytest.mark.parametrize("Bs", [17, 33])
@pytest.mark.parametrize("form", ["ns", "ns_skew"])
def test_stage_and_filter_bit_exact(mr, oracle_mod, form, Bs, name):  # noqa: F811
    o, g, dt = load(mr, oracle_mod, form, Bs, name, "fp64")
    o.rk4(0.0, dt)
    g.rk_step(0.0, dt)
    ob, f = assert_same_tree(o, g)
    assert np.array_equal(f, ob["fields"])
    o.filter()
    g.filter()
    ob, f = assert_same_tree(o, g)
    assert np.array_equal(f, ob["fields"])
    assert o.errors == 0


@pytest.mark.parametrize("precision", ["fp32", "fp32_acc64"])
@pytest.mark.parametrize("name", sorted(TREES))
@pytest.mark.parametrize("Bs", [17, 33])
@pytest.mark.parametrize("form", ["ns", "ns_skew"])
def test_fp32_stages_within_rounding(mr, oracle_mod, form, Bs, name, precision):  # noqa: F811
    o, g, dt = load(mr, oracle_mod, form, Bs, name, precision)
    o.rk4(0.0, dt)
    g.rk_step(0.0, dt)
    ob, f = assert_same_tree(o, g)
    assert np.linalg.norm(f - ob["fields"]) <= 1e-5 * np.linalg.norm(ob["fields"])
