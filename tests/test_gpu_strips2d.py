"""2D advection stage with gathered ghost strips against the oracle: one CTA and
one warp per block, both block sizes, trees where a strip can go wrong (level 1:
a block's neighbours on both sides are the same block; random adaptive trees:
coarser, equal and finer neighbours across edges and corners), random nodal values.

FP64: bit for bit.  FP32 stages: one RK4 step at CFL 0.1 amplifies the rounding of
its four stages (a few u = 2^-24 of the values, difference weights of size
<= 1.5 / dx) by less than 1, which leaves some tens of u: relative L2 within 1e-5.
"""
import numpy as np
import pytest

from tests import treegen
from tests.test_gpu_parity import assert_same_tree, cfg2d, make_pair, mr  # noqa: F401

pytestmark = pytest.mark.gpu

TREES = {"level1": lambda: sorted(treegen.uniform_tree(2, 1)), "level3": lambda: sorted(treegen.uniform_tree(2, 3)),
         "random4": lambda: sorted(treegen.random_graded_tree(2, 1, 4, 6, 9)),
         "random5": lambda: sorted(treegen.random_graded_tree(2, 2, 5, 8, 4))}
FORMS = [(17, 0), (17, 1), (33, 0)]  # block size, one warp per block


def step(mr, oracle_mod, Bs, form, rhs, name, precision, staging=1):  # noqa: F811
    lvl, crd = treegen.as_arrays(TREES[name]())
    f = np.random.default_rng(11).standard_normal((len(lvl), 1, Bs, Bs)).astype(np.float32).astype(np.float64)
    c = cfg2d(Bs=Bs, Jmin=1, Jmax=5, ic="none", rhs=rhs, rhs_params=(5.0,) if rhs == "swirl" else (0.9, -0.7, 0.0))
    o, g = make_pair(mr, oracle_mod, c, precision)
    g.set_tuning(0, form)
    g.set_warp_form(4, staging)
    o.set_blocks(lvl, crd, f)
    g.set_blocks(lvl, crd, f)
    dt = 0.1 / ((Bs - 1) * (1 << int(lvl.max())))
    o.rk4(0.3, dt)
    g.rk_step(0.3, dt)
    ob, f = assert_same_tree(o, g)
    assert o.errors == 0
    return ob["fields"], f


@pytest.mark.parametrize("name", sorted(TREES))
@pytest.mark.parametrize("rhs", ["adv", "swirl"])
@pytest.mark.parametrize("Bs,form", FORMS)
def test_stage_bit_exact(mr, oracle_mod, Bs, form, rhs, name):  # noqa: F811
    want, got = step(mr, oracle_mod, Bs, form, rhs, name, "fp64")
    assert np.array_equal(got, want)


@pytest.mark.parametrize("precision,staging", [("fp32", 1), ("fp32", 0), ("fp32_acc64", 1)])
@pytest.mark.parametrize("name", sorted(TREES))
@pytest.mark.parametrize("Bs,form", FORMS)
def test_fp32_stages_within_rounding(mr, oracle_mod, Bs, form, name, precision, staging):  # noqa: F811
    want, got = step(mr, oracle_mod, Bs, form, "adv", name, precision, staging)
    assert np.linalg.norm(got - want) <= 1e-5 * np.linalg.norm(want)
