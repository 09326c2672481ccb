"""The coarsening threshold at the ends of its range, normalised and not: the flags are the
oracle's, which compares the detail with eps (strictly below; no detail is below a NaN)."""
import math

import numpy as np
import pytest

from tests import treegen
from tests.test_gpu_parity import cfg2d, make_pair, mr  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("norm_kind", [0, 1])
@pytest.mark.parametrize("eps", [math.nan, -math.nan, math.inf, 0.0, -1.0, 5e-324])
def test_flags_at_odd_thresholds(mr, oracle_mod, eps, norm_kind):  # noqa: F811
    lvl, crd = treegen.as_arrays(sorted(treegen.random_graded_tree(2, 1, 4, 6, 9)))
    f = np.random.default_rng(3).standard_normal((len(lvl), 1, 17, 17))
    f[: len(lvl) // 2] = 1.0  # details of exactly zero in the first half
    o, g = make_pair(mr, oracle_mod, cfg2d(Jmin=1, Jmax=4, eps=eps, ic="none", norm_kind=norm_kind))
    o.set_blocks(lvl, crd, f)
    g.set_blocks(lvl, crd, f)
    o.details()
    o.flags(0)
    g.adapt("flags_only")
    want = o.blocks()["flag"]
    assert np.array_equal(g.get_flags()[0], want)
    assert (want == -2).any() == (eps > 0)
