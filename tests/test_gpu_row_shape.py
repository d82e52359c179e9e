"""CTA shapes of the FP32 row passes: the default rule, 256 threads x 8 values
per line and 128 x 16 (fl_plan_set_row_shape 0, 1, 2), and the tuner's choice
where the rule already takes 256 x 8 in every pass."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1802_03770_gb300 import _lib  # noqa: E402
from paper_1802_03770_gb300.api import Plan, solve_batched  # noqa: E402


def outputs(p, u):
    return p.apply(u), p.precond(u)


# default: 256 x 8 (up to two CTAs per SM), 128 x 16 (more)
@pytest.mark.parametrize("n,default", [((160, 160), 1), ((300, 257), 1), ((1024, 1024), 2), ((700, 1001), 2)])
def test_every_shape_can_be_asked_for(n, default):
    """Each shape runs its own stage plan: same numbers to FP32 rounding (2e-5 of
    the FP64 passes, the parity tests' bound), other bits; the default is one
    of the two."""
    p = Plan(2, n, 1.0 / (max(n) + 1), 1.3)
    u = torch.tensor(np.random.default_rng(12).standard_normal(p.N, dtype=np.float32), device="cuda:0")
    got = []
    for shape in (0, 1, 2):
        p.set_row_shape(shape)
        assert p.row_shape() == shape
        got.append(outputs(p, u))
    for ys, ref in zip(zip(*got), outputs(p, u.double())):
        for y in ys:
            assert float((y.double() - ref).norm()) <= 2e-5 * float(ref.norm())
        assert not torch.equal(ys[1], ys[2])
        assert torch.equal(ys[0], ys[default])
    for bad in (-1, 3):
        with pytest.raises(_lib.FracLapError, match="INVALID_ARG"):
            p.set_row_shape(bad)


def test_tuning_again_changes_no_lockstep_result():
    """On grids where the rule takes 256 x 8 in every row pass the tuner has
    nothing to time: it names that shape every time, and a lockstep batch of
    tuned plans gives the same bits after every tuning."""
    sides = [131, 160, 200]
    plans = [Plan(2, (n, n), 1.0 / (n + 1), 1.1) for n in sides]
    fs = [torch.tensor(np.random.default_rng(n).standard_normal(n * n), device="cuda:0") for n in sides]
    first = None
    for _ in range(6):
        for p in plans:
            p.autotune()
            assert p.row_shape() == 1
            p.set_tiles([0] * 6)
        us, infos = solve_batched(plans, fs, tol=1e-8)
        us = [u.clone() for u in us]
        its = [i["iterations"] for i in infos]
        if first is None:
            first = us, its
        assert its == first[1]
        assert all(torch.equal(a, b) for a, b in zip(us, first[0]))
