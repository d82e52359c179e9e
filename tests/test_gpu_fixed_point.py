"""FP64 passes on 64-bit fixed-point lines (apply and preconditioner) against
the oracle: every line length's edge, the ends of the FP64 range, lines of
zeros and non-finite inputs.

Tolerance of the applies: an FP64 FFT of up to 2^24 points has a relative
2-norm error below 5e-16 (0.6 2^-53 sqrt(log2 N) and a factor of 1.5); the
oracle and the device each do two of them and the symbol's largest value
amplifies both, so they agree to 4 x 5e-16 x max|symbol| ||u||, taken
twice."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import precond as oprec  # noqa: E402
from oracle.operator import Plan as OPlan  # noqa: E402
from paper_1802_03770_gb300.api import Plan  # noqa: E402

EPS = 4e-15


def dev(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda:0")


def pair(d, n, alpha):
    """A plan with h = 1 and the oracle's operator with the plan's constants
    (the oracle's own agree with them to 1e-12 only)."""
    p, op = Plan(d, n, 1.0, alpha), OPlan(d, n, 1.0, alpha)
    k = p.describe()
    op.C, op.A1, op.A2, op.A3 = k["c_alpha_d"], k["lattice_zeta"], k["window_corr"], 0.0
    return op, p


def field(n, seed):
    rng = np.random.default_rng(seed)
    u = rng.standard_normal(n)
    # a few decades of dynamic range between the lines, one line of zeros
    u *= 10.0 ** rng.integers(-6, 3, size=n[:-1] + (1,))
    if n[0] > 2:
        u[n[0] // 2] = 0.0
    return u


# padded lengths 16 .. 8192 (one stage to four), tiles cut short, odd sizes
SIZES = [(1, (1,)), (1, (8,)), (1, (4096,)), (2, (1, 5)), (2, (9, 8)), (2, (33, 16)), (2, (64, 65)), (2, (130, 257)),
         (2, (513, 31)), (2, (3, 2049)), (2, (1025, 7)), (3, (9, 17, 5)), (3, (33, 8, 65)), (3, (2, 129, 16))]


@pytest.mark.parametrize("d,n", SIZES)
@pytest.mark.parametrize("alpha", [0.4, 1.7])
def test_apply_matches_oracle(d, n, alpha):
    op, p = pair(d, n, alpha)
    u = field(n, 3)
    y = p.apply(dev(u)).cpu().numpy().reshape(n)
    assert np.linalg.norm(y - op.apply(u)) <= EPS * np.abs(op.kernel_hat()).max() * np.linalg.norm(u)


@pytest.mark.parametrize("power", [-1000, 900, 1000])
@pytest.mark.parametrize("d,n", [(2, (40, 33)), (3, (9, 17, 12))])
def test_apply_at_the_ends_of_the_range(d, n, power):
    """u near the subnormal numbers and near the largest: the apply is
    homogeneous."""
    op, p = pair(d, n, 1.2)
    u = np.ldexp(np.random.default_rng(1).uniform(-1, 1, n), power)
    ref = op.apply(np.ldexp(u, -power))
    y = np.ldexp(p.apply(dev(u)).cpu().numpy().reshape(n), -power)
    tol = EPS * np.abs(op.kernel_hat()).max() * np.linalg.norm(np.ldexp(u, -power))
    assert np.linalg.norm(y - ref) <= tol


@pytest.mark.parametrize("d,n", [(2, (9, 8)), (2, (64, 65)), (2, (130, 257)), (2, (1023, 31)), (3, (9, 17, 5)),
                                 (3, (33, 70, 65))])
@pytest.mark.parametrize("shift,scale", [(0.0, 1.0), (1.0, 1e-3)])
def test_precond_matches_oracle(d, n, shift, scale):
    """The chirp-z sine transforms amplify an FFT's error by at most the
    condition of the chirp kernel's transform (below 10): 20 x EPS."""
    op, p = pair(d, n, 1.3)
    r = field(n, 5)
    z = p.precond(dev(r), shift=shift, scale=scale).cpu().numpy().reshape(n)
    ref = oprec.solve_box(op, r, shift, scale)
    lam = oprec.eigenvalues(op)
    assert np.linalg.norm(z - ref) <= 20 * EPS / (shift + scale * lam.min()) * np.linalg.norm(r)


@pytest.mark.parametrize("d,n", [(1, (50,)), (2, (40, 33)), (3, (9, 17, 12))])
def test_zero_and_non_finite_inputs(d, n):
    p = Plan(d, n, 1.0, 1.2)
    u = np.zeros(n)
    assert not p.apply(dev(u)).any() and not p.precond(dev(u)).any()
    for bad in (np.nan, np.inf, -np.inf):
        u = field(n, 7)
        u.flat[u.size // 3] = bad
        assert not torch.isfinite(p.apply(dev(u))).any()
        assert not torch.isfinite(p.precond(dev(u))).any()
