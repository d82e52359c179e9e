"""Errors of the FP32 passes against the FP64 ones, not above those of the forms
that their transforms replaced: sines by Rader's convolution (n + 1 prime) against
the chirp convolution, in-place transforms and the 256 x 8 row shape against
autosort stages of 16 values per thread.

The bounds are the replaced forms' own root mean square errors, measured on these
grids over 48 to 200 standard-normal fields (preconditioner: shift 1 and scale
1e-3); over the 24 of these tests the mean moves by under 1 %."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1802_03770_gb300.api import Plan  # noqa: E402

CHIRP_ERROR = {(40, 40): 2.29e-7, (130, 130): 2.36e-7, (136, 136): 2.49e-7, (192, 192): 2.88e-7, (256, 256): 3.00e-7,
               (40, 126, 130): 3.50e-7, (130, 130, 130): 3.11e-7, (256, 256, 256): 3.82e-7}


def precond_error(n):
    p = Plan(len(n), n, 1.0 / (max(n) + 1), 1.3)
    rng = np.random.default_rng(11)
    sq = []
    for _ in range(24 if p.N < 5e6 else 4):
        r = torch.tensor(rng.standard_normal(p.N, dtype=np.float32), device="cuda:0")
        z = p.precond(r, shift=1.0, scale=1e-3).double()
        ref = p.precond(r.double(), shift=1.0, scale=1e-3)
        sq.append(float(((z - ref).norm() / ref.norm()) ** 2))
    p.close()
    return np.sqrt(np.mean(sq))


@pytest.mark.parametrize("n", sorted(CHIRP_ERROR, key=lambda n: (len(n), n)))
def test_prime_length_error_not_above_the_chirps(n):
    assert precond_error(n) <= CHIRP_ERROR[n]


# the preconditioner in the 256 x 8 row shape, chirp convolutions
ROWS_ERROR = {(160, 160): 2.50e-7, (180, 200): 2.81e-7, (200, 200): 2.81e-7}
# the apply: 256 x 8 rows, strided passes in place
APPLY_ERROR = {(130, 130): 1.46e-7, (160, 160): 1.54e-7, (200, 200): 1.65e-7, (255, 255): 1.82e-7,
               (160, 160, 160): 1.81e-7, (200, 200, 200): 1.93e-7, (256, 256, 256): 2.11e-7}


@pytest.mark.parametrize("n", sorted(ROWS_ERROR))
def test_row_shape_error_not_above_the_wide_rows(n):
    assert precond_error(n) <= ROWS_ERROR[n]


@pytest.mark.parametrize("n", sorted(APPLY_ERROR, key=lambda n: (len(n), n)))
def test_apply_error_not_above_the_autosort_passes(n):
    p = Plan(len(n), n, 1.0 / (max(n) + 1), 1.3)
    rng = np.random.default_rng(14)
    sq = []
    for _ in range(24 if p.N < 1e6 else 4):
        u = torch.tensor(rng.standard_normal(p.N, dtype=np.float32), device="cuda:0")
        y, ref = p.apply(u).double(), p.apply(u.double())
        sq.append(float(((y - ref).norm() / ref.norm()) ** 2))
    p.close()
    assert np.sqrt(np.mean(sq)) <= APPLY_ERROR[n]
