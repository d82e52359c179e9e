"""Edges of the launch rules of the preconditioner and row passes, against the
oracle: rows per segment of the tridiagonal pass (8, 16 and 32), the FP32 row
shape by grid size, and the interface solve of an occluded domain by the size
of the hole's boundary.

Tolerances as in the parity tests: 2e-5 relative for FP32; for the FP64
preconditioner 1e-11 (its operators' condition, below 1e4 here, times FP64
rounding and a factor of ten)."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import precond as oprec  # noqa: E402
from oracle.operator import Plan as OPlan  # noqa: E402
from paper_1802_03770_gb300.api import Plan  # noqa: E402


def dev(a, dtype):
    return torch.tensor(np.ascontiguousarray(a).ravel(), dtype=dtype, device="cuda:0")


def rel(a, b):
    return np.linalg.norm(a.ravel() - b.ravel()) / np.linalg.norm(b)


@pytest.mark.parametrize("n", [(1, 40), (31, 9), (32, 9), (33, 9), (256, 7), (257, 7), (512, 5), (513, 5), (1023, 6),
                               (1024, 3), (9, 17, 6), (257, 5, 6)])
@pytest.mark.parametrize("shift,scale", [(0.0, 1.0), (1.0, 1e-3), (1.0, 1e-30)])
def test_tridiagonal_segments(n, shift, scale):
    d = len(n)
    h = 1.0 / (max(n) + 1)
    op, p = OPlan(d, n, h, 1.3), Plan(d, n, h, 1.3)
    r = np.random.default_rng(2).standard_normal(n).astype(np.float32).astype(np.float64)
    ref = oprec.solve_box(op, r, shift, scale)
    for dtype, tol in ((torch.float64, 1e-11), (torch.float32, 2e-5)):
        z = p.precond(dev(r, dtype), shift=shift, scale=scale).cpu().numpy()
        assert rel(z, ref) <= tol, (dtype, rel(z, ref))


# rows of 512 .. 2048 points at 303 .. 305 CTAs, of 256 points at 152 and 153
@pytest.mark.parametrize("n", [(606, 600), (608, 600), (612, 600), (304, 1000), (1215, 300), (1218, 300),
                               (2432, 100), (2436, 100), (150, 200), (3, 130)])
def test_row_shape_by_grid(n):
    h = 1.0 / (max(n) + 1)
    op, p = OPlan(2, n, h, 1.2), Plan(2, n, h, 1.2)
    u = np.random.default_rng(4).standard_normal(n).astype(np.float32).astype(np.float64)
    assert rel(p.apply(dev(u, torch.float32)).cpu().numpy(), op.apply(u)) <= 2e-5
    if n[0] <= 1024:
        z = p.precond(dev(u, torch.float32)).cpu().numpy()
        assert rel(z, oprec.solve_box(op, u)) <= 2e-5


# holes of k points in a row, away from the edge: all k are of the hole's boundary
@pytest.mark.parametrize("k", [1, 2, 15, 16, 17, 31, 32, 33, 64, 65, 97])
@pytest.mark.parametrize("shift,scale", [(0.0, 1.0), (1.0, 1e-3)])
def test_interface_solve_sizes(k, shift, scale):
    n, h = (24, 120), 1.0 / 121
    mask = np.ones(n, dtype=bool)
    mask[11, 7:7 + k] = False
    op, p = OPlan(2, n, h, 1.6, mask=mask), Plan(2, n, h, 1.6, mask=mask)
    r = np.random.default_rng(6).standard_normal(n).astype(np.float32).astype(np.float64)
    ref = oprec.solve_domain(op, r, shift, scale)
    for dtype, tol in ((torch.float64, 1e-11), (torch.float32, 2e-5)):
        z = p.precond(dev(r, dtype), shift=shift, scale=scale).cpu().numpy()
        assert rel(z, np.where(mask, ref, 0.0)) <= tol


# last axis 2^k - 1 (sines by the odd extension, two rows per line), odd and even numbers of rows, and its neighbours
@pytest.mark.parametrize("n", [(1, 7), (5, 7), (4, 15), (7, 31), (33, 63), (9, 127), (64, 255), (3, 511), (6, 1023),
                               (5, 2047), (2, 4095), (5, 126), (5, 128), (5, 9, 31), (4, 31, 31)])
def test_odd_extension_rows(n):
    d = len(n)
    h = 1.0 / (max(n) + 1)
    op, p = OPlan(d, n, h, 1.3), Plan(d, n, h, 1.3)
    r = np.random.default_rng(8).standard_normal(n).astype(np.float32).astype(np.float64)
    for shift, scale in ((0.0, 1.0), (1.0, 1e-3)):
        ref = oprec.solve_box(op, r, shift, scale)
        for dtype, tol in ((torch.float64, 1e-11), (torch.float32, 2e-5)):
            z = p.precond(dev(r, dtype), shift=shift, scale=scale).cpu().numpy()
            assert rel(z, ref) <= tol, (dtype, rel(z, ref))


# iterations between reads of the device state: caps inside, at and past the captured graph's four
@pytest.mark.parametrize("cap", [1, 3, 4, 5, 7, 8, 13, 40])
def test_iteration_cap(cap):
    n = (31, 40)
    p = Plan(2, n, 1.0 / 41, 1.3)
    b = dev(np.random.default_rng(9).standard_normal(n), torch.float64)
    _, info = p.solve(b, tol=1e-300, maxit=cap, mode=0, raise_on_fail=False)
    assert info["iterations"] == cap


# axes with n + 1 prime (FP32: Rader's convolution): the shortest lines, one stage and several, full and partial CTAs and
# tiles, the last and the middle axis, generators of all residues and of half of them; FP64 stays with its own form
@pytest.mark.parametrize("n", [(1, 10), (5, 12), (300, 16), (33, 40), (17, 96), (3, 130), (65, 192), (40, 256), (5, 640),
                               (4, 768), (2, 1012), (3, 2028), (2, 4092), (4, 16, 9), (3, 96, 33), (2, 256, 256),
                               (3, 192, 35), (2, 12, 1000)])
@pytest.mark.parametrize("masked", [False, True])
def test_prime_sines(n, masked):
    d = len(n)
    h = 1.0 / (max(n) + 1)
    rng = np.random.default_rng(10)
    mask = None
    if masked:
        mask = np.ones(n, dtype=bool)
        mask[(0,) * (d - 1) + (slice(2, 5),)] = False
    op, p = OPlan(d, n, h, 1.3, mask=mask), Plan(d, n, h, 1.3, mask=mask)
    r = rng.standard_normal(n).astype(np.float32).astype(np.float64)
    for shift, scale in ((0.0, 1.0), (1.0, 1e-3)):
        ref = oprec.solve_domain(op, r, shift, scale) if masked else oprec.solve_box(op, r, shift, scale)
        if masked:
            ref = np.where(mask, ref, 0.0)
        for dtype, tol in ((torch.float64, 1e-11), (torch.float32, 2e-5)):
            z = p.precond(dev(r, dtype), shift=shift, scale=scale).cpu().numpy()
            assert rel(z, ref) <= tol, (dtype, rel(z, ref))


# tridiagonal segments about 24 rows
@pytest.mark.parametrize("n", [(544, 6), (545, 6), (700, 9), (768, 5), (769, 5)])
def test_tridiagonal_segments_24(n):
    test_tridiagonal_segments(n, 1.0, 1e-3)
