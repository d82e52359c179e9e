"""Device memory of a plan's sine-transform tables: only what its passes read.

One row of n points padded to 8192: n + 1 = 4095 composite (chirp convolution,
all its tables), 4096 = 2^12 (odd extension, none) and 4093 prime (Rader's
convolution in FP32: no FP32 chirp, half the kernel spectrum, no tables of a
strided pass).  The fields differ by a point or two."""

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1802_03770_gb300.api import Plan  # noqa: E402


def workspace(n):
    p = Plan(1, (n,), 1.0 / (n + 1), 1.3)
    b = p.describe()["workspace_bytes"]
    p.close()
    return b


def test_tables_by_form_of_the_sine_transform():
    n, L = 4094, 8192
    fields = 4 * 1024
    chirp32, chirp64, spectrum32, spectrum64 = 8 * n, 16 * n, 2 * 8 * L, 16 * L
    full = workspace(n)
    assert workspace(4095) <= full - (chirp32 + chirp64 + spectrum32 + spectrum64) + fields
    assert workspace(4092) <= full - (chirp32 + spectrum32 // 2) + 2 * n + fields
