"""Allocation-free volume average at the edges of its launch rule: one block (up to 4096 values), the
first sizes beyond, partial rounds, and more rows than one round of the full grid.

Reference: the same sum in extended precision on the host.  Tolerance: n eps sum |w f|, the bound of
any summation order (n terms, eps = 2^-53), far above what blocked sums reach.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("ncomp", [1, 2, 3, 5, 7, 8, 9])
@pytest.mark.parametrize("n", [1, 2, 31, 255, 454, 456, 1365, 1366, 4096, 4097, 65_537, 400_001])
def test_every_row_and_component_counts_once(gspm_lib, n, ncomp):
    rng = np.random.default_rng(100 * ncomp + n % 97)
    f = rng.standard_normal((n, ncomp))
    w = rng.random(n)
    out = torch.full((ncomp,), float("nan"), dtype=torch.float64, device="cuda")
    gspm_lib.volume_avg_noalloc(torch.tensor(f, device="cuda"), torch.tensor(w, device="cuda"), out)
    prod = w[:, None].astype(np.longdouble) * f
    bound = n * 2.0 ** -53 * np.abs(prod).sum(0)
    assert np.all(np.abs(out.cpu().numpy() - prod.sum(0)) <= bound)
