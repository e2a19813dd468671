"""Shielding averages over rows of every length that changes how many lanes share a cell, for few and many
cells, against the definitions in FP64."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 33, 4097, 40001])
@pytest.mark.parametrize("npix", [1, 2, 8, 9, 12, 24, 25, 48, 108, 192])
def test_rows(oracle, n, npix):
    import torch
    from paper_1708_06142_gb300.treesolver import TreeSolver
    rng = np.random.default_rng(n + npix)
    cols = np.stack([10.0 ** rng.uniform(-2, 1.5, (n, npix)), 10.0 ** rng.uniform(12, 21, (n, npix)),
                     10.0 ** rng.uniform(10, 19, (n, npix))], 1).astype(np.float32)
    tab = rng.uniform(0.01, 1.0, (7, 5))
    kw = dict(k_av=0.9, k_h2=1.0, b5=2.0, k_co=1.0, co_table=tab, lg_co=(11.0, 18.0), lg_h2=(13.0, 20.0))
    out = torch.full((n + 1, 3), -7.0, device="cuda")
    ts = TreeSolver(0)
    ts.column_shielding(torch.from_numpy(cols).cuda(), out[:n], **kw)
    ts.sync()
    got = out.cpu().numpy().astype(np.float64)
    ref = oracle.column_shielding(cols.astype(np.float64), **kw)
    # FP32 exponentials and logarithms of arguments up to ~100: a few 2^-24 of each, as in the other tests
    np.testing.assert_allclose(got[:n, 0], ref[:, 0], rtol=2e-5, atol=2e-6)
    np.testing.assert_allclose(got[:n, 1], ref[:, 1], rtol=1e-5, atol=1e-7)
    np.testing.assert_allclose(got[:n, 2], ref[:, 2], rtol=1e-4, atol=1e-6)
    assert np.all(got[n] == -7.0)
