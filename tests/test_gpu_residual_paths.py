"""The allocation-free residual where its thread blocking has edges: odd rows
(one cell a thread), an odd number of rows (a last pair of one row), level
counts that are no multiple of the levels a thread walks, one vector across,
arrays that start between two vectors, and no residual array."""
import math

import numpy as np
import pytest

from .test_zz_no_alloc import _reference_residual

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(4, 3, 2), (3, 4, 3), (5, 5, 5), (64, 16, 8), (66, 17, 9), (65, 33, 7), (34, 18, 4)])
@pytest.mark.parametrize("offset,write", [(0, True), (1, True), (0, False)])
def test_residual_edges(stp_lib, shape, offset, write):
    """Against b - stp_eval(laplacian): both form the same second differences
    in FP64, so they agree to a few units of rounding, 1e-12."""
    torch = pytest.importorskip("torch")
    nx, ny, nz = shape
    cfg = dict(nx=nx, ny=ny, nz=nz, Lx=2 * math.pi, Ly=math.pi, Lz=2.0, nu=0.01, dt=1e-3, stretch=1.5)
    rng = np.random.default_rng(31)
    p, b = rng.standard_normal((nz, ny, nx)), rng.standard_normal((nz, ny, nx))
    r_ref = _reference_residual(stp_lib, cfg, p, b)
    n_ref = float(np.sqrt(np.sum(r_ref * r_ref)))

    def put(a):
        t = torch.empty(a.size + offset, dtype=torch.float64, device="cuda")[offset:].view(a.shape)
        return t.copy_(torch.from_numpy(a))

    tp, tb = put(p), put(b)
    tr = put(np.full(p.shape, np.nan)) if write else None
    n = stp_lib.poisson_residual_noalloc(cfg, tp, tb, tr)
    assert abs(n - n_ref) <= 1e-12 * n_ref
    if write:
        assert np.abs(tr.cpu().numpy() - r_ref).max() <= 1e-12 * np.abs(r_ref).max()
