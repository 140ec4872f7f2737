"""The cloth step at the edges of its tiles of 32 x 8 vertices."""

import numpy as np
import pytest
import torch

import synth
from oracle import cloth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nsdf(nsdf_lib):
    import paper_2110_01614_gb300 as m
    return m


@pytest.mark.parametrize("nx,ny", [(1, 1), (1, 9), (9, 1), (32, 8), (33, 9), (31, 7), (2, 65),
                                   (121, 3), (130, 33)])
def test_cloth_step_matches_oracle(nsdf, nx, ny):
    """One vertex, single rows and columns, one short of, at and past each edge
    (the bound of the square-grid test: 2e-6 at this spacing)."""
    hx, hz = 2.0 / 63, 1.5 / 63
    i, j = np.meshgrid(np.arange(ny), np.arange(nx), indexing="ij")
    idx = i * nx + j
    pairs = [(idx[:, :-1], idx[:, 1:], hx), (idx[:-1], idx[1:], hz),
             (idx[:-1, :-1], idx[1:, 1:], np.hypot(hx, hz)),
             (idx[:-1, 1:], idx[1:, :-1], np.hypot(hx, hz))]
    S = np.concatenate([np.stack([a.ravel(), b.ravel()], 1) for a, b, _ in pairs])
    rest = np.concatenate([np.full(a.size, r) for a, _, r in pairs])
    s = synth.Stream(5)
    X = np.zeros((nx * ny, 4), np.float32)
    X[:, 0], X[:, 1], X[:, 2] = hx * j.ravel(), 0.6, hz * i.ravel()
    X[:, :3] += s.normal(3 * nx * ny, std=1e-3).reshape(-1, 3).astype(np.float32)
    X[:, 3] = np.arange(nx * ny)
    Xp = X.copy()
    Xp[:, 1] += 1e-3
    ref = cloth.verlet_step(X, Xp, S, rest, 1e5, 1e-3)
    x, xp = torch.from_numpy(X).cuda(), torch.from_numpy(Xp).cuda()
    nsdf.nsdf_cloth_step(x, xp, nx, ny, hx, hz, 1e5, 9.81, 1e-3)
    torch.cuda.synchronize()
    got = xp.cpu().numpy()
    np.testing.assert_allclose(got[:, :3], ref, atol=2e-6)
    np.testing.assert_array_equal(got[:, 3], X[:, 3])
    assert torch.equal(x.cpu(), torch.from_numpy(X))
