"""Springs at rest: a flat cloth whose edges are exactly as long as their rest lengths
feels no force, not even a rounding (x_new = 2 x - x_prev + dt^2 F with x_prev = 2 x,
no gravity and dt = 1 leaves F itself)."""

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(64, 64), (33, 7), (2, 2), (1, 40)])
@pytest.mark.parametrize("h", [0.75, 1.0, 0.4375])
def test_a_cloth_at_rest_stays(nsdf_lib, nx, ny, h):
    import paper_2110_01614_gb300 as nsdf
    i, j = np.meshgrid(np.arange(ny), np.arange(nx), indexing="ij")
    X = np.zeros((nx * ny, 4), np.float32)
    X[:, 0], X[:, 2] = h * j.ravel(), h * i.ravel()
    x = torch.from_numpy(X).cuda()
    out = (2.0 * x).contiguous()
    nsdf.nsdf_cloth_step(x, out, nx, ny, h, h, 1e5, 0.0, 1.0)
    torch.cuda.synchronize()
    assert float(out[:, :3].abs().max()) == 0.0
