"""The mesh distance on both sides of its rules (faces of the smallest tree, points up
to which the leaf budget is the small one) gives the answers of brute force."""

import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


def spindle(faces):
    """A closed mesh: two caps over a ring of faces / 2 vertices."""
    k = faces // 2
    a = 2 * np.pi * np.arange(k) / k
    r = 0.5 + 0.05 * np.sin(3 * a)
    V = np.concatenate([np.stack([r * np.cos(a), r * np.sin(a), 0 * a], 1), [[0, 0, 0.5], [0, 0, -0.5]]])
    i, j = np.arange(k), (np.arange(k) + 1) % k
    F = np.concatenate([np.stack([i, j, 0 * i + k], 1), np.stack([j, i, 0 * i + k + 1], 1)])
    return V.astype(np.float32), F.astype(np.int32)


@pytest.mark.parametrize("faces,n", [(190, 500), (192, 500), (194, 1), (192, 48640), (192, 48641),
                                     (600, 48640), (600, 48641)])
def test_agrees_with_brute_force(nsdf_lib, faces, n):
    import paper_2110_01614_gb300 as nsdf
    V, F = (torch.from_numpy(x).cuda() for x in spindle(faces))
    P = torch.from_numpy(synth.uniform_cube_points(n, 3)).float().cuda()
    P[: n // 2, :3] = V[F[torch.arange(n // 2, device="cuda") % faces].long()].mean(1) * 1.002
    tree, brute = torch.full((2, n), 7.0, device="cuda")
    nsdf.nsdf_mesh_sdf(V, F, P, tree)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):                       # captured calls take brute force
        nsdf.nsdf_mesh_sdf(V, F, P, brute)
    g.replay()
    torch.cuda.synchronize()
    tree, brute = tree.cpu().numpy(), brute.cpu().numpy()
    np.testing.assert_allclose(np.abs(tree), np.abs(brute), rtol=4 * 2.0 ** -23, atol=1e-7)
    far = np.abs(brute) > 1e-6
    np.testing.assert_array_equal(np.signbit(tree[far]), np.signbit(brute[far]))
