"""The mesh distance at sizes where products of FP32 coordinates overflow or
underflow: the answers of the brute-force kernel, and signs that do not depend on
the unit of length (a scale by a power of two is exact)."""

import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nsdf(nsdf_lib):
    import paper_2110_01614_gb300 as m
    return m


def distances(nsdf, V, F, P):
    V = torch.from_numpy(np.ascontiguousarray(V, np.float32)).cuda()
    F = torch.from_numpy(np.ascontiguousarray(F, np.int32)).cuda()
    P = torch.from_numpy(np.ascontiguousarray(P, np.float32)).cuda()
    tree, brute = torch.full((2, P.shape[0]), 7.0, device="cuda")
    nsdf.nsdf_mesh_sdf(V, F, P, tree)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):              # a captured call takes the brute-force kernel
        nsdf.nsdf_mesh_sdf(V, F, P, brute)
    g.replay()
    torch.cuda.synchronize()
    return tree.cpu().numpy(), brute.cpu().numpy()


def points(n, few):
    """Around the middle of the body, where every triangle is about as near, and anywhere."""
    P = synth.uniform_cube_points(n, 3).astype(np.float32)
    P[: n // 2, :3] *= np.float32(0.05)
    return P[:16] if few else P


@pytest.mark.parametrize("few", [True, False])
@pytest.mark.parametrize("scale", [2.0 ** 33, 2.0 ** 50, 2.0 ** 62])
def test_overflowing_products_leave_the_upper_bound(nsdf, scale, few):
    V, F = synth.displaced_icosphere(level=3, seed=7)
    P = points(20000, few)
    P[:, :3] *= np.float32(scale)
    tree, brute = distances(nsdf, V.astype(np.float32) * np.float32(scale), F, P)
    np.testing.assert_allclose(np.abs(tree), np.abs(brute), rtol=4 * 2.0 ** -23)


@pytest.mark.parametrize("n", [8, 20000])
@pytest.mark.parametrize("radius", [2.0 ** 33, 1.9e19])
def test_no_computable_distance_is_not_infinite(nsdf, radius, n):
    """Close to the middle of a sphere whose triangle tests all overflow, the result
    is the root of what the distance starts from, as by brute force."""
    V, F = synth.displaced_icosphere(level=3, seed=7)
    V = V / np.linalg.norm(V, axis=1, keepdims=True) * radius
    P = synth.uniform_cube_points(n, 3).astype(np.float32)
    P[:, :3] *= np.float32(1e-4 * radius)
    tree, brute = distances(nsdf, V, F, P)
    assert np.isfinite(brute).all()
    np.testing.assert_allclose(np.abs(tree), np.abs(brute), rtol=4 * 2.0 ** -23)


@pytest.mark.parametrize("power", [-30, -40, -44, -48, -56, -64])
def test_signs_do_not_depend_on_the_unit(nsdf, power):
    V, F = synth.displaced_icosphere(level=3, seed=7)
    V = V.astype(np.float32)
    P = points(20000, False)
    near = V[F[:, 0]] * np.float32(0.999)
    P[-len(near):, :3] = near
    ref = distances(nsdf, V, F, P)[0]
    s = np.float32(2.0 ** power)
    P[:, :3] *= s
    got = distances(nsdf, V * s, F, P)[0]
    assert 0.02 < np.signbit(ref).mean() < 0.98
    np.testing.assert_array_equal(np.signbit(got), np.signbit(ref))
