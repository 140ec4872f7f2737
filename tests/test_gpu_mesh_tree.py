"""The bounding-box tree of nsdf_mesh_sdf against the brute-force kernel and the oracle.

A call that is captured into a CUDA graph takes the brute-force kernel (the
tree needs an allocation), so one function gives both answers.  The triangle
test is the same code in both and its minimum is taken over the same triangle,
hence equal distances up to a rounding of the final operations (4 ulp allowed
for another contraction of products and sums); signs are equal wherever the
point is further than 1e-6 from the surface.
"""

import numpy as np
import pytest
import torch

import synth
from oracle import mesh

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nsdf(nsdf_lib):
    import paper_2110_01614_gb300 as m
    return m


def both(nsdf, V, F, P):
    """(tree, brute force) distances; the tree is used where it applies."""
    V = torch.from_numpy(np.ascontiguousarray(V, np.float32)).cuda()
    F = torch.from_numpy(np.ascontiguousarray(F, np.int32)).cuda()
    P = torch.as_tensor(P).cuda()
    tree, brute = torch.full((2, P.shape[0]), 7.0, device="cuda")
    nsdf.nsdf_mesh_sdf(V, F, P, tree)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        nsdf.nsdf_mesh_sdf(V, F, P, brute)
    g.replay()
    torch.cuda.synchronize()
    return tree.cpu().numpy(), brute.cpu().numpy()


def agree(tree, brute):
    np.testing.assert_allclose(np.abs(tree), np.abs(brute), rtol=4 * 2.0 ** -23, atol=1e-7)
    far = ~(np.abs(brute) <= 1e-6)
    np.testing.assert_array_equal(np.signbit(tree[far]), np.signbit(brute[far]))


def points(V, F, n, seed):
    """Random points, points above and below vertices, edge midpoints and face
    centres (the ray passes exactly through them), and points near the surface."""
    V32 = np.asarray(V, np.float32)
    s = synth.Stream(seed)
    k = (s.u64(n) % np.uint64(len(F))).astype(np.int64)
    a, b, c = (V32[F[k, i]] for i in range(3))
    at = np.concatenate([a, (a + b) * np.float32(0.5), (a + b + c) * np.float32(1 / 3)])
    z = s.uniform(len(at), -1.0, 1.0).astype(np.float32)
    ray = at.copy()
    ray[:, 2] = z
    near = at + s.normal(at.size, std=1e-4).reshape(at.shape).astype(np.float32)
    P = np.zeros((n + 3 * len(at), 4), np.float32)
    P[:n, :3] = s.uniform(3 * n, -1.0, 1.0).reshape(n, 3)
    P[n:, :3] = np.concatenate([at, ray, near])
    return P


def scenes():
    V1, F1 = synth.displaced_icosphere(level=1, seed=3)       # 80 faces: below the tree's rule
    V2, F2 = synth.displaced_icosphere(level=2, seed=7)       # 320 faces, one box block
    V4, F4 = synth.displaced_icosphere(level=4, seed=7)       # 5,120 faces, several box blocks
    yield "few faces", V1, F1
    yield "small", V2, F2
    yield "several blocks", V4, F4
    yield "inverted", V2, F2[:, ::-1]
    yield "soup", V2[F2.reshape(-1)], np.arange(F2.size).reshape(-1, 3)
    yield "bad indices", V2, np.vstack([F2, [[0, 1, len(V2)], [-1, 2, 3]]])
    yield "nested", np.vstack([V2, 0.5 * V2]), np.vstack([F2, F2 + len(V2)])
    yield "hollow", np.vstack([V2, 0.5 * V2]), np.vstack([F2, F2[:, ::-1] + len(V2)])
    yield "apart", np.vstack([0.4 * V4, 0.4 * V4 + 0.5]), np.vstack([F4, F4 + len(V4)])
    # vertical walls and axis-aligned faces: a box cut into 12 * 4**3 faces
    V, F = synth.box_mesh()
    V, F = np.asarray(V, np.float64), np.asarray(F)
    for _ in range(3):
        a, b, c = (V[F[:, i]] for i in range(3))
        n = len(V)
        V = np.concatenate([V, (a + b) / 2, (b + c) / 2, (c + a) / 2])
        ab, bc, ca = (n + i * len(F) + np.arange(len(F)) for i in range(3))
        F = np.concatenate([np.stack(x, 1) for x in ((F[:, 0], ab, ca), (F[:, 1], bc, ab),
                                                     (F[:, 2], ca, bc), (ab, bc, ca))])
    yield "box", V, F
    yield "degenerate", V2, np.vstack([F2, [[4, 4, 9], [7, 7, 7]]])
    yield "open", V2, F2[:-3]                                 # left to the brute-force kernel
    yield "flat scale", V2 * np.array([1.0, 1e-3, 1.0]), F2


@pytest.mark.parametrize("name,V,F", list(scenes()), ids=[s[0] for s in scenes()])
def test_tree_agrees_with_brute_force(nsdf, name, V, F):
    inside = F[((F >= 0) & (F < len(V))).all(axis=1)]
    agree(*both(nsdf, V, F, points(V, inside, 700, 11)))


@pytest.mark.parametrize("level", [2, 3])
def test_tree_matches_oracle(nsdf, level):
    V, F = synth.displaced_icosphere(level=level, seed=5)
    V32 = V.astype(np.float32).astype(np.float64)
    P = points(V, F, 400, 12)
    ref = mesh.signed_distance(P[:, :3].astype(np.float64), V32, F)
    got = both(nsdf, V, F, P)[0]
    np.testing.assert_allclose(got, ref, atol=2e-6, rtol=1e-5)
    far = np.abs(ref) > 1e-6
    np.testing.assert_array_equal(np.sign(got[far]), np.sign(ref[far]))


def test_odd_values_agree(nsdf):
    """Points and vertices that are not finite or very large."""
    V, F = synth.displaced_icosphere(level=2, seed=7)
    P = synth.uniform_cube_points(16, 3)
    P[0, 0], P[1, 1], P[2, 2] = np.nan, np.inf, -np.inf
    P[3, :3], P[4, :3] = -1e6, np.nan
    agree(*both(nsdf, V, F, P))
    # a point so far out that FP32 solid angles overflow is outside all the same
    far = P[:1].copy()
    far[0, :3] = 1e20
    assert both(nsdf, V, F, far)[0][0] > 1e18
    V = V.copy()
    V[5, 1] = np.nan
    agree(*both(nsdf, V, F, P))


def test_voxel_build_equals_mesh_sdf_of_its_nodes(nsdf):
    V, F = synth.displaced_icosphere(level=3, seed=7)
    V = torch.from_numpy(V.astype(np.float32)).cuda()
    F = torch.from_numpy(F.astype(np.int32)).cuda()
    n = 17
    grid = torch.empty(n ** 3, device="cuda")
    nsdf.nsdf_voxel_build(V, F, n, (-1.0,) * 3, (1.0,) * 3, grid)
    c = (-1.0 + 0.125 * torch.arange(n)).cuda()
    z, y, x = torch.meshgrid(c, c, c, indexing="ij")
    P = torch.stack([x, y, z, torch.zeros_like(x)], -1).reshape(-1, 4).contiguous()
    out = torch.empty(n ** 3, device="cuda")
    nsdf.nsdf_mesh_sdf(V, F, P, out)
    torch.cuda.synchronize()
    assert torch.equal(grid, out)


def test_two_streams_share_no_scratch(nsdf):
    """Calls on two streams at once, each with its own mesh, give each call's own answer."""
    meshes, outs, refs = [], [], []
    P = torch.from_numpy(synth.uniform_cube_points(20000, 4)).cuda()
    for k in range(2):
        V, F = synth.displaced_icosphere(level=3, seed=7 + k)
        meshes.append((torch.from_numpy(V.astype(np.float32)).cuda(),
                       torch.from_numpy(F.astype(np.int32)).cuda()))
        outs.append(torch.empty(20000, device="cuda"))
        refs.append(torch.empty(20000, device="cuda"))
        nsdf.nsdf_mesh_sdf(*meshes[k], P, refs[k])
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in range(2)]
    for _ in range(20):
        for k in range(2):
            nsdf.nsdf_mesh_sdf(*meshes[k], P, outs[k], stream=streams[k])
    torch.cuda.synchronize()
    for k in range(2):
        assert torch.equal(outs[k], refs[k])
