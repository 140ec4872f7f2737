"""FP32 query kernel: both tile shapes, ragged tiles, every width, networks of
one and two layers.  A point's result does not depend on the tile it falls in
(both shapes sum the columns in the same order), so small calls (the small
tiles) repeat a large call (the large tiles) bit for bit; a sample of the points
is compared with the FP64 oracle at the FP32 form's bounds (1e-5, 1e-4 rad)."""

import numpy as np
import pytest
import torch

import synth
from oracle import mlp

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nsdf(nsdf_lib):
    import paper_2110_01614_gb300 as m
    return m


@pytest.mark.parametrize("arch,n", [
    (synth.Arch(3, 32, 4, 2, 100.0), 300_001), (synth.Arch(3, 64, 1, -1, 100.0), 100_001),
    (synth.Arch(3, 64, 3, 1, 100.0), 200_003), (synth.Arch(3, 128, 2, -1, 100.0), 100_007),
    (synth.Arch(3, 256, 3, 2, 100.0), 50_021), (synth.Arch(3, 512, 2, 1, 100.0), 20_011)])
def test_shapes_agree_and_match_oracle(nsdf, arch, n):
    blob = synth.geometric_init(arch, 3)
    net = nsdf.NeuralSDF(arch, nsdf.NSDF_FP32).load(blob)
    P = torch.from_numpy(synth.uniform_cube_points(n, 5)).cuda()
    ref = net.query(P)
    for m in (1, 31, 33, 64, 65, 129, 1000):
        lo = n - m                                   # the last, ragged tile of the large call
        assert torch.equal(net.query(P[lo:].clone()), ref[lo:])
        assert torch.equal(net.query(P[:m].clone()), ref[:m])
    net.close()
    idx = np.concatenate([np.arange(200), np.arange(n - 200, n)])
    f, N, _, _ = mlp.collide(blob, arch, P.cpu().numpy()[idx], 0.0)
    got = ref.cpu().numpy()[idx].astype(np.float64)
    assert np.abs(got[:, 3] - f).max() <= 1e-5
    ang = np.arctan2(np.linalg.norm(np.cross(got[:, :3], N), axis=1),
                     np.einsum("ij,ij->i", got[:, :3], N))
    assert ang.max() <= 1e-4
