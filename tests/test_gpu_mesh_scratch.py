"""The memory that the mesh distance keeps between calls: bounded, given back when a
context is destroyed, and shared safely by threads and streams."""

import threading

import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

KEEP = 64 << 20


@pytest.fixture(scope="module")
def nsdf(nsdf_lib):
    import paper_2110_01614_gb300 as m
    return m


def scene(level, seed, n):
    V, F = synth.displaced_icosphere(level=level, seed=seed)
    return (torch.from_numpy(V).float().cuda(), torch.from_numpy(F).int().cuda(),
            torch.from_numpy(synth.uniform_cube_points(n, seed)).cuda(), torch.empty(n, device="cuda"))


def used():
    torch.cuda.synchronize()
    free, total = torch.cuda.mem_get_info()
    return total - free


def test_kept_memory_is_bounded_and_given_back(nsdf):
    small, large = scene(3, 7, 1000), scene(5, 7, 1 << 20)
    many = torch.zeros(3 << 20, 4, device="cuda"), torch.empty(3 << 20, device="cuda")
    nsdf.nsdf_mesh_sdf(*small)
    arch = synth.Arch(3, 64, 3, -1, 100.0)
    ctx = nsdf.NeuralSDF(arch, nsdf.NSDF_FP32)
    ctx.close()
    before = used()
    nsdf.nsdf_mesh_sdf(*large)
    nsdf.nsdf_mesh_sdf(large[0], large[1], *many)
    for _ in range(3):
        nsdf.nsdf_mesh_sdf(*small)
        assert used() - before <= KEEP
    ctx = nsdf.NeuralSDF(arch, nsdf.NSDF_FP32)
    ctx.close()
    assert used() <= before


def test_threads_and_streams(nsdf):
    scenes = [scene(3, 7 + k, 5000 + 999 * k) for k in range(6)]
    refs = []
    for s in scenes:
        nsdf.nsdf_mesh_sdf(*s)
        torch.cuda.synchronize()
        refs.append(s[3].clone())
    wrong = []

    def work(k):
        stream = torch.cuda.Stream()
        V, F, P, _ = scenes[k]
        for i in range(30):
            out = torch.full_like(refs[k], 7.0)
            torch.cuda.current_stream().synchronize()
            nsdf.nsdf_mesh_sdf(V, F, P, out, stream=stream)
            if i % 5 == 0:
                stream.synchronize()
                c = nsdf.NeuralSDF(synth.Arch(3, 64, 2, -1, 100.0), nsdf.NSDF_FP32)
                c.close()                       # empties the pool beside the other threads' calls
            stream.synchronize()
            if not torch.equal(out, refs[k]):
                wrong.append((k, i))

    threads = [threading.Thread(target=work, args=(k,)) for k in range(len(scenes))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong
