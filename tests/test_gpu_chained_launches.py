"""The kernels of a step start while the one in front of them drains: a captured step, with AnnCA and the query side of the selector
on a second stream, has to give the bits of the same calls made one after the other with the device idle in between."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("heads,dim,n,fp32", [(1, 64, 65, True), (3, 128, 520, False)])
def test_captured_step_equals_serial_step(heads, dim, n, fp32):
    import torch

    from paper_2602_01801_b200 import fastar

    g = torch.Generator(device="cuda").manual_seed(5)
    dt = torch.float32 if fp32 else torch.bfloat16

    def normal(rows):
        return torch.randn(heads, rows, dim, generator=g, device="cuda").to(dt)

    lsh = np.random.default_rng(5).standard_normal((32, dim)).astype(np.float32)
    k0, v0, kp, vp, q = normal(2 * n), normal(2 * n), normal(48), normal(48), normal(n)
    near = k0[:, :n] + 0.1 * normal(n)                     # half of the chunk is found in the cache, the rest appended
    v1 = normal(n)
    k1 = torch.where(torch.arange(n, device="cuda")[:, None] % 2 == 0, near, normal(n))

    def fresh():
        c = fastar.Cache(heads, dim, 4096, 64, lsh, max_tokens=2 * n, max_prompt_tokens=48, max_frames=2, fp32=fp32)
        c.update(k0, v0, n, 2.0, outputs=False)
        return c

    serial = fresh()
    want = []
    for call in (lambda: serial.update(k1, v1, n, 0.9), lambda: serial.annsa(q, 64, 3), lambda: serial.annca(q, kp, vp, n, 8)):
        torch.cuda.synchronize()
        r = call()
        torch.cuda.synchronize()
        want += [r[k] for k in ("match", "sim", "dest", "stats", "out") if k in r]

    cache, side = fresh(), torch.cuda.Stream()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        main = torch.cuda.current_stream()
        side.wait_stream(main)
        with torch.cuda.stream(side):
            cache.annsa_prepare(q, 64)
            ca = cache.annca(q, kp, vp, n, 8)
        up = cache.update(k1, v1, n, 0.9)
        main.wait_stream(side)
        sa = cache.annsa(q, 64, 3)
    graph.replay()
    torch.cuda.synchronize()
    got = [up[k] for k in ("match", "sim", "dest", "stats")] + [sa["out"], ca["out"]]
    assert cache.status() == fastar.OK
    assert int(got[3].reshape(-1)[0]) > 0                  # something matched
    for a, b in zip(got, want):
        assert torch.equal(a, b)
