"""Tensors whose rows do not start on 16-byte boundaries are refused on the host, before anything is launched, whichever tensor of a
call it is; views at a boundary, with other strides than a dense tensor's, are accepted."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fp32,search_bits", [(False, 16), (False, 8), (True, 16)])
def test_rows_off_a_boundary_are_refused(fp32, search_bits):
    import torch

    from paper_2602_01801_b200 import fastar

    H, d, n = 2, 64, 70
    dt = torch.float32 if fp32 else torch.bfloat16
    g = torch.Generator(device="cuda").manual_seed(1)

    def rows(offset=0, pad=0):
        """[H][n][d] whose storage starts `offset` elements into an allocation, rows `pad` elements apart."""
        return torch.randn(offset + H * n * (d + pad), generator=g, device="cuda").to(dt)[offset:].view(H, n, d + pad)[..., :d]

    cache = fastar.Cache(H, d, 256, 64, np.random.default_rng(1).standard_normal((32, d)).astype(np.float32), max_tokens=n,
                         max_prompt_tokens=n, max_frames=1, fp32=fp32, search_bits=search_bits)
    calls = dict(
        update=lambda k, v: cache.update(k, v, n, 0.9),
        probe=lambda q, k, v: cache.update(k, v, n, 0.9, probe=q),
        prepare=lambda q: cache.annsa_prepare(q, 64),
        annsa=lambda q: cache.annsa(q, 64, 1, out=torch.empty_like(q.contiguous())),
        segment=lambda k, v: cache.annsa_segment(rows(), k, v, 64, 1),
        annca=lambda k, v: cache.annca(rows(), k, v, n, 5),
        lsh=lambda k, v: cache.annca_lsh(rows(), k, v, n))
    good = 16 // rows().element_size()
    for name, call in calls.items():
        args = call.__code__.co_argcount
        launches = cache.launch_count()
        for bad in range(args):
            for offset in (1, good // 2, good + 1):
                with pytest.raises(fastar.FastarError) as e:
                    call(*[rows(offset if i == bad else 0) for i in range(args)])
                assert e.value.status == fastar.ERR_INVALID_ARG, name
        if not (name == "annsa" or name == "prepare"):
            with pytest.raises(fastar.FastarError):
                call(*[rows(0, 1)] * args)
        if name in ("update", "probe", "prepare", "annsa"):
            assert cache.launch_count() == launches, name
        call(*[rows(good if name != "annsa" else 0)] * args)
        if name != "annsa":
            call(*[rows(0, good)] * args)
    assert cache.status() == fastar.OK


@pytest.mark.parametrize("fp32", [False, True])
def test_a_refused_call_leaves_the_prepared_queries(fp32):
    import torch

    from paper_2602_01801_b200 import fastar

    H, d, n = 2, 64, 70
    q = torch.randn(H, n, d, device="cuda", dtype=torch.float32 if fp32 else torch.bfloat16)
    cache = fastar.Cache(H, d, 512, 64, np.random.default_rng(1).standard_normal((32, d)).astype(np.float32), max_tokens=n, fp32=fp32)
    cache.update(q, q, n, 2.0)

    def launches(call):
        before = cache.launch_count()
        out = call()["out"]
        return cache.launch_count() - before, out

    off = torch.empty(H * n * d + 1, device="cuda", dtype=q.dtype)[1:].view(H, n, d)
    plain, want = launches(lambda: cache.annsa(q, 64, 3))
    for refused in (lambda: cache.annsa(q, 96, 3), lambda: cache.annsa(q, 64, 0), lambda: cache.annsa(q, 64, 3, out=off),
                    lambda: cache.annsa_segment(q, q[:, :0], q[:, :0], 64, 3)):
        cache.annsa_prepare(q, 64)
        with pytest.raises(fastar.FastarError):
            refused()
        prepared, out = launches(lambda: cache.annsa(q, 64, 3))
        assert prepared == plain - 1
        assert torch.equal(out, want)
    assert cache.status() == fastar.OK
