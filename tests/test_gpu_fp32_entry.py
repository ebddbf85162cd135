"""fp32 updates whose tensors the hash rounds on its way: the cache bit for bit as from the rounded tensors, for few and many heads, single tokens and
remainders, contiguous and interleaved layouts, with and without a probe."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("H,n", [(1, 1), (1, 257), (7, 65), (40, 3), (40, 130), (5, 1333)])
@pytest.mark.parametrize("probe,interleaved", [(False, False), (True, True)])
def test_fp32_update_equals_the_rounded_one(d, H, n, probe, interleaved):
    import torch
    from paper_2602_01801_b200 import fastar
    g = torch.Generator(device="cuda").manual_seed(d + H + n)
    lsh = np.random.default_rng(1).standard_normal((32, d)).astype(np.float32)

    def new():
        shape = (n, H, d + 8) if interleaved else (H, n, d)
        x = torch.randn(*shape, generator=g, device="cuda")
        return x.transpose(0, 1)[..., :d] if interleaved else x
    caches = [fastar.Cache(H, d, 4096, 128, lsh, max_tokens=n, fp32=fp32) for fp32 in (True, False)]
    k0 = new()
    for step in range(2):
        k, v, q = (k0 if step == 0 else k0 + 0.01 * new()), new(), new()
        if interleaved and step:                           # the sum is contiguous: back into the layout of the others
            k = torch.empty(n, H, d + 8, device="cuda").transpose(0, 1)[..., :d].copy_(k)
        for cache in caches:
            as_is = lambda x: x if cache is caches[0] else x.bfloat16().contiguous()
            cache.update(as_is(k), as_is(v), n, 0.9, probe=as_is(q) if probe else None)
            assert cache.status() == 0
    a, b = (cache.export_state() for cache in caches)
    assert a["count"].max() == 2 and all(np.array_equal(a[x], b[x]) for x in a)
