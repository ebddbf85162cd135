"""The bounds that the attention takes the logits by: exactly those of the slots that are live in a block, after every way into the cache and
out of it."""
import math

import numpy as np
import pytest

from paper_2602_01801_b200 import synth

pytestmark = pytest.mark.gpu


def _check(cache):
    s, b = cache.export_state(), cache.export_bounds()
    k = (s["k"].astype(np.uint32) << 16).view(np.float32).astype(np.float64)
    with np.errstate(invalid="ignore", over="ignore"):
        norms = np.sqrt((k ** 2).sum(2))
        norms = np.where(np.isfinite(norms) & (norms ** 2 < 3.4e38), norms, np.inf)
    m = np.log2(np.maximum(s["count"], 1))
    live = np.arange(cache.CAP) < s["len"][:, None]
    for name, x in (("norm", norms), ("log2m", m), ("joint", norms * math.log2(math.e) + m)):
        want = np.where(live, x, 0.0).reshape(cache.H, -1, cache.PT).max(2)
        # fp32 sums of the squares, two reciprocals and a root
        assert np.allclose(b[name], want, rtol=1e-5, atol=0.0), name
    return {name: x.max(1) for name, x in b.items()}


@pytest.mark.parametrize("d,pt", [(64, 64), (128, 128)])
@pytest.mark.parametrize("representative,bits,fp32,weighted", [("last", 16, False, False), ("mean", 8, False, True), ("last", 1, True, False)])
def test_bounds_are_those_of_the_live_slots(d, pt, representative, bits, fp32, weighted):
    import torch
    from paper_2602_01801_b200 import fastar
    rng = np.random.default_rng(d + bits)
    H, n, cap = 3, 128, 384
    cache = fastar.Cache(H, d, cap, pt, rng.standard_normal((32, d)).astype(np.float32), max_tokens=n, search_bits=bits, fp32=fp32, n_sink=8,
                         representative=representative, weighted_histograms=weighted)
    up = (lambda x: torch.from_numpy(x).cuda()) if fp32 else fastar.to_device
    new = lambda scale=1.0: synth.round_bf16((scale * rng.standard_normal((H, n, d))).astype(np.float32))
    assert not _check(cache)["norm"].any()                                # nothing live
    first = new()
    first[0, 70] *= 512.0                                                     # far longer than the rest
    first[1, 71] *= 2.0 ** 100                                                # |k|^2 beyond the range
    first[2, 72, 3] = np.nan
    cache.update(up(first), up(new()), n, 2.0)
    b = _check(cache)
    assert b["norm"][0] > 1000 and np.isinf(b["norm"][1:]).all()
    merged = first.copy()
    merged[:, 70:73] = 0.0                                                    # zeros match nothing
    for _ in range(3):                                                        # multiplicities up to four
        cache.update(up(merged), up(new()), n, 0.9)
    assert (_check(cache)["log2m"] >= 1.9).all()
    for _ in range(4):                                                        # appended, and the oldest slots replaced
        cache.update(up(new(0.5)), up(new()), n, 2.0)
        b = _check(cache)
    assert (b["norm"] < 50).all()
    # what does not fit is refused: the cache and its bounds as before
    small = fastar.Cache(1, d, 128, pt, rng.standard_normal((32, d)).astype(np.float32), max_tokens=n, n_sink=100)
    k = fastar.to_device(new()[:1])
    small.update(k, k, n, 2.0)
    before = _check(small)
    small.update((k * 64)[:, :64], k[:, :64], n, 2.0)
    assert small.status() == fastar.ERR_CAPACITY
    after = _check(small)
    assert all(np.array_equal(before[x], after[x]) for x in before)
    # an import: rows past a head's length don't count
    k, lens = new(), np.array([5, 0, n])
    k[:, 5:] *= 3.0
    k[0, 9] = np.inf
    k[0, 5] *= 100.0
    cache.import_state(fastar.bf16_bits(k), fastar.bf16_bits(new()), lens, rng.integers(1, 999, (H, n)).astype(np.int32))
    b = _check(cache)
    assert b["norm"][0] < 50 and b["norm"][1] == 0
