"""The correspondence search at the edges of its tiles: 256-row units of two 128-row tiles (the last may hold one, or one row),
128-key tiles, work cut into equal pieces across units and heads, ragged and empty caches."""
import numpy as np
import pytest

from paper_2602_01801_b200 import synth

pytestmark = pytest.mark.gpu


def _case(d, pt, n, lengths, seed):
    """Keys around shared centroids, so that maxima are contested; a third of the cached keys are exact copies of earlier ones."""
    rng = np.random.default_rng(seed)
    H, cap = len(lengths), -(-max(max(lengths), n, 128) // 128) * 128 + 256
    cent = rng.standard_normal((H, 24, d))
    new = synth.round_bf16((cent[:, rng.integers(0, 24, n)] + 0.3 * rng.standard_normal((H, n, d))).astype(np.float32))
    old = cent[:, rng.integers(0, 24, cap)] * rng.uniform(0.5, 2.0, (1, cap, 1)) + 0.3 * rng.standard_normal((H, cap, d))
    old = synth.round_bf16(old.astype(np.float32))
    for j in range(128, cap, 3):
        old[:, j] = old[:, j - 128]
    return H, cap, new, old


@pytest.mark.parametrize("probe", [False, True])
@pytest.mark.parametrize("d,pt,n,lengths", [
    (128, 128, 1, (1,)), (64, 64, 128, (128, 0, 127)), (128, 64, 129, (129, 640)), (128, 128, 256, (255, 1, 0, 3000)),
    (64, 128, 257, (5000, 129, 4096)), (128, 128, 385, (6000,) * 7), (64, 64, 1000, (2049, 2048, 2047)), (128, 128, 2600, (9000, 12000)),
    # many heads whose second unit is one tile (the other group of warps sits it out), more keys than one wave may touch (96 MB)
    (128, 64, 300, (700, 129, 0, 1500) * 10), (128, 128, 300, (52000, 50000, 49999, 51000, 50001, 50000, 52001, 50000)),
])
def test_search_edges(d, pt, n, lengths, probe):
    import torch
    from paper_2602_01801_b200 import fastar
    H, cap, new, old = _case(d, pt, n, lengths, n + d)
    rng = np.random.default_rng(3)
    cache = fastar.Cache(H, d, cap, pt, rng.standard_normal((32, d)).astype(np.float32), max_tokens=n)
    bits = fastar.bf16_bits(old)
    cache.import_state(bits, bits, np.array(lengths))
    q = synth.round_bf16(new + rng.standard_normal(new.shape).astype(np.float32)) if probe else new
    tau = 0.5
    res = cache.update(fastar.to_device(new), fastar.to_device(new), n, tau, probe=fastar.to_device(q) if probe else None)
    assert cache.status() == 0
    for h, L in enumerate(lengths):
        match, sim = res["match"][h].cpu().numpy(), res["sim"][h].cpu().numpy()
        if L == 0:
            assert (match == -1).all() and (sim == 0).all()
            continue
        k, c = new[h].astype(np.float64), old[h, :L].astype(np.float64)
        cos = (k / np.linalg.norm(k, axis=1, keepdims=True)) @ (c / np.linalg.norm(c, axis=1, keepdims=True)).T
        score = q[h].astype(np.float64) @ c.T if probe else cos
        best = score.argmax(1)                                   # the lowest slot among exact copies
        rows = np.arange(n)
        # fp32 sums of d products: d 2^-24 relative to sum |q_i k_i| <= |q| |k| (1e-5 for a cosine, times the norms for a probe)
        scale = np.linalg.norm(q[h], axis=1) * np.linalg.norm(c, axis=1).max() if probe else 1.0
        slack = d * 2.0 ** -24 * scale
        clear = score[rows, best] - np.where(score < score[rows, best][:, None], score, -np.inf).max(1) > 2 * slack
        got = match >= 0
        assert np.abs(sim - cos[rows, best])[clear | ~np.bool_(probe)].max() <= 2e-5
        assert np.array_equal(match[got & clear], best[got & clear])
        assert (score[rows, match] >= score[rows, best] - 2 * slack)[got].all()
        far = np.abs(cos[rows, best] - tau) > 1e-4
        assert np.array_equal(got[far & clear], (cos[rows, best] >= tau)[far & clear])


@pytest.mark.parametrize("heads,n,cap", [(1, 1, 128), (1, 1, 32768), (5, 17, 16384), (3, 40, 4224)])
def test_few_tokens_against_a_long_cache(heads, n, cap):
    """The words that an update accumulates into are cleared over the whole cache, however few tokens it has: the same tokens are
    merged again and again into slots from the first to the last of every head, once each time."""
    from paper_2602_01801_b200 import fastar
    rng = np.random.default_rng(cap + n)
    keys = synth.round_bf16(rng.standard_normal((heads, cap, 64)).astype(np.float32))
    bits = fastar.bf16_bits(keys)
    cache = fastar.Cache(heads, 64, cap, 64, rng.standard_normal((32, 64)).astype(np.float32), max_tokens=n)
    cache.import_state(bits, bits, np.full(heads, cap))
    slots = np.linspace(0, cap - 1, n).astype(int) if n > 1 else np.array([cap - 1])
    for rep in range(1, 4):
        new = fastar.to_device(np.ascontiguousarray(keys[:, slots]))
        res = cache.update(new, new, n, 0.999)
        assert cache.status() == 0
        assert (res["match"].cpu().numpy() == slots).all()
        assert (res["stats"].cpu().numpy()[:, :3] == [n, n, 0]).all()
        want = np.ones((heads, cap), np.int32)
        want[:, slots] += rep
        assert np.array_equal(cache.export_state(kv=False)["count"], want)
