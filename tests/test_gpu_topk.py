"""Block and prompt top-k against a stable sort of the same scores: rows at the limits of the register tiles (128, 512, 1152, 2048
entries), one entry, everything kept, forced blocks, many equal scores."""
import numpy as np
import pytest

from paper_2602_01801_b200 import synth

pytestmark = pytest.mark.gpu


def _kept(score, k):
    return np.sort(np.lexsort((np.arange(len(score)), -score.astype(np.int64)))[:k])


@pytest.mark.parametrize("capacity,length,keep,sink,recent", [(128, 1, 1, 0, 0), (8192, 8192, 127, 0, 0), (8320, 8257, 5, 2, 3),
                                                              (32768, 32700, 64, 1, 0), (32896, 32833, 513, 0, 1),
                                                              (73728, 73700, 1, 0, 0), (73856, 70000, 300, 4, 4),
                                                              (131072, 131072, 700, 1, 1)])
def test_block_topk(capacity, length, keep, sink, recent):
    from paper_2602_01801_b200 import fastar
    rng = np.random.default_rng(length)
    d, nq = 64, 130
    cache = fastar.Cache(1, d, capacity, 64, rng.standard_normal((32, d)).astype(np.float32), max_tokens=nq)
    k = synth.round_bf16(rng.standard_normal((1, length, d)).astype(np.float32))
    cache.import_state(fastar.bf16_bits(k), fastar.bf16_bits(k), np.array([length]))
    cache.set_forced_blocks(sink, recent)
    r = cache.annsa(fastar.to_device(synth.round_bf16(rng.standard_normal((1, nq, d)).astype(np.float32))), 64, keep, debug=True)
    assert cache.status() == 0
    if "sel" not in r:                                     # all blocks kept: dense, nothing is ranked
        assert keep >= capacity // 64
        return
    n = -(-length // 64)
    score, sel = r["scores"][0].cpu().numpy(), r["sel"][0].cpu().numpy()
    assert int(r["nsel"][0]) == min(keep, n)
    for a in range(sel.shape[0]):
        s = score[a, :n].astype(np.int64)
        i = np.arange(n)
        s = np.where((i < sink) | (i >= n - recent), s + (1 << 30), s)
        assert np.array_equal(sel[a, : min(keep, n)], _kept(s, min(keep, n)))


@pytest.mark.parametrize("prompt,keep", [(1, 1), (128, 128), (129, 7), (512, 511), (513, 64), (1024, 1000)])
def test_prompt_topk(prompt, keep):
    from paper_2602_01801_b200 import fastar
    rng = np.random.default_rng(prompt)
    d, nq = 64, 40
    cache = fastar.Cache(2, d, 128, 64, rng.standard_normal((32, d)).astype(np.float32), max_tokens=nq, max_prompt_tokens=prompt, max_frames=3)
    kp = rng.integers(-1, 2, (2, prompt, d)).astype(np.float32)      # small integers: exact scores, ties
    q = np.zeros((2, nq, d), np.float32)
    q[:, :, :2] = rng.integers(-1, 2, (2, nq, 2))
    r = cache.annca(fastar.to_device(q), fastar.to_device(kp), fastar.to_device(kp), 17, keep, debug=True)
    assert cache.status() == 0
    for h in range(2):
        for f in range(3):
            want = (q[h, 17 * f: 17 * f + 17] @ kp[h].T).max(0)
            assert np.array_equal(np.rint(r["rel"][h, f].cpu().numpy() * 8.0), want)
            assert np.array_equal(r["sel"][h, f].cpu().numpy(), _kept(want, keep))


@pytest.mark.parametrize("H,capacity,nq", [(1, 4224, 130), (29, 16640, 130), (40, 16640, 130)])
def test_block_scores_of_few_and_many_heads(H, capacity, nq):
    """The grid of the block scores on both sides of one CTA per SM (2, 145 and 200 CTAs): same-bucket pairs counted from the codes."""
    import torch
    from paper_2602_01801_b200 import fastar
    rng = np.random.default_rng(H)
    d, pt, length = 64, 64, capacity - 7
    cache = fastar.Cache(H, d, capacity, pt, rng.standard_normal((32, d)).astype(np.float32), max_tokens=nq)
    k = synth.round_bf16(rng.standard_normal((H, length, d)).astype(np.float32))
    cache.import_state(fastar.bf16_bits(k), fastar.bf16_bits(k), np.full(H, length))
    r = cache.annsa(fastar.to_device(synth.round_bf16(rng.standard_normal((H, nq, d)).astype(np.float32))), 128, 1, debug=True)
    assert cache.status() == 0
    kc = torch.from_numpy(cache.export_state(kv=False)["code"][:, :length].astype(np.int64)).cuda()
    qc = r["qcode"].long() & 0xFFFFFFFF

    def histograms(code, block):
        n = -(-code.shape[1] // block)
        at = (torch.arange(code.shape[1], device="cuda") // block * 1024)[None, :, None] + 256 * torch.arange(4, device="cuda") + (code[..., None] >> (8 * torch.arange(4, device="cuda")) & 255)
        out = torch.zeros(H, n * 1024, device="cuda", dtype=torch.float64)
        return out.scatter_add_(1, at.reshape(H, -1), torch.ones_like(at.reshape(H, -1), dtype=torch.float64)).reshape(H, n, 1024)
    hk = histograms(kc, pt)
    assert torch.equal(r["scores"][:, :, : hk.shape[1]].double(), histograms(qc, 128) @ hk.mT)
