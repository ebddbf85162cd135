"""Where planning and ranking change their kernels: numbers of tokens at the edges of the one-kernel planner, the largest slot numbers that
it takes, groups of many members; prompts ranked by the relevance kernel and behind it, block scores of few rows and of more."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,length,capacity", [(1, 1, 128), (33, 200, 256), (1024, 40, 1152), (1025, 700, 2048), (2049, 300, 4096), (4097, 5000, 9216),
                                               (8192, 100, 8320), (8193, 100, 8320), (3000, 65000, 65536), (3000, 65000, 65664)])
def test_matched_and_fresh_tokens_find_their_places(n, length, capacity):
    from paper_2602_01801_b200 import fastar, synth
    rng = np.random.default_rng(n + length)
    H, d = 2, 64
    keys = synth.round_bf16(rng.standard_normal((H, length, d)).astype(np.float32))
    values = synth.round_bf16(rng.standard_normal((H, length, d)).astype(np.float32))
    count = rng.integers(1, 5, (H, length)).astype(np.int32)
    lens = np.array([length, length - 1 if length > 1 else 1])
    cache = fastar.Cache(H, d, capacity, 64, rng.standard_normal((32, d)).astype(np.float32), max_tokens=n)
    pad = lambda x: np.concatenate([x, np.zeros((H, capacity - length) + x.shape[2:], x.dtype)], 1)
    cache.import_state(fastar.bf16_bits(pad(keys)), fastar.bf16_bits(pad(values)), lens, pad(count))
    # a token is a cached key (its cosine to it is 1, to any other far below) or a fresh vector; the last fresh ones fill the cache
    room = capacity - length
    slot = np.stack([rng.integers(0, lens[h], n) for h in range(H)])
    fresh = rng.random((H, n)) < min(0.4, 0.8 * room / n)
    new = synth.round_bf16(rng.standard_normal((H, n, d)).astype(np.float32))
    k = np.where(fresh[..., None], new, np.take_along_axis(keys, slot[..., None], 1))
    v = synth.round_bf16(rng.standard_normal((H, n, d)).astype(np.float32))
    res = cache.update(fastar.to_device(k), fastar.to_device(v), n, 0.95)
    assert cache.status() == 0
    state = cache.export_state()
    for h in range(H):
        want = np.where(fresh[h], lens[h] + np.cumsum(fresh[h]) - 1, slot[h])
        assert np.array_equal(res["dest"][h].cpu().numpy(), want)
        assert np.array_equal(res["match"][h].cpu().numpy(), np.where(fresh[h], -1, slot[h]))
        st = res["stats"][h].cpu().numpy()
        assert list(st[:3]) == [int((~fresh[h]).sum()), len(np.unique(slot[h][~fresh[h]])), int(fresh[h].sum())]
        members = np.bincount(want, minlength=capacity)
        old = np.concatenate([count[h, : lens[h]], np.zeros(capacity - lens[h], np.int32)])
        assert np.array_equal(state["count"][h], old + members)
        total = np.zeros((capacity, d))
        total[: lens[h]] = values[h, : lens[h]].astype(np.float64) * count[h, : lens[h], None]
        np.add.at(total, want, v[h].astype(np.float64))
        live = np.flatnonzero(members)
        got = fastar.bits_to_f32(state["v"][h])[live]
        mean = total[live] / (old + members)[live, None]
        # one rounding to bf16, of sums in fp32
        assert (np.abs(got - mean) <= 2.0 ** -8 * np.abs(mean) + 1e-5).all()


@pytest.mark.parametrize("H,nq,frame,n_prompt,keep", [(1, 1, 1, 1, 1), (2, 600, 300, 80, 24), (3, 700, 11, 129, 40), (40, 300, 100, 513, 64), (2, 4000, 4000, 1024, 33)])
def test_prompt_ranked_inside_the_relevance_kernel(H, nq, frame, n_prompt, keep):
    import torch
    from paper_2602_01801_b200 import fastar
    g = torch.Generator(device="cuda").manual_seed(nq)
    cache = fastar.Cache(H, 128, 1024, 128, np.random.default_rng(1).standard_normal((32, 128)).astype(np.float32), max_tokens=nq, max_prompt_tokens=n_prompt,
                         max_frames=64)
    q, k, v = (torch.randn(H, m, 128, device="cuda", generator=g).bfloat16() for m in (nq, n_prompt, n_prompt))
    k[:, n_prompt // 2:] = k[:, : n_prompt - n_prompt // 2]            # equal relevances: the lower index is kept
    for _ in range(2):                                                # the maxima and the counters are back at zero
        got = cache.annca(q, k, v, frame, keep)["out"]
        ref = cache.annca(q, k, v, frame, keep, debug=True)           # ranked by a kernel of its own, behind the maxima's decoding
        assert torch.equal(got, ref["out"])
    assert cache.status() == 0


@pytest.mark.parametrize("nq,blocks,forced", [(1, 1, 0), (128 * 20, 64, 0), (128 * 20 + 1, 64, 0), (1300, 37, 2), (700, 65, 0)])
def test_block_scores_ranked_by_their_own_kernel_or_behind_it(nq, blocks, forced):
    import torch
    from oracle import fastar_oracle as O
    from paper_2602_01801_b200 import fastar
    rng = np.random.default_rng(nq)
    H, d, cap = 2, 64, 64 * -(-blocks // 2) * 2
    cache = fastar.Cache(H, d, cap, 64, rng.standard_normal((32, d)).astype(np.float32), max_tokens=max(nq, 64))
    keys = fastar.bf16_bits(rng.standard_normal((H, cap, d)).astype(np.float32))
    cache.import_state(keys, keys, np.array([64 * blocks, 64 * max(1, blocks - 3) - 5]))
    keep = max(1, blocks // 3)
    if forced:
        cache.set_forced_blocks(forced, forced)
    r = cache.annsa(fastar.to_device(rng.standard_normal((H, nq, d)).astype(np.float32)), 128, keep, debug=True)
    assert cache.status() == 0
    for h in range(H):
        live = -(-(64 * blocks if h == 0 else 64 * max(1, blocks - 3) - 5) // 64)
        kept = min(keep, live)
        assert int(r["nsel"][h]) == kept
        scores, sel = r["scores"][h].cpu().numpy()[:, :live], r["sel"][h].cpu().numpy()
        for b in range(scores.shape[0]):
            rank = scores[b].copy()
            rank[:forced] += 1e9
            if forced:
                rank[max(0, live - forced):] = np.where(rank[max(0, live - forced):] < 1e9, rank[max(0, live - forced):] + 1e9, rank[max(0, live - forced):])
            want = np.sort(np.lexsort((np.arange(live), -rank))[:kept])
            assert np.array_equal(sel[b, :kept], want)


@pytest.mark.parametrize("H,nq,frame,n_prompt,keep", [(1, 1, 1, 1, 1), (4, 4736, 592, 512, 33), (4, 4737, 4737, 300, 20), (2, 80, 10, 128, 17), (2, 90, 10, 129, 40),
                                                      (3, 700, 233, 257, 64), (3, 700, 234, 513, 24), (37, 512, 256, 256, 9), (1, 640, 10, 1024, 30)])
def test_kept_prompt_tokens_are_those_of_the_largest_relevance(H, nq, frame, n_prompt, keep):
    """On both sides of where the relevance kernel ranks (8 frames, 512 tokens, 148 tiles): attention over the tokens that the relevances in 64 bits
    keep.  Frames whose last kept token is ahead by less than fp32 sums can tell are left out."""
    import math

    import torch
    from paper_2602_01801_b200 import fastar
    g = torch.Generator(device="cuda").manual_seed(nq + n_prompt)
    d = 128
    cache = fastar.Cache(H, d, 1024, 128, np.random.default_rng(1).standard_normal((32, d)).astype(np.float32), max_tokens=nq, max_prompt_tokens=n_prompt, max_frames=64)
    q, k, v = (torch.randn(H, m, d, device="cuda", generator=g).bfloat16() for m in (nq, n_prompt, n_prompt))
    out, again = (cache.annca(q, k, v, frame, keep)["out"] for _ in range(2))          # the maxima and the counters are back at zero
    assert cache.status() == 0 and torch.equal(out, again)
    compared = frames = 0
    for f in range(-(-nq // frame)):
        s = q[:, f * frame: f * frame + frame].double() @ k.double().transpose(1, 2) / math.sqrt(d)
        rel, kept = torch.sort(s.amax(1), dim=1, descending=True)
        for h in range(H):
            frames += 1
            if keep < n_prompt and rel[h, keep - 1] - rel[h, keep] < 1e-5:       # sums of 128 products of size 1: 128 * 2^-24
                continue
            compared += 1
            at = kept[h, :keep]
            want = torch.softmax(s[h][:, at], -1) @ v[h, at].double()
            got = out[h, f * frame: f * frame + frame].double()
            # rounding of the probabilities and of the output
            assert (got - want).abs().max() <= 2.0 ** -7 * v[h].abs().max()
    assert compared >= 0.9 * frames


@pytest.mark.parametrize("H,nq,block_q,tables,bits", [(1, 1, 64, 4, 8), (3, 320, 64, 4, 8), (40, 1000, 64, 1, 3), (39, 1010, 64, 4, 8), (40, 1200, 128, 4, 8), (3, 129, 128, 2, 5)])
def test_histograms_of_query_blocks(H, nq, block_q, tables, bits):
    """One block, an odd number of them (a pass of two has one), more than a CTA has in one pass; the scores are the products of the blocks'
    histograms by the codes of queries and keys."""
    import torch
    from paper_2602_01801_b200 import fastar
    g = torch.Generator(device="cuda").manual_seed(nq)
    d, cap = 64, 256
    cache = fastar.Cache(H, d, cap, 64, np.random.default_rng(1).standard_normal((tables * bits, d)).astype(np.float32), tables, bits, max_tokens=max(nq, cap))
    k, q = (torch.randn(H, m, d, device="cuda", generator=g).bfloat16() for m in (cap, nq))
    cache.update(k, k, cap, 2.0)
    for _ in range(2):
        r = cache.annsa(q, block_q, 2, debug=True)
        keys = torch.from_numpy(cache.export_state(kv=False)["code"].astype(np.int64)).cuda()

        def histogram(codes, rows):
            n = -(-codes.shape[1] // rows)
            h = torch.zeros(H, n, tables << bits, device="cuda", dtype=torch.float64)
            for t in range(tables):
                at = (torch.arange(codes.shape[1], device="cuda") // rows * (tables << bits) + (t << bits))[None] + ((codes >> 8 * t) & 255)
                h.view(H, -1).scatter_add_(1, at, torch.ones_like(at, dtype=torch.float64))
            return h

        want = histogram(r["qcode"].long() & 0xFFFFFFFF, block_q) @ histogram(keys, 64).transpose(1, 2)
        assert torch.equal(r["scores"].double(), want)
    assert cache.status() == 0
