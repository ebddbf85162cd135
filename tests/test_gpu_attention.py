"""The attention kernel's tile loop: one to many key tiles (the four soft-max groups, the hand-over of the running maximum between
them), maxima that rise late or by far, weighted slots, an un-cached segment, ragged query blocks; many items per CTA, blocks without a
live slot, values at the ends of their range."""
import math

import numpy as np
import pytest

from paper_2602_01801_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rise", [0.0, 6.0, 60.0])
@pytest.mark.parametrize("d,pt,nq,length,seg", [(128, 128, 1, 1, 0), (128, 128, 129, 128, 0), (128, 64, 200, 65, 0), (64, 128, 128, 300, 7),
                                                (64, 64, 77, 1000, 130), (128, 128, 300, 4200, 300), (128, 64, 64, 700, 64)])
def test_tiles_and_maxima(d, pt, nq, length, seg, rise):
    import torch
    from paper_2602_01801_b200 import fastar
    rng = np.random.default_rng(length + d)
    H, cap = 2, -(-max(length, nq, 128) // 128) * 128 + 128
    q = synth.round_bf16(rng.standard_normal((H, nq, d)).astype(np.float32))
    # the logit of key j against every query grows with j by about `rise` from the first key to the last: q . mean direction
    u = q.mean((0, 1)) / np.linalg.norm(q.mean((0, 1)))
    q = synth.round_bf16(q + 3.0 * u)
    ramp = (np.arange(cap + seg) / max(1, length + seg - 1)) * rise * math.sqrt(d) / 3.0
    k = synth.round_bf16((0.5 * rng.standard_normal((H, cap + seg, d)) + ramp[None, :, None] * u).astype(np.float32))
    v = synth.round_bf16(rng.standard_normal((H, cap + seg, d)).astype(np.float32))
    count = rng.integers(1, 9, (H, cap)).astype(np.int32)
    lens = np.array([length, max(0, length - 61)])
    cache = fastar.Cache(H, d, cap, pt, rng.standard_normal((32, d)).astype(np.float32), max_tokens=max(nq, seg, 1))
    cache.import_state(fastar.bf16_bits(k[:, :cap]), fastar.bf16_bits(v[:, :cap]), lens, count)
    dq = fastar.to_device(q)
    if seg:
        out = cache.annsa_segment(dq, fastar.to_device(k[:, cap:]), fastar.to_device(v[:, cap:]), 128, cap // pt)["out"]
    else:
        out = cache.annsa(dq, 128, cap // pt)["out"]
    assert cache.status() == 0
    for h in range(H):
        L = int(lens[h])
        kk = np.concatenate([k[h, :L], k[h, cap:]]).astype(np.float64)
        vv = np.concatenate([v[h, :L], v[h, cap:]]).astype(np.float64)
        got = out[h].float().cpu().numpy()
        if len(kk) == 0:
            assert (got == 0).all()
            continue
        s = q[h].astype(np.float64) @ kk.T / math.sqrt(d) + np.log(np.concatenate([count[h, :L], np.ones(seg)]))
        p = np.exp(s - s.max(1, keepdims=True))
        want = (p / p.sum(1, keepdims=True)) @ vv
        # probabilities and output rounded to 8 significant bits (2^-8 each), sums in fp32: 2^-7 of the largest value averaged
        assert np.abs(got - want).max() <= 2.0 ** -7 * np.abs(vv).max()
        assert np.linalg.norm(got - want) <= 1e-2 * np.linalg.norm(want)


@pytest.mark.parametrize("d,pt,seg", [(128, 128, 0), (128, 64, 0), (64, 128, 190), (64, 64, 70), (128, 64, 129)])
def test_many_items_on_a_cta(d, pt, seg):
    """400 items on 148 CTAs, with what one item leaves to the next: numbers of sub-tiles that no count of groups or stages divides,
    empty heads between others, maxima that rise in some items and fall from one item to the next."""
    import torch
    from paper_2602_01801_b200 import fastar
    rng = np.random.default_rng(d + pt + seg)
    H, nq, cap = 40, 10 * 128 - 50, 1408
    lens = np.resize([1, 65, 0, 5 * pt, cap, 3 * pt + 1, 700, 129, 0, pt + 64, 11 * 64 + 3], H)
    q = rng.standard_normal((H, -(-nq // 128), 128, d)) * rng.choice([1.0, 30.0], (H, -(-nq // 128), 1, 1))
    q = synth.round_bf16(q.reshape(H, -1, d)[:, :nq].astype(np.float32))
    k, v = (synth.round_bf16(rng.standard_normal((H, cap + seg, d)).astype(np.float32)) for _ in range(2))
    k[::3] *= (2.0 ** np.linspace(-3, 2, cap + seg).round())[None, :, None].astype(np.float32)      # exact in bf16
    count = rng.integers(1, 9, (H, cap)).astype(np.int32)
    cache = fastar.Cache(H, d, cap, pt, rng.standard_normal((32, d)).astype(np.float32), max_tokens=nq)
    cache.import_state(fastar.bf16_bits(k[:, :cap]), fastar.bf16_bits(v[:, :cap]), lens, count)
    if seg:
        out = cache.annsa_segment(fastar.to_device(q), fastar.to_device(k[:, cap:]), fastar.to_device(v[:, cap:]), 128, cap // pt)["out"]
    else:
        out = cache.annsa(fastar.to_device(q), 128, cap // pt)["out"]
    assert cache.status() == 0
    for h in range(H):
        L = int(lens[h])
        got = out[h].float().cpu().numpy()
        if L + seg == 0:
            assert (got == 0).all()
            continue
        s = q[h].astype(np.float64) @ np.concatenate([k[h, :L], k[h, cap:]]).T / math.sqrt(d)
        s += np.log(np.concatenate([count[h, :L], np.ones(seg)]))
        p = np.exp(s - s.max(1, keepdims=True))
        want = (p / p.sum(1, keepdims=True)) @ np.concatenate([v[h, :L], v[h, cap:]])
        # as above: rounding of the probabilities and of the output
        assert np.abs(got - want).max() <= 2.0 ** -7 * np.abs(v).max(), f"head {h}"
        assert np.linalg.norm(got - want) <= 1e-2 * np.linalg.norm(want), f"head {h}"


@pytest.mark.parametrize("d,pt,seg", [(128, 128, 0), (128, 64, 70), (64, 128, 200), (64, 64, 0)])
def test_listed_blocks_without_a_live_slot(d, pt, seg):
    """A caller's list may name blocks past a head's live slots: they add nothing, wherever in the list they stand, also for an empty
    head and where nothing live is listed.  More items than two rounds of the CTAs, so that an item follows others on its CTA."""
    import torch
    from oracle import fastar_oracle as O
    from paper_2602_01801_b200 import fastar
    rng = np.random.default_rng(d + pt)
    H, nq, cap, keep = 40, 10 * 128, 1024, 3
    nb = cap // pt
    lens = np.resize([cap, 0, 1, 65, pt, 3 * pt + 1, cap - 1], H)
    q = rng.standard_normal((H, nq // 128, 128, d)) * rng.choice([1.0, 60.0], (H, nq // 128, 1, 1))      # maxima far apart between items
    q = synth.round_bf16(q.reshape(H, nq, d).astype(np.float32))
    k, v = (synth.round_bf16(rng.standard_normal((H, cap + seg, d)).astype(np.float32)) for _ in range(2))
    count = rng.integers(1, 9, (H, cap)).astype(np.int32)
    cache = fastar.Cache(H, d, cap, pt, rng.standard_normal((32, d)).astype(np.float32), max_tokens=nq)
    cache.import_state(fastar.bf16_bits(k[:, :cap]), fastar.bf16_bits(v[:, :cap]), lens, count)
    sel = np.stack([[rng.permutation(nb)[:keep] for _ in range(nq // 128)] for _ in range(H)]).astype(np.int32)
    sel[:, ::2] = np.sort(sel[:, ::2], axis=2)[:, :, ::-1]                                # dead blocks first
    sel[3, 1], sel[5, 2] = nb - 1, nb - 1                                                 # nothing but dead blocks
    args = dict(sel_in=torch.from_numpy(sel).cuda(), nsel_in=torch.full((H,), keep, dtype=torch.int32, device="cuda"))
    dq = fastar.to_device(q)
    if seg:
        out = cache.annsa_segment(dq, fastar.to_device(k[:, cap:]), fastar.to_device(v[:, cap:]), 128, keep, **args)["out"]
    else:
        out = cache.annsa(dq, 128, keep, **args)["out"]
    assert cache.status() == 0
    for h in range(H):
        hc = O.HeadCache(cap, d)
        L = int(lens[h])
        hc.load(k[h, :L].astype(np.float64), v[h, :L].astype(np.float64), m=count[h, :L].astype(np.int64), now=1)
        want = O.sparse_attention_with_segment(q[h], hc, sel[h], 128, pt, k[h, cap:], v[h, cap:])
        got = out[h].float().cpu().numpy()
        assert np.isfinite(got).all()
        # as above: rounding of the probabilities and of the output
        assert np.abs(got - want).max() <= 2.0 ** -7 * np.abs(v).max(), f"head {h}"


@pytest.mark.parametrize("pt", [64, 128])
@pytest.mark.parametrize("d,magnitude", [(64, 110), (128, 110), (128, -100)])
def test_range_of_the_values(d, pt, magnitude):
    """Values near the ends of bf16's range under maxima that rise with every sub-tile of 64 keys, by 18 to 25 binary orders each time:
    the output is a mean of the values and stays finite and as exact as for ordinary ones."""
    import torch
    from paper_2602_01801_b200 import fastar
    rng = np.random.default_rng(d + pt)
    n, steps = 768, 12
    rise = np.cumsum(np.concatenate([[0.0], rng.uniform(18.0, 25.0, steps - 1)]))
    unit = math.sqrt(d) / math.log2(math.e) / 8.0          # q = 8 e0: this much of a key's first component is one binary order
    k = 0.01 * rng.standard_normal((1, n, d))
    k[0, :, 0] = np.repeat(rise, 64) * unit
    k, q = synth.round_bf16(k.astype(np.float32)), np.zeros((1, 130, d), np.float32)
    q[:, :, 0], q[:, :, 1] = 8.0, synth.round_bf16(rng.standard_normal(130).astype(np.float32))
    v = synth.round_bf16((rng.standard_normal((1, n, d)) * 2.0 ** magnitude).astype(np.float32))
    cache = fastar.Cache(1, d, n, pt, rng.standard_normal((32, d)).astype(np.float32), max_tokens=n)
    cache.import_state(fastar.bf16_bits(k), fastar.bf16_bits(v), np.array([n]))
    for last in (n, 640, 192):                             # the segment entry as well: the last keys from there
        kk, vv = k[:, :last], v[:, :last]
        if last == n:
            out = cache.annsa(fastar.to_device(q), 128, n // pt)["out"]
        else:
            cache.import_state(fastar.bf16_bits(k[:, :last - 128]), fastar.bf16_bits(v[:, :last - 128]), np.array([last - 128]))
            out = cache.annsa_segment(fastar.to_device(q), fastar.to_device(k[:, last - 128:last]), fastar.to_device(v[:, last - 128:last]),
                                      128, n // pt)["out"]
        assert cache.status() == 0
        s = q[0].astype(np.float64) @ kk[0].T.astype(np.float64) / math.sqrt(d)
        p = np.exp(s - s.max(1, keepdims=True))
        want = (p / p.sum(1, keepdims=True)) @ vv[0].astype(np.float64)
        got = out[0].float().cpu().numpy().astype(np.float64)
        assert np.isfinite(got).all()
        assert np.abs(got - want).max() <= 2.0 ** -7 * np.abs(vv).max()
        assert np.linalg.norm(got - want) <= 1e-2 * np.linalg.norm(want)


@pytest.mark.parametrize("d,pt,H,nq,lens,seg,keep", [
    (128, 128, 1, 100, [40 * 128 - 5], 0, 0),                      # one item for all CTAs
    (64, 64, 1, 64, [1030 * 64], 0, 0),                            # as many parts as an item gets
    (128, 64, 3, 300, [9 * 64, 0, 31 * 64 + 1], 200, 0),           # unequal heads, one of them with nothing but the segment
    (64, 128, 7, 22 * 128 - 60, [17 * 128, 0, 1, 129, 24 * 128, 9 * 128, 300], 0, 0),      # a full round and six items
    (128, 128, 5, 44 * 128, [24 * 128], 0, 0),                     # 72 items: the ends of two in one CTA
    (128, 128, 2, 500, [60 * 128], 0, 33),                         # lists of blocks, and a segment behind them
    (64, 64, 3, 700, [40 * 64 - 9, 64, 40 * 64], 100, 21),
])
def test_items_cut_by_key_tiles(d, pt, H, nq, lens, seg, keep):
    """The items of a last round that does not fill the SMs are cut: parts of all lengths, empty heads between them, the same result by
    a second call (the counters of the parts are back at zero)."""
    import torch
    from paper_2602_01801_b200 import fastar
    rng = np.random.default_rng(d + pt + H)
    lens = np.resize(lens, H)
    cap = -(-max(int(lens.max()), 128) // 128) * 128
    cap += cap // 2 // 128 * 128 if H == 7 else 0                  # fewer live blocks than the launch knows of
    q = synth.round_bf16((rng.standard_normal((H, nq, d)) * rng.choice([1.0, 20.0], (H, nq, 1))).astype(np.float32))
    k, v = (synth.round_bf16(rng.standard_normal((H, cap + seg, d)).astype(np.float32)) for _ in range(2))
    count = rng.integers(1, 9, (H, cap)).astype(np.int32)
    cache = fastar.Cache(H, d, cap, pt, rng.standard_normal((32, d)).astype(np.float32), max_tokens=nq)
    cache.import_state(fastar.bf16_bits(k[:, :cap]), fastar.bf16_bits(v[:, :cap]), lens, count)
    args, nqb = {}, -(-nq // 128)
    if keep:
        sel = np.stack([[rng.permutation(cap // pt)[:keep] for _ in range(nqb)] for _ in range(H)]).astype(np.int32)
        args = dict(sel_in=torch.from_numpy(sel).cuda(), nsel_in=torch.full((H,), keep, dtype=torch.int32, device="cuda"))
    dq, dk, dv = fastar.to_device(q), fastar.to_device(k[:, cap:]), fastar.to_device(v[:, cap:])
    blocks = keep or cap // pt
    out, again = (cache.annsa_segment(dq, dk, dv, 128, blocks, **args)["out"] if seg else cache.annsa(dq, 128, blocks, **args)["out"] for _ in range(2))
    assert cache.status() == 0
    assert torch.equal(out, again)
    for h in range(H):
        for b in range(0, nqb, max(1, nqb // 6)):
            slots = np.concatenate([np.arange(s * pt, s * pt + pt) for s in (sel[h, b] if keep else range(cap // pt))])
            slots = slots[slots < lens[h]]
            got = out[h, b * 128: b * 128 + 128].float().cpu().numpy()
            if len(slots) + seg == 0:
                assert (got == 0).all()
                continue
            kk, vv = (np.concatenate([x[h, slots], x[h, cap:]]) for x in (k, v))
            s = q[h, b * 128: b * 128 + 128].astype(np.float64) @ kk.T / math.sqrt(d) + np.log(np.concatenate([count[h, slots], np.ones(seg)]))
            p = np.exp(s - s.max(1, keepdims=True))
            want = (p / p.sum(1, keepdims=True)) @ vv
            # as above: rounding of the probabilities and of the output
            assert np.abs(got - want).max() <= 2.0 ** -7 * np.abs(vv).max(), f"head {h}, block {b}"
            assert np.linalg.norm(got - want) <= 1e-2 * np.linalg.norm(want), f"head {h}, block {b}"


@pytest.mark.parametrize("d,pt", [(64, 64), (64, 128), (128, 64), (128, 128)])
@pytest.mark.parametrize("whole_rounds", [False, True])
def test_not_a_number_stays_in_its_rows(d, pt, whole_rounds):
    """A query of NaN, a cached key of NaN: exactly the rows that they reach are NaN, whether items are cut by key tiles (a few of them) or not
    (as many as there are SMs)."""
    import torch
    from paper_2602_01801_b200 import fastar
    rng = np.random.default_rng(d + pt)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    H, keep, blocks = 2, 33, 60
    nq = 128 * (sms // H if whole_rounds else 3) - 28
    nqb = -(-nq // 128)
    q, k, v = (synth.round_bf16(rng.standard_normal((H, m, d)).astype(np.float32)) for m in (nq, blocks * pt, blocks * pt))
    q[0, 5, 3] = np.nan
    q[1, nq - 1] = np.inf
    k[1, 7 * pt + 9, d - 1] = np.nan
    lens = np.array([blocks * pt - 3, blocks * pt])
    cap = -(-blocks * pt // 128) * 128
    cache = fastar.Cache(H, d, cap, pt, rng.standard_normal((32, d)).astype(np.float32), max_tokens=nq)
    cache.import_state(fastar.bf16_bits(k), fastar.bf16_bits(v), lens)
    sel = np.stack([[np.sort(rng.permutation(blocks)[:keep]) for _ in range(nqb)] for _ in range(H)]).astype(np.int32)
    nsel = torch.full((H,), keep, dtype=torch.int32, device="cuda")
    out = cache.annsa(fastar.to_device(q), 128, keep, sel_in=torch.from_numpy(sel).cuda(), nsel_in=nsel)["out"].float().cpu().numpy()
    assert cache.status() == 0
    with np.errstate(invalid="ignore"):
        for h in range(H):
            for b in {0, 1, nqb // 2, nqb - 1}:
                rows = slice(b * 128, min(nq, b * 128 + 128))
                at = (sel[h, b][:, None] * pt + np.arange(pt)).reshape(-1)
                at = at[at < lens[h]]
                s = q[h, rows].astype(np.float64) @ k[h, at].T.astype(np.float64) / math.sqrt(d)
                p = np.exp(s - s.max(1, keepdims=True))
                want = (p / p.sum(1, keepdims=True)) @ v[h, at]
                nan = np.isnan(want)
                assert nan.any() == (7 in sel[1, b] if h == 1 and b < nqb - 1 else h == 1 or b == 0)
                assert np.array_equal(np.isnan(out[h, rows]), nan)
                # rounding of the probabilities and of the output
                assert np.abs(out[h, rows] - want)[~nan].max(initial=0) <= 2.0 ** -7 * np.abs(v[h]).max()


@pytest.mark.parametrize("d,pt,H,nqb,tiles,lens,seg", [
    (128, 128, 1, 3, 128, [512], 0),                               # room for 128 tiles, four are there
    (128, 128, 1, 3, 128, [15 * 128], 0),                          # the most that is not cut, and the least that is
    (128, 128, 1, 3, 128, [15 * 128 + 1], 0),
    (64, 64, 6, 3, 160, [0, 1, 64 * 7, 64 * 19, 64 * 15 - 1, 64 * 4], 0),
    (64, 64, 6, 3, 160, [0, 1, 64 * 7, 64 * 60, 64 * 15 - 1, 64 * 160], 0),        # cut, heads of nothing and of a few keys too
    (128, 64, 6, 3, 100, [64 * 9, 0, 5, 64 * 7, 0, 64 * 3 + 3], 130),
    (128, 64, 6, 3, 100, [64 * 9, 64 * 100, 5, 64 * 40, 0, 64 * 30 + 3], 130),
    (128, 128, 8, 11, 80, [128 * 50, 128 * 5 - 1, 128 * 3, 100, 128 * 40, 0, 128 * 6, 128], 0),      # 88 items, cut if dealt to all CTAs
    (128, 128, 8, 11, 80, [128 * 80, 128 * 56 - 1, 128 * 57, 100, 128 * 80, 0, 128 * 56, 128 * 70], 0),
    (64, 64, 11, 9, 140, [64 * 140, 64, 64 * 127, 64 * 128, 64 * 100, 64 * 140, 64 * 3, 0, 64 * 140, 64 * 130, 64 * 135], 0),      # 99 items
    (64, 128, 11, 17, 40, [128 * 9, 128 * 10, 128 * 2, 1, 0, 1, 128 * 3, 128 * 4, 128 * 8, 128 * 4, 128 * 3], 0),      # a full round and 39
    (64, 128, 11, 17, 40, [128 * 40, 128 * 11, 128 * 12, 128 * 12 + 1, 0, 1, 128 * 30, 128 * 40, 128 * 8, 128 * 40, 128 * 13], 0),
])
def test_items_of_caches_that_are_not_full(d, pt, H, nqb, tiles, lens, seg):
    """Whether items are cut is decided by the keys that are there, not by the room for them: on both sides of the decision, with heads of no,
    few and many tiles in one call; the same by a second call."""
    import torch
    from paper_2602_01801_b200 import fastar
    g = torch.Generator(device="cuda").manual_seed(d + H * tiles)
    cap, nq = -(-tiles * pt // 128) * 128, nqb * 128 - 31
    normal = lambda *shape: torch.randn(*shape, generator=g, device="cuda").bfloat16()
    q, k, v, sk, sv = (normal(H, m, d) for m in (nq, cap, cap, max(seg, 1), max(seg, 1)))
    cache = fastar.Cache(H, d, cap, pt, np.random.default_rng(1).standard_normal((32, d)).astype(np.float32), max_tokens=nq)
    cache.import_state(fastar.bf16_bits(k.float().cpu().numpy()), fastar.bf16_bits(v.float().cpu().numpy()), np.array(lens))
    call = (lambda: cache.annsa_segment(q, sk, sv, 128, cap // pt)["out"]) if seg else (lambda: cache.annsa(q, 128, cap // pt)["out"])
    out, again = call(), call()
    assert cache.status() == 0
    assert torch.equal(out, again)
    for h in range(H):
        kk, vv = (torch.cat([x[h, : lens[h]], y[h, :seg]]).double() for x, y in ((k, sk), (v, sv)))
        if len(kk) == 0:
            assert (out[h] == 0).all()
            continue
        want = torch.softmax(q[h].double() @ kk.T / math.sqrt(d), -1) @ vv
        # rounding of the probabilities and of the output
        assert (out[h].double() - want).abs().max() <= 2.0 ** -7 * vv.abs().max()
        assert (out[h].double() - want).norm() <= 1e-2 * want.norm()


@pytest.mark.parametrize("d,pt", [(64, 64), (64, 128), (128, 64), (128, 128)])
@pytest.mark.parametrize("tiles", [7, 8, 9, 21])
def test_bounds_of_the_logits(d, pt, tiles):
    """Heads whose largest norms and multiplicities bound every logit near an item's first ones, and heads where they do not: a last key
    that towers over the others, values near the end of bf16's range, rows of very unequal norms, keys and values of zero.  The same for keys
    that came by updates, by an import, and as a segment."""
    import torch
    from paper_2602_01801_b200 import fastar
    rng = np.random.default_rng(d + pt + tiles)
    H, nq, n = 8, 200, tiles * 64
    cap = -(-n // 128) * 128 + 128
    q, k, v = (rng.standard_normal((H, m, d)).astype(np.float32) for m in (nq, n, n))
    count = np.ones((H, n), np.int32)
    q[1, ::3] *= 30.0                                      # rows of a warp far apart
    q[2, :, 0] = np.abs(q[2, :, 0]) + 4.0
    k[2, n - 1] = 0.0
    k[2, n - 1, 0] = 12.0 * math.sqrt(d)                   # the last key, 50 binary orders and more above the others
    v[3] *= 2.0 ** 100                                     # 8 binary orders of room, and logits that rise by about 20
    q[3, :, 0], k[3, :, 0] = 4.0, np.linspace(0.0, 3.5 * math.sqrt(d) / math.log2(math.e), n)
    count[4] = rng.integers(1, 5000, n)
    k[5, n // 2:], v[5, : n // 2] = 0.0, 0.0
    v[6] = 0.0
    v[7] *= 2.0 ** -100
    k[7] *= 3.0
    q, k, v = (synth.round_bf16(x) for x in (q, k, v))
    lsh = rng.standard_normal((32, d)).astype(np.float32)
    dq, dk, dv = (fastar.to_device(x) for x in (q, k, v))

    def check(out, times, but=-1):
        for h in range(H):
            if h == but:
                continue
            s = q[h].astype(np.float64) @ k[h].T.astype(np.float64) / math.sqrt(d) + np.log(times[h])
            p = np.exp(s - s.max(1, keepdims=True))
            want = (p / p.sum(1, keepdims=True)) @ v[h].astype(np.float64)
            got = out[h].float().cpu().numpy().astype(np.float64)
            assert np.isfinite(got).all(), f"head {h}"
            # as above: rounding of the probabilities and of the output
            assert np.abs(got - want).max() <= 2.0 ** -7 * np.abs(v[h]).max(), f"head {h}"
            assert np.linalg.norm(got - want) <= 1e-2 * np.linalg.norm(want), f"head {h}"

    def new():
        return fastar.Cache(H, d, cap, pt, lsh, max_tokens=max(n, nq))
    cache = new()
    cache.import_state(fastar.bf16_bits(k), fastar.bf16_bits(v), np.full(H, n), count)
    check(cache.annsa(dq, 128, cap // pt)["out"], count)
    cut = n // 2 + 5
    cache.import_state(fastar.bf16_bits(k[:, :cut]), fastar.bf16_bits(v[:, :cut]), np.full(H, cut), count[:, :cut])
    check(cache.annsa_segment(dq, dk[:, cut:], dv[:, cut:], 128, cap // pt)["out"], np.where(np.arange(n) < cut, count, 1))
    cache = new()
    for a, b in ((0, cut), (cut, n)):                      # (a threshold that nothing reaches: appended)
        cache.update(dk[:, a:b], dv[:, a:b], n, 2.0)
    check(cache.annsa(dq, 128, cap // pt)["out"], np.ones((H, n)))
    cache.update(dk[:, :cut], dv[:, :cut], n, 0.999)       # every key finds itself: multiplicities of two, the same mean values
    check(cache.annsa(dq, 128, cap // pt)["out"], np.broadcast_to(np.where(np.arange(n) < cut, 2, 1), (H, n)), but=5)      # (keys of zero find nothing)
    assert cache.status() == 0


@pytest.mark.parametrize("d,pt", [(64, 64), (64, 128), (128, 64), (128, 128)])
@pytest.mark.parametrize("size", [1.0, 1.5, 2.0, 4.0])
def test_items_without_maxima_are_as_exact_as_with(d, pt, size):
    """Keys in the order of their clusters, logits of `size` times the usual: a row's own cluster comes late, so where the maximum is looked for it
    may be raised there, and a row's largest probability is a power of two behind a raise.  Looking for it is forced by one more key, of a norm that
    no bound admits, against which every query has a logit of minus thousands: the error without that key is not larger than with it."""
    import torch
    from paper_2602_01801_b200 import fastar
    g = torch.Generator(device="cuda").manual_seed(d + pt)
    normal = lambda *shape: torch.randn(*shape, generator=g, device="cuda")
    H, n, nq = 2, 4095, 512
    centre = normal(H, 64, d) * math.sqrt(size)
    k = centre[:, torch.arange(n + 1, device="cuda") * 64 // (n + 1)] + 0.5 * normal(H, n + 1, d)
    q = centre[:, torch.randint(0, 64, (nq,), generator=g, device="cuda")] + 0.5 * normal(H, nq, d)
    q[..., 0], k[..., 0] = 4.0, 0.0
    k[:, n], k[:, n, 0] = 0.0, -(2.0 ** 20)
    q, k, v = q.bfloat16(), k.bfloat16(), normal(H, n + 1, d).bfloat16()
    want = torch.softmax(q.double() @ k[:, :n].double().mT / math.sqrt(d), -1) @ v[:, :n].double()
    errors = []
    for m in (n, n + 1):
        cache = fastar.Cache(H, d, 4096, pt, np.random.default_rng(1).standard_normal((32, d)).astype(np.float32), max_tokens=n + 1)
        cache.update(k[:, :m], v[:, :m], m, 2.0)
        out = cache.annsa(q, 128, 4096 // pt)["out"].double()
        assert cache.status() == 0
        errors.append(float((out - want).norm() / want.norm()))
    # the same probabilities up to the exponentials' 2e-7, which round to another bf16 number once in some ten thousand times
    assert errors[0] <= 1.001 * errors[1]


@pytest.mark.parametrize("d,pt", [(64, 64), (64, 128), (128, 64), (128, 128)])
@pytest.mark.parametrize("source", ["import", "update", "merge", "segment"])
def test_a_late_key_that_only_its_bound_gives_away(d, pt, source):
    """One key, behind all others, 200 binary orders above the first logits: without its bound the item would not look for a maximum, and the
    exponential would leave fp32's range.  The key comes by an import, by a second update, by a merge (in the place of a short key of its
    direction), or with a segment."""
    import torch
    from paper_2602_01801_b200 import fastar
    rng = np.random.default_rng(d + pt)
    H, n, nq = 2, 13 * 64, 200
    order = math.sqrt(d) / math.log2(math.e) / 8.0         # q = 8 e0: so much of a key's first component is one binary order
    q = 0.01 * rng.standard_normal((H, nq, d))
    q[:, :, 0] = 8.0
    k, v = 0.3 * rng.standard_normal((H, n, d)), rng.standard_normal((H, n, d))
    k[:, :, 0] = rng.uniform(-0.5, 0.5, (H, n)) * order
    k[:, n - 1] = 0.0
    k[:, n - 1, 0] = 200.0 * order
    q, k, v = (synth.round_bf16(x.astype(np.float32)) for x in (q, k, v))
    assert (8.0 * k[:, n - 1, 0] / math.sqrt(d) * math.log2(math.e) > 150.0).all()        # 2^150 and more, relative to the others
    cap = n + 192
    cache = fastar.Cache(H, d, cap // 128 * 128, pt, rng.standard_normal((32, d)).astype(np.float32), max_tokens=n)
    dk, dv, blocks = fastar.to_device(k), fastar.to_device(v), cap // 128 * 128 // pt
    if source == "import":
        cache.import_state(fastar.bf16_bits(k), fastar.bf16_bits(v), np.full(H, n))
    elif source == "merge":
        short = k.copy()
        short[:, n - 1, 0] = 1.0
        cache.update(fastar.to_device(short), dv, n, 2.0)
        assert (cache.update(dk[:, n - 64:], dv[:, n - 64:], 64, 0.999)["match"] >= 0).all()
    else:
        cache.update(dk[:, :n - 64], dv[:, :n - 64], n, 2.0)
        if source == "update":
            cache.update(dk[:, n - 64:], dv[:, n - 64:], 64, 2.0)
    if source == "segment":
        out = cache.annsa_segment(fastar.to_device(q), dk[:, n - 64:], dv[:, n - 64:], 128, blocks)["out"]
    else:
        out = cache.annsa(fastar.to_device(q), 128, blocks)["out"]
    assert cache.status() == 0
    out = out.float().cpu().numpy()
    assert np.isfinite(out).all()
    # nothing else has any weight (2^-150), and a mean of equal values is that value
    assert np.array_equal(out, np.broadcast_to(v[:, n - 1:], out.shape))
