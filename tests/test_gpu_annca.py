"""AnnCA at the edges of its tiles: one row, frames shorter than a tile and across tile borders, prompt groups of one to eight tiles,
more units than CTAs; two calls in a row (the second must not see the first one's maxima)."""
import numpy as np
import pytest

from oracle import fastar_oracle as O
from paper_2602_01801_b200 import synth
from tests import parity as P

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("heads,d,nq,frame_len,prompt,keep,bits", [
    (1, 64, 1, 1, 1, 1, 16), (2, 128, 129, 129, 129, 5, 16), (3, 128, 300, 37, 513, 64, 16), (1, 64, 640, 64, 1024, 65, 16),
    (2, 128, 64, 1, 200, 3, 16), (40, 64, 520, 260, 32, 8, 16), (2, 128, 300, 100, 130, 129, 8), (1, 64, 257, 256, 400, 64, 8),
    # gathered key tiles: two, a remainder of one token, more than the rings have stages
    (3, 128, 200, 200, 512, 256, 16), (2, 128, 300, 150, 1024, 1000, 16), (2, 64, 129, 129, 700, 641, 16)])
def test_relevance_selection_attention(heads, d, nq, frame_len, prompt, keep, bits):
    from paper_2602_01801_b200 import fastar

    rng = np.random.default_rng(nq + prompt)
    frames = -(-nq // frame_len)
    cache = fastar.Cache(heads, d, 128, 64, rng.standard_normal((32, d)).astype(np.float32), max_tokens=nq, max_prompt_tokens=prompt,
                         max_frames=frames, search_bits=bits)
    for scale in (1.0, 0.25):                              # the second call's maxima are the smaller ones
        Q, Kp, Vp = (synth.round_bf16(scale * rng.standard_normal((heads, n, d)).astype(np.float32)) for n in (nq, prompt, prompt))
        r = cache.annca(fastar.to_device(Q), fastar.to_device(Kp), fastar.to_device(Vp), frame_len, keep, debug=True)
        assert cache.status() == fastar.OK
        codes = cache.export_annca_codes(nq, prompt) if bits == 8 else None
        out = r["out"].float().cpu().numpy()
        for h in sorted({0, heads // 2, heads - 1}):
            sel = r["sel"][h].cpu().numpy()
            P.check_prompt_selection(Q[h], Kp[h], frame_len, keep, sel, r["rel"][h].cpu().numpy(),
                                     codes=(codes["q"][h][:, :d], codes["prompt"][h][:, :d]) if bits == 8 else None)
            P.check_attention(out[h], O.annca(Q[h], Kp[h], Vp[h], frame_len, keep, sel=sel)["out"], f"AnnCA head {h}")


def test_reset_on_another_stream_leaves_the_relevance_alone():
    """AnnCA uses its own scratch and reads no cache state: a reset (or an import, which begins with one) that runs meanwhile on another
    stream does not change what it selects."""
    import torch

    from paper_2602_01801_b200 import fastar

    g = torch.Generator(device="cuda").manual_seed(3)
    H, d, nq, prompt, keep = 8, 128, 2048, 256, 8
    q, kp, vp = (torch.randn(H, n, d, generator=g, device="cuda").bfloat16() for n in (nq, prompt, prompt))
    cache = fastar.Cache(H, d, 256, 128, np.random.default_rng(3).standard_normal((32, d)).astype(np.float32), max_tokens=nq,
                         max_prompt_tokens=prompt, max_frames=4)
    def call():
        return cache.annca(q, kp, vp, nq // 4, keep, debug=True)["sel"]

    want = call()
    main, side, gate = torch.cuda.current_stream(), torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(gate):                          # both streams find their work queued when they start
        torch.cuda._sleep(40_000_000)
        start = gate.record_event()
    main.wait_event(start)
    side.wait_event(start)
    got = []
    for _ in range(60):
        with torch.cuda.stream(side):
            cache.reset()
            cache.reset()
        got.append(call())
    torch.cuda.synchronize()
    assert cache.status() == fastar.OK
    assert all(torch.equal(x, want) for x in got)


@pytest.mark.parametrize("d,keep", [(128, 70), (64, 9)])
def test_frame_longer_than_the_call(d, keep):
    """A frame length beyond the queries means one frame, up to the largest integer."""
    import torch

    from paper_2602_01801_b200 import fastar

    g = torch.Generator(device="cuda").manual_seed(d)
    H, nq, prompt = 3, 200, 96
    q, kp, vp = (torch.randn(H, n, d, generator=g, device="cuda").bfloat16() for n in (nq, prompt, prompt))
    cache = fastar.Cache(H, d, 128, 64, np.random.default_rng(3).standard_normal((32, d)).astype(np.float32), max_tokens=nq,
                         max_prompt_tokens=prompt, max_frames=2)
    for call in (lambda f: cache.annca(q, kp, vp, f, keep, debug=True), lambda f: cache.annca_lsh(q, kp, vp, f, debug=True)):
        want = call(nq)
        for frame_len in (nq + 1, 2 ** 30, 2 ** 31 - 128, 2 ** 31 - 1):
            got = call(frame_len)
            assert cache.status() == fastar.OK
            assert torch.equal(got["out"], want["out"])
            n = want["nsel"].max() if "nsel" in want else keep
            assert torch.equal(got["sel"][..., :n], want["sel"][..., :n])
