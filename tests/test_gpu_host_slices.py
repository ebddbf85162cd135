"""The host-tensor step in slices of heads: outputs and cache as by the device calls, bit for bit, where the heads do not divide evenly, with
every search and a probe, over two steps (one clock for all slices).
(Even numbers of key tiles: which of the attention's four groups adds up a sub-tile depends on the sub-tiles of the items before.)"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,n,d,fp32,bits,probe,capacity,keep", [(12, 4200, 128, False, 16, False, 8448, 8), (5, 5000, 128, True, 16, True, 10112, 10),
                                                                 (3, 8200, 128, False, 8, False, 8448, 6), (1, 4096, 64, True, 8, True, 4352, 99)])
def test_host_step_by_slices_equals_the_device_calls(H, n, d, fp32, bits, probe, capacity, keep):
    import torch
    from paper_2602_01801_b200 import fastar
    g = torch.Generator().manual_seed(H * n)
    dtype, np_, frame = (torch.float32 if fp32 else torch.bfloat16), 70, n // 2
    lsh = np.random.default_rng(n).standard_normal((32, d)).astype(np.float32)
    host, dev = (fastar.Cache(H, d, capacity, 128, lsh, max_tokens=n, max_prompt_tokens=np_, max_frames=3, fp32=fp32, search_bits=bits) for _ in range(2))
    rand = lambda m: torch.randn(H, m, d, generator=g).to(dtype).pin_memory()
    kp, vp = rand(np_), rand(np_)
    k0 = rand(n)
    for step in range(2):
        # the second step finds most of the first one's keys again, appends a few and, where the cache is full, evicts
        k, v, q = (k0 if step == 0 else torch.where(torch.rand(H, n, 1, generator=g) < 0.9, k0, rand(n)).pin_memory()), rand(n), rand(n)
        sa, ca = torch.empty_like(q).pin_memory(), torch.empty_like(q).pin_memory()
        host.step_host(k, v, q, kp, vp, sa, ca, frame, 0.9, 128, keep, 20, probe=probe)
        dk, dv, dq = k.cuda(), v.cuda(), q.cuda()
        dev.update(dk, dv, frame, 0.9, probe=dq if probe else None)
        assert torch.equal(sa, dev.annsa(dq, 128, keep)["out"].cpu())
        assert torch.equal(ca, dev.annca(dq, kp.cuda(), vp.cuda(), frame, 20)["out"].cpu())
        assert host.status() == dev.status()
        a, b = host.export_state(), dev.export_state()
        assert all(np.array_equal(a[x], b[x]) for x in a)
    with pytest.raises(fastar.FastarError):
        host.step_host(k, v, q, kp, vp, sa, ca, frame, 0.9, 96, keep, 20)
    c = host.export_state()
    assert all(np.array_equal(a[x], c[x]) for x in a)          # refused before anything was queued


@pytest.mark.parametrize("H,n,d,fp32,probe,capacity,keep", [(20, 3111, 128, False, False, 6272, 5), (12, 4725, 128, False, False, 9600, 7),
                                                            (5, 5001, 128, True, True, 10112, 9), (3, 8201, 128, False, False, 8448, 67),
                                                            (11, 8201, 64, True, False, 16640, 3)])
def test_host_step_of_odd_numbers_of_tokens(H, n, d, fp32, probe, capacity, keep):
    """Slices that begin at odd heads of odd numbers of tokens, on both paths of the planner (up to 8192 tokens and above), odd numbers of kept
    blocks, and a last round that the device call may cut by key tiles and a slice may not: the cache bit for bit as by the device calls, the
    outputs against attention in 64 bits over what the device call selects."""
    import math

    import torch
    from paper_2602_01801_b200 import fastar
    g = torch.Generator().manual_seed(H * n)
    dtype, np_, frame, keep_prompt = (torch.float32 if fp32 else torch.bfloat16), 77, n // 2 + 1, 21
    lsh = np.random.default_rng(n).standard_normal((32, d)).astype(np.float32)
    host, dev = (fastar.Cache(H, d, capacity, 128, lsh, max_tokens=n, max_prompt_tokens=np_, max_frames=2, fp32=fp32) for _ in range(2))
    rand = lambda m: torch.randn(H, m, d, generator=g).to(dtype).pin_memory()
    kp, vp, k0 = rand(np_), rand(np_), rand(n)
    bf = lambda x: x.bfloat16().double()

    def check(got, q, k, v, bias):
        s = q @ k.transpose(-1, -2) / math.sqrt(d) + bias
        want = torch.softmax(s, -1) @ v
        # probabilities and output are rounded to bf16
        assert (got.double() - want).abs().max() <= 2.0 ** -7 * v.abs().max()
        assert (got.double() - want).norm() <= 1e-2 * want.norm()

    for step in range(2):
        k, v, q = (k0 if step == 0 else torch.where(torch.rand(H, n, 1, generator=g) < 0.9, k0, rand(n)).pin_memory()), rand(n), rand(n)
        sa, ca = torch.empty_like(q).pin_memory(), torch.empty_like(q).pin_memory()
        host.step_host(k, v, q, kp, vp, sa, ca, frame, 0.9, 128, keep, keep_prompt, probe=probe)
        dk, dv, dq, dkp, dvp = (x.cuda() for x in (k, v, q, kp, vp))
        dev.update(dk, dv, frame, 0.9, probe=dq if probe else None)
        assert host.status() == 0 and dev.status() == 0
        a, b = host.export_state(), dev.export_state()
        assert all(np.array_equal(a[x], b[x]) for x in a)
        r, c = dev.annsa(dq, 128, keep, debug=True), dev.annca(dq, dkp, dvp, frame, keep_prompt, debug=True)
        for h in range(H):
            keys, values = (torch.from_numpy(fastar.bits_to_f32(a[x][h])).cuda().double() for x in "kv")
            bias = torch.from_numpy(a["count"][h]).cuda().double().log()
            for blk in {0, n // 300, (n - 1) // 128}:
                rows = slice(blk * 128, min(n, blk * 128 + 128))
                at = torch.arange(capacity, device="cuda")
                if keep < capacity // 128:
                    at = (r["sel"][h, blk, : int(r["nsel"][h])].long()[:, None] * 128 + torch.arange(128, device="cuda")).reshape(-1)
                at = at[at < int(a["len"][h])]
                for got in (sa[h, rows].cuda(), r["out"][h, rows]):
                    check(got, bf(dq[h, rows]), keys[at], values[at], bias[at])
            for f in range(2):
                rows, sel = slice(f * frame, min(n, f * frame + 128)), c["sel"][h, f].long()
                for got in (ca[h, rows].cuda(), c["out"][h, rows]):
                    check(got, bf(dq[h, rows]), bf(dkp[h])[sel], bf(dvp[h])[sel], 0.0)
