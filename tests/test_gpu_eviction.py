"""Eviction order against a sort by (stamp, slot): caches up to and beyond what the planner keeps in registers, ages of more than 16
bits, sinks, one victim and the largest chunk, a chunk that does not fit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("capacity,free,n,sink,stamps,now", [(128, 0, 1, 0, 5, 9), (1024, 100, 700, 16, 3, 4), (16512, 0, 16384, 128, 40, 41),
                                                             (32768, 1, 300, 0, 200, 201), (32896, 0, 513, 7, 2, 3),
                                                             (2048, 0, 1024, 0, 100000, 100001), (2048, 0, 2000, 100, 6, 6)])
def test_oldest_slots_are_evicted(capacity, free, n, sink, stamps, now):
    from paper_2602_01801_b200 import fastar
    rng = np.random.default_rng(capacity + n)
    H, d = 2, 64
    length = capacity - free
    cache = fastar.Cache(H, d, capacity, 64, rng.standard_normal((32, d)).astype(np.float32), max_tokens=n, n_sink=sink)
    bits = fastar.bf16_bits(rng.standard_normal((H, length, d)).astype(np.float32))
    stamp = rng.integers(0, stamps, (H, length)).astype(np.int32)
    cache.import_state(bits, bits, np.array([length, length]), np.ones((H, length), np.int32), stamp, now=now)
    new = fastar.to_device(rng.standard_normal((H, n, d)).astype(np.float32))
    r = cache.update(new, new, n, 2.0)                       # a threshold above 1: nothing is merged
    appended = min(free, n)
    for h in range(H):
        slots = np.arange(length)
        may = slots[(slots >= sink) & (stamp[h] < now)]
        dest = r["dest"][h].cpu().numpy()
        if len(may) < n - appended:
            assert (dest == -1).all()
            continue
        victims = may[np.lexsort((may, stamp[h][may]))][: n - appended]
        assert np.array_equal(dest, np.concatenate([length + np.arange(appended), victims]))
    assert (cache.status() == fastar.OK) == bool((r["stats"][:, 6] == 1).all())
