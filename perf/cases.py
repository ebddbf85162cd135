"""What the speed of this library is measured on: the calls that an autoregressive video generator makes per layer.

Per generated chunk such a program runs TempCache's update, AnnSA over the cache and AnnCA over the prompt (a step);
while a chunk is being denoised it runs AnnSA over the cache and the chunk's own keys, and AnnCA, once per denoising
step; and it runs AnnSA alone where the cache is only read.  The sizes are those of the repository's own workloads
(`synth.py`): the tiny single-head step, the small ragged test case, the 12-head layer with 3 x 1560-token chunks, its
long rollout at the cache's capacity, the 40-head layer with 3 x 3600-token chunks and the length sweep.

Inputs follow the cluster / drift model of `synth.py`, drawn on the GPU: per-head centroids, a spatially coherent
cluster map that shifts by `shift` cells per frame, keys and queries = centroid + sigma * noise, a share `resample` of
every frame's tokens replaced by fresh vectors (they match nothing and are appended), prompt tokens of which `relevant`
per frame lie near the frame's most populous clusters.

A state holds `ring` consecutive chunks, and every pass takes the next one, as a rollout does.  After a whole round
the chunks come again: where the cache is large enough the fresh tokens of the first round are then found in it and
merged; `rollout_full` keeps a ring long enough that they have been evicted by then, so every pass appends and evicts.
"""
import math

import numpy as np
import torch

from paper_2602_01801_b200 import fastar

# kind:      step      update, AnnSA, AnnCA one after the other on the current stream
#            overlap   the same step with AnnCA and the query side of AnnSA's selector on a second stream
#            host      the same step through the host-tensor entry point
#            denoise   AnnSA over [cache, the chunk's own keys] and AnnCA; the cache is only read
#            attend    AnnSA alone; the cache is only read
# tokens of a frame = grid_h * grid_w, of a chunk = frames * that; cached = tokens appended un-merged before the first
# pass, warm = chunks merged after that (to fill the cache); keep >= capacity / block is dense attention
_BASE = dict(kind="step", heads=12, dim=128, grid_h=30, grid_w=52, frames=3, clusters=256, sigma=0.1, resample=0.1, shift=1.0,
             prompt=512, relevant=16, capacity=32768, block=128, keep=32, keep_prompt=64, cached=28080, warm=0, ring=4,
             search_bits=16, probe=False, fp32=False, tau=0.9)


def _case(name, **kw):
    return dict(_BASE, name=name, **kw)


def listed():
    return [
        # the smallest call: one head, 256 new tokens, fp32 tensors; latency and launches are everything
        _case("tiny_fp32", heads=1, dim=64, grid_h=16, grid_w=16, frames=1, clusters=32, prompt=32, relevant=4, capacity=1280, block=64,
              keep=4, keep_prompt=8, cached=1024, ring=8, fp32=True),
        # a small layer with ragged tails everywhere (600 tokens, 80 prompt tokens)
        _case("small_ragged", heads=2, grid_h=12, grid_w=25, frames=2, clusters=24, prompt=80, relevant=6, capacity=2048, keep=4,
              keep_prompt=24, cached=1200, ring=8),
        # frame-sequential update, one frame per call, the correspondence read off the queries (query probe)
        _case("frame_probe", frames=1, cached=14040, capacity=16384, keep=16, ring=8, probe=True),
        # head dimension 64: one point of the length sweep as a whole step
        _case("step_d64", heads=8, dim=64, grid_h=64, grid_w=64, frames=1, cached=16384, capacity=20480, keep=16),
        # the 12-head layer, the ordinary step
        _case("layer_step", ring=4),
        # the same layer with the 8-bit search, the method's default quantiser
        _case("layer_step_8bit", search_bits=8, ring=4),
        # long rollout at the cache's capacity: every pass evicts; AnnCA beside the update on a second stream
        _case("rollout_full", kind="overlap", sigma=0.05, resample=0.05, shift=0.5, warm=26, ring=140),
        # the same layer fed from and read back to host memory
        _case("layer_host", kind="host", ring=2),
        # one denoising step of the 12-head layer: the chunk's own 4680 keys are attended beside the cache
        _case("layer_denoise", kind="denoise", ring=2),
        # dense attention over a short cache (what early chunks and dense layers run)
        _case("dense_16k", kind="attend", heads=8, grid_h=64, grid_w=64, frames=1, cached=16384, capacity=16384, keep=128, ring=2),
        # block-sparse attention over the longest cache of the sweep, head dimension 64
        _case("sparse_128k_d64", kind="attend", heads=8, dim=64, grid_h=64, grid_w=64, frames=1, cached=131072, capacity=135168, keep=64,
              ring=2),
        # the largest: a 40-head layer, 10800 tokens against 64800 cached keys
        _case("world_step", heads=40, grid_h=45, grid_w=80, clusters=512, capacity=65536, keep_prompt=32, cached=64800, ring=3),
    ]


def _cost(c):
    """Multiply-adds of the search and the attention, the measure that keeps a drawn case below the largest listed one."""
    n = c["frames"] * c["grid_h"] * c["grid_w"]
    seg = n if c["kind"] == "denoise" else 0
    search = 0 if c["kind"] in ("denoise", "attend") else c["cached"]
    return c["heads"] * n * c["dim"] * (search + 2 * (min(c["cached"], c["keep"] * c["block"]) + seg))


def draw(rng):
    """One more case: the same kinds of call, sizes spread over the logarithm of their range."""
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    while True:
        kind = rng.choice(("step", "step", "step", "overlap", "host", "denoise", "attend", "attend"))
        block = rng.choice((128, 128, 128, 64))
        frames = rng.randint(1, 3)
        gh, gw = log(8, 64), log(16, 80)
        n = frames * gh * gw
        cached = log(1024, 131072 if kind == "attend" else 65536)
        capacity = -(-max(cached + rng.randint(0, 4096), n + 256) // 128) * 128
        nblk = -(-cached // block)
        prompt = log(32, 512)
        small = cached <= 8192
        c = dict(_BASE, kind=kind, heads=log(1, 40), dim=rng.choice((64, 128, 128)), grid_h=gh, grid_w=gw, frames=frames,
                 clusters=log(24, 512), sigma=rng.choice((0.05, 0.1)), resample=rng.choice((0.05, 0.1)), shift=rng.choice((0.5, 1.0)),
                 prompt=prompt, relevant=max(1, min(16, prompt // (4 * frames))), capacity=capacity, block=block,
                 keep=max(1, nblk // rng.choice((4, 8, 16, 32))) if rng.random() < 0.85 else capacity // block,
                 keep_prompt=max(1, prompt // rng.choice((4, 8, 16))), cached=cached, ring=3,
                 search_bits=rng.choice((16, 16, 8)), probe=kind == "step" and rng.random() < 0.2, fp32=small and rng.random() < 0.3,
                 warm=0)
        if n <= 10800 and _cost(c) <= _cost(listed()[-1]) and c["heads"] * capacity <= 40 * 65536:
            return c


class _Video:
    """The cluster / drift model on the GPU, seeded."""

    def __init__(self, c, seed):
        self.c = c
        self.dev = torch.device("cuda", torch.cuda.current_device())
        self.g = torch.Generator(device=self.dev).manual_seed(int(seed))
        self.dtype = torch.float32 if c["fp32"] else torch.bfloat16
        H, C, d, gh, gw = c["heads"], c["clusters"], c["dim"], c["grid_h"], c["grid_w"]
        self.centroids = self._normal(H, C, d)
        y = torch.rand(C, generator=self.g, device=self.dev) * gh
        x = torch.rand(C, generator=self.g, device=self.dev) * gw
        dy = (torch.arange(gh, device=self.dev)[:, None, None] + 0.5 - y).abs()
        dx = (torch.arange(gw, device=self.dev)[None, :, None] + 0.5 - x).abs()
        self.map0 = (torch.minimum(dy, gh - dy) ** 2 + torch.minimum(dx, gw - dx) ** 2).argmin(-1)

    def _normal(self, *shape):
        return torch.randn(*shape, generator=self.g, device=self.dev)

    def frame_map(self, t):
        return torch.roll(self.map0, int(self.c["shift"] * t), dims=1).reshape(-1)

    def chunk(self, i):
        """(q, k, v) of chunk i, each [heads][tokens][dim]."""
        c, f = self.c, self.c["frames"]
        m = torch.cat([self.frame_map(i * f + t) for t in range(f)])
        base = self.centroids[:, m]
        k = base + c["sigma"] * self._normal(*base.shape)
        q = base + c["sigma"] * self._normal(*base.shape)
        fresh = torch.rand(base.shape[:2], generator=self.g, device=self.dev)[..., None] < c["resample"]
        new = self._normal(*base.shape)
        k = torch.where(fresh, new, k)
        q = torch.where(fresh, new + c["sigma"] * self._normal(*base.shape), q)
        v = self._normal(*base.shape)
        return tuple(x.to(self.dtype) for x in (q, k, v))

    def prompt(self):
        """(k_prompt, v_prompt): random tokens, `relevant` per frame near the frame's most populous clusters."""
        c = self.c
        kp, vp = self._normal(c["heads"], c["prompt"], c["dim"]), self._normal(c["heads"], c["prompt"], c["dim"])
        pos = torch.randperm(c["prompt"], generator=self.g, device=self.dev)
        for f in range(c["frames"]):
            top = torch.bincount(self.frame_map(f), minlength=c["clusters"]).argsort(descending=True)[: c["relevant"]]
            at = pos[f * c["relevant"]: f * c["relevant"] + len(top)]
            kp[:, at] = 0.8 * self.centroids[:, top] + 0.6 * kp[:, at]
        return kp.to(self.dtype), vp.to(self.dtype)


def prepare(case, seed):
    c = case
    video = _Video(c, seed)
    n = c["frames"] * c["grid_h"] * c["grid_w"]
    lsh = np.random.default_rng(seed).standard_normal((32, c["dim"])).astype(np.float32)
    cache = fastar.Cache(c["heads"], c["dim"], c["capacity"], c["block"], lsh, max_tokens=n, max_prompt_tokens=c["prompt"],
                         max_frames=c["frames"], fp32=c["fp32"], search_bits=c["search_bits"])
    frame_len = c["grid_h"] * c["grid_w"]
    left, i = c["cached"], 0
    while left > 0:                              # the history, appended un-merged (a threshold above 1 merges nothing)
        _, k, v = video.chunk(i)
        m = min(left, n)
        cache.update(k[:, :m], v[:, :m], frame_len, 2.0, outputs=False)
        left, i = left - m, i + 1
    chunks = []
    for j in range(max(c["ring"], c["warm"])):
        chunks.append(video.chunk(i + j))
        if j < c["warm"]:
            cache.update(chunks[j][1], chunks[j][2], frame_len, c["tau"], outputs=False)
    kp, vp = video.prompt()
    s = dict(case=c, cache=cache, chunks=chunks[: c["ring"]], at=c["warm"] % c["ring"], kp=kp, vp=vp, frame_len=frame_len)
    if c["kind"] == "overlap":
        q = chunks[0][0]
        s.update(side=torch.cuda.Stream(device=q.device), sa=torch.empty_like(q), ca=torch.empty_like(q))
    if c["kind"] == "host":
        s["chunks"] = [tuple(x.cpu().pin_memory() for x in t) for t in s["chunks"]]
        s.update(kp=kp.cpu().pin_memory(), vp=vp.cpu().pin_memory(), sa=torch.empty_like(s["chunks"][0][0]).pin_memory(),
                 ca=torch.empty_like(s["chunks"][0][0]).pin_memory())
    if cache.status() != fastar.OK:
        raise RuntimeError("building the cache failed")
    return s


def run(state):
    s = state
    c, cache, fl = s["case"], s["cache"], s["frame_len"]
    q, k, v = s["chunks"][s["at"]]
    s["at"] = (s["at"] + 1) % len(s["chunks"])
    kind = c["kind"]
    if kind == "attend":
        return cache.annsa(q, c["block"], c["keep"])["out"]
    if kind == "denoise":
        sa = cache.annsa_segment(q, k, v, c["block"], c["keep"])["out"]
        return sa, cache.annca(q, s["kp"], s["vp"], fl, c["keep_prompt"])["out"]
    if kind == "host":
        cache.step_host(k, v, q, s["kp"], s["vp"], s["sa"], s["ca"], fl, c["tau"], c["block"], c["keep"], c["keep_prompt"])
        return s["sa"], s["ca"]
    if kind == "overlap":
        main, side = torch.cuda.current_stream(), s["side"]
        side.wait_stream(main)
        with torch.cuda.stream(side):
            cache.annsa_prepare(q, c["block"])
            prepared = side.record_event()
            cache.annca(q, s["kp"], s["vp"], fl, c["keep_prompt"], out=s["ca"])
        res = cache.update(k, v, fl, c["tau"])
        main.wait_event(prepared)
        cache.annsa(q, c["block"], c["keep"], out=s["sa"])
        main.wait_stream(side)
        return dict(res, sa=s["sa"], ca=s["ca"])
    res = cache.update(k, v, fl, c["tau"], probe=q if c["probe"] else None)
    sa = cache.annsa(q, c["block"], c["keep"])["out"]
    ca = cache.annca(q, s["kp"], s["vp"], fl, c["keep_prompt"])["out"]
    return dict(res, sa=sa, ca=ca)


def work(case):
    """Per pass.  Search: every new key against every cached one; AnnSA: every query against its kept keys (and the
    segment); AnnCA: relevance of every prompt token, attention over the kept ones.  Bytes: tensors in and out once, the
    cached keys once for the search, the cached keys and values that attention can reach once, merged rows once."""
    c = case
    H, d, n = c["heads"], c["dim"], c["frames"] * c["grid_h"] * c["grid_w"]
    L, kept = c["cached"], min(c["cached"], c["keep"] * c["block"])
    esz = 4 if c["fp32"] else 2
    nblocks = -(-n // c["block"])
    reach = min(L, nblocks * kept)
    flops = 4.0 * n * kept * d
    nbytes = 2.0 * n * d * esz + 2.0 * reach * d * 2
    if c["kind"] == "denoise":
        flops += 4.0 * n * n * d
        nbytes += 2.0 * n * d * esz
    if c["kind"] != "attend":
        flops += 2.0 * n * c["prompt"] * d + 4.0 * n * min(c["prompt"], c["keep_prompt"]) * d
        nbytes += 2.0 * n * d * esz + 2.0 * c["prompt"] * d * esz
    if c["kind"] in ("step", "overlap", "host"):
        flops += 2.0 * n * L * d
        nbytes += 2.0 * n * d * esz + L * d * (1 if c["search_bits"] == 8 else 2) + 4.0 * n * d * 2
    return {"bytes": H * nbytes, "flops": H * flops}


def tolerance(case):
    """Against the same attention in 64 bits the outputs are off by 0.0022 (probabilities and output rounded to bf16, fp32
    accumulation), single values by 0.015 of the root mean square; of the slots found, 0.0002 differ from a 64-bit search
    (similarities that agree to fp32 rounding).  Four times that."""
    return {"rel": 0.009, "max": 0.06, "differ": 0.001}
