"""The decode step at the edges of its tiles (64 tokens), of a warp's share of a tile (16) and of
a CTA's range, over the cluster sizes the planner takes, against the oracle. Some key rows overflow:
their logits are far below (or -inf in fp32), a whole warp's tokens among them, and weigh nothing. In
fp32 every padding of the group, and a range too long for the roomier of the kernel's two layouts. Units
longer than the launch's bound are skipped and left as they are, whatever the length seen beforehand."""
import math

import numpy as np
import pytest
import torch

import oracle
from gpu_harness import SCORE_ATOL, SCORE_RTOL
from paper_2608_08569_gb300 import (DEV_LEN_HINT, CacheDesc, allocate_cache, allocate_paged_cache,
                                    voxzip_anchor_fuse, voxzip_anchor_fuse_paged, voxzip_decode_step,
                                    voxzip_decode_step_paged, voxzip_get_status)

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_08569_gb300 import build
    build.build_library()
    oracle.build()
    voxzip_get_status()


EDGES = [0, 1, 14, 15, 16, 17, 31, 32, 47, 48, 62, 63, 64, 65, 126, 127, 128, 129, 255, 256, 511, 512, 1023, 2047, 2049]


@pytest.mark.parametrize("D,Hq,Hkv", [(128, 32, 4), (64, 16, 1), (128, 16, 1)])
@pytest.mark.parametrize("capacity", [66, 520, 2100])
@pytest.mark.parametrize("low_rows", [False, True])
def test_decode_edges(D, Hq, Hkv, capacity, low_rows):
    _check(torch.bfloat16, D, Hq, Hkv, capacity, sorted({min(e, capacity - 1) for e in EDGES}), low_rows, 2e-2)


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("G", [1, 2, 3, 4, 7, 8, 9, 16])
@pytest.mark.parametrize("capacity", [66, 2100])
def test_decode_edges_fp32(D, G, capacity):
    _check(torch.float32, D, 2 * G, 2, capacity, sorted({min(e, capacity - 1) for e in EDGES}), capacity == 66, 1e-4)


@pytest.mark.parametrize("G,n", [(16, 50000), (9, 55000), (1, 300001)])
def test_decode_long_fp32(G, n):
    _check(torch.float32, 64, G, 1, n + 5, [n], False, 1e-4)


@pytest.mark.parametrize("paged", [False, True])
@pytest.mark.parametrize("n", [640, 2333])
def test_decode_many_units(paged, n):
    """768 units of ragged lengths: clusters in several rounds, each asking L2 for a later one's rows.
    Against the same arithmetic in fp64 on the device."""
    B, L, Hq, H, D, dt = 4, 48, 32, 4, 128, torch.bfloat16
    C = (n + 64) // 64 * 64
    desc = CacheDesc(B, L, Hq, H, D, C, dt)
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    lens = torch.randint(1, n + 1, (B, L, H), generator=g, device="cuda", dtype=torch.int32)
    lens[0], lens[1, :, :2], lens[2, 5] = n, n - 63, 0
    k, v = (torch.randn(B, L, H, C, D, generator=g, device="cuda").to(dt) for _ in range(2))
    score = torch.rand(B, L, H, C, generator=g, device="cuda")
    before = score.clone()
    pos = torch.zeros(B, L, H, C, dtype=torch.int32, device="cuda")
    q = torch.randn(L, B, Hq, D, generator=g, device="cuda").to(dt)
    kn, vn = (torch.randn(L, B, H, D, generator=g, device="cuda").to(dt) for _ in range(2))
    npos, out, ln = torch.full((B,), 9, dtype=torch.int32, device="cuda"), torch.empty_like(q), lens.clone()
    if paged:
        pages = B * L * H * (C // 64)
        order = torch.randperm(pages, generator=g, device="cuda")
        pc = allocate_paged_cache(desc, pages)
        pc["k_pool"][order], pc["v_pool"][order] = k.view(pages, 64, D), v.view(pages, 64, D)
        pc["page_table"].copy_(order.view(pc["page_table"].shape))
        pc["free_count"].zero_()
        pc.update(score=score, pos=pos, len=ln)
        voxzip_decode_step_paged(desc, pc, 0, L, q, kn, vn, npos, 0.99, out, max_len=n + 1)
    else:
        voxzip_decode_step(desc, 0, L, q, kn, vn, npos, k, v, score, pos, ln, 0.99, out, max_len=n + 1)
    assert voxzip_get_status() == 0
    assert torch.equal(ln, lens + 1)
    slot = torch.arange(C, device="cuda")
    for l in range(L):
        m = lens[:, l].long()
        at = m[..., None, None].expand(B, H, 1, D)
        kl = k[:, l].double().scatter(2, at, kn[l].double()[:, :, None])
        vl = v[:, l].double().scatter(2, at, vn[l].double()[:, :, None])
        x = q[l].double().view(B, H, Hq // H, D) @ kl.transpose(-1, -2) / math.sqrt(D)
        p = torch.softmax(x.masked_fill((slot > m[..., None])[:, :, None], -math.inf), -1)
        assert ((p @ vl).reshape(B, Hq, D) - out[l].double()).abs().max() <= 2e-2
        old = before[:, l].double().masked_fill(slot == m[..., None], 0.0)
        want = torch.where(slot <= m[..., None], 0.99 * old + p.sum(2), before[:, l].double())
        torch.testing.assert_close(score[:, l].double(), want, rtol=SCORE_RTOL, atol=SCORE_ATOL)


def _cache(desc, paged):
    """An empty cache, and a function that gives its K or V rows as [B][L][Hkv][C][D]."""
    if not paged:
        c = allocate_cache(desc)
        return c, lambda x: c[x]
    units, mp = desc.batch * desc.layers * desc.kv_heads, desc.capacity // 64
    c = allocate_paged_cache(desc, units * mp)
    return c, lambda x: c[x + "_pool"][c["page_table"].long().clamp(min=0)].reshape(
        desc.batch, desc.layers, desc.kv_heads, desc.capacity, desc.head_dim)


def _step(desc, c, paged, q, kn, vn, npos, out, max_len):
    if paged:
        voxzip_decode_step_paged(desc, c, 0, desc.layers, q, kn, vn, npos, 0.99, out, max_len=max_len)
    else:
        voxzip_decode_step(desc, 0, desc.layers, q, kn, vn, npos, c["k"], c["v"], c["score"], c["pos"], c["len"], 0.99,
                           out, max_len=max_len)


def _unit_against_oracle(u, q, kn, vn, out, score, K, n):
    f = lambda t: t.to("cpu", torch.float64).numpy()
    o = oracle.decode_step(u, f(q), f(kn), f(vn), 70000, 0.99, 1 / math.sqrt(q.shape[-1]))
    assert np.abs(f(out) - o).max() <= 2e-2, n
    np.testing.assert_allclose(f(score[:n + 1]), u.score[:n + 1], rtol=SCORE_RTOL, atol=SCORE_ATOL)
    np.testing.assert_array_equal(f(K[:n + 1]), u.K[:n + 1])


@pytest.mark.parametrize("paged", [False, True])
@pytest.mark.parametrize("D,G", [(128, 8), (64, 16)])
@pytest.mark.parametrize("bound,short,long", [(130, [0, 63, 64, 100, 129], [400, 1000, 4100]), (64, [1, 62], [45000])])
def test_units_above_the_bound_are_skipped(paged, D, G, bound, short, long):
    """max_len below the length of some units, by a few tiles and by hundreds: those keep their length,
    rows, positions and scores, the status word says so and nothing else, and the others take the step."""
    lens, H, dt = [x for p in zip(short, long) for x in p] + short[len(long):], 2, torch.bfloat16
    B, C = len(lens), (max(lens) + 128) // 64 * 64
    desc = CacheDesc(B, 1, G * H, H, D, C, dt)
    g = torch.Generator(device="cuda")
    g.manual_seed(D + bound)
    c, rows = _cache(desc, paged)
    if paged:  # every unit holds all its pages
        c["page_table"].copy_(torch.randperm(c["pages"], generator=g, device="cuda").view(c["page_table"].shape))
        c["free_count"].zero_()
    for x in ("k_pool", "v_pool") if paged else ("k", "v"):
        c[x].normal_(generator=g)
    c["score"].uniform_(generator=g)
    c["pos"].copy_(torch.arange(C, dtype=torch.int32, device="cuda"))
    c["len"].copy_(torch.tensor(lens, dtype=torch.int32, device="cuda")[:, None, None].expand(B, 1, H))
    before = {x: rows(x).clone() for x in ("k", "v")} | {x: c[x].clone() for x in ("score", "pos", "len")}
    q = torch.randn(1, B, G * H, D, generator=g, device="cuda").to(dt)
    kn, vn = (torch.randn(1, B, H, D, generator=g, device="cuda").to(dt) for _ in range(2))
    out = torch.empty_like(q)
    _step(desc, c, paged, q, kn, vn, torch.full((B,), 70000, dtype=torch.int32, device="cuda"), out, bound)
    assert voxzip_get_status() == DEV_LEN_HINT
    after = {x: rows(x) for x in ("k", "v")}
    f = lambda t: t.to("cpu", torch.float64).numpy()
    for b, n in enumerate(lens):
        if n in long:
            assert torch.equal(c["len"][b], before["len"][b])
            for x, y in ((c["score"], "score"), (c["pos"], "pos"), (after["k"], "k"), (after["v"], "v")):
                assert torch.equal(x[b], before[y][b])
            continue
        assert (c["len"][b] == n + 1).all()
        for h in range(H):
            u = oracle.UnitCache.from_rows(C, f(before["k"][b, 0, h, :n]), f(before["v"][b, 0, h, :n]),
                                           before["pos"][b, 0, h, :n].cpu().numpy(), f(before["score"][b, 0, h, :n]))
            _unit_against_oracle(u, q[0, b, h * G:(h + 1) * G], kn[0, b, h], vn[0, b, h],
                                 out[0, b, h * G:(h + 1) * G], c["score"][b, 0, h], after["k"][b, 0, h], n)


@pytest.mark.parametrize("paged", [False, True])
def test_a_short_prompt_after_a_long_one(paged):
    """Stage 1 of a long prompt, a step, stage 1 of a short prompt and a step bounded by it, back to back:
    whatever length the last launch has seen before it waited, it works on the short prompt's."""
    B, H, G, D, dt, long, short = 2, 2, 8, 128, torch.bfloat16, 20000, 40
    C = (long + 128) // 64 * 64
    desc = CacheDesc(B, 1, G * H, H, D, C, dt)
    g = torch.Generator(device="cuda")
    g.manual_seed(9)
    c, rows = _cache(desc, paged)
    q = torch.randn(2, 1, B, G * H, D, generator=g, device="cuda").to(dt)
    kn, vn = (torch.randn(2, 1, B, H, D, generator=g, device="cuda").to(dt) for _ in range(2))
    npos, out = torch.full((B,), 70000, dtype=torch.int32, device="cuda"), torch.empty_like(q)
    i32 = lambda x: torch.tensor(x, dtype=torch.int32, device="cuda")
    kv = [[torch.randn(B, 1, H, n, D, generator=g, device="cuda").to(dt) for _ in range(2)] for n in (long, short)]
    ints = [(i32([n] * B), i32([0] * B), i32([0] * B), i32([0] * (B + 1)), i32([]), i32([]), i32([]))
            for n in (long, short)]
    torch.cuda.synchronize()
    for t, n in enumerate((long, short)):
        if paged:
            voxzip_anchor_fuse_paged(desc, c, *kv[t], *ints[t])
        else:
            voxzip_anchor_fuse(desc, *kv[t], *ints[t], c["k"], c["v"], c["score"], c["pos"], c["len"])
        _step(desc, c, paged, q[t], kn[t], vn[t], npos, out[t], n + 1)
    assert voxzip_get_status() == 0
    assert (c["len"] == short + 1).all()
    f = lambda t: t.to("cpu", torch.float64).numpy()
    for b in range(B):
        for h in range(H):
            u = oracle.UnitCache.from_rows(C, f(kv[1][0][b, 0, h]), f(kv[1][1][b, 0, h]), np.arange(short, dtype=np.int32),
                                           np.zeros(short))
            _unit_against_oracle(u, q[1, 0, b, h * G:(h + 1) * G], kn[1, 0, b, h], vn[1, 0, b, h],
                                 out[1, 0, b, h * G:(h + 1) * G], c["score"][b, 0, h], rows("k")[b, 0, h], short)


def _check(dt, D, Hq, Hkv, capacity, lens, low_rows, tol):
    B, G = len(lens), Hq // Hkv
    desc = CacheDesc(B, 1, Hq, Hkv, D, capacity, dt)
    g = torch.Generator(device="cuda")
    g.manual_seed(capacity + D)
    c = allocate_cache(desc)
    for x in ("k", "v"):
        c[x].normal_(generator=g)
    c["score"].uniform_(generator=g)
    c["pos"].copy_(torch.arange(capacity, dtype=torch.int32, device="cuda"))
    q = torch.randn(1, B, Hq, D, generator=g, device="cuda").to(dt)
    if low_rows:  # logits of about -1e38 (finite) and below the fp32 range, 16 to 31 whole warps' worth
        q[..., 0] = 4.0
        c["k"][:, :, :, 16:32, 0] = -3e38
        c["k"][:, :, :, 40:52, 0] = -3e38
        c["k"][:, :, :, 96:128, 0] = -1e37
    kn, vn = (torch.randn(1, B, Hkv, D, generator=g, device="cuda").to(dt) for _ in range(2))
    c["len"].copy_(torch.tensor(lens, dtype=torch.int32, device="cuda")[:, None, None].expand(B, 1, Hkv))
    before = {x: y.clone() for x, y in c.items()}
    npos = torch.full((B,), 70000, dtype=torch.int32, device="cuda")
    out = torch.empty_like(q)
    voxzip_decode_step(desc, 0, 1, q, kn, vn, npos, c["k"], c["v"], c["score"], c["pos"], c["len"], 0.99, out)
    assert voxzip_get_status() == 0
    f = lambda t: t.to("cpu", torch.float64).numpy()
    for b, n in enumerate(lens):
        for h in range(Hkv):
            u = oracle.UnitCache.from_rows(capacity, f(before["k"][b, 0, h, :n]), f(before["v"][b, 0, h, :n]),
                                           before["pos"][b, 0, h, :n].cpu().numpy(), f(before["score"][b, 0, h, :n]))
            o = oracle.decode_step(u, f(q[0, b, h * G:(h + 1) * G]), f(kn[0, b, h]), f(vn[0, b, h]), 70000, 0.99,
                                   1 / math.sqrt(D))
            assert np.abs(f(out[0, b, h * G:(h + 1) * G]) - o).max() <= tol, (n, h)
            np.testing.assert_allclose(f(c["score"][b, 0, h, :n + 1]), u.score[:n + 1], rtol=SCORE_RTOL,
                                       atol=SCORE_ATOL)
            np.testing.assert_array_equal(f(c["k"][b, 0, h, :n + 1]), u.K[:n + 1])
            assert int(c["len"][b, 0, h]) == n + 1
            assert torch.equal(c["score"][b, 0, h, n + 1:], before["score"][b, 0, h, n + 1:])
