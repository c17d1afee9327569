"""The decode step at the edges of its tiles (64 tokens), of a warp's share of a tile (16) and of
a CTA's range, over the cluster sizes the planner takes, against the oracle. Some key rows overflow:
their logits are far below (or -inf in fp32), a whole warp's tokens among them, and weigh nothing. In
fp32 every padding of the group, and a range too long for the roomier of the kernel's two layouts."""
import math

import numpy as np
import pytest
import torch

import oracle
from gpu_harness import SCORE_ATOL, SCORE_RTOL
from paper_2608_08569_gb300 import (CacheDesc, allocate_cache, allocate_paged_cache, voxzip_decode_step,
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
