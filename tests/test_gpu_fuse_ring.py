"""Stage 1 at the edges of its kernels: spans shorter than, equal to and many times a ring stage,
runs of output rows around a work item's, embedding widths around the column ranges of a row, short, empty
and skipped sequences beside long ones. Rows, positions, slot maps and lengths are the oracle's bit for bit. A ring
whose waits give up leaves every unit that it did not finish empty."""
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

import oracle
from paper_2608_08569_gb300 import (DEV_BAD_SPANS, CacheDesc, EmbedDesc, allocate_cache, allocate_paged_cache,
                                    voxzip_anchor_fuse, voxzip_anchor_fuse_paged, voxzip_embed_fuse,
                                    voxzip_get_status)

pytestmark = pytest.mark.gpu

TEXT = 5   # text tokens before the audio


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_08569_gb300 import build
    build.build_library()
    oracle.build()
    voxzip_get_status()


def _sequence(kind, rng):
    """(in_len, audio_len, spans) with spans as (start, end, groups) in prompt tokens."""
    if kind == "empty":
        return 0, 0, []
    if kind == "bad":            # spans out of order: the sequence is skipped
        return 60, 40, [(20, 30, 1), (10, 15, 1)]
    if kind == "one":
        return TEXT + 1, 1, [(TEXT, TEXT + 1, 3)]
    if kind == "copied":         # no span: every row is copied
        return TEXT + 64, 60, []
    lens = {"small": [1, 2, 3, 4, 5, 7, 8, 9, 15, 16, 17], "long": [33, 1, 200, 64, 31, 96, 1000],
            "random": list(rng.integers(1, 13, 150))}[kind]
    t, spans = TEXT, []
    for l in lens:
        t += int(rng.integers(0, 3))                      # now and then a gap of background
        spans.append((t, t + int(l), int(rng.integers(1, 4))))
        t += int(l)
    return t + 9, t + 2 - TEXT, spans


KINDS = ["small", "empty", "long", "one", "bad", "random", "copied"]


def _batch(rng):
    seqs = [_sequence(k, rng) for k in KINDS]
    off = np.cumsum([0] + [len(s[2]) for s in seqs])
    flat = np.array([x for s in seqs for x in s[2]], np.int32).reshape(-1, 3)
    i32 = lambda x: torch.as_tensor(np.asarray(x), dtype=torch.int32, device="cuda")
    ints = (i32([s[0] for s in seqs]), i32([min(TEXT, s[0]) for s in seqs]), i32([s[1] for s in seqs]), i32(off),
            i32(flat[:, 0].copy()), i32(flat[:, 1].copy()), i32(flat[:, 2].copy()))
    return seqs, ints, max(s[0] for s in seqs) + 3, max(sum(x[2] for x in s[2]) for s in seqs)


def _expect(seq, x, anchor, bf16, capacity, keep=True):
    s, e, g = (np.array([y[i] for y in seq[2]], np.int32) for i in range(3))
    f = lambda t: t.double().cpu().numpy()
    return oracle.stage1(f(x[:seq[0]]), seq[0], min(TEXT, seq[0]), seq[1], s, e, g,
                         anchor=None if anchor is None else f(anchor), cache_is_bf16=bf16, capacity=capacity,
                         keep_background=keep)


@pytest.mark.parametrize("dtype,D", [(torch.bfloat16, 128), (torch.float32, 128), (torch.float32, 64),
                                     (torch.bfloat16, 64)])
@pytest.mark.parametrize("anchors", [False, True])
@pytest.mark.parametrize("paged", [False, True])
def test_rows(dtype, D, anchors, paged):
    seqs, ints, stride, A = _batch(np.random.default_rng(7))
    B, L, H, C = len(seqs), 2, 3, (stride + 63) // 64 * 64
    desc = CacheDesc(B, L, 2 * H, H, D, C, dtype)
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    rnd = lambda n: torch.randn(B, L, H, n, D, generator=g, device="cuda").to(dtype)
    k, v = rnd(stride), rnd(stride)
    ak, av = (rnd(A), rnd(A)) if anchors else (None, None)
    smap = torch.full((B, stride), -7, dtype=torch.int32, device="cuda")
    if paged:
        c = allocate_paged_cache(desc, B * L * H * (C // 64 + 1))
        voxzip_anchor_fuse_paged(desc, c, k, v, *ints, slot_map=smap, anchor_k=ak, anchor_v=av)
        table = c["page_table"].long().clamp(min=0)
        kc, vc = (c[x][table].reshape(B, L, H, C, D) for x in ("k_pool", "v_pool"))
    else:
        c = allocate_cache(desc)
        voxzip_anchor_fuse(desc, k, v, *ints, c["k"], c["v"], c["score"], c["pos"], c["len"], slot_map=smap,
                           anchor_k=ak, anchor_v=av)
        kc, vc = c["k"], c["v"]
    assert voxzip_get_status() == DEV_BAD_SPANS
    for b, seq in enumerate(seqs):
        for l in range(L):
            for h in range(H):
                if KINDS[b] in ("bad", "empty"):
                    assert int(c["len"][b, l, h]) == 0
                    continue
                for x, a, y in ((k, ak, kc), (v, av, vc)):
                    r = _expect(seq, x[b, l, h], None if a is None else a[b, l, h], dtype == torch.bfloat16, C)
                    n = r["n"]
                    assert int(c["len"][b, l, h]) == n
                    np.testing.assert_array_equal(y[b, l, h, :n].double().cpu().numpy(), r["stored"])
                np.testing.assert_array_equal(c["pos"][b, l, h, :n].cpu().numpy(), r["pos"])
                assert not c["score"][b, l, h].any()
                if not paged:
                    assert not y[b, l, h, n:].any()


@pytest.mark.parametrize("dtype,width", [(torch.bfloat16, w) for w in (248, 256, 264, 504, 512, 1000, 1024, 1032, 2048,
                                                                       2056, 4096, 4608)] +
                         [(torch.float32, w) for w in (124, 128, 260, 1028, 2048)])
@pytest.mark.parametrize("text,keep", [(True, True), (False, True), (True, False)])
def test_embedding_rows(dtype, width, text, keep):
    seqs, ints, stride, A = _batch(np.random.default_rng(11))
    B, C = len(seqs), stride
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    e_in = torch.randn(B, stride, width, generator=g, device="cuda").to(dtype)
    e_text = torch.randn(B, A, width, generator=g, device="cuda").to(dtype) if text else None
    out = torch.zeros(B, C, width, dtype=dtype, device="cuda")
    pos = torch.full((B, C), -7, dtype=torch.int32, device="cuda")
    ln = torch.full((B,), -7, dtype=torch.int32, device="cuda")
    voxzip_embed_fuse(EmbedDesc(B, width, C, dtype), e_in, *ints, out, pos, ln, e_text=e_text, keep_background=keep)
    assert voxzip_get_status() == DEV_BAD_SPANS
    for b, seq in enumerate(seqs):
        if KINDS[b] in ("bad", "empty"):
            assert int(ln[b]) == 0 and not out[b].any()
            continue
        r = _expect(seq, e_in[b], e_text[b] if text else None, dtype == torch.bfloat16, C, keep)
        n = r["n"]
        assert int(ln[b]) == n
        np.testing.assert_array_equal(out[b, :n].double().cpu().numpy(), r["stored"])
        np.testing.assert_array_equal(pos[b, :n].cpu().numpy(), r["pos"])
        assert not out[b, n:].any() and (pos[b, n:] == -7).all()


@pytest.mark.parametrize("paged", [False, True])
@pytest.mark.parametrize("host", ["k", "v"])
def test_only_one_of_the_two_prefills_in_host_memory(paged, host):
    """K in pinned host memory and V on the device, or the other way round: the same rows."""
    seqs, ints, stride, _ = _batch(np.random.default_rng(17))
    B, L, H, D, C = len(seqs), 1, 2, 128, (stride + 63) // 64 * 64
    desc = CacheDesc(B, L, 2 * H, H, D, C, torch.bfloat16)
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    dev = [torch.randn(B, L, H, stride, D, generator=g, device="cuda").bfloat16() for _ in range(2)]
    mixed = [x.cpu().pin_memory() if y == host else x for x, y in zip(dev, "kv")]
    got = []
    for k, v in (dev, mixed):
        if paged:
            c = allocate_paged_cache(desc, B * L * H * (C // 64 + 1))
            voxzip_anchor_fuse_paged(desc, c, k, v, *ints, workspace=torch.empty(1 << 22, dtype=torch.uint8, device="cuda"))
            table = c["page_table"].long().clamp(min=0)
            rows = [c[x][table].reshape(B, L, H, C, D) for x in ("k_pool", "v_pool")]
        else:
            c = allocate_cache(desc)
            voxzip_anchor_fuse(desc, k, v, *ints, c["k"], c["v"], c["score"], c["pos"], c["len"])
            rows = [c["k"], c["v"]]
        assert voxzip_get_status() == DEV_BAD_SPANS
        got.append((c["len"], c["pos"], rows))
    (la, pa, ra), (lb, pb, rb) = got
    assert torch.equal(la, lb) and la.any()
    for b in range(B):
        n = int(la[b, 0, 0])
        assert torch.equal(pa[b, ..., :n], pb[b, ..., :n])
        for x, y in zip(ra, rb):
            assert torch.equal(x[b, :, :, :n], y[b, :, :, :n])


GIVES_UP = """
import sys
import torch
import paper_2608_08569_gb300._native as N
N.LIB_PATH = sys.argv[1]
from paper_2608_08569_gb300 import (DEV_TIMEOUT, CacheDesc, allocate_cache, allocate_paged_cache, voxzip_anchor_fuse,
                                    voxzip_anchor_fuse_paged, voxzip_get_status)
i32 = lambda x: torch.tensor(x, dtype=torch.int32, device="cuda")
B, L, H, n, D = 2, 3, 2, 5000, 128
ints = (i32([n, 40]), i32([0, 0]), i32([0, 0]), i32([0, 0, 0]), i32([]), i32([]), i32([]))
for dtype in (torch.bfloat16, torch.float32):
    desc = CacheDesc(B, L, 2 * H, H, D, 5056, dtype)
    k = torch.ones(B, L, H, n, D, dtype=dtype, device="cuda")
    c, p = allocate_cache(desc), allocate_paged_cache(desc, B * L * H * 80)
    c["len"].fill_(7), p["len"].fill_(7)
    voxzip_anchor_fuse(desc, k, k, *ints, c["k"], c["v"], c["score"], c["pos"], c["len"])
    assert voxzip_get_status() == DEV_TIMEOUT
    assert not c["len"].any(), c["len"]
    voxzip_anchor_fuse_paged(desc, p, k, k, *ints)
    assert voxzip_get_status() == DEV_TIMEOUT
    assert not p["len"].any(), p["len"]
"""


@pytest.mark.skipif("VOXZIP_CHECKED" in os.environ, reason="builds a library of its own")
def test_a_wait_that_gives_up_leaves_its_units_empty(tmp_path):
    """A build whose waits for rows give up at once (the loads in flight are still waited for before a warp
    leaves): the status word says so, and no unit keeps an earlier request's length."""
    from paper_2608_08569_gb300 import build as B
    objs = [os.path.join(B.BUILD_DIR, os.path.basename(s)[:-3] + ".o") for s in B._sources()]
    if not all(os.path.exists(o) for o in objs):
        B.build_library(force=True)
    src, obj, lib = os.path.join(B.CSRC, "anchor_fuse.cu"), str(tmp_path / "anchor_fuse.o"), str(tmp_path / "lib.so")
    cmds = [[B._nvcc(), *B.ARCH, *B.NVCC_FLAGS, "-DVOXZIP_FUSE_WAIT_LIMIT=0u", "-c", src, "-o", obj],
            [B._nvcc(), *B.ARCH, "-shared", "-cudart", "shared", "-Xlinker", "-rpath,/usr/local/cuda/lib64", "-o", lib, obj,
             *[o for o in objs if os.path.basename(o) != "anchor_fuse.o"]],
            [sys.executable, "-c", GIVES_UP, lib]]
    for cmd in cmds:
        r = subprocess.run(cmd, cwd=B.ROOT, capture_output=True, text=True, timeout=600)
        assert r.returncode == 0, r.stderr[-3000:]
