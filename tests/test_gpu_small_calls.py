"""Small encode calls (one kernel for every codebook shape, which re-decides its
own codes) against large ones (a kernel per shape, queue and fix-up kernel).

Every shape the library takes, row counts around the warp tile, contiguous,
scattered and out-of-range slots, rows that need the exact path, zero rows and
non-finite rows: the records must be the same bytes, and so must the records of
a large call whose queue has no room.
"""
import pytest

pytestmark = pytest.mark.gpu

SHAPES = [(n, b, m) for n in (2, 4, 8, 16, 32, 48, 56, 64, 128, 256)
          for b, m in ((4, 0), (4, 1), (8, 0), (8, 1), (32, 2))]
LARGE_TILES = 65536


def _rows(torch, d, dtype, rows):
    """Gaussian rows with channel scales; the first 400 hold rows that take the rare paths."""
    g = torch.Generator(device="cuda")
    g.manual_seed(d)
    x = torch.randn((rows, d), generator=g, device="cuda")
    x *= torch.exp(torch.randn((1, d), generator=g, device="cuda"))
    x[3] = 0
    x[7] = 1.0
    x[11] = 0
    x[11, d // 2] = -3.0
    x[13, ::2] = 0
    x[17] = float("nan")
    x[19, 1] = float("inf")
    x[100:200] = torch.randint(-2, 3, (100, d), generator=g, device="cuda").float()   # ties at edges and midpoints
    x[200:300] *= torch.exp2(torch.linspace(-36, 50, 100, device="cuda"))[:, None]
    x[300:400, 1:] = x[300:400, :1] * 2.0**-30
    return x.to(torch.bfloat16 if dtype == "bf16" else torch.float32)


def _view(torch, tac, cache):
    """The planes of a device cache as rows: angle, norm, header (or None)."""
    c, n = cache.cfg, cache.capacity
    ab, nb = tac.angle_row_bytes(c), tac.norm_row_bytes(c)
    off = tac.header_offset(c, n)
    hdr = None if c.norm_mode == tac.NORM_FP32 else cache.norms[off: off + 8 * n].reshape(n, 8)
    return cache.codes[: n * ab].reshape(n, ab), cache.norms[: n * nb].reshape(n, nb), hdr


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("d", [16, 32, 64, 128])
def test_small_calls_match_large_ones(tac_gpu, d, dtype):
    import torch
    tac = tac_gpu
    rw = 32 // (d // 16)
    rows = LARGE_TILES * rw + 3
    x = _rows(torch, d, dtype, rows)
    # seven rows in eight of those not compared are zero: the re-decision queue then
    # holds every entry (which codes a full one leaves to whole rows varies)
    g = torch.Generator(device="cuda")
    g.manual_seed(d + 2)
    x[1000: rows - 1000][torch.rand(rows - 2000, generator=g, device="cuda") < 0.875] = 0
    pieces = [(0, 400), (400, 1), (401, rw - 1), (500, rw), (600, rw + 1), (700, 5 * rw + 3), (rows - 1000, 1000)]
    pieces = [(a, k) for a, k in pieces if k > 0]
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    for n, b, m in SHAPES:
        cfg = tac.layer_cfg(d, n, b, m, 0, 2, 1)
        big = tac.Cache.empty(cfg, rows)
        st = torch.zeros(1, dtype=torch.int32, device="cuda")
        tac.encode_multi([tac.EncodeJob(cfg, x, big, None, st)])
        want = _view(torch, tac, big)
        jobs, at, stats = [], [], []
        for i, (a, k) in enumerate(pieces):
            cap, slot, sel = k, None, torch.arange(k, device="cuda")
            if i % 2:                                   # scattered, two rows dropped
                cap = 3 * k + 5
                slot = torch.randperm(cap, generator=g, device="cuda")[:k]
                if k > 4:
                    slot[1], slot[k - 2] = -1, cap
                sel = slot
            cache = tac.Cache.empty(cfg, cap)
            s = torch.zeros(1, dtype=torch.int32, device="cuda")
            jobs.append(tac.EncodeJob(cfg, x[a:a + k], cache, slot, s))
            at.append((a, k, sel, cap))
            stats.append(s)
        if tac.launch_count(jobs) == 1:
            tac.encode_multi(jobs)
        else:                                           # scattered records that share words: no small call
            assert tac.launch_count(jobs[0::2]) == 1
            tac.encode_multi(jobs[0::2])
            tac.encode_multi(jobs[1::2])
        torch.cuda.synchronize()
        assert int(st) == tac.TAC_E_NONFINITE
        for (a, k, sel, cap), j, s in zip(at, jobs, stats):
            ok = (sel >= 0) & (sel < cap)
            for got, ref in zip(_view(torch, tac, j.cache), want):
                if ref is not None:
                    assert torch.equal(got[sel[ok]], ref[a:a + k][ok]), (n, b, m, a, k)
            assert int(s) == (tac.TAC_E_NONFINITE if a == 0 else 0)


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("d", [16, 32, 64, 128])
def test_large_scattered_calls_match_dense_ones(tac_gpu, d, dtype):
    """A call by shape whose rows go to a permutation of slots, some of them out of
    range: the dense call's records, and nothing else is written.  Seven rows in eight
    are zero, so that the re-decision queue holds every entry (which codes a full one
    leaves to whole rows differs from run to run)."""
    import torch
    import parity
    tac = tac_gpu
    rows = (parity.SMALL_LIMIT + 1) * (32 // (d // 16)) + 3
    cap = rows + 1000
    x = _rows(torch, d, dtype, rows)
    g = torch.Generator(device="cuda")
    g.manual_seed(d + 1)
    x[400:][torch.rand(rows - 400, generator=g, device="cuda") < 0.875] = 0
    slot = torch.randperm(cap, generator=g, device="cuda")[:rows]
    slot[::97], slot[5::101], slot[rows - 1] = -1, cap, cap + 5
    ok = (slot >= 0) & (slot < cap)
    free = torch.ones(cap, dtype=torch.bool, device="cuda")
    free[slot[ok]] = False
    for n, b, m in SHAPES:
        cfg = tac.layer_cfg(d, n, b, m, 0, 3, 0)
        dense, scat = tac.Cache.empty(cfg, rows), tac.Cache.empty(cfg, cap)
        scat.codes.fill_(0xA5)
        scat.norms.fill_(0xA5)
        jobs = [tac.EncodeJob(cfg, x, scat, slot)]
        assert tac.launch_count(jobs) == 2
        ws = torch.zeros(tac.encode_workspace_bytes(jobs)[0], dtype=torch.uint8, device="cuda")
        tac.encode_multi(jobs, workspace=ws)
        tac.encode_multi([tac.EncodeJob(cfg, x, dense)])
        assert int(ws[:8].view(torch.int64)) <= rows * (d // 2) // 512 + 1024
        for got, ref in zip(_view(torch, tac, scat), _view(torch, tac, dense)):
            if ref is not None:
                assert torch.equal(got[slot[ok]], ref[ok]), (n, b, m)
                assert bool((got[free] == 0xA5).all()), (n, b, m)


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("d", [16, 32, 64, 128])
def test_subnormal_pairs_match_large_calls(tac_gpu, d, dtype):
    """Pairs whose |E| + |O| is a subnormal number (its hardware reciprocal is
    infinite) get a code inside the codebook and leave their neighbours' codes
    alone: rows of subnormals, one subnormal element in a row whose even elements
    cancel, and the same beside ordinary rows, against the large call."""
    import torch
    tac = tac_gpu
    rw = 32 // (d // 16)
    rows = LARGE_TILES * rw
    g = torch.Generator(device="cuda")
    g.manual_seed(7 * d)
    x = torch.zeros((rows, d), device="cuda")
    sub = 2.0**-130
    x[0, 0], x[1, 1], x[2, d - 1] = sub, -sub, sub
    x[3:20] = torch.randn((17, d), generator=g, device="cuda") * sub
    for i in range(20, 60):                             # E = 0 in half of the pairs, O subnormal
        j = 2 * int(torch.randint(1, d // 2, (1,), generator=g, device="cuda"))
        x[i, 0], x[i, j], x[i, 1 + 2 * (i % (d // 2))] = 1.0, -1.0 if i & 1 else 1.0, sub if i & 2 else -3 * sub
    for i in range(60, 80):                             # the same with the halves exchanged
        x[i, 1], x[i, 3], x[i, 2 * (i % (d // 2))] = 2.0, 2.0, sub
    x[80:100] = torch.randn((20, d), generator=g, device="cuda")
    x[80:100:3, ::2] = sub
    x = x.to(torch.bfloat16 if dtype == "bf16" else torch.float32)
    for n, b, m in [s for s in SHAPES if s[1:] in ((4, 1), (8, 0), (32, 2))]:
        cfg = tac.layer_cfg(d, n, b, m, 0, 1, 0)
        big, few = tac.Cache.empty(cfg, rows), tac.Cache.empty(cfg, 101)
        tac.encode_multi([tac.EncodeJob(cfg, x, big)])
        tac.encode_multi([tac.EncodeJob(cfg, x[:101], few)])
        torch.cuda.synchronize()
        for got, ref in zip(_view(torch, tac, few), _view(torch, tac, big)):
            assert ref is None or torch.equal(got, ref[:101]), (n, b, m)


@pytest.mark.parametrize("n,b,m", [(64, 8, 0), (256, 4, 1), (56, 32, 2)])
def test_large_call_without_queue_room(tac_gpu, n, b, m):
    """The minimum workspace: every queued code's row is re-decided whole."""
    import torch
    tac, d = tac_gpu, 128
    rows = LARGE_TILES * 4 + 1
    x = _rows(torch, d, "bf16", rows)
    cfg = tac.layer_cfg(d, n, b, m, 0, 0, 0)
    caches = [tac.Cache.empty(cfg, rows) for _ in range(2)]
    for cache, ws in zip(caches, (None, "min")):
        jobs = [tac.EncodeJob(cfg, x, cache)]
        if ws:
            ws = torch.empty(tac.encode_workspace_bytes(jobs)[1], dtype=torch.uint8, device="cuda")
        tac.encode_multi(jobs, workspace=ws)
    torch.cuda.synchronize()
    for a, c in zip(_view(torch, tac, caches[0]), _view(torch, tac, caches[1])):
        assert a is None or torch.equal(a, c)
