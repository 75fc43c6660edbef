"""Gathered decode (decode_multi with a slot table): every record copy size and the tile edges.

A gathered row must be the bits of the same record decoded by a contiguous
call, and a slot outside the cache must decode to zeros, for each record row
size (16-, 8- and 4-byte copies, and the odd widths below them) and for row
counts around the warp tile and the prefetch depth.
"""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [16, 32, 64, 128])
@pytest.mark.parametrize("n,b,mode", [(64, 8, 0), (128, 4, 1), (256, 32, 2), (32, 8, 1), (2, 4, 0), (56, 32, 2)])
@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
def test_gather_matches_contiguous_decode(tac_gpu, d, n, b, mode, dtype):
    import torch
    tac = tac_gpu
    tdt = torch.bfloat16 if dtype == "bf16" else torch.float32
    g = torch.Generator(device="cuda")
    g.manual_seed(d * 1000 + n)
    cap = 777
    x = torch.randn((cap, d), generator=g, device="cuda")
    cfg = tac.layer_cfg(d, n, b, mode, 0, 3, 1)
    cache = tac.encode(x, cfg)
    dense = tac.decode(cache, cfg, dtype=tdt)
    rw = 32 // (d // 16)
    jobs, want = [], []
    for rows in (1, rw - 1, rw, rw + 1, 3 * rw, 5 * rw + 1, 1500):
        if rows < 1:
            continue
        slot = torch.randint(0, cap, (rows,), generator=g, device="cuda")
        if rows > 2:
            slot[1], slot[rows - 1] = -1, cap
        y = torch.full((rows, d), 7.0, dtype=tdt, device="cuda")
        ok = (slot >= 0) & (slot < cap)
        want.append(torch.where(ok[:, None], dense[slot.clamp(0, cap - 1)], torch.zeros((), dtype=tdt, device="cuda")))
        jobs.append(tac.DecodeJob(cfg, cache, y, slot))
    jobs.append(tac.DecodeJob(cfg, cache, torch.empty_like(dense)))     # a contiguous job in the same launch
    want.append(dense)
    tac.decode_multi(jobs)
    torch.cuda.synchronize()
    for j, ref in zip(jobs, want):
        assert torch.equal(j.y.abs(), ref.abs()) and torch.equal(j.y[ref != 0], ref[ref != 0])
