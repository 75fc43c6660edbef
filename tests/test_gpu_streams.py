"""Batched calls with several kernel shapes run their launches concurrently on
the caller's stream and helper streams joined back by events.

The call must still be ordered on the caller's stream (work queued after it on
that stream sees its results) and must be capturable into a CUDA graph once the
helper streams exist.  Reference results come from the same calls with a device
synchronization after each.
"""
import pytest

import workloads

pytestmark = pytest.mark.gpu


# tokens of a block (each call: 9 warp tiles a token): a small call, one whose five
# launches get shares of the SMs, and one whose launches get the whole GPU each,
# the fix-ups after a second fork and join
SIZES = {"small": 96, "shares": 8000, "whole": 12000}


def _jobs(tac, size):
    import torch
    tokens = SIZES[size]
    enc, dec = [], []
    # four kernel shapes: K/V x base/boosted codebooks, plus a d = 64 job
    specs = [(0, 0, 128, (256, 8, 0)), (0, 1, 128, (256, 4, 1)), (9, 0, 128, (64, 8, 0)),
             (9, 1, 128, (64, 4, 1)), (3, 0, 64, (128, 8, 0))]
    for layer, kv, d, (n, b, mode) in specs:
        cfg = tac.layer_cfg(d, n, b, mode, 0, layer, kv)
        src = workloads.CONFIGS["mistral7b" if d == 128 else "llama1b"]
        x = workloads.block(src, layer, kv, tokens=tokens, device="cuda")
        cache = tac.Cache.empty(cfg, x.shape[0], device="cuda")
        enc.append(tac.EncodeJob(cfg, x, cache))
        dec.append(tac.DecodeJob(cfg, cache, torch.empty_like(x)))
    assert tac.launch_count(enc) == (2 if size == "small" else 2 * 5)
    if size != "small":
        whole = 9 * tokens >= 640 * torch.cuda.get_device_properties(0).multi_processor_count
        assert whole == (size == "whole")
    return enc, dec


def _reference(tac, enc, dec):
    """Codes, norms and rows from calls with a synchronization after each, the records
    checked against small calls over pieces of the rows."""
    import torch
    tac.encode_multi(enc)
    torch.cuda.synchronize()
    tac.decode_multi(dec)
    torch.cuda.synchronize()
    for j in enc:
        for a in (0, j.x.shape[0] - 500):
            c = tac.Cache.empty(j.cfg, 500)
            tac.encode_multi([tac.EncodeJob(j.cfg, j.x[a:a + 500], c)])
            ab, nb = tac.angle_row_bytes(j.cfg), tac.norm_row_bytes(j.cfg)
            assert torch.equal(c.codes[: 500 * ab], j.cache.codes[a * ab:(a + 500) * ab])
            assert torch.equal(c.norms[: 500 * nb], j.cache.norms[a * nb:(a + 500) * nb])
    return [(j.cache.codes.clone(), j.cache.norms.clone()) for j in enc], [j.y.clone() for j in dec]


def _clear(enc, dec):
    for j in enc:
        j.cache.codes.zero_()
        j.cache.norms.zero_()
    for j in dec:
        j.y.zero_()


def _check(tac, enc, records, want):
    import torch
    for j, (codes, norms), (wc, wn) in zip(enc, records, want):
        assert torch.equal(codes, wc)
        used = tac.norms_bytes(j.cfg, j.cache.capacity)
        pad = (j.cache.capacity * tac.norm_row_bytes(j.cfg), tac.header_offset(j.cfg, j.cache.capacity))
        assert torch.equal(norms[: pad[0]], wn[: pad[0]]) and torch.equal(norms[pad[1]: used], wn[pad[1]: used])


@pytest.mark.parametrize("size", list(SIZES))
def test_multi_calls_ordered_on_caller_stream(tac_gpu, size):
    import torch
    tac = tac_gpu
    enc, dec = _jobs(tac, size)
    want, want_y = _reference(tac, enc, dec)
    s = torch.cuda.Stream()
    _clear(enc, dec)
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        tac.encode_multi(enc, stream=s)
        records = [(j.cache.codes.clone(), j.cache.norms.clone()) for j in enc]   # queued on s right after the call
        tac.decode_multi(dec, stream=s)
        ys = [j.y.clone() for j in dec]
    s.synchronize()
    _check(tac, enc, records, want)
    for a, b in zip(ys, want_y):
        assert torch.equal(a, b)


@pytest.mark.parametrize("size", list(SIZES))
def test_multi_calls_capture_into_graph(tac_gpu, size):
    import torch
    tac = tac_gpu
    enc, dec = _jobs(tac, size)
    want, want_y = _reference(tac, enc, dec)            # also creates the helper streams
    ecall, dcall = tac.encode_multi_prepared(enc), tac.decode_multi_prepared(dec)
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        ecall(torch.cuda.current_stream())
        dcall(torch.cuda.current_stream())
    _clear(enc, dec)
    torch.cuda.synchronize()
    for _ in range(2):
        g.replay()
        torch.cuda.synchronize()
        _check(tac, enc, [(j.cache.codes, j.cache.norms) for j in enc], want)
        for j, b in zip(dec, want_y):
            assert torch.equal(j.y, b)
