"""Attention from records at the edges of the kernel's tiles: every norm storage
of K and V, batches of 32 and units of 256 tokens and their remainders, jobs that
span several CTAs and CTAs that span several jobs, and value rows whose scale
varies by 2^40 from token to token (the running scales of the accumulators).

Same oracle and tolerance as test_gpu_attend.
"""
import math

import numpy as np
import pytest

import parity
import test_gpu_attend as base

pytestmark = pytest.mark.gpu

NORMS = [(4, 0), (4, 1), (8, 0), (8, 1), (32, 2)]


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("nq", [3, 7])
def test_norm_storage_and_batch_edges(tac_gpu, orc, d, nq):
    ns = [2, 16, 48, 128, 256]
    spec = []
    for i, kn in enumerate(NORMS):
        for j, vn in enumerate(NORMS):
            T = (1, 31, 32, 33, 255, 256, 257, 600)[(5 * i + j) % 8]
            spec.append(dict(d=d, T=T, nq=nq, k=(ns[(i + j) % 5], *kn), v=(ns[(2 * i + j) % 5], *vn), seed=10 * i + j))
    base._check(orc, tac_gpu, spec)


@pytest.mark.parametrize("nq", [1, 8])
def test_jobs_across_ctas(tac_gpu, orc, nq):
    """More units than CTAs fit on the device at once, of jobs of very different lengths."""
    lens = [9000, 1, 70001, 256, 5000, 31, 12345, 513]
    spec = [dict(d=128, T=T, nq=nq, k=(64, 8, 0), v=(64, 4, 1), seed=i) for i, T in enumerate(lens)]
    base._check(orc, tac_gpu, spec)


@pytest.mark.parametrize("order", ["up", "down", "mixed"])
def test_value_scales_per_token(tac_gpu, orc, order):
    """The output is compared row by row against sum_t p_t |v^_t|, so tokens that
    weigh little because their values are small must not disturb the others: the
    error of an output element stays below 2^-18 of that sum (fp32 scores of
    magnitude below 2^5 carry 2^-20, each weight and value 2^-22)."""
    import torch
    tac, d, T, nq = tac_gpu, 128, 700, 4
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    e = torch.linspace(-20, 20, T, device="cuda")
    if order == "down":
        e = e.flip(0)
    elif order == "mixed":
        e = e[torch.randperm(T, generator=g, device="cuda")]
    xk = torch.randn((T, d), generator=g, device="cuda")
    xv = torch.randn((T, d), generator=g, device="cuda") * torch.exp2(torch.round(e))[:, None]
    kcfg, vcfg = tac.layer_cfg(d, 64, 8, 0, 0, 1, 0), tac.layer_cfg(d, 64, 8, 0, 0, 1, 1)
    kc, vc = tac.encode(xk, kcfg), tac.encode(xv, vcfg)
    # the first query attends to everything, the others ever more sharply to tokens
    # of small values: along (a multiple of) the mean of their keys
    small = xk[e < -10].mean(0)
    q = torch.stack([0.2 * torch.randn(d, generator=g, device="cuda")] +
                    [s * small * d / small.norm() ** 2 for s in (0.02, 0.05, 0.1)])
    out = torch.empty_like(q)
    tac.attend_multi([tac.AttendJob(kcfg, kc, vcfg, vc, T, q, out, 1.0 / math.sqrt(d))])
    torch.cuda.synchronize()
    kh = base._oracle_rows(orc, tac, kcfg, kc, T)
    vh = base._oracle_rows(orc, tac, vcfg, vc, T)
    q64 = parity.to_f64(q)
    s = q64 @ kh.T / math.sqrt(d)
    p = np.exp(s - s.max(1, keepdims=True))
    p /= p.sum(1, keepdims=True)
    want = orc.attend(q64, kh, vh, 1.0 / math.sqrt(d))
    size = p @ np.linalg.norm(vh, axis=1)           # sum_t p_t ||v^_t||
    err = np.abs(parity.to_f64(out) - want).max(1)
    assert np.all(err <= 2.0**-18 * size), err / size


def _job(torch, tac, d, T, nq, seed, dtype):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    kcfg, vcfg = tac.layer_cfg(d, 64, 8, 0, 0, 1, 0), tac.layer_cfg(d, 64, 4, 1, 0, 1, 1)
    kc, vc = (tac.encode(torch.randn((T, d), generator=g, device="cuda"), c) for c in (kcfg, vcfg))
    q = (2 * torch.randn((nq, d), generator=g, device="cuda")).to(dtype)
    return tac.AttendJob(kcfg, kc, vcfg, vc, T, q, torch.zeros_like(q), 1.0 / math.sqrt(d))


@pytest.mark.parametrize("d,nq", [(64, 4), (128, 1), (128, 8)])
def test_outputs_do_not_depend_on_the_other_jobs(tac_gpu, d, nq):
    """The same bits from a job alone and in batches whose units are dealt to the
    CTAs in other ways (more units than CTAs, fewer, the job first or last), among jobs
    of more and of fewer queries."""
    import torch
    tac = tac_gpu
    jobs = [_job(torch, tac, d, T, nq, i, torch.float32) for i, T in enumerate([20000, 300, 4097, 33, 70000, 1000])]
    alone = []
    for j in jobs:
        tac.attend_multi([j])
        alone.append(j.out.clone())
    fill = [_job(torch, tac, d, T, m, 50 + i, torch.float32)
            for i, (T, m) in enumerate([(511, nq), (30000, 8), (30000, 1), (7, 5), (90000, 2)])]
    for batch in (jobs, jobs[::-1], fill[:1] + jobs[1:4], fill + jobs, jobs + fill, jobs[:2] + fill + jobs[2:]):
        for j in jobs:
            j.out.zero_()
        tac.attend_multi(batch)
        torch.cuda.synchronize()
        for j, want in zip(jobs, alone):
            if any(j is b for b in batch):
                assert torch.equal(j.out, want), (j.tokens, len(batch))


def _fwht(x, dtype):
    """Unnormalized Walsh-Hadamard butterfly over the last axis, in `dtype`."""
    import torch
    x, d = x.to(dtype), x.shape[-1]
    for h in [1 << i for i in range(d.bit_length() - 1)]:
        v = x.reshape(*x.shape[:-1], d // (2 * h), 2, h)
        x = torch.stack([v[..., 0, :] + v[..., 1, :], v[..., 0, :] - v[..., 1, :]], -2).reshape(x.shape)
    return x


def _plain(q, rk, ak, rv, av, scale, signs, dtype):
    """The kernel's op with every operation in `dtype`: rotated queries, scores against
    r (cos, sin), base-2 softmax, weighted values, one transform of the output."""
    import torch
    d = q.shape[-1]
    cs = lambda r, a: torch.stack([r.to(dtype) * torch.cos(a).to(dtype), r.to(dtype) * torch.sin(a).to(dtype)], -1).flatten(-2)
    qr = _fwht(q.to(dtype) * signs[0].to(dtype), dtype) * (scale * math.log2(math.e) / math.sqrt(d))
    s = (qr[..., :, None, :] * cs(rk, ak)[..., None, :, :]).sum(-1)
    p = torch.exp2(s - s.amax(-1, keepdim=True))
    y = (p[..., None] * cs(rv, av)[..., None, :, :]).sum(-2) / p.sum(-1, keepdim=True)
    return _fwht(y, dtype) / math.sqrt(d) * signs[1].to(dtype)


@pytest.mark.parametrize("T", [1, 2, 5, 20, 33, 130, 300, 1500])
@pytest.mark.parametrize("d,nq", [(64, 2), (128, 8)])
def test_error_no_larger_than_that_of_fp32_arithmetic(tac_gpu, d, nq, T):
    """Outputs against 64 bits (2-norm over 16 jobs of fp32 norms) are no further off
    than the same op in fp32 throughout, by more than the spread of such a ratio
    (each side a few thousand rounding errors; pairwise sums in the fp32 one, whose
    error is the least fp32 arithmetic can have).  Jobs of more than 256 tokens keep
    two parts of a value: the residue's rounding (0.44 * 2^-23 of the record's scale
    in the mean square) is about as large as that error and adds to the 0.75 of it
    that three parts leave: sqrt(1 + 0.75^2) = 1.25."""
    import torch
    tac, n, jobs = tac_gpu, 256, 16
    g = torch.Generator(device="cuda")
    g.manual_seed(100 * d + T)
    cfg = [tac.layer_cfg(d, n, 32, tac.NORM_FP32, 0, 1, kv) for kv in (0, 1)]
    signs = [torch.tensor(parity.signs_pm1(c.signs, d), dtype=torch.float64, device="cuda") for c in cfg]
    order = torch.tensor([4 * (v % (d // 16)) + (v // (d // 16)) % 4 + d // 4 * (v // (d // 4)) for v in range(d // 2)],
                         device="cuda")
    q = 2 * torch.randn((jobs, nq, d), generator=g, device="cuda")
    out = torch.zeros_like(q)
    r, a, job = [[], []], [[], []], []
    for i in range(jobs):
        caches = []
        for kv in (0, 1):
            c = tac.Cache.empty(cfg[kv], T)
            k = torch.randint(0, n, (T, d // 2), generator=g, device="cuda", dtype=torch.uint8)
            v = torch.sqrt(torch.empty((T, d // 2), device="cuda").exponential_(0.5, generator=g))
            c.codes[: k.numel()] = k.reshape(-1)
            c.norms[: 4 * v.numel()] = v.reshape(-1).view(torch.uint8)
            pairs = torch.empty((2, T, d // 2), dtype=torch.float64, device="cuda")
            pairs[0][:, order], pairs[1][:, order] = v.double(), k.double() * (2 * math.pi / n)
            r[kv].append(pairs[0]), a[kv].append(pairs[1])
            caches.append(c)
        job.append(tac.AttendJob(cfg[0], caches[0], cfg[1], caches[1], T, q[i], out[i], 1.0 / math.sqrt(d)))
    tac.attend_multi(job)
    args = [torch.stack(x) for kv in (0, 1) for x in (r[kv], a[kv])]
    want, fp32 = (_plain(q, *args, 1.0 / math.sqrt(d), signs, t) for t in (torch.float64, torch.float32))
    torch.cuda.synchronize()
    err, lim = (float((x.double() - want).norm() / want.norm()) for x in (out, fp32))
    assert err <= (1.15 if T <= 256 else 1.25) * lim, (err, lim)


def test_attend_captured_into_graph(tac_gpu):
    """A prepared call (both kernels, the second launched while the first runs)
    replays from a CUDA graph to the bits of the direct call, over new queries."""
    import torch
    tac = tac_gpu
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    jobs = []
    for d, T, nq in ((128, 1000, 4), (128, 33, 4), (64, 2000, 7)):
        caches = []
        for kv, (n, b, m) in ((0, (64, 8, 0)), (1, (64, 4, 1))):
            cfg = tac.layer_cfg(d, n, b, m, 0, 1, kv)
            caches.append((cfg, tac.encode(torch.randn((T, d), generator=g, device="cuda"), cfg)))
        q = torch.randn((nq, d), generator=g, device="cuda")
        jobs.append(tac.AttendJob(*caches[0], *caches[1], T, q, torch.empty_like(q), 1.0 / math.sqrt(d)))
    call = tac.attend_multi_prepared(jobs)
    call()
    torch.cuda.synchronize()
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        call(torch.cuda.current_stream())
    for _ in range(3):
        for j in jobs:
            j.q.copy_(torch.randn(j.q.shape, generator=g, device="cuda"))
        call()
        torch.cuda.synchronize()
        want = [j.out.clone() for j in jobs]
        for j in jobs:
            j.out.zero_()
        graph.replay()
        torch.cuda.synchronize()
        for j, w in zip(jobs, want):
            assert torch.equal(j.out, w)
