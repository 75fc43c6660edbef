"""The binding's packed job arrays hold the bytes that setting the structs' fields gives."""
import numpy as np
import pytest
import torch


class _Tensor:
    """What the binding reads of a device tensor."""

    def __init__(self, ptr, shape, dtype=torch.bfloat16, row_stride=None):
        self.ptr, self.shape, self.dtype, self.is_cuda = ptr, shape, dtype, True
        self.strides = (row_stride or shape[-1], 1)

    def data_ptr(self):
        return self.ptr

    def stride(self, i):
        return self.strides[i]


class _Int(int):
    """Takes the field by field path."""


@pytest.mark.parametrize("d,n,b,m,words", [(128, 64, 8, 0, 4), (64, 56, 32, 2, 2), (16, 2, 4, 1, 1), (32, 256, 8, 1, 4)])
def test_packed_jobs_equal_fields(tac_host, d, n, b, m, words):
    tac = tac_host
    signs = np.arange(7, 7 + words, dtype=np.uint32) * 0x9E3779B9
    for rows, stride, slot, status, dt in ((5, d, None, None, torch.bfloat16), (1, 3 * d, 4096, 8, torch.float32),
                                           (0, d, 16, None, torch.bfloat16), (7, d + 16, None, 12, torch.float32)):
        enc, dec = [], []
        for kind in (int, _Int):
            cfg = tac.LayerCfg(kind(d), kind(n), kind(b), kind(m), signs)
            cache = tac.Cache(cfg, kind(2**40 + 3), _Tensor(2**47 + 16, (1,)), _Tensor(32, (1,)))
            x = _Tensor(2**46 + 64, (rows, d), dt, stride)
            sl = None if slot is None else _Tensor(slot, (rows,))
            st = None if status is None else _Tensor(status, (1,))
            enc.append(tac.EncodeJob(cfg, x, cache, sl, st))
            dec.append(tac.DecodeJob(cfg, cache, x, sl))
        a, b2 = (bytes(tac._enc_array([j, j])) for j in enc)
        assert a == b2
        a, b2 = (bytes(tac._dec_array([j, j])) for j in dec)
        assert a == b2
