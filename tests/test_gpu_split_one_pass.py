"""GPU: the one-pass AUTO split (split as E4M3, redone as E5M2 when a word is out of range) and the two item widths
of the load-time kernels, bit for bit against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import paper_2609_34380_b200 as dps
from paper_2609_34380_b200 import workloads
from tests.helpers import to_np_bytes, to_np_words

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
# one item; one block of 8192 weights and its neighbours; several blocks with a partial one; thousands of blocks
SHAPES = [(1, 16), (511, 16), (512, 16), (513, 16), (37, 1008), (8200, 4112)]


def place(words, offset_bytes):
    """The tensor at a base address that is `offset_bytes` past a 256-byte boundary (16: not on a 32-byte boundary)."""
    buf = torch.empty(words.numel() * 2 + 256, dtype=torch.uint8, device=DEV)
    w = buf[offset_bytes:offset_bytes + words.numel() * 2].view(torch.float16).view(words.shape)
    w.copy_(words)
    assert w.data_ptr() % 32 == offset_bytes % 32
    return w


@pytest.mark.parametrize("offset", [0, 16])
@pytest.mark.parametrize("rows,cols", SHAPES)
def test_auto_split(rows, cols, offset):
    base = workloads.weights(rows, cols, 31 + rows, device=DEV)
    n = rows * cols
    for at in (None, 0, n // 2, n - 1):                   # no word out of range; one at the start, inside, at the end
        w = place(base, offset)
        if at is not None:
            w.view(-1)[at] = -1.751
        wn = to_np_words(w)
        p_ref, r_ref, enc_ref = oracle.split(wn, dps.DPS_ENC_AUTO)
        p, r, enc = dps.dps_split_weights(w)
        assert enc == enc_ref == (dps.DPS_ENC_E4M3 if at is None else dps.DPS_ENC_E5M2)
        assert np.array_equal(to_np_bytes(p), p_ref) and np.array_equal(to_np_bytes(r), r_ref)
        out = place(torch.zeros_like(base), offset)
        dps.dps_reconstruct(p, r, enc, out)
        assert np.array_equal(to_np_words(out), wn)
        dps.dps_reconstruct(p, None, enc, out)
        assert np.array_equal(to_np_words(out), oracle.fast_words(p_ref, enc_ref))
