"""GPU: chains of linears that are two launches (whole rounds of CTA pairs, the rest of the rows) or have wide token tiles, each output the next
input: back to back and with the device drained after every launch, bit for bit, and the first layer against the oracle at sampled entries.  The
two launches of a linear overlap each other and their neighbours; the consumer must see the rows of both."""
import re

import numpy as np
import pytest
import torch

import oracle
import paper_2609_34380_b200 as dps
from paper_2609_34380_b200 import workloads
from tests.helpers import TIGHT_BOUND, launch_lines, split_both, to_np_words
from tests.test_gpu_chained_launches import _chain

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
ROUND = 74 * 256
TALL = [(ROUND + 272, 8192), (8192, ROUND + 272)]        # one round and two row tiles, the second of them partly filled
# (modes, tokens, the shapes in rotation, what the first shape's launches say)
CHAINS = [((1,), 24, TALL, r"pair .*N=18944 .*\n.*N=272 "), ((0, 1), 64, TALL, r"pair .*N=18944 .*\n.*N=272 "), ((0, 1), 100, TALL, r"pair .*N=18944 .*\n.*N=272 "),
          ((0, 1), 1240, [(4096, 4096)], r"tokens=320 .*tail=1x"), ((0, 1), 1490, [(4096, 4096)], r"tokens=384 .*tail=1x"),
          ((0, 1), 1110, [(8192, 2048), (2048, 8192)], r"tokens=384 .*tail=3x")]


@pytest.mark.parametrize("modes,M,shapes,says", CHAINS)
def test_back_to_back_chain_equals_drained_chain(modes, M, shapes, says):
    planes, first = [], None
    for i, (N, K) in enumerate(shapes * 2):              # two matrices of each shape
        w = workloads.weights(N, K, 8100 + i, device=DEV)
        w = (w.float() * (1.0 / (w.float().std().item() * K ** 0.5))).to(torch.float16)      # the chain's magnitudes stay level
        if first is None:
            p, r, enc, *first = split_both(w, dps.DPS_ENC_AUTO, DEV)
        else:
            p, r, enc = dps.dps_split_weights(w, dps.DPS_ENC_AUTO)
        planes.append((p, r, enc))
        del w
    planes *= 6 // len(planes) + 1
    N, K = shapes[0]
    x0 = workloads.activations(M, K, 8200 + M, device=DEV)
    ms, ns = workloads.sample_entries(M, N, 2048, 8300)
    for mode in modes:
        assert re.search(says, "\n".join(launch_lines([(mode, M, N, K)])))
        drained = _chain(planes, x0, mode, drain=True)
        for attempt in range(3):
            for layer, (a, b) in enumerate(zip(_chain(planes, x0, mode, drain=False), drained, strict=True)):
                assert torch.equal(a.view(torch.int16), b.view(torch.int16)), f"layer {layer}, attempt {attempt}, mode {mode}"
        assert torch.isfinite(drained[-1].float()).all() and float(drained[-1].float().abs().max()) > 0.0
        ref = oracle.linear_at(mode, planes[0][2], to_np_words(x0), *first, ms, ns)
        got = drained[0].cpu().double().numpy()[ms, ns]
        # (the bound is of the largest output; the sample's largest is no more than that)
        assert np.max(np.abs(got - ref)) <= TIGHT_BOUND * np.max(np.abs(ref))
    assert dps.dps_stream_status() == dps.DPS_OK
