"""GPU: activations handed from both CTAs of a pair to the MMAs: new activations in every call, and a token's result does not
depend on which CTA of the pair fetched it."""
import pytest
import torch

import paper_2609_34380_b200 as dps
from paper_2609_34380_b200 import workloads

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


# several tiles per pair and slots used many times over; K split over pairs; a ragged K
@pytest.mark.parametrize("N,K,M", [(9216, 4096, 512), (2048, 8192, 256), (4104, 2064, 320)])
def test_fresh_activations_and_moved_tokens(N, K, M):
    w = workloads.weights(N, K, 81, device=DEV)
    p, r, enc = dps.dps_split_weights(w)
    fast = dps.dps_reconstruct(p, None, enc)
    gen = torch.Generator(device=DEV)
    gen.manual_seed(82)
    moved = torch.arange(M, device=DEV).roll(M // 2 + 1)
    for mode, weights in ((dps.DPS_MODE_FAST, fast), (dps.DPS_MODE_FULL, w)):
        for _ in range(12):
            x = torch.randn((M, K), generator=gen, device=DEV).to(torch.float16)
            y = dps.dps_linear(mode, enc, x, p, r)
            z = dps.dps_linear(mode, enc, x[moved].contiguous(), p, r)
            assert torch.equal(z, y[moved])               # the same sums in the same order, wherever the token sits
            ref = x.double() @ weights.double().T
            assert bool(((y.double() - ref).abs().max() <= 2e-3 * ref.abs().max()))
    assert dps.dps_stream_status() == dps.DPS_OK
