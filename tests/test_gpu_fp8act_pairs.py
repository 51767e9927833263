"""GPU: the FP8-activation linear on CTA pairs, at the edges of its 256-row x 16..256-token tiles."""
import pytest
import torch

import oracle
import paper_2609_34380_b200 as dps
from paper_2609_34380_b200 import workloads
from tests.helpers import assert_close_to_oracle, split_both, to_np_words

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


# rows: within the first CTA of a pair, just into the second, a full tile and eight rows more; tokens: one, below and above
# the smallest tile, around 256, several token tiles of uneven width; K: below, at and above one block and the ring
@pytest.mark.parametrize("N,K,M", [(8, 16, 1), (128, 128, 16), (136, 144, 17), (256, 768, 255), (264, 784, 256), (520, 896, 257),
                                   (1032, 912, 600), (19208, 272, 40)])
def test_edges_of_the_pair_tiles(N, K, M):
    for enc_req in (dps.DPS_ENC_AUTO, dps.DPS_ENC_E5M2):
        p, _, enc, p_ref, _ = split_both(workloads.weights(N, K, 51, device=DEV), enc_req, DEV)
        x = workloads.activations(M, K, 52, device=DEV)
        q, scale = dps.dps_quantize_activations(x)
        guard = torch.full((M + 2, N), 7.0, dtype=torch.float16, device=DEV)
        dps.dps_linear_fp8act(enc, q, scale, p, guard[1:M + 1])
        ref = oracle.linear_fp8act(enc, *oracle.quantize_activations(to_np_words(x)), p_ref, threads=8)
        assert_close_to_oracle(guard[1:M + 1], ref, f"pairs N={N} K={K} M={M} enc={enc}")
        assert bool((guard[0] == 7.0).all()) and bool((guard[M + 1] == 7.0).all())
    assert dps.dps_stream_status() == dps.DPS_OK
