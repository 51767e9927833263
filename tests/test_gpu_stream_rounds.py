"""GPU: the streaming decode kernel over every split of K into rounds of 512 and batches of rounds: below one round, whole
batches of every length, short last batches, ragged ends."""
import pytest
import torch

import oracle
import paper_2609_34380_b200 as dps
from paper_2609_34380_b200 import workloads
from tests.helpers import assert_close_to_oracle, split_both, to_np_words

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
KS = [16, 496, 512, 528, 1024, 1552, 2048, 2576, 3072, 3088, 3584, 4096, 4112, 4608, 5648, 6656, 7184, 8192, 8336, 11008]


@pytest.mark.parametrize("K", KS)
def test_rounds(K):
    N = 40
    for enc_req in (dps.DPS_ENC_AUTO, dps.DPS_ENC_E5M2, dps.DPS_ENC_E5M2_RN):
        p, r, enc, p_ref, r_ref = split_both(workloads.weights(N, K, 71, device=DEV), enc_req, DEV)
        for M in (1, 8, 12):                              # 12: two token groups (small matrices stay on this kernel)
            x = workloads.activations(M, K, 72 + M, device=DEV)
            for mode in (dps.DPS_MODE_FAST, dps.DPS_MODE_FULL):
                y = dps.dps_linear(mode, enc, x, p, r if mode else None)
                ref = oracle.linear(mode, enc, to_np_words(x), p_ref, r_ref, threads=8)
                assert_close_to_oracle(y, ref, f"K={K} M={M} enc={enc} mode={mode}")
                assert torch.equal(y, dps.dps_linear(mode, enc, x, p, r if mode else None))
    assert dps.dps_stream_status() == dps.DPS_OK
