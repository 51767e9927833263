"""GPU: grouped launches of 12 to 47 rows per expert that CTA pairs serve (many row tiles over the experts, short K), against the oracle: mixed encodings,
rounded nests, skewed routing (an expert with several token tiles, one without rows)."""
import numpy as np
import pytest
import torch

import oracle
import paper_2609_34380_b200 as dps
from paper_2609_34380_b200 import workloads
from tests.helpers import assert_close_to_oracle, split_both, to_np_words

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


# row tiles of 256 over all experts: 76 and 226 (fewer rounds of pairs than waves of tiles), 600 (nine)
@pytest.mark.parametrize("E,N,K,rows", [(2, 37 * 256 + 8, 80, 13), (2, 112 * 256 + 136, 48, 25), (12, 49 * 256 + 520, 144, 46)])
@pytest.mark.parametrize("skewed", [False, True])
def test_few_rows_per_expert_on_pairs(E, N, K, rows, skewed):
    A = E * rows
    rng = np.random.default_rng(rows)
    eor = (rng.integers(0, E, A) if not skewed else np.where(rng.random(A) < 0.8, 0, rng.integers(0, max(1, E - 1), A))).astype(np.int32)
    requests = [dps.DPS_ENC_AUTO, dps.DPS_ENC_E5M2, dps.DPS_ENC_E4M3_RN, dps.DPS_ENC_E5M2_RN]
    planes = [split_both(workloads.weights(N, K, 40 + e, device=DEV), requests[e % 4], DEV) for e in range(E)]
    p, r, encs = torch.stack([t[0] for t in planes]), torch.stack([t[1] for t in planes]), [t[2] for t in planes]
    x = workloads.activations(A, K, 3, device=DEV)
    for mode in (dps.DPS_MODE_FAST, dps.DPS_MODE_FULL):
        y = dps.dps_moe_linear(mode, encs, x, None, torch.from_numpy(eor).to(DEV), p, r if mode else None)
        ref, rc = oracle.moe_linear(mode, encs, to_np_words(x), None, eor, np.stack([t[3] for t in planes]), np.stack([t[4] for t in planes]), threads=8)
        assert rc == oracle.OK
        assert_close_to_oracle(y, ref, f"E={E} N={N} K={K} rows={rows} mode={mode}")
        assert torch.equal(y, dps.dps_moe_linear(mode, encs, x, None, torch.from_numpy(eor).to(DEV), p, r if mode else None))
    assert dps.dps_stream_status() == dps.DPS_OK
