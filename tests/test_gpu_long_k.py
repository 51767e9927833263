"""GPU: 33 to 64 tokens on a matrix with a long K, which the CTA pairs serve where they fill the chip: the smallest such matrix and its
neighbours on both sides, the family on both sides of every edge."""
import pytest
import torch

import oracle
import paper_2609_34380_b200 as dps
from paper_2609_34380_b200 import workloads
from tests.helpers import assert_close_to_oracle, launch_lines, split_both, to_np_words

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("M,N,K", [(33, 5120, 16384), (64, 5128, 16400), (32, 5120, 16384), (64, 5112, 16384), (33, 5120, 16368)])
def test_long_k(M, N, K):
    p, r, enc, p_ref, r_ref = split_both(workloads.weights(N, K, 7, device=DEV), dps.DPS_ENC_AUTO, DEV)
    x = workloads.activations(M, K, 9, device=DEV)
    for mode in (dps.DPS_MODE_FAST, dps.DPS_MODE_FULL):
        y = dps.dps_linear(mode, enc, x, p, r if mode else None)
        assert_close_to_oracle(y, oracle.linear(mode, enc, to_np_words(x), p_ref, r_ref, threads=8), f"M={M} N={N} K={K} mode={mode}")
        assert torch.equal(y, dps.dps_linear(mode, enc, x, p, r if mode else None))
    assert dps.dps_stream_status() == dps.DPS_OK


def test_family_at_the_edges():
    # 20, 22 | 23, 26 | 27, 33 | 34, 45 | 46, 74 | 75 tiles of 256 rows, and the bounds on tokens, rows and K
    cases = [(64, 256 * t, 16384) for t in (20, 22, 23, 26, 27, 33, 34, 45, 46, 74, 75)]
    cases += [(33, 5120, 16384), (32, 5120, 16384), (64, 5112, 16384), (33, 5120, 16368), (40, 8456, 28672)]
    pairs = [True, True, False, False, True, True, False, False, True, True, False, True, False, False, False, False]
    for mode in (dps.DPS_MODE_FAST, dps.DPS_MODE_FULL):
        lines = launch_lines([(mode, *c) for c in cases])
        assert [line.startswith("[dps] pair ") for line in lines] == pairs, "\n".join(lines)
