"""GPU: 9-16 tokens on both sides of the rule that picks the kernel family: the smaller side of the matrix (1536) and its size (2^25)."""
import pytest
import torch

import oracle
import paper_2609_34380_b200 as dps
from paper_2609_34380_b200 import workloads
from tests.helpers import assert_close_to_oracle, split_both, to_np_words

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("N,K", [(1536, 2064), (2056, 1536), (1544, 2064), (2056, 1552), (3088, 1552)])
def test_both_families(N, K):
    for enc_req in (dps.DPS_ENC_AUTO, dps.DPS_ENC_E5M2, dps.DPS_ENC_E4M3_RN):
        p, r, enc, p_ref, r_ref = split_both(workloads.weights(N, K, 61, device=DEV), enc_req, DEV)
        for M in (8, 9, 13, 16, 17):
            x = workloads.activations(M, K, 62 + M, device=DEV)
            for mode in (dps.DPS_MODE_FAST, dps.DPS_MODE_FULL):
                y = dps.dps_linear(mode, enc, x, p, r if mode else None)
                ref = oracle.linear(mode, enc, to_np_words(x), p_ref, r_ref, threads=8)
                assert_close_to_oracle(y, ref, f"N={N} K={K} M={M} enc={enc} mode={mode}")
                assert torch.equal(y, dps.dps_linear(mode, enc, x, p, r if mode else None))
    assert dps.dps_stream_status() == dps.DPS_OK


def test_wide_flat_matrices_are_the_tiles(monkeypatch, capfd):
    """Just below and just above 2^25 weights with a side of 256: the tiles print a launch line, the streaming kernel does not."""
    monkeypatch.setenv("DPS_DEBUG", "1")
    K, M = 256, 9
    for N, tiles in ((131064, False), (131072, True)):
        p, r, enc, p_ref, r_ref = split_both(workloads.weights(N, K, 63, device=DEV), dps.DPS_ENC_AUTO, DEV)
        x = workloads.activations(M, K, 64, device=DEV)
        for mode in (dps.DPS_MODE_FAST, dps.DPS_MODE_FULL):
            capfd.readouterr()
            y = dps.dps_linear(mode, enc, x, p, r)
            assert ("[dps] umma " in capfd.readouterr().err) == tiles
            ref = oracle.linear(mode, enc, to_np_words(x), p_ref, r_ref, threads=8)
            assert_close_to_oracle(y, ref, f"N={N} mode={mode}")
    assert dps.dps_stream_status() == dps.DPS_OK
