"""GPU: routing and gather in one launch, at the edges: one row, the last number of rows it takes and the first it does not (which
the two launches serve, with and without their table of experts), many experts, activations longer than a block asks for ahead."""
import numpy as np
import pytest
import torch

import oracle
import paper_2609_34380_b200 as dps
from paper_2609_34380_b200 import workloads
from tests.helpers import assert_close_to_oracle, to_np_words
from tests.test_gpu_moe_routing import DEV, problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("E,A,N,K,gathered", [(1, 1, 8, 16, True), (3, 40, 16, 8208, True), (1000, 300, 8, 16, True), (5, 1024, 72, 144, True),
                                              (2, 512, 136, 144, False), (5, 1025, 72, 144, True), (257, 4500, 8, 32, True)])
def test_rows_at_the_edges(E, A, N, K, gathered):
    p, r, encs, p_ref, r_ref = problem(E, N, K, 500)
    rng = np.random.default_rng(3 + A)
    eor = rng.integers(0, E, A).astype(np.int32)
    T = 29 if gathered else A
    tor = rng.integers(0, T, A).astype(np.int32) if gathered else None
    x = workloads.activations(T, K, 8, device=DEV)
    for mode in (dps.DPS_MODE_FAST, dps.DPS_MODE_FULL):
        y = dps.dps_moe_linear(mode, encs, x, torch.from_numpy(tor).to(DEV) if gathered else None, torch.from_numpy(eor).to(DEV), p,
                               r if mode else None)
        ref, rc = oracle.moe_linear(mode, encs, to_np_words(x), tor if gathered else np.arange(A, dtype=np.int32), eor, p_ref, r_ref, threads=8)
        assert rc == oracle.OK
        assert_close_to_oracle(y, ref, f"E={E} A={A} N={N} K={K} mode={mode}")
    assert dps.dps_stream_status() == dps.DPS_OK
