"""GPU: the routing pre-pass (rows grouped 1024 at a time, stable) and the grouped linear on CTA pairs, at their edges."""
import numpy as np
import pytest
import torch

import oracle
import paper_2609_34380_b200 as dps
from paper_2609_34380_b200 import binding, workloads
from tests.helpers import assert_close_to_oracle, split_both, to_np_words

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
ENCS = [dps.DPS_ENC_AUTO, dps.DPS_ENC_E5M2, dps.DPS_ENC_E4M3_RN, dps.DPS_ENC_E5M2_RN]


def problem(E, N, K, seed):
    parts = [split_both(workloads.weights(N, K, seed + e, device=DEV), ENCS[e % 4], DEV) for e in range(E)]
    stack = lambda i, f: f([q[i] for q in parts])
    return stack(0, torch.stack), stack(1, torch.stack), [q[2] for q in parts], stack(3, np.stack), stack(4, np.stack)


# rows: one, around a warp, around the 1024 rows placed at a time, more; experts: few rows and many rows per expert (pairs
# from 48 on: tiles of 16 to 256 tokens), one expert, more experts than the table holds
@pytest.mark.parametrize("E,A,N,K", [(1, 1, 8, 16), (3, 33, 136, 144), (2, 96, 264, 272), (5, 1023, 520, 144), (4, 1025, 264, 400),
                                     (7, 2500, 72, 128), (1, 700, 264, 144), (257, 600, 16, 32)])
def test_random_routing(E, A, N, K):
    p, r, encs, p_ref, r_ref = problem(E, N, K, 300)
    rng = np.random.default_rng(7 + A)
    eor = rng.integers(0, E, A).astype(np.int32)
    if E > 2:
        eor[eor == E - 1] = 0                             # an expert without rows, one with a double share
    tor = rng.integers(0, 37, A).astype(np.int32)
    x = workloads.activations(37, K, 8, device=DEV)
    for mode in (dps.DPS_MODE_FAST, dps.DPS_MODE_FULL):
        args = (mode, encs, x, torch.from_numpy(tor).to(DEV), torch.from_numpy(eor).to(DEV), p, r if mode else None)
        y = dps.dps_moe_linear(*args)
        ref, rc = oracle.moe_linear(mode, encs, to_np_words(x), tor, eor, p_ref, r_ref, threads=8)
        assert rc == oracle.OK
        assert_close_to_oracle(y, ref, f"E={E} A={A} N={N} K={K} mode={mode}")
        assert torch.equal(y, dps.dps_moe_linear(*args))
    assert dps.dps_stream_status() == dps.DPS_OK


def test_invalid_rows_of_many_are_left_alone():
    E, A, N, K = 4, 1500, 136, 144
    p, r, encs, p_ref, r_ref = problem(E, N, K, 400)
    rng = np.random.default_rng(9)
    eor, tor = rng.integers(0, E, A).astype(np.int32), rng.integers(0, 50, A).astype(np.int32)
    eor[::97], tor[5::101] = E, -1
    bad = (eor == E) | (tor < 0)
    x = workloads.activations(50, K, 10, device=DEV)
    y = torch.full((A, N), 7.0, dtype=torch.float16, device=DEV)
    dps.dps_moe_linear(dps.DPS_MODE_FULL, encs, x, torch.from_numpy(tor).to(DEV), torch.from_numpy(eor).to(DEV), p, r, y)
    assert dps.dps_stream_status() == binding.DPS_ERR_DATA
    good = np.flatnonzero(~bad)
    ref, rc = oracle.moe_linear(dps.DPS_MODE_FULL, encs, to_np_words(x), tor[good], eor[good], p_ref, r_ref, threads=8)
    assert rc == oracle.OK
    assert_close_to_oracle(y[torch.from_numpy(good).to(DEV)], ref, "valid rows")
    assert bool((y[torch.from_numpy(np.flatnonzero(bad)).to(DEV)] == 7.0).all())
