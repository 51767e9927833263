"""GPU: grouped launches of 12 to 47 rows per expert on either side of the border between CTA pairs and 128-row tiles (row tiles over the experts),
against the oracle: mixed encodings, rounded nests, skewed routing (an expert with several token tiles, one without rows), token tiles of 64 to 128.
Which kernel ran is read off the lines that the library prints on request; it reads its knobs once per process, so a case is a child
process: this file executed as a script."""
import os
import re
import subprocess
import sys

import pytest

REPO = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
# experts, N, K, rows per expert; token tile of the pairs in fast and full mode, 0: the 128-row tiles.  Row tiles of 256, rounds of 74 pairs against turns of the
# 128-row tiles (two per wave of 296):
CASES = [(2, 37 * 256 + 8, 80, 13, 0, 0),         # 76, two against two
         (2, 112 * 256 + 136, 48, 25, 0, 0),      # 226, four against four
         (2, 80 * 256 + 8, 80, 13, 0, 96),        # 162, three against four; fast mode has too few rows
         (3, 60 * 256 + 136, 48, 25, 64, 96),     # 183, three against four
         (8, 18 * 256 + 8, 80, 25, 0, 0),         # 152, three against two: 37 tiles of 128 rows an expert are one wave
         (12, 49 * 256 + 520, 144, 46, 64, 96),   # 624, nine
         (24, 25 * 256 + 8, 144, 13, 0, 96),      # 624, nine
         (4, 16 * 256 - 8, 3088, 30, 96, 128)]    # 64, one against two


def _run(E, N, K, rows, skewed):
    import numpy as np
    import torch

    import oracle
    import paper_2609_34380_b200 as dps
    from paper_2609_34380_b200 import workloads
    from tests.helpers import assert_close_to_oracle, split_both, to_np_words

    dev = "cuda:0"
    A = E * rows
    rng = np.random.default_rng(rows)
    eor = (rng.integers(0, E, A) if not skewed else np.where(rng.random(A) < 0.8, 0, rng.integers(0, max(1, E - 1), A))).astype(np.int32)
    requests = [dps.DPS_ENC_AUTO, dps.DPS_ENC_E5M2, dps.DPS_ENC_E4M3_RN, dps.DPS_ENC_E5M2_RN]
    planes = [split_both(workloads.weights(N, K, 40 + e, device=dev), requests[e % 4], dev) for e in range(E)]
    p, r, encs = torch.stack([t[0] for t in planes]), torch.stack([t[1] for t in planes]), [t[2] for t in planes]
    x = workloads.activations(A, K, 3, device=dev)
    for mode in (dps.DPS_MODE_FAST, dps.DPS_MODE_FULL):
        y = dps.dps_moe_linear(mode, encs, x, None, torch.from_numpy(eor).to(dev), p, r if mode else None)
        ref, rc = oracle.moe_linear(mode, encs, to_np_words(x), None, eor, np.stack([t[3] for t in planes]), np.stack([t[4] for t in planes]), threads=8)
        assert rc == oracle.OK
        assert_close_to_oracle(y, ref, f"E={E} N={N} K={K} rows={rows} mode={mode}")
        assert torch.equal(y, dps.dps_moe_linear(mode, encs, x, None, torch.from_numpy(eor).to(dev), p, r if mode else None))
    assert dps.dps_stream_status() == dps.DPS_OK
    print("passed")


@pytest.mark.gpu
@pytest.mark.parametrize("E,N,K,rows,fast,full", CASES)
@pytest.mark.parametrize("skewed", [False, True])
def test_few_rows_per_expert_on_either_kernel(E, N, K, rows, fast, full, skewed):
    out = subprocess.run([sys.executable, os.path.abspath(__file__), *map(str, (E, N, K, rows, int(skewed)))], cwd=REPO,
                         env=dict(os.environ, DPS_DEBUG="1", PYTHONPATH=REPO), capture_output=True, text=True, timeout=600)
    assert out.returncode == 0 and "passed" in out.stdout, out.stdout[-2000:] + out.stderr[-4000:]
    on_pairs = re.findall(r"\[dps\] pair grouped full=(\d) .*? tokens=(\d+) ", out.stderr)
    assert on_pairs == [(str(mode), str(tokens)) for mode, tokens in ((0, fast), (1, full)) if tokens for _ in range(2)], out.stderr[-2000:]


if __name__ == "__main__":
    _run(*map(int, sys.argv[1:]))
