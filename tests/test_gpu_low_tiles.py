"""GPU: 9 to 32 tokens, more 128-row tiles than SMs: lower tiles.  The matrix heights on both sides of the rule's edges (one
wave of tiles and two; the shortest K), a last tile of few rows; and pinned heights that end inside every quarter of the
lanes, with K below and beyond the ring, in child processes, since the library reads the knob once."""
import os
import re
import subprocess
import sys

import pytest
import torch

import oracle
import paper_2609_34380_b200 as dps
from paper_2609_34380_b200 import workloads
from tests import test_gpu_pair_linear as checks
from tests.helpers import assert_close_to_oracle, launch_lines, split_both, to_np_words

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("M,N,K,enc", [(13, 18944, 48, dps.DPS_ENC_E5M2), (16, 18952, 2064, dps.DPS_ENC_AUTO), (32, 22024, 272, dps.DPS_ENC_E4M3_RN),
                                       (17, 27648, 144, dps.DPS_ENC_E5M2_RN), (9, 37896, 2064, dps.DPS_ENC_E5M2), (24, 40008, 16, dps.DPS_ENC_AUTO),
                                       (12, 20008, 6720, dps.DPS_ENC_AUTO), (32, 22024, 1552, dps.DPS_ENC_E4M3_RN),
                                       (24, 40008, 1536, dps.DPS_ENC_E5M2)])
def test_heights_around_the_rule(M, N, K, enc):
    p, r, enc, p_ref, r_ref = split_both(workloads.weights(N, K, 5, device=DEV), enc, DEV)
    x = workloads.activations(M, K, 6, device=DEV)
    for mode in (dps.DPS_MODE_FAST, dps.DPS_MODE_FULL):
        guard = torch.full((M + 2, N), 7.0, dtype=torch.float16, device=DEV)
        y = guard[1:M + 1]
        dps.dps_linear(mode, enc, x, p, r if mode else None, y)
        ref = oracle.linear(mode, enc, to_np_words(x), p_ref, r_ref, threads=8)
        assert_close_to_oracle(y, ref, f"M={M} N={N} K={K} enc={enc} mode={mode}")
        assert bool((guard[0] == 7.0).all()) and bool((guard[M + 1] == 7.0).all())
        assert torch.equal(y, dps.dps_linear(mode, enc, x, p, r if mode else None))
    assert dps.dps_stream_status() == dps.DPS_OK


@pytest.mark.parametrize("rows", [64, 72, 104, 120])
def test_pinned_heights_in_child_process(rows):
    env = dict(os.environ, DPS_FORCE_PATH="umma", DPS_TILE_ROWS=str(rows), PYTHONPATH=checks.REPO)
    shapes = ["8,16,1", "136,80,17", "264,1040,25", "1032,2720,32", "1032,272,16"]
    out = subprocess.run([sys.executable, os.path.abspath(checks.__file__), *shapes], cwd=checks.REPO, env=env, capture_output=True, text=True, timeout=900)
    assert out.returncode == 0, out.stdout[-2000:] + out.stderr[-4000:]
    assert "all 30 cases passed" in out.stdout


def test_heights_launched():
    """On both sides of the rule's edges: 148 tiles of 128 rows, K = 1536, the modes' and widths' limits, 2^27 weights in fast mode; and pinned."""
    cases = {(1, 12, 18944, 2048): 128, (1, 12, 18952, 2048): 88, (1, 32, 22016, 1536): 88, (1, 32, 22016, 1520): 128, (1, 24, 22016, 768): 128,
             (1, 16, 57344, 1536): 104, (1, 17, 57344, 1536): 128, (1, 33, 22016, 2048): 128, (0, 13, 40000, 4096): 96, (0, 17, 40000, 4096): 128,
             (0, 13, 32760, 4096): 128, (0, 13, 38016, 3520): 128, (0, 13, 38016, 3536): 96}
    lines = launch_lines(list(cases))
    assert heights(lines) == list(cases.values())
    # lower tiles never split K, so their set-up makes no occupancy queries
    for line, rows in zip(lines, cases.values()):
        assert line.endswith(" split=1 capacity=" + ",".join("0" * 8)) == (rows < 128), line
    assert heights(launch_lines([(1, 32, 1032, 272), (0, 16, 1032, 272)], DPS_FORCE_PATH="umma", DPS_TILE_ROWS="104")) == [104, 104]


def heights(lines):
    return [int(re.search(r" rows=(\d+) ", line).group(1)) for line in lines]
