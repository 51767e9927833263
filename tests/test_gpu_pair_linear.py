"""GPU: the dense linear on CTA pairs against the oracle, at the edges of its tiles: rows within the first CTA of a pair, just
into the second, beyond a whole tile; one token to several token tiles; K below, at and above one plane unit and the ring;
more tiles than pairs; a last round cut into pieces.

DPS_FORCE_PATH / DPS_PAIR_TOKENS / DPS_PAIR_SPLIT pin the family, the tile width and the K split; the library reads them once
per process, so each forced run is a child process: this file executed as a script.
"""
import os
import re
import subprocess
import sys

import pytest

REPO = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
# (N, K, M)
SHAPES = [(8, 16, 1), (128, 64, 16), (136, 80, 17), (256, 128, 100), (264, 1040, 255), (520, 720, 257), (1032, 272, 600), (512, 2064, 31)]
MANY = [(19208, 144, 70), (4096, 208, 1300)]
# tile width, pairs that share a tile (0: the library's choice)
VARIANTS = [(0, 0), (16, 1), (112, 1), (192, 1), (256, 1), (48, 2), (256, 2), (16, 4), (256, 4)]


def _run(shapes):
    import torch

    import oracle
    import paper_2609_34380_b200 as dps
    from paper_2609_34380_b200 import workloads
    from tests.helpers import assert_close_to_oracle, split_both, to_np_words

    dev = "cuda:0"
    count = 0
    for (N, K, M) in shapes:
        for enc_req in (dps.DPS_ENC_AUTO, dps.DPS_ENC_E5M2, dps.DPS_ENC_E4M3_RN):
            p, r, enc, p_ref, r_ref = split_both(workloads.weights(N, K, 17 + N, device=dev), enc_req, dev)
            x = workloads.activations(M, K, 19 + M, device=dev)
            for mode in (dps.DPS_MODE_FAST, dps.DPS_MODE_FULL):
                guard = torch.full((M + 2, N), 7.0, dtype=torch.float16, device=dev)
                y = guard[1:M + 1]
                dps.dps_linear(mode, enc, x, p, r if mode else None, y)
                ref = oracle.linear(mode, enc, to_np_words(x), p_ref, r_ref, threads=8)
                assert_close_to_oracle(y, ref, f"pairs N={N} K={K} M={M} enc={enc} mode={mode}")
                assert bool((guard[0] == 7.0).all()) and bool((guard[M + 1] == 7.0).all())
                assert torch.equal(y, dps.dps_linear(mode, enc, x, p, r if mode else None))   # run-to-run bits
                count += 1
    assert dps.dps_stream_status() == dps.DPS_OK
    print(f"all {count} cases passed")


# 80 tiles of 256 tokens: one round and 6 to 14 tiles more on 74 to 66 pairs, each cut into at least 4 pieces; the last token
# tile has 108 tokens, which end inside a piece
CUT = (2440, 1040, 1900)


@pytest.mark.gpu
def test_last_round_in_pieces_in_child_process():
    env = dict(os.environ, DPS_FORCE_PATH="pair", DPS_PAIR_TOKENS="256", DPS_PAIR_SPLIT="1", DPS_DEBUG="1", PYTHONPATH=REPO)
    out = subprocess.run([sys.executable, os.path.abspath(__file__), ",".join(map(str, CUT))], cwd=REPO, env=env,
                         capture_output=True, text=True, timeout=900)
    assert out.returncode == 0, out.stdout[-2000:] + out.stderr[-4000:]
    assert "all 6 cases passed" in out.stdout
    parts = [int(p) for p in re.findall(r"\[dps\] pair full=.*? tail=(\d+)x", out.stderr)]
    assert len(parts) == 12 and min(parts) > 1, out.stderr[-2000:]


@pytest.mark.gpu
@pytest.mark.parametrize("tokens,split", VARIANTS)
def test_pair_kernel_in_child_process(tokens, split):
    env = dict(os.environ, DPS_FORCE_PATH="pair", PYTHONPATH=REPO)
    if tokens:
        env.update(DPS_PAIR_TOKENS=str(tokens), DPS_PAIR_SPLIT=str(split))
    shapes = SHAPES + (MANY if tokens in (0, 192) else [])
    out = subprocess.run([sys.executable, os.path.abspath(__file__)] + [",".join(map(str, s)) for s in shapes], cwd=REPO, env=env,
                         capture_output=True, text=True, timeout=900)
    assert out.returncode == 0, out.stdout[-2000:] + out.stderr[-4000:]
    assert f"all {len(shapes) * 3 * 2} cases passed" in out.stdout


if __name__ == "__main__":
    _run([tuple(map(int, a.split(","))) for a in sys.argv[1:]])
