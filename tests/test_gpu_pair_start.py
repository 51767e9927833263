"""GPU: the CTA-pair linear where its start and its end can go wrong: a ring that is loaded before the pair meets and holds more, as many
or fewer units than K has; the units asked of L2 ahead, across the end of a tile and past the last one; partial sums of three ranges of K."""
import os
import subprocess
import sys

import pytest

from tests import test_gpu_pair_linear as pairs

REPO = pairs.REPO
# (N, K, M): K shorter than the ring, equal to it, longer; 76 row tiles on 74 pairs (a second tile); one and two token tiles of 192 to 256 tokens
SHAPES = [(264, 16, 192), (520, 256, 250), (264, 400, 224), (264, 1040, 440), (19208, 656, 200)]


@pytest.mark.gpu
@pytest.mark.parametrize("tokens,split,shapes", [(0, 0, SHAPES), (256, 3, [(264, 784, 255), (136, 1040, 33)]), (64, 3, [(520, 784, 31), (8, 2064, 64)])])
def test_start_and_end_in_child_process(tokens, split, shapes):
    env = dict(os.environ, DPS_FORCE_PATH="pair", PYTHONPATH=REPO)
    if tokens:
        env.update(DPS_PAIR_TOKENS=str(tokens), DPS_PAIR_SPLIT=str(split))
    out = subprocess.run([sys.executable, os.path.abspath(pairs.__file__)] + [",".join(map(str, s)) for s in shapes], cwd=REPO, env=env,
                         capture_output=True, text=True, timeout=900)
    assert out.returncode == 0, out.stdout[-2000:] + out.stderr[-4000:]
    assert f"all {len(shapes) * 3 * 2} cases passed" in out.stdout
