"""GPU: CTA pairs with tiles of 320 and 384 tokens (two MMAs of half the tokens per step of A) against the oracle: tokens that end in the first
half, at its edge, in the second, in another tile; K of one step to many; more tiles than pairs; a last round cut into pieces.

DPS_FORCE_PATH / DPS_PAIR_TOKENS pin family and width; the library reads them once per process, so each run is a child process: the other
file's script.
"""
import os
import re
import subprocess
import sys

import pytest

from tests import test_gpu_pair_linear as checks

# (N, K, M)
SHAPES = [(8, 16, 257), (128, 64, 320), (136, 80, 385), (256, 400, 513), (264, 1040, 700), (512, 2064, 1000), (19208, 144, 400)]
# 15 row tiles of 5 or 6 token tiles: one round and a few tiles more, cut into pieces; the last token tile ends inside one
CUT = (3840, 528, 1700)


@pytest.mark.gpu
@pytest.mark.parametrize("tokens", [320, 384])
def test_wide_tiles_in_child_process(tokens):
    env = dict(os.environ, DPS_FORCE_PATH="pair", DPS_PAIR_TOKENS=str(tokens), DPS_DEBUG="1", PYTHONPATH=checks.REPO)
    shapes = SHAPES + [CUT]
    out = subprocess.run([sys.executable, os.path.abspath(checks.__file__)] + [",".join(map(str, s)) for s in shapes], cwd=checks.REPO,
                         env=env, capture_output=True, text=True, timeout=900)
    assert out.returncode == 0, out.stdout[-2000:] + out.stderr[-4000:]
    assert f"all {len(shapes) * 3 * 2} cases passed" in out.stdout
    launches = re.findall(r"\[dps\] pair full=.*? M=(\d+) .*?tokens=(\d+) .*?tail=(\d+)x", out.stderr)
    assert launches and {int(t) for _, t, _ in launches} == {tokens}, out.stderr[-2000:]
    assert max(int(p) for m, _, p in launches if int(m) == CUT[2]) > 1, out.stderr[-2000:]
