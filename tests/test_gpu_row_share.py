"""GPU: a matrix of whole rounds of CTA pairs and a rest that is launched by itself, against the oracle: one row group to many in the rest, the widths of
both families, K of a few steps (pinned by DPS_ROW_CUT, in a child process: the library reads its knobs once); and, at sizes of the rule, the
launches on both sides of its edges."""
import os
import subprocess
import sys

import pytest

from tests import test_gpu_pair_linear as checks
from tests.helpers import launch_lines

pytestmark = pytest.mark.gpu
ROUND = 74 * 256
# (N, K, M): a rest of 8 rows, of one decode tile and a bit, of several row tiles; one round and two; token widths up to 256
SHAPES = [(ROUND + 8, 144, 17), (ROUND + 136, 272, 33), (2 * ROUND + 2440, 80, 64), (ROUND + 264, 1040, 70), (ROUND + 520, 144, 129), (2 * ROUND + 8, 16, 256)]


def test_pinned_cut_in_child_process():
    env = dict(os.environ, DPS_ROW_CUT="1", DPS_DEBUG="1", PYTHONPATH=checks.REPO)
    out = subprocess.run([sys.executable, os.path.abspath(checks.__file__), *(",".join(map(str, s)) for s in SHAPES)], cwd=checks.REPO, env=env,
                         capture_output=True, text=True, timeout=900)
    assert out.returncode == 0, out.stdout[-2000:] + out.stderr[-4000:]
    assert f"all {len(SHAPES) * 3 * 2} cases passed" in out.stdout
    lines = [line for line in out.stderr.splitlines() if line.startswith("[dps] ")]
    whole = [i for i, line in enumerate(lines) if line.startswith("[dps] pair") and any(f" N={n * ROUND} " in line for n in (1, 2))]
    assert whole == list(range(0, len(lines), 2)) and len(lines) == len(SHAPES) * 3 * 2 * 2 * 2      # two launches a call, two calls a case


def test_launches_at_the_edges():
    def families(mode, M, N, K):
        return [(line.split()[1], int(line.split(" N=")[1].split()[0])) for line in launch_lines([(mode, M, N, K)])]

    assert families(1, 64, 86 * 256, 5120) == [("pair", ROUND), ("umma", 12 * 256)]
    assert families(1, 64, 112 * 256, 5120) == [("pair", 112 * 256)]
    assert families(0, 64, 86 * 256, 4096) == [("umma", 86 * 256)]
    assert families(1, 24, 75 * 256, 8192) == [("pair", ROUND), ("umma", 256)]
    assert families(1, 16, 75 * 256, 8192) == [("umma", 75 * 256)]
    assert families(0, 48, 60 * 256, 4096) == [("pair", 60 * 256)]
    assert families(0, 48, 48 * 256, 4096) == [("umma", 48 * 256)]
