"""A dense linear that is two launches (whole rounds of CTA pairs, the rest of the rows): what can fail in front of the second is done before the first is
enqueued, so that a call that fails there has enqueued nothing."""
import re
import shutil
import subprocess
from pathlib import Path

import pytest

CSRC = Path(__file__).resolve().parents[1] / "paper_2609_34380_b200" / "csrc"
PROGRAM = r"""
#include "two_launches.h"
#include <cstdio>
#include <cstdlib>
int main(int, char** argv) {
    const int bad_prepare = atoi(argv[1]), bad_first = atoi(argv[2]), bad_second = atoi(argv[3]);
    const int e = dps::launch_two([&] { printf("first "); return bad_first; },
                                  [&](bool only) { printf(only ? "prepare " : "second "); return only ? bad_prepare : bad_second; });
    printf("%d", e);
}
"""


@pytest.mark.parametrize("bad,want", [((0, 0, 0), "prepare first second 0"), ((7, 0, 0), "prepare 7"), ((0, 8, 0), "prepare first 8"), ((0, 0, 9), "prepare first second 9")])
def test_nothing_is_enqueued_in_front_of_a_failed_preparation(tmp_path, bad, want):
    gxx = shutil.which("g++")
    assert gxx
    (tmp_path / "two.cpp").write_text(PROGRAM)
    subprocess.run([gxx, "-std=c++17", "-I", str(CSRC), str(tmp_path / "two.cpp"), "-o", str(tmp_path / "two")], check=True)
    assert subprocess.run([str(tmp_path / "two"), *map(str, bad)], text=True, capture_output=True, check=True).stdout == want


def test_a_preparation_makes_every_tensor_map_and_launches_nothing():
    for file, launcher in (("pair_linear.cu", "launch_enc"), ("umma_linear.cu", "launch_tn")):
        text = (CSRC / file).read_text()
        body = text[text.index(f"cudaError_t {launcher}("):]
        body = body[:body.index("\n}\n")]
        at = body.index("if (prepare_only) return cudaSuccess;")
        assert "setup.run" in body[:at] and "make_map_2d" in body[:at] and "cudaLaunchKernelEx" not in body[:at], file
        assert "cudaLaunchKernelEx" in body[at:] and not re.search(r"make_map_2d|return cudaErrorInvalid", body[at:]), file
