"""A dense linear that is two launches (whole rounds of CTA pairs, the rest of the rows): what can fail in front of the second is done before the first is
enqueued, so that a call that fails there has enqueued nothing."""
import re
from pathlib import Path

import pytest

from tests.helpers import host_program

CSRC = Path(__file__).resolve().parents[1] / "paper_2609_34380_b200" / "csrc"
PROGRAM = r"""
#include "two_launches.h"
#include <cstdio>
int main() {
    int bad_prepare, bad_first, bad_second;
    while (scanf("%d %d %d", &bad_prepare, &bad_first, &bad_second) == 3) {
        const int e = dps::launch_two([&] { printf("2 "); return bad_first; }, [&](bool only) { printf(only ? "1 " : "3 "); return only ? bad_prepare : bad_second; });
        printf("%d\n", e);
    }
}
"""


def test_nothing_is_enqueued_in_front_of_a_failed_preparation(tmp_path):
    # what was done (1: the second launch prepared, 2: the first launch, 3: the second), then the error
    wanted = {(0, 0, 0): (1, 2, 3, 0), (7, 0, 0): (1, 7), (0, 8, 0): (1, 2, 8), (0, 0, 9): (1, 2, 3, 9)}
    assert host_program(tmp_path, PROGRAM)(list(wanted)) == list(wanted.values())


def test_a_preparation_makes_every_tensor_map_and_launches_nothing():
    for file, launcher in (("pair_linear.cu", "launch_enc"), ("umma_linear.cu", "launch_tn")):
        text = (CSRC / file).read_text()
        body = text[text.index(f"cudaError_t {launcher}("):]
        body = body[:body.index("\n}\n")]
        at = body.index("if (prepare_only) return cudaSuccess;")
        assert "setup.run" in body[:at] and "make_map_2d" in body[:at] and "cudaLaunchKernelEx" not in body[:at], file
        assert "cudaLaunchKernelEx" in body[at:] and not re.search(r"make_map_2d|return cudaErrorInvalid", body[at:]), file
