"""Kernels that start while their predecessor still runs must not read its output through the non-coherent path: in a kernel that
waits for the preceding grid, only the weight planes (model state, not that grid's output) may be __restrict__.  The streaming
kernel's x is the one exception; its reason and its price stand beside that kernel."""
import re
from pathlib import Path

CSRC = Path(__file__).resolve().parents[1] / "paper_2609_34380_b200" / "csrc"


def early_kernels():
    for path in sorted(CSRC.glob("*.cu")):
        for part in re.split(r"(?=__global__ void)", path.read_text())[1:]:
            if "grid_dependency_wait()" in part[:part.index("\n}\n")]:
                yield path.name, part[:part.index("{")]


def test_only_planes_are_restrict_in_early_launched_kernels():
    early = list(early_kernels())
    assert {f for f, _ in early} >= {"decode_mma.cu", "fp8act.cu", "gemv.cu", "moe.cu", "umma_linear.cu", "pair_linear.cu"}
    for file, head in early:
        marked = set(re.findall(r"__restrict__\s+(\w+)", head))
        allowed = {"P", "Rp", "x", "y"} if file == "decode_mma.cu" else {"P", "Rp"}
        assert marked <= allowed, f"{file}: {marked} in {head}"
