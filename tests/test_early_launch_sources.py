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


def test_pair_set_up_meets_again_before_its_aligned_barriers():
    """Lane 0 of a warp initialises barriers alone; what follows (bar.sync, barrier.cluster.arrive.aligned, tcgen05.alloc) is for whole warps."""
    text = (CSRC / "pair_linear.cu").read_text()
    set_up = text[text.index("if (warp == 0) {\n        if (lane == 0) {"):text.index("    cluster_wait();")]
    parted = [m.start() for m in re.finditer(r"lane == 0\)", set_up)]
    assert len(parted) == 2
    for at in parted:
        after = set_up[at:]
        meets = after.index("__syncwarp()")
        assert all(meets < after.index(b) for b in ("named_barrier", "cluster_arrive") if b in after), after[:meets]
    # between the second warp's set-up and the block's barrier
    tail = set_up[parted[1]:]
    assert tail.index("__syncwarp()") < tail.index("tmem_alloc_pair")


def test_fp8_epilogue_waits_itself_for_the_scales_it_reads():
    """The scales are the preceding kernel's output, read with ordinary loads: the warps that read them wait for that kernel, not another warp for them."""
    text = (CSRC / "fp8act.cu").read_text()
    kernel = text[text.index("fp8act_linear_kernel("):]
    kernel = kernel[:kernel.index("\n}\n")]
    reads = [m.start() for m in re.finditer(r"prm\.scale\[", kernel)]
    role = kernel.index("// ---------------- epilogue")
    assert reads and all(role < at for at in reads)
    assert "grid_dependency_wait()" in kernel[role:reads[0]]
