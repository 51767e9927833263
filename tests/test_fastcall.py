"""The native marshalling of dps_linear: what it does not take goes the ctypes way and is refused there as before."""
import pytest
import torch

import paper_2609_34380_b200 as dps
from paper_2609_34380_b200 import binding, build, workloads


def test_module_loads_and_passes_host_tensors_on():
    build.build_fastcall()
    binding.library()
    if binding._fast_linear is None:                      # the library was loaded before the module existed
        binding._load_fastcall(binding.library())
    x, p = torch.zeros((2, 16), dtype=torch.float16), torch.zeros((8, 16), dtype=torch.uint8)
    assert binding._fast_linear(0, 1, x, p, None, None) is None
    assert binding._fast_linear(0, 1, x, "p", None, None) is None
    assert binding._fast_linear(0, 1, x) is None
    with pytest.raises(ValueError):
        dps.dps_linear(0, 1, x, p, None)


@pytest.mark.gpu
def test_same_results_and_same_refusals():
    assert binding.FASTCALL_PATH.exists()
    w = workloads.weights(136, 144, 1, device="cuda:0")
    p, r, enc = dps.dps_split_weights(w)
    x = workloads.activations(5, 144, 2, device="cuda:0")
    assert binding._fast_linear is not None
    for mode in (dps.DPS_MODE_FAST, dps.DPS_MODE_FULL):
        y = dps.dps_linear(mode, enc, x, p, r)
        assert y.dtype == torch.float16 and y.shape == (5, 136) and y.device == x.device
        by_hand = dps.dps_linear(mode, enc, x, p, r, stream=torch.cuda.current_stream())       # the ctypes way
        out = torch.full_like(y, 7.0)
        assert dps.dps_linear(mode, enc, x, p, r, out) is out
        assert torch.equal(y, by_hand) and torch.equal(y, out)
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):                         # the current stream, not the default one
        side.wait_stream(torch.cuda.default_stream())
        z = dps.dps_linear(dps.DPS_MODE_FULL, enc, x, p, r)
    side.synchronize()
    assert torch.equal(z, y)
    assert dps.dps_linear(dps.DPS_MODE_FULL, enc, x[:0], p, r).shape == (0, 136)
    for bad, error in [((dps.DPS_MODE_FULL, enc, x, p, None), dps.DpsError), ((5, enc, x, p, r), dps.DpsError),
                       ((0, 77, x, p, r), dps.DpsError), ((0, enc, x[:, ::2], p, r), ValueError), ((0, enc, x.float(), p, r), TypeError),
                       ((0, enc, x.cpu(), p, r), ValueError), ((0, enc, x[:, :128].contiguous(), p, r), ValueError),
                       ((0, enc, x.t().contiguous().t(), p, r), ValueError)]:
        with pytest.raises(error):
            dps.dps_linear(*bad)
