"""The native marshalling: what it does not take goes the ctypes way and is refused there as before."""
import ctypes
import subprocess
import sysconfig
import threading
import time

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


@pytest.fixture
def plain_call():
    """A call that the native entry takes, and a way to put another function in the place of the library's; undone afterwards."""
    w = workloads.weights(136, 144, 1, device="cuda:0")
    p, r, enc = dps.dps_split_weights(w)
    x = workloads.activations(5, 144, 2, device="cuda:0")
    assert binding._fast_linear is not None
    set_linear = binding._fast_linear.__self__.set_linear
    yield (enc, x, p, r), lambda fn: set_linear(ctypes.cast(fn, ctypes.c_void_p).value)
    set_linear(ctypes.cast(binding.library().dps_linear, ctypes.c_void_p).value)


@pytest.mark.gpu
def test_plain_calls_are_taken_and_go_to_the_current_stream(plain_call):
    (enc, x, p, r), _ = plain_call
    y = binding._fast_linear(dps.DPS_MODE_FULL, enc, x, p, r, None)
    assert isinstance(y, torch.Tensor)
    out = torch.zeros_like(y)
    torch.cuda.synchronize()
    graph, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(graph, stream=side):            # a launch on another stream is not in the graph
        assert binding._fast_linear(dps.DPS_MODE_FULL, enc, x, p, r, out) is out
    torch.cuda.synchronize()
    assert bool((out == 0).all())
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, y)


@pytest.mark.gpu
def test_other_threads_run_while_the_call_blocks(plain_call):
    (enc, x, p, r), put = plain_call
    put(ctypes.CDLL(None).sleep)                          # sleep(mode) seconds, then status 0
    ticks, stop = [], threading.Event()

    def tick():
        while not stop.wait(0.01):
            ticks.append(time.monotonic())
    thread = threading.Thread(target=tick)
    thread.start()
    try:
        begin = time.monotonic()
        assert isinstance(dps.dps_linear(1, enc, x, p, r), torch.Tensor)
        end = time.monotonic()
    finally:
        stop.set()
        thread.join()
    assert end - begin > 0.9
    assert sum(begin + 0.1 < t < end - 0.1 for t in ticks) > 20


@pytest.mark.gpu
def test_a_failed_call_is_reported_and_not_made_again(plain_call):
    (enc, x, p, r), put = plain_call
    calls = []

    def fails(*args):
        calls.append(args)
        return binding.DPS_ERR_CUDA
    fn = ctypes.CFUNCTYPE(ctypes.c_int, *binding.library().dps_linear.argtypes)(fails)
    put(fn)
    before = dps.dps_launch_count()
    with pytest.raises(dps.DpsError) as caught:
        dps.dps_linear(dps.DPS_MODE_FULL, enc, x, p, r)
    assert caught.value.status == binding.DPS_ERR_CUDA
    assert len(calls) == 1 and dps.dps_launch_count() == before


def test_a_module_of_another_version_is_not_taken(monkeypatch):
    build.build_fastcall()
    lib = binding.library()
    monkeypatch.setattr(binding, "_fast_linear", None)
    monkeypatch.setattr(torch, "__version__", "2.99.0")
    binding._load_fastcall(lib)
    assert binding._fast_linear is None
    monkeypatch.undo()
    binding._load_fastcall(lib)
    assert binding._fast_linear is not None


OLDER = r"""
#include <Python.h>
static PyObject* nothing(PyObject* self, PyObject* arg) { Py_RETURN_NONE; }
static PyMethodDef methods[] = {{"set_linear", nothing, METH_O, 0}, {"linear", nothing, METH_O, 0}, {0, 0, 0, 0}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_fastcall", 0, -1, methods};
PyMODINIT_FUNC PyInit__fastcall(void) { return PyModule_Create(&module); }
"""


def test_a_module_that_lacks_an_entry_is_not_taken(monkeypatch, tmp_path):
    lib = binding.library()
    (tmp_path / "older.c").write_text(OLDER)
    subprocess.run(["gcc", "-shared", "-fPIC", "-I", sysconfig.get_paths()["include"], str(tmp_path / "older.c"), "-o", str(tmp_path / "older.so")], check=True)
    monkeypatch.setattr(binding, "_fast_linear", None)
    monkeypatch.setattr(binding, "_native", None)
    monkeypatch.setattr(binding, "fastcall_path", lambda: tmp_path / "older.so")
    binding._load_fastcall(lib)
    assert binding._fast_linear is None and binding._native is None


def test_the_module_is_named_by_its_source(monkeypatch, tmp_path):
    here = binding.fastcall_path()
    other = tmp_path / "fastcall.cpp"
    other.write_bytes(binding.FASTCALL_SOURCE.read_bytes() + b"\n")
    monkeypatch.setattr(binding, "FASTCALL_SOURCE", other)
    assert binding.fastcall_path() != here and binding.fastcall_path().parent == here.parent


def test_other_entries_pass_on_what_they_do_not_take():
    build.build_fastcall()
    if binding._native is None:
        binding._load_fastcall(binding.library())
    native, h, b = binding._native, torch.zeros((8, 16), dtype=torch.float16), torch.zeros((8, 16), dtype=torch.uint8)
    assert native.split_weights(h, 0, None, None) is None and native.split_weights("w", 0, None, None) is None
    assert native.reconstruct(b, b, 1, None) is None and native.reconstruct(b, b, "1", None) is None
    assert native.moe_linear(0, [1], h, None, h, b, None, None, None) is None
    assert native.moe_linear(0, [1] * 2000, h, None, h, b, None, None, b) is None
    with pytest.raises(ValueError):
        dps.dps_split_weights(h)
    with pytest.raises(ValueError):
        dps.dps_reconstruct(b, None, 1)


@pytest.mark.gpu
def test_other_entries_answer_as_the_other_path_does():
    w = workloads.weights(24, 144, 3, device="cuda:0")
    stream = torch.cuda.current_stream()                  # an explicit stream: the ctypes way
    p, r, enc = dps.dps_split_weights(w)
    q, s, enc2 = dps.dps_split_weights(w, stream=stream)
    assert isinstance(enc, int) and enc == enc2 and torch.equal(p, q) and torch.equal(r, s) and p.shape == w.shape
    out = torch.empty_like(p)
    assert dps.dps_split_weights(w, dps.DPS_ENC_E5M2, out, r)[0] is out
    r = s
    assert torch.equal(dps.dps_reconstruct(p, r, enc), w)
    assert torch.equal(dps.dps_reconstruct(p, None, enc), dps.dps_reconstruct(p, None, enc, stream=stream))
    bad = torch.full_like(w, 4.0)
    with pytest.raises(dps.DpsError) as caught:
        dps.dps_split_weights(bad, dps.DPS_ENC_E4M3)
    assert caught.value.status == binding.DPS_ERR_DATA
    x = workloads.activations(3, 144, 4, device="cuda:0")
    tok, exp = (torch.tensor(v, dtype=torch.int32, device="cuda:0") for v in ([0, 0, 2, 1], [0, 1, 1, 0]))
    planes, res = torch.stack([p, p]), torch.stack([r, r])
    ws = torch.empty(dps.dps_moe_workspace_bytes(4, 2, 144), dtype=torch.uint8, device="cuda:0")
    for mode in (dps.DPS_MODE_FAST, dps.DPS_MODE_FULL):
        args = (mode, [enc, enc], x, tok, exp, planes, res if mode else None)
        y = dps.dps_moe_linear(*args, workspace=ws)
        assert torch.equal(y, dps.dps_moe_linear(*args, workspace=ws, stream=stream)) and torch.equal(y, dps.dps_moe_linear(*args))
        mine = torch.empty_like(y)
        assert dps.dps_moe_linear(*args, y=mine, workspace=ws) is mine and torch.equal(mine, y)
    for wrong, error in [(dict(workspace=ws[:16]), dps.DpsError), (dict(workspace=ws.cpu()), ValueError)]:
        with pytest.raises(error):
            dps.dps_moe_linear(dps.DPS_MODE_FAST, [enc, enc], x, tok, exp, planes, None, **wrong)
    with pytest.raises(dps.DpsError):
        dps.dps_moe_linear(dps.DPS_MODE_FULL, [enc, 77], x, tok, exp, planes, res, workspace=ws)


@pytest.mark.gpu
def test_other_entries_take_the_current_stream():
    """All three beside a busy default stream: their answers are there once their own stream is through, and they wait for what is on it."""
    w = workloads.weights(64, 272, 3, device="cuda:0")
    p0, r0, enc = dps.dps_split_weights(w)
    x, token, expert = workloads.activations(5, 272, 4, device="cuda:0"), None, torch.tensor([1, 0, 1, 0, 0], dtype=torch.int32, device="cuda:0")
    planes, res = torch.stack([p0, p0]), torch.stack([r0, r0])
    ws = torch.empty(dps.dps_moe_workspace_bytes(5, 2, 272), dtype=torch.uint8, device="cuda:0")
    want = dps.dps_moe_linear(dps.DPS_MODE_FULL, [enc, enc], x, token, expert, planes, res, workspace=ws)
    side, done = torch.cuda.Stream(), torch.cuda.Event()
    source, late, answers = torch.zeros_like(w), torch.zeros_like(x), {}
    torch.cuda.synchronize()
    with torch.cuda.stream(side):
        torch.cuda._sleep(20_000_000)                    # 10 ms in front of the inputs: a call on another stream would read the zeros
        source.copy_(w)
        late.copy_(x)
        answers["reconstruct"] = dps.dps_reconstruct(p0, r0, enc)
        answers["moe"] = dps.dps_moe_linear(dps.DPS_MODE_FULL, [enc, enc], late, token, expert, planes, res, workspace=ws)
        started = not side.query()
        done.record()
        p, r, got = dps.dps_split_weights(source, dps.DPS_ENC_E5M2)
    torch.cuda._sleep(2_000_000_000)                     # a second on the default stream, which none of the answers waits for
    side.synchronize()
    assert started and done.query() and not torch.cuda.default_stream().query()
    with torch.cuda.stream(side):
        q, s, _ = dps.dps_split_weights(w, dps.DPS_ENC_E5M2, stream=side)
        assert got == dps.DPS_ENC_E5M2 and torch.equal(p, q) and torch.equal(r, s)
        assert torch.equal(answers["reconstruct"], w) and torch.equal(answers["moe"], want)
    torch.cuda.synchronize()
