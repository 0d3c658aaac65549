"""The binding's native fast path against its Python path (taken when a stream is given), and what neither may accept."""
import ctypes
import subprocess
import threading
import time

import numpy as np
import pytest
import torch

from oracle import direct
from paper_2208_00763_b200 import binding as hk
from paper_2208_00763_b200 import inputs
from gpu_util import assert_exact, dev

pytestmark = pytest.mark.gpu


def _both(call, **kw):
    """The call's result by the native path and by the Python path."""
    return call(**kw), call(stream=torch.cuda.current_stream(), **kw)


def test_both_paths_give_the_same():
    f, g = inputs.conv1d_case(5003, 5, 4, 4, False, True, seed=1)
    for y in _both(lambda **kw: hk.conv1d(dev(f), dev(g), 4, 4, False, True, **kw)):
        assert y.dtype == torch.int32 and y.shape == (5007,)
        assert_exact(y, direct.conv1d_full(f, g), "conv1d")
    f2, g2 = inputs.conv1d_case(5003, 5, 2, 2, False, False, seed=2)
    dense = torch.from_numpy(inputs.to_dense(f2, 2)).cuda()
    for y in _both(lambda **kw: hk.conv1d_dense(dense, 5003, dev(g2), 2, 2, False, False, **kw)):
        assert_exact(y, direct.conv1d_full(f2, g2), "conv1d_dense")
    for word in (32, 64):
        a, b = _both(lambda **kw: hk.pack(dev(f), 4, False, 10, 3, word, **kw))
        assert a.dtype == b.dtype and torch.equal(a, b)
    x, w = inputs.conv2d_case(2, 6, 8, 10, 5, 3, 4, 4, True, True, seed=3)
    ref = direct.conv2d_nchw(x, w, 1)
    space = torch.empty(hk.conv2d_workspace_bytes(2, 6, 8, 10, 5, 3, 1), dtype=torch.uint8, device="cuda")
    for rq, want, dtype in ((None, ref, torch.int32), ((5, -8, 7), direct.requant(ref, 5, -8, 7), torch.int8)):
        for ws in (None, space):
            for y in _both(lambda **kw: hk.conv2d(dev(x), dev(w), 1, 4, 4, True, True, requant=rq, workspace=ws, **kw)):
                assert y.dtype == dtype
                assert_exact(y, want, "conv2d")
    for bits in (8, 4):
        a, b = _both(lambda **kw: hk.conv2d_dense(dev(x).reshape(-1), x.shape, 8, dev(w).reshape(-1), w.shape, 8, 1, 4, 4, True, True,
                                                  requant=(5, -8, 7), out_store_bits=bits, **kw))
        assert a.dtype == b.dtype and a.shape == b.shape and torch.equal(a, b)


def test_caller_output_and_current_stream():
    f, g = inputs.conv1d_case(70001, 3, 4, 4, False, False, seed=4)
    d_f, d_g = dev(f), dev(g)
    out = torch.empty(70003, dtype=torch.int32, device="cuda")
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        out.fill_(-1)
        assert hk.conv1d(d_f, d_g, 4, 4, False, False, out=out) is out       # on `side`, after the fill
    side.synchronize()
    assert_exact(out, direct.conv1d_full(f, g), "side stream")


def test_errors_are_those_of_the_python_path():
    f, g = dev(np.zeros(100, dtype=np.int64)), dev(np.zeros(3, dtype=np.int64))
    for bad in (torch.empty(101, dtype=torch.int32, device="cuda"), torch.empty(102, dtype=torch.float32, device="cuda"),
                torch.empty(204, dtype=torch.int32, device="cuda")[::2], torch.empty(102, dtype=torch.int32)):
        with pytest.raises(ValueError):
            hk.conv1d(f, g, 4, 4, False, False, out=bad)
    for bad in (f.cpu(), f.float(), torch.zeros(200, dtype=torch.int8, device="cuda")[::2]):
        with pytest.raises(ValueError):
            hk.conv1d(bad, g, 4, 4, False, False)
        with pytest.raises(ValueError):
            hk.pack(bad, 4, False, 10, 3)
    with pytest.raises(hk.HikonvError) as err:
        hk.conv1d(f, g, 9, 4, False, False)
    assert err.value.status == hk.ERR_INVALID_ARG
    x, w = torch.zeros((1, 4, 6, 6), dtype=torch.int8, device="cuda"), torch.zeros((2, 4, 3, 3), dtype=torch.int8, device="cuda")
    with pytest.raises(ValueError):
        hk.conv2d(x, torch.zeros((2, 5, 3, 3), dtype=torch.int8, device="cuda"), 1, 4, 4, True, True)
    with pytest.raises(ValueError):
        hk.conv2d(x, w, 1, 4, 4, True, True, out=torch.empty((1, 2, 6, 6), dtype=torch.int8, device="cuda"))
    with pytest.raises(hk.HikonvError) as err:
        hk.conv2d(x, w, 1, 4, 4, True, True, workspace=torch.empty(16, dtype=torch.uint8, device="cuda"))
    assert err.value.status == hk.ERR_WORKSPACE
    with pytest.raises(hk.HikonvError) as err:
        hk.conv2d(x, w, 5, 4, 4, True, True)
    assert err.value.status == hk.ERR_UNSUPPORTED
    with pytest.raises(hk.HikonvError) as err:
        hk.conv2d(x, w, 1, 4, 4, True, True, stride=2)
    assert err.value.status == hk.ERR_UNSUPPORTED
    with pytest.raises(ValueError):
        hk.conv2d_dense(x.reshape(-1), (1, 4, 6, 7), 8, w.reshape(-1), w.shape, 8, 1, 4, 4, True, True)


def test_other_threads_run_during_a_library_call(tmp_path):
    # the native path bound to a stand-in that sleeps: a second Python thread must get on meanwhile
    src, so = tmp_path / "slow.c", tmp_path / "slow.so"
    src.write_text("#include <time.h>\nint slow(void) { struct timespec t = {0, 300000000}; nanosleep(&t, 0); return 0; }\n")
    subprocess.run(["gcc", "-shared", "-fPIC", "-o", str(so), str(src)], check=True)
    slow = ctypes.cast(ctypes.CDLL(str(so)).slow, ctypes.c_void_p).value
    f, g = torch.zeros(64, dtype=torch.int8, device="cuda"), torch.zeros(3, dtype=torch.int8, device="cuda")
    x, w = torch.zeros((1, 4, 6, 6), dtype=torch.int8, device="cuda"), torch.zeros((2, 4, 3, 3), dtype=torch.int8, device="cuda")
    calls = {"hikonv_conv1d": lambda: hk.conv1d(f, g, 4, 4, False, False),
             "hikonv_conv1d_dense": lambda: hk.conv1d_dense(f.view(torch.uint8), 64, g, 4, 4, False, False),
             "hikonv_pack": lambda: hk.pack(f, 4, False, 10, 3),
             "hikonv_conv2d": lambda: hk.conv2d(x, w, 1, 4, 4, True, True),
             "hikonv_conv2d_dense": lambda: hk.conv2d_dense(x.reshape(-1), x.shape, 8, w.reshape(-1), w.shape, 8, 1, 4, 4, True, True)}
    for name, call in calls.items():
        call()
        hk._fast.bind(name, slow)
        try:
            done, ticks = threading.Event(), []

            def tick():
                while not done.is_set():
                    ticks.append(time.monotonic())
                    time.sleep(0.01)

            other = threading.Thread(target=tick)
            other.start()
            t0 = time.monotonic()
            call()
            t1 = time.monotonic()
            done.set()
            other.join()
        finally:
            hk._fast.bind(name, ctypes.cast(getattr(hk.lib(), name), ctypes.c_void_p).value)
        assert t1 - t0 > 0.25 and sum(t0 + 0.05 < t < t1 - 0.05 for t in ticks) >= 3, name
