"""Training stops at the step whose tensor-core wait ran out: once the flag is up, a step changes neither
parameters nor moments. The flag is set by hand; no wait is made to run out."""
import ctypes
import re
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

P = 128 * 32 + 128 + 128 * 128 + 128 + 128 + 1


class MlpTrain(ctypes.Structure):
    _fields_ = [(f, ctypes.c_void_p) for f in ("params", "m", "v", "X", "target", "Xb", "H1", "H2", "dH2", "dH1", "dy",
                                               "W1b", "W2b")] + [("R", ctypes.c_int64), ("err", ctypes.c_void_p)]


@pytest.fixture(scope="module")
def lib():
    from paper_2508_21287_gb300 import build
    path = build.build()
    names = subprocess.run(["nm", "-D", "--defined-only", path], capture_output=True, text=True).stdout
    so = ctypes.CDLL(path)
    get = lambda f: getattr(so, re.search(r" T (_ZN3dmk\d+%s\w*)" % f, names).group(1))
    fns = {f: get(f) for f in ("mlp_train_bytes", "mlp_train_layout", "mlp_train_begin", "mlp_train_step")}
    fns["mlp_train_bytes"].restype = ctypes.c_int64
    return fns


@pytest.mark.parametrize("n", [16, 300])
def test_no_step_once_the_flag_is_up(lib, n):
    torch = pytest.importorskip("torch")
    gen = torch.Generator(device="cuda").manual_seed(n)
    state = [torch.randn(P, generator=gen, device="cuda") * 0.05, torch.zeros(P, device="cuda"), torch.zeros(P, device="cuda")]
    X, t = torch.randn(n, 32, generator=gen, device="cuda"), torch.randn(n, generator=gen, device="cuda")
    idx = torch.arange(n, dtype=torch.int32, device="cuda")
    work = torch.zeros(lib["mlp_train_bytes"](n), dtype=torch.uint8, device="cuda")
    err, loss = torch.zeros(2, dtype=torch.int32, device="cuda"), torch.zeros(1, device="cuda")
    T = MlpTrain(params=state[0].data_ptr(), m=state[1].data_ptr(), v=state[2].data_ptr(), X=X.data_ptr(),
                 target=t.data_ptr(), err=err.data_ptr())
    stream = torch.cuda.current_stream().cuda_stream
    lib["mlp_train_layout"](ctypes.byref(T), ctypes.c_void_p(work.data_ptr()), n)
    assert lib["mlp_train_begin"](ctypes.byref(T), ctypes.c_void_p(stream)) == 0

    def step(k):
        assert lib["mlp_train_step"](ctypes.byref(T), ctypes.c_void_p(idx.data_ptr()), n, ctypes.c_void_p(loss.data_ptr()),
                                     ctypes.c_float(1e-3), k, ctypes.c_void_p(stream)) == 0
        torch.cuda.synchronize()
        return [x.cpu().numpy().copy() for x in state]

    start = [x.cpu().numpy().copy() for x in state]
    one = step(1)
    assert not np.array_equal(one[0], start[0]) and err.tolist() == [0, 1]
    err[0] = 1
    for k in (2, 3):
        assert all(np.array_equal(a, b) for a, b in zip(step(k), one)) and err.tolist() == [1, 1]
    err[0] = 0  # down again: the next step is taken
    assert not np.array_equal(step(2)[0], one[0]) and err.tolist() == [0, 2]
