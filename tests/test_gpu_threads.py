"""Solves on one host thread while another host thread uses the same device: neither may see an
error of the other's, and the solution is the one of a solve alone, bit for bit."""
import ctypes
import threading

import numpy as np
import pytest

from paper_1804_08593_gb300 import inputs
from tests.gpu_common import cuda, host, lib

pytestmark = pytest.mark.gpu


def _blocking_stream():
    """A stream that synchronises with the legacy stream (torch's own streams do not)."""
    import torch
    from paper_1804_08593_gb300 import dwf
    rt = ctypes.CDLL(dwf.LIB_PATH)     # its CUDA runtime
    p = ctypes.c_void_p()
    assert rt.cudaStreamCreate(ctypes.byref(p)) == 0
    return torch.cuda.ExternalStream(p.value), lambda: rt.cudaStreamDestroy(p)


def _beside(other, solve, times):
    """Results of `times` solves while another thread repeats `other`, and that thread's errors."""
    import torch
    stop, errors = threading.Event(), []
    buf = torch.zeros(16, device="cuda")
    torch.cuda.synchronize()
    step = {"device_wait": torch.cuda.synchronize, "legacy_stream": lambda: buf.add_(1.0)}[other]

    def loop():
        while not stop.is_set():
            try:
                step()
            except Exception as e:
                errors.append(str(e).split("\n")[0])
                return

    t = threading.Thread(target=loop)
    t.start()
    try:
        out = [solve() for _ in range(times)]
    finally:
        stop.set()
        t.join()
    torch.cuda.synchronize()
    return out, errors


@pytest.mark.parametrize("blocking", [False, True])
@pytest.mark.parametrize("other", ["device_wait", "legacy_stream"])
@pytest.mark.parametrize("prec", ["f64", "f32"])
def test_cg_beside_another_thread(prec, other, blocking):
    import torch
    dwf = lib()
    dims, Ls = (4, 4, 4, 4), 8
    rng = np.random.default_rng(29)
    U, phi = cuda(inputs.gauge_links(dims, 0.2, rng)), cuda(inputs.even_source(dims, Ls, rng))
    stream, free = _blocking_stream() if blocking else (torch.cuda.Stream(), lambda: None)
    torch.cuda.synchronize()
    h = dwf.dwf_create(dims, Ls, 1.8, 0.1, 1.0, 0.0, U, stream)

    def solve():
        x = torch.zeros_like(phi)
        torch.cuda.current_stream().synchronize()
        dwf.dwf_cg(h, phi, x, 1e-10, 5000, prec)
        return host(x)

    alone = solve()
    got, errors = _beside(other, solve, 8)
    assert not errors, errors
    assert all(np.array_equal(g, alone) for g in got)
    h.close()
    free()


@pytest.mark.parametrize("blocking", [False, True])
@pytest.mark.parametrize("other", ["device_wait", "legacy_stream"])
@pytest.mark.parametrize("flexible", [False, True])
def test_mspcg_beside_another_thread(flexible, other, blocking):
    import torch
    dwf = lib()
    dims, Ls = (8, 4, 4, 8), 8
    rng = np.random.default_rng(37)
    U, phi = cuda(inputs.gauge_links(dims, 0.2, rng)), cuda(inputs.even_source(dims, Ls, rng))
    stream, free = _blocking_stream() if blocking else (torch.cuda.Stream(), lambda: None)
    torch.cuda.synchronize()
    h = dwf.dwf_create(dims, Ls, 1.8, 0.1, 1.5, 0.5, U, stream)

    def solve():
        x = torch.zeros_like(phi)
        torch.cuda.current_stream().synchronize()
        st = dwf.dwf_mspcg(h, (4, 4, 4, 4), 4, "f16", "f32", phi, x, 1e-10, 2000,
                           local_op=dwf.LOCAL_EXACT, flexible=flexible)
        assert st["true_residual"] <= 1e-10
        return host(x)

    for _ in range(4):     # the local solver's launch variant is decided
        alone = solve()
    got, errors = _beside(other, solve, 8)
    assert not errors, errors
    assert all(np.array_equal(g, alone) for g in got)
    h.close()
    free()


@pytest.mark.parametrize("form", ["stages", "persistent"])
def test_batch_beside_another_thread(form, monkeypatch):
    import torch
    dwf = lib()
    monkeypatch.setenv("DWF_BATCH_FORM", form)
    rng = np.random.default_rng(41)
    probs = []
    for dims, Ls, mf in (((4, 4, 4, 4), 4, 0.1), ((4, 4, 4, 8), 8, 0.05), ((4, 6, 2, 6), 8, 0.2)):
        phi = cuda(inputs.even_source(dims, Ls, rng))
        probs.append(dict(dims=dims, Ls=Ls, M5=1.8, mf=mf, b=1.5, c=0.5, phi=phi,
                          links=cuda(inputs.gauge_links(dims, 0.3, rng)), x=torch.zeros_like(phi)))
    torch.cuda.synchronize()

    def solve():
        st = dwf.dwf_batch_solve(probs, 1e-10, 20000)
        assert all(s["true_residual"] <= 1e-10 for s in st)
        return [host(p["x"]) for p in probs]

    solve()                # the chunk's launch shape is decided
    alone = solve()
    got, errors = _beside("device_wait", solve, 8)
    assert not errors, errors
    assert all(np.array_equal(a, b) for g in got for a, b in zip(g, alone))
