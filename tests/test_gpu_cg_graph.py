"""Plain CG on small lattices replays recorded iterations: only where a solve is long enough to
earn the recording back, and with the bits of the same iterations launched one by one."""
import numpy as np
import pytest

from paper_1804_08593_gb300 import inputs
from tests.gpu_common import cuda, host, lib

pytestmark = pytest.mark.gpu


def _problem(dims, Ls, b, c):
    rng = np.random.default_rng(31)
    return (cuda(inputs.gauge_links(dims, 0.3, rng)), cuda(inputs.even_source(dims, Ls, rng)),
            (dims, Ls, 1.8, 0.1, b, c))


@pytest.mark.parametrize("maxit,replayed", [(16, False), (23, False), (24, True), (56, True)])
def test_short_solves_record_no_graph(maxit, replayed):
    """Chunks of 8, 16, 32 iterations: a graph of 8 is recorded after the first chunk, if at least
    16 more may follow."""
    import torch
    from torch.profiler import ProfilerActivity, profile
    dwf = lib()
    U, phi, p = _problem((4, 4, 4, 4), 8, 1.5, 0.5)
    h = dwf.dwf_create(*p, U, torch.cuda.Stream())
    x = torch.zeros_like(phi)
    activities = [ProfilerActivity.CPU, ProfilerActivity.CUDA]
    with profile(activities=activities):   # a process's first profile is empty
        torch.cuda.synchronize()
    with profile(activities=activities) as prof:
        st = dwf.dwf_cg(h, phi, x, 1e-12, maxit, "f64", raise_on_fail=False)
    assert st["iterations"] == maxit
    names = [e.name for e in prof.events()]
    assert any("LaunchKernel" in n for n in names)
    assert any("GraphLaunch" in n for n in names) == replayed


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("dims,Ls,b,c", [((4, 4, 4, 4), 8, 1.0, 0.0), ((4, 4, 4, 4), 4, 1.5, 0.5),
                                         ((6, 6, 6, 10), 10, 1.5, 0.5), ((8, 8, 8, 16), 8, 1.5, 0.5)])
def test_replayed_iterations_are_the_launched_ones(dims, Ls, b, c, prec):
    """The profiler switch launches every iteration by itself."""
    import torch
    dwf = lib()
    U, phi, p = _problem(dims, Ls, b, c)
    out = {}
    for direct in (False, True):
        h = dwf.dwf_create(*p, U, torch.cuda.Stream())
        dwf.dwf_profile_enable(h, direct)
        x = torch.zeros_like(phi)
        torch.cuda.synchronize()
        st = dwf.dwf_cg(h, phi, x, 1e-10, 5000, prec, history=5000)
        out[direct] = host(x), st["history"]
    assert np.array_equal(out[False][0], out[True][0])
    assert out[False][1] == out[True][1]
