"""FP64 stages with whole hops at the Ls whose CTAs have 16 sites (6 and 10: two CTAs share a
32-site tile), on lattices large enough for the launch rule to take them, which the kernel names
of the call show (the last template argument: thread groups per site, 1 for whole hops)."""
import re

import numpy as np
import pytest

from oracle import dwf_oracle as o
from paper_1804_08593_gb300 import inputs
from tests.gpu_common import TOL, cuda, host, lib, rand_even, rel

pytestmark = pytest.mark.gpu

DIMS = (12, 12, 12, 12)


def _handle(Ls, mf, b, c, seed):
    dwf = lib()
    rng = np.random.default_rng(seed)
    U = inputs.gauge_links(DIMS, 0.3, rng)
    p = o.DWFParams(DIMS, Ls, 1.8, mf, b, c)
    return dwf, rng, U, p, dwf.dwf_create(DIMS, Ls, p.M5, mf, b, c, cuda(U))


def _stage_kernels(call):
    """(Ls, post, groups) of every FP64 stage that `call` launches."""
    import torch
    from torch.profiler import ProfilerActivity, profile
    activities = [ProfilerActivity.CPU, ProfilerActivity.CUDA]
    with profile(activities=activities):   # a process's first profile is empty
        torch.cuda.synchronize()
    with profile(activities=activities) as prof:
        call()
    pat = re.compile(r"stage64_kernel<(\d+), \w+, \w+, (\d+), (\d+)>")
    return {tuple(int(v) for v in m.groups()) for m in (pat.search(e.name) for e in prof.events())
            if m}


@pytest.mark.parametrize("Ls,b,c,post", [(6, 1.5, 0.5, 4), (10, 1.5, 0.5, 4), (10, 1.0, 0.0, 4),
                                         (6, 0.5, 1.5, 1), (10, 0.5, 1.5, 1)])
def test_whole_hops_match_oracle(Ls, b, c, post):
    """post 4: by recurrence; b = 0.5, c = 1.5 has |beta/alpha| > 1: the dense matrices (1)."""
    dwf, rng, U, p, h = _handle(Ls, 0.07, b, c, 43)
    x = rand_even(rng, DIMS, Ls)
    out = cuda(np.zeros_like(x))
    dx = cuda(x)
    seen = _stage_kernels(lambda: dwf.dwf_apply(h, "MdagM", dx, out, "f64"))
    assert (Ls, post, 1) in seen and all(k[0] == Ls and k[2] == 1 for k in seen), seen
    assert rel(host(out), o.mdagm(U, x, p)) <= TOL["f64"]


@pytest.mark.parametrize("Ls", [6, 10])
def test_cg_with_16_site_ctas(Ls):
    """The solve's sums run over two CTAs per tile."""
    dwf, rng, U, p, h = _handle(Ls, 0.2, 1.5, 0.5, 47)
    phi = inputs.even_source(DIMS, Ls, rng)
    x = cuda(np.zeros_like(phi))
    st = dwf.dwf_cg(h, cuda(phi), x, 1e-10, 5000, "f64")
    assert st["true_residual"] <= 1e-10
    assert o.true_residual(U, host(x), phi, p) <= 1.5e-10
