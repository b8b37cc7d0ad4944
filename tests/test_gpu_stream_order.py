"""Device memory that goes from torch to the library is used in the order of torch's stream.

The library runs a default-stream context on a non-blocking stream of its own.  A log-potential
that an earlier kernel is still writing, and a block of torch's pool that an earlier kernel is
still reading when it becomes dlogZ_dv or the workspace, must not be touched before that kernel
is done.  `busy` keeps the caller's stream occupied for some tens of milliseconds; without the
order the library's kernels, which take well under one, would be first.

Log Z sums worldlines in FP64 in the order of arrival (1e-12), the gradients in FP32 (1e-5 of
scale)."""
import contextlib

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

PARAMS = (1.0, 4.0, 1.0, 0.05, 0.5)


def lattice():
    from paper_2510_13866_gb300 import Lattice

    lat = Lattice(16, [1, 2, 3], precision="fp32")
    lat.set_params(*PARAMS)
    return lat


def busy():
    import torch

    a = torch.full((4096, 4096), 1.0 / 4096, device="cuda")
    for _ in range(16):
        a = a @ a
    return a


@pytest.mark.parametrize("made,called", [("default", "default"), ("default", "side"), ("side", "default"), ("side", "side")])
def test_log_potential_written_by_a_queued_kernel(made, called):
    import torch

    side = torch.cuda.Stream()
    on = lambda which: torch.cuda.stream(side) if which == "side" else contextlib.nullcontext()
    with on(made):
        lat = lattice()
    _, M, _ = lat._shapes()[0]
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    new = 0.5 * torch.randn(3 * 2 * M * 256, generator=g, device="cuda")
    torch.cuda.synchronize()
    lz0, dv0, dt0 = lat.log_weight_grad(v=new)
    torch.cuda.synchronize()
    v = torch.zeros_like(new)
    busy()  # a first matrix product sets its library up and would wait for that
    torch.cuda.synchronize()
    with on(called):
        busy()
        v.copy_(new)
        lz, dv, dt = lat.log_weight_grad(v=v)
    torch.cuda.synchronize()
    assert np.abs(lz - lz0).max() <= 1e-12 * np.abs(lz0).max()
    assert np.abs(dt - dt0).max() <= 1e-5 * np.abs(dt0).max()
    assert (dv - dv0).abs().max() <= 1e-5 * dv0.abs().max()
    lat.close()


@pytest.mark.parametrize("what", ["gradient", "workspace"])
def test_pool_block_that_a_queued_kernel_reads(what):
    import torch

    lat = lattice()
    if what == "gradient":
        _, M, _ = lat._shapes()[0]
        lat.log_weight_grad()
        n, dtype = 3 * 2 * M * 256, torch.float32
    else:
        n, dtype = lat.workspace_size() + 256, torch.uint8
    busy()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    old = torch.full((n,), 7, dtype=dtype, device="cuda")
    sink = torch.empty_like(old)
    busy()
    sink.copy_(old)
    del old  # its block is the next one of this size
    if what == "gradient":
        lat.log_weight_grad()
    else:
        lat.prepare()
    torch.cuda.synchronize()
    assert bool((sink == 7).all())
    lat.close()
