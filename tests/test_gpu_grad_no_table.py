"""The adjoint of a given log-potential without the memory for its exp(v) table: the exponentials are
taken at each use, with the same results (the sums over worldlines come in the order of arrival:
log Z 1e-12, the gradients 1e-5 of scale in FP32, 1e-12 in FP64)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,tol", [("fp32", 1e-5), ("fp64", 1e-12)])
def test_exponentials_at_each_use(prec, tol):
    import torch

    from paper_2510_13866_gb300 import Lattice

    Ls = [3, 16, 32, 48] + [64] * 12
    M, dtype = 1000, torch.float32 if prec == "fp32" else torch.float64

    def lattice():
        lat = Lattice(Ls, range(len(Ls)), precision=prec)
        for c, L in enumerate(Ls):
            lat.set_params(1.0, 4.0, M * 0.01, 0.01, 2.0 / (L * L), chain=c)
        return lat

    lat = lattice()
    n = sum(2 * M * L * L for L in Ls)
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    v = 0.3 * torch.randn(n, generator=g, device="cuda", dtype=dtype)
    for c, L in enumerate(Ls[:4]):  # and some masked sites, not on the worldlines
        x = torch.from_numpy(lat.get_state(c)[1][:, 0, 0]).long()
        o = sum(2 * M * k * k for k in Ls[:c])
        part = v[o:o + 2 * M * L * L].view(2, M, L * L)
        keep = part[[0, 1], :, x].clone()
        part[torch.rand(part.shape, generator=g, device="cuda") < 0.1] = -float("inf")
        part[[0, 1], :, x] = keep
    want = lat.log_weight_grad(v=v)
    lat.close()
    lat = lattice()
    lat.log_weight_grad()  # the scratch, and dlogZ_dv's block in torch's pool
    torch.cuda.empty_cache()
    spare = torch.empty(n, dtype=dtype, device="cuda")
    table = n * v.element_size()
    fill = torch.empty(torch.cuda.mem_get_info()[0] - table * 3 // 4, dtype=torch.uint8, device="cuda")
    del spare  # for dlogZ_dv
    try:
        assert torch.cuda.mem_get_info()[0] < table
        got = lat.log_weight_grad(v=v)
    finally:
        del fill
        torch.cuda.empty_cache()
    assert np.abs(got[0] - want[0]).max() <= 1e-12 * np.abs(want[0]).max()
    assert np.isfinite(want[2]).all() and np.abs(got[2] - want[2]).max() <= tol * np.abs(want[2]).max()
    assert (got[1] - want[1]).abs().max() <= tol * want[1].abs().max()
    lat.close()
