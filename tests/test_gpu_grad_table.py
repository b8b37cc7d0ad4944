"""The adjoint with a given log-potential: exp(v) comes from a table in the kernels' reading
order (lines of even slices along x, of odd ones along y; 16-byte chunks on wide lattices), and
d log Z / d t from neighbours within a lane's own line, in both parities of M and at segment
starts.  One context holds chains of every kernel form and of sizes that would leave an
unpadded table misaligned (2 M N = 126 elements at L = 3, M = 7).

Tolerances as for the field's own potential: FP32 with checkpoints in FP32 1e-5 on log Z and
1e-4 of scale on the gradients, FP64 1e-10.
"""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,M,stride", [("fp32", 7, 3), ("fp32", 8, 1), ("fp32", 5, 0), ("fp32", 1, 0),
                                           ("fp64", 7, 3), ("fp64", 4, 2)])
def test_given_log_potential_on_uneven_chains(prec, M, stride):
    import torch

    from paper_2510_13866_gb300 import Lattice

    Ls = [3, 16, 6, 48, 2, 24, 32, 12, 64, 8, 4]
    nsig = [3, 5, 4, 3, 1, 3, 2, 3, 1, 4, 2]
    params = [(1.0, 4.0, M * 0.1, 0.1, 2.0 * n / (L * L)) for L, n in zip(Ls, nsig)]
    lat = Lattice(Ls, list(range(11)), precision=prec)
    for c, p in enumerate(params):
        lat.set_params(*p, chain=c)
    lat.sweep(1)
    lat.set_checkpoint(stride, bf16=False)
    rng = np.random.default_rng(17)
    dtype = np.float32 if prec == "fp32" else np.float64
    v = [rng.normal(0.0, 0.5, size=(2, M, L * L)).astype(dtype) for L in Ls]
    lz, dv, dt = lat.log_weight_grad(v=torch.from_numpy(np.concatenate([a.ravel() for a in v])).cuda())
    dv = dv.double().cpu().numpy()
    tol_z, tol_g = (1e-5, 1e-4) if prec == "fp32" else (1e-10, 1e-10)
    o = 0
    for c, L in enumerate(Ls):
        n = 2 * M * L * L
        got = dv[o:o + n].reshape(2, M, L * L)
        o += n
        orc = oracle.Chain(L, *params[c], c)
        s, x, _, _ = lat.get_state(c)
        orc.s[:] = s
        orc.x[:] = x
        rz, rdv, rdt = orc.grad(v[c].astype(np.float64))
        assert abs(lz[c] - rz) <= tol_z * max(1.0, abs(rz)), (L, lz[c], rz)
        assert np.abs(got - rdv).max() <= tol_g * max(1.0, np.abs(rdv).max()), L
        assert abs(dt[c] - rdt) <= tol_g * max(1.0, abs(rdt)), (L, dt[c], rdt)
    lat.close()
