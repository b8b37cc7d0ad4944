"""The adjoint with masked sites: a log-potential of -inf, or one whose exponential vanishes or is
denormal in the context's precision, at some sites of every kind of slice -- the anchor's, a
segment's first, last and inner ones.  Everything is finite and equal to the oracle's.

Tolerances as for a given log-potential without masks: FP32 with checkpoints in FP32 1e-5 on
log Z and 1e-4 of scale on the gradients, BF16 checkpoints 2^-6 of scale, FP64 1e-10.
"""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

LS, NSIG = [3, 8, 16, 32, 12, 48], [2, 6, 5, 4, 3, 2]


@pytest.mark.parametrize("prec,bf16,M,stride", [("fp32", False, 9, 3), ("fp32", True, 9, 3), ("fp32", False, 8, 1),
                                                ("fp32", True, 10, 0), ("fp64", False, 9, 3), ("fp64", False, 6, 1)])
@pytest.mark.parametrize("low", [-np.inf, -735.0, -95.0, -80.0, "mixed"])
def test_masked_sites(prec, bf16, M, stride, low):
    import torch

    from paper_2510_13866_gb300 import Lattice

    params = [(1.0, 4.0, M * 0.1, 0.1, 2.0 * n / (L * L)) for L, n in zip(LS, NSIG)]
    lat = Lattice(LS, list(range(len(LS))), precision=prec)
    for c, p in enumerate(params):
        lat.set_params(*p, chain=c)
    lat.sweep(1)
    lat.set_checkpoint(stride, bf16=bf16)
    rng = np.random.default_rng(23)
    dtype = np.float32 if prec == "fp32" else np.float64
    v, state = [], []
    for c, L in enumerate(LS):
        s, x, _, _ = lat.get_state(c)
        state.append((s, x))
        a = rng.normal(0.0, 0.5, size=(2, M, L * L))
        mask = rng.random(a.shape) < 0.3
        for sg in range(2):
            mask[sg][:, x[sg, :, 0]] = False  # a path that stays at its anchor: log Z far above the rounding
        values = rng.choice([-np.inf, -1e4, -95.0, -80.0, -45.0, -41.0], size=a.shape) if low == "mixed" else low
        v.append(np.where(mask, values, a).astype(dtype))
    lz, dv, dt = lat.log_weight_grad(v=torch.from_numpy(np.concatenate([a.ravel() for a in v])).cuda())
    dv = dv.double().cpu().numpy()
    tol_z, tol_g = (1e-10, 1e-10) if prec == "fp64" else (1e-5, 2.0 ** -6 if bf16 else 1e-4)
    o = 0
    for c, L in enumerate(LS):
        n = 2 * M * L * L
        got = dv[o:o + n].reshape(2, M, L * L)
        o += n
        orc = oracle.Chain(L, *params[c], c)
        orc.s[:], orc.x[:] = state[c]
        rz, rdv, rdt = orc.grad(v[c].astype(np.float64))
        assert abs(lz[c] - rz) <= tol_z * max(1.0, abs(rz)), (L, lz[c], rz)
        assert np.abs(got - rdv).max() <= tol_g * max(1.0, np.abs(rdv).max()), L
        assert abs(dt[c] - rdt) <= tol_g * max(1.0, abs(rdt)), (L, dt[c], rdt)
    lat.close()
