"""The windowed backward draw (ffbs_window.cuh) against the draw from whole slices.

A wide FP32 chain that streams f draws its worldlines from windows around them; the same chain
with FP32 checkpoints of f (`set_ffbs_storage("f32")`) recomputes the same f and draws from whole
slices.  Both make the same draw, so worldlines, fields, log-weights, their error estimates and
the diagnostic counters are equal bit for bit, whichever way each slice was answered.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def sweeps(L, nsig, M, dtau, storage, t=1.0, U=4.0, block=0, perm=False, scatter=False, n=3, seeds=(3, 4, 5, 6, 7)):
    from paper_2510_13866_gb300 import Lattice

    lat = Lattice(L, seeds, precision="fp32")
    lat.set_params(t, U, M * dtau, dtau, 2.0 * nsig / (L * L))
    if block:
        lat.set_block(block)
    if perm:
        lat.set_permutations(True)
    lat.set_ffbs_storage(storage)
    if scatter:
        # worldlines whose slices lie anywhere: block ends far from where the message is large
        for c in range(len(seeds)):
            x = np.random.default_rng(100 + c).integers(0, L * L, size=(2, nsig, M))
            lat.set_state(c, x=x)
    out = []
    for _ in range(n):
        out += [w.copy() for w in lat.sweep(1, logw=True)] + list(lat.logw_error())
    for c in range(len(seeds)):
        s, x, a, _ = lat.get_state(c)
        out += [s, x, np.array(a)]
    for o in lat.measure():
        out += [np.array([o[k] for k in ("density", "double_occ", "m2")]),
                np.array([o[k] for k in ("n_samples", "n_degenerate", "n_nonpositive", "n_inexact", "n_perm_accepted")])]
        # sums over worldlines in the order of arrival
        out.append(("sum", o["ekin"]))
    lat.close()
    return out


def assert_same(a, b):
    assert len(a) == len(b)
    for u, v in zip(a, b):
        if isinstance(u, tuple):
            assert abs(u[1] - v[1]) <= 1e-12 * max(1.0, abs(u[1]))
        else:
            assert np.array_equal(u, v, equal_nan=True)


@pytest.mark.parametrize("L,nsig,M,dtau,kw", [
    (48, 5, 20, 0.05, {}),                              # odd count: a half-empty CTA; full batches
    (48, 7, 13, 0.1, dict(block=5)),                    # odd M, blocks that do not divide it
    (48, 6, 24, 0.05, dict(perm=True, U=8.0)),
    (48, 4, 12, 0.05, dict(block=4, scatter=True)),     # draws on the rounding floor: whole slices
    (64, 5, 21, 0.05, {}),
    (64, 3, 16, 0.1, dict(perm=True, block=6)),
    (64, 4, 12, 1 / 32, dict(U=20.0, scatter=True, block=3)),
    (64, 300, 5, 0.05, {}),                             # more units than CTAs
    (128, 3, 11, 0.05, {}),
    (128, 2, 10, 0.125, dict(block=4)),                 # the widest window (no margin to spare)
    (128, 2, 10, 0.05, dict(scatter=True, block=3)),
])
def test_window_draws_equal_whole_slice_draws(L, nsig, M, dtau, kw):
    assert_same(sweeps(L, nsig, M, dtau, "stream", **kw), sweeps(L, nsig, M, dtau, "f32", **kw))


@pytest.mark.parametrize("L,M,dtau,t", [(64, 1, 0.05, 1.0), (64, 2, 0.05, 1.0), (48, 3, 0.05, 1.0), (48, 4, 0.05, 0.0),
                                        (64, 6, 0.05, 3.0), (128, 4, 0.2, 1.0)])
def test_window_edges(L, M, dtau, t):
    """One to four slices (fewer than the windows loaded ahead), no hopping, and hops too long
    for a window (t dtau above 0.14: whole slices in both)."""
    assert_same(sweeps(L, 3, M, dtau, "stream", t=t), sweeps(L, 3, M, dtau, "f32", t=t))


def test_workspace_without_extra_slots_gives_the_same_sweep():
    """hqmc_workspace_size asks for several scratch slots per CTA where units outnumber CTAs; an attached
    workspace of the size without them is accepted and draws the same, a smaller one is refused."""
    import ctypes as C

    import torch

    from paper_2510_13866_gb300 import Lattice, hqmc

    def run(fraction):
        lat = Lattice(64, [5], precision="fp32", torch_memory=False)
        lat.set_params(1.0, 4.0, 0.25, 0.05, 1400 / 4096)  # 1400 units of one worldline, M = 5
        n = int(lat.workspace_size() * fraction) // 256 * 256
        ws = torch.empty(n + 256, dtype=torch.uint8, device="cuda")
        p = (ws.data_ptr() + 255) // 256 * 256
        rc = hqmc.lib().hqmc_attach_workspace(lat._ctx, C.c_void_p(p), n)
        out = None if rc else [lat.sweep(2, logw=True)[0].copy(), lat.get_state(0)[1]]
        lat.close()
        return rc, out

    rc, full = run(1.0)
    assert rc == 0
    rc, small = run(0.65)
    assert rc == 0
    assert all(np.array_equal(a, b) for a, b in zip(full, small))
    assert run(0.2)[0] == -2  # HQMC_ERR_NOMEM
