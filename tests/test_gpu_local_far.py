"""Local moves of worldlines whose neighbouring slices lie far apart.  G of the direction that does
not move can then underflow in FP64 (L = 128, t dtau = 0.05: G(64)^2 is below 1e-340): R is 0/0 and
the move is refused, although the factors of the moving direction alone would accept it.

The reference takes R in FP64 from the oracle's ratio with the propagator's power series, whose
terms are all positive: the oracle's own table is a cosine sum, which ends in rounding noise at
1e-17.  Decisions lie further than 1e-9 from their edge (checked), so the moves are equal.  Both
forms of the sweep: one length, and with a chain of another length beside it."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def ring(L, z):
    """exp(z A) of the ring's adjacency A, first row."""
    term = np.zeros(L)
    term[0] = 1.0
    g = term.copy()
    for n in range(1, 3 * L):
        term = (np.roll(term, 1) + np.roll(term, -1)) * (z / n)
        g += term
    return g


def reference_sweep(orc, g):
    """The local moves of one sweep on orc.x; returns (accepted, least distance from an edge)."""
    L, M, W = orc.L, orc.M, orc.slice_potentials()
    accepted, edge = 0, np.inf
    for color in range(3):
        for sg in range(2):
            for p in range(orc.Nsig):
                x, wl = orc.x[sg, p], sg * orc.Nsig + p
                for l in range(M):
                    if oracle.local_color(M, l) != color:
                        continue
                    u0, u1 = (oracle.uniform(orc.seed, orc.sweep_count, 4, wl, 2 * l + k) for k in (0, 1))
                    new = oracle.local_step(L, int(x[l]), int(4 * u0))
                    R = oracle.local_ratio(L, M, g, W[sg, l], int(x[l - 1]), int(x[l]), int(x[(l + 1) % M]), new)
                    if np.isfinite(R):
                        edge = min(edge, abs(u1 - R))
                    if u1 < R:
                        x[l] = new
                        accepted += 1
    return accepted, edge


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("companion", [False, True])
@pytest.mark.parametrize("L,dy,dtau", [(128, 64, 0.05), (128, 56, 0.05), (64, 32, 1e-4), (32, 16, 0.05)])
def test_far_neighbours(L, dy, dtau, companion, prec):
    from paper_2510_13866_gb300 import Lattice

    M, nsig = 6, 40
    par = (1.0, 4.0, M * dtau, dtau, 2.0 * nsig / (L * L))
    lat = Lattice([L] + [4] * companion, [9] + [10] * companion, precision=prec)
    lat.set_params(*par, chain=0)
    if companion:
        lat.set_params(1.0, 4.0, 0.5, 0.1, 1.0, chain=1)
    orc = oracle.Chain(L, *par, 9)
    ix, iy = np.random.default_rng(2).integers(0, L, (2, 2, nsig))
    odd = np.arange(M) % 2
    orc.x[:] = (ix[..., None] + odd) % L + L * ((iy[..., None] + dy * odd) % L)
    lat.set_state(0, s=orc.s, x=orc.x)
    lat.local_sweep(1)
    accepted, edge = reference_sweep(orc, ring(L, dtau))
    assert edge > 1e-9
    assert np.array_equal(lat.get_state(0)[1], orc.x)
    assert lat.measure()[0]["n_local_accepted"] == accepted
    lat.close()
