"""The local sweep's two forms -- both colours in one launch for closed loops of one length, a
launch per colour otherwise -- make the same moves: equal worldlines, fields, occupations,
accepted counts and link sums, at slice counts where a worldline's pairs leave warps ragged,
fill several rounds of a CTA, or vanish (M = 1, 2, 3), and next to chains of another length."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def chain_run(L, M, nsig, companion, n=3, U=4.0, dtau=0.1):
    """Two chains alone (one length: the fused form), or with a chain of another M."""
    from paper_2510_13866_gb300 import Lattice

    Ls = [L, L] + ([L] if companion else [])
    lat = Lattice(Ls, list(range(40, 40 + len(Ls))), precision="fp32")
    for c in range(2):
        lat.set_params(1.0, U, M * dtau, dtau, 2.0 * nsig / (L * L), chain=c)
    if companion:
        lat.set_params(1.0, U, (M + 1) * dtau, dtau, 2.0 * nsig / (L * L), chain=2)
    lat.local_sweep(n)
    out = [lat.get_state(c)[:2] for c in range(2)]
    obs = lat.measure()[:2]
    lat.close()
    return out, obs


@pytest.mark.parametrize("L,M,nsig,U", [
    (4, 1, 5, 4.0), (4, 2, 8, 4.0), (6, 3, 7, 4.0), (8, 20, 32, 20.0), (16, 81, 33, 4.0), (8, 645, 3, 4.0),
    (12, 1500, 2, 8.0), (32, 40, 100, 4.0), (128, 6, 3, 4.0), (8, 12, 9, -4.0), (3, 17, 4, 2.0),
])
def test_forms_make_the_same_moves(L, M, nsig, U):
    (a, oa), (b, ob) = chain_run(L, M, nsig, False, U=U), chain_run(L, M, nsig, True, U=U)
    for (s0, x0), (s1, x1) in zip(a, b):
        assert np.array_equal(s0, s1) and np.array_equal(x0, x1)
    for p, q in zip(oa, ob):
        for k in ("n_local_accepted", "n_samples", "density", "double_occ", "m2"):
            assert p[k] == q[k], k
        assert abs(p["ekin"] - q["ekin"]) <= 1e-13 * max(1.0, abs(p["ekin"]))
