"""A wide class of short and long hops (windows for some of its chains), and a hop that is changed in
place between sweeps (the class goes from windows to none and back): the draws equal those from
FP32 checkpoints, which read whole slices, bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def run(L, hops, storage):
    """hops: per sweep, the hopping of every chain."""
    from paper_2510_13866_gb300 import Lattice

    nsig, M = 5, 7
    lat = Lattice(L, range(20, 20 + len(hops[0])), precision="fp32")
    out = []
    for k, row in enumerate(hops):
        for c, t in enumerate(row):
            lat.set_params(t, 4.0, M * 0.05, 0.05, 2.0 * nsig / (L * L), chain=c)
        if k == 0:
            lat.set_ffbs_storage(storage)
        for _ in range(2):  # the second one replays the first one's graph
            out += [w.copy() for w in lat.sweep(1, logw=True)]
    for c in range(len(hops[0])):
        out += list(lat.get_state(c)[:2])
    lat.close()
    return out


@pytest.mark.parametrize("L", [48, 64, 128])
@pytest.mark.parametrize("hops", [[(1.0, 4.0, 3.3)], [(4.0, 4.0)], [(1.0, 1.0), (4.0, 4.0), (1.0, 1.0)], [(4.0, 4.0), (4.0, 1.0), (4.0, 4.0)]])
def test_classes_with_and_without_windows(L, hops):
    a, b = run(L, hops, "stream"), run(L, hops, "f32")
    assert all(np.array_equal(u, v) for u, v in zip(a, b))
