"""The wide kernel's extra scratch slots are asked for only where units wait to be drawn -- Hirsch
chains with short hops -- and only out of memory that leaves room for others."""
import ctypes as C

import pytest

pytestmark = pytest.mark.gpu

UNITS, M = 1400, 20  # more units of one worldline than CTAs of L = 64


def lattice(L=64, U=4.0, t=1.0):
    from paper_2510_13866_gb300 import Lattice

    lat = Lattice(L, [5], precision="fp32", torch_memory=False)
    lat.set_params(t, U, M * 0.05, 0.05, UNITS / (L * L))
    return lat


def attach(lat, n):
    import torch

    from paper_2510_13866_gb300 import hqmc

    ws = torch.empty(n + 256, dtype=torch.uint8, device="cuda")
    rc = hqmc.lib().hqmc_attach_workspace(lat._ctx, C.c_void_p((ws.data_ptr() + 255) // 256 * 256), n)
    if rc == 0:
        lat.sweep(1)
    lat.close()
    return rc


@pytest.mark.parametrize("L,U,t,spare", [(64, 4.0, 1.0, True), (128, 4.0, 1.0, True), (64, -4.0, 1.0, False),
                                         (64, 4.0, 4.0, False), (128, -4.0, 1.0, False), (128, 4.0, 4.0, False)])
def test_slots_only_where_units_wait(L, U, t, spare):
    """Two slots or more: a workspace of 0.7 of the size holds the layout without the extra ones (HQMC_OK).
    One slot: nothing to leave out (HQMC_ERR_NOMEM)."""
    lat = lattice(L, U, t)
    assert attach(lat, int(0.7 * lat.workspace_size()) // 256 * 256) == (0 if spare else -2)


def test_slots_leave_room_on_a_full_device():
    import torch

    lat = lattice()
    wide = lat.workspace_size()
    torch.cuda.empty_cache()
    left = wide + (64 << 20)
    fill = torch.empty(torch.cuda.mem_get_info()[0] - left, dtype=torch.uint8, device="cuda")
    try:
        assert torch.cuda.mem_get_info()[0] >= wide  # all of it would fit, with next to nothing left
        narrow = lat.workspace_size()
    finally:
        del fill
        torch.cuda.empty_cache()
    assert narrow < 0.7 * wide
    assert lat.workspace_size() == wide
    lat.close()
