"""The rule that puts large mixed groups on the three-launch plane stage looks at the
whole group: every member block runs the same plane kernel, whatever its own members.
Host only: the stage's column storage is part of a block's workspace, so the workspace
of a handle tells how many of its blocks run it."""
import numpy as np
import pytest

dns = pytest.importorskip("paper_2306_12739_gb300")


def _bytes(mx, my, mz, E, plane):
    g = dict(flow="couette", mx=mx, my=my, mz=mz, lx=2 * np.pi, lz=np.pi, re=500.0, dt=0.01, members=E)
    h = dns.dns_create(dns.make_config([g], "mixed", plane=plane), 0)
    try:
        return dns.dns_workspace_size(h)
    finally:
        dns.dns_destroy(h)


# (grid, members, blocks): (My - 2) Mx Mz members around 1.5 million, uneven blocks
@pytest.mark.parametrize("mx,my,mz,E,split", [
    (48, 49, 48, 14, True),     # 1.516 M, blocks of 5, 5, 4
    (48, 49, 48, 13, False),    # 1.408 M, blocks of 5, 4, 4
    (64, 33, 64, 12, True),     # 1.524 M, blocks of 4
    (64, 33, 64, 11, False),    # 1.397 M, blocks of 6, 5
    (32, 49, 32, 31, False),    # 1.492 M, blocks of 5, 5, 5, 4, 4, 4, 4
    (32, 49, 32, 35, True)])    # 1.684 M, blocks of 5, 5, 5, 4, 4, 4, 4, 4
def test_every_block_of_a_group_runs_the_same_plane_kernel(mx, my, mz, E, split):
    want = _bytes(mx, my, mz, E, "split" if split else "lines")
    other = _bytes(mx, my, mz, E, "lines" if split else "split")
    assert want != other
    assert _bytes(mx, my, mz, E, "default") == want
