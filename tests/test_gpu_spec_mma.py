"""The fused stage in parity blocks with its products on mma.sync (fused_eo_ff on
groups whose operator fragments fit): mixed against FP64 at the edges of its 16-row
and 4-column tiles (odd and even Ny from the smallest grid to the largest, member
counts off the tiles and over one CTA's members), both nonlinear forms, and the
one- and two-warp forms of a tile bit for bit."""
import numpy as np
import pytest

import dns_synth

pytestmark = pytest.mark.gpu
dns = pytest.importorskip("paper_2306_12739_gb300")


def _group(mx, my, mz, E, form="advective"):
    return dict(flow="poiseuille", mx=mx, my=my, mz=mz, lx=2 * np.pi, lz=np.pi, re=1650.0, dt=0.004, members=E,
                member_block=E, form=form)


def _run(g, st, n, precision, **kw):
    ens = dns.Ensemble([g], precision=precision, **kw)
    ens.set_state(0, *(st[k] for k in ("v", "eta", "U", "W")))
    ens.step(n)
    got = ens.get_state(0)
    ens.close()
    return got


@pytest.mark.parametrize("mx,my,mz,E,form", [
    (16, 5, 16, 1, "advective"), (16, 18, 32, 3, "advective"), (32, 34, 16, 5, "rotational"),
    (16, 35, 16, 9, "advective"), (32, 65, 32, 2, "rotational"), (16, 66, 16, 17, "advective"),
    (16, 67, 16, 3, "advective"), (32, 98, 16, 4, "advective"), (16, 129, 32, 5, "advective")])
def test_mma_stage_matches_fp64(mx, my, mz, E, form):
    g = _group(mx, my, mz, E, form)
    st = dns_synth.make_state(mx, my, mz, g["lx"], g["lz"], g["flow"], E, 120, 5e-2)
    ref = _run(g, st, 10, "fp64")
    got = _run(g, st, 10, "mixed", helm="fused_eo_ff")
    # the mixed path's budget: 1e-6 per field and member, the mean flow as one field
    for e in range(E):
        for a, r in ((got[0], ref[0]), (got[1], ref[1]), (np.stack(got[2:], 1), np.stack(ref[2:], 1))):
            assert np.abs(a[e] - r[e]).max() < 1e-6 * np.abs(r[e]).max()


def test_one_and_two_warp_forms_agree_bitwise():
    """48 members of a small grid run one warp per tile, one member two."""
    g = _group(32, 33, 32, 48)
    st = dns_synth.make_state(32, 33, 32, g["lx"], g["lz"], g["flow"], 48, 130, 5e-2)
    kw = dict(helm="fused_eo_ff", plane="lines")
    whole = _run(g, st, 3, "mixed", **kw)
    one = _run(dict(g, members=1, member_block=1), {k: st[k][7:8] for k in st}, 3, "mixed", **kw)
    for a, b in zip(whole, one):
        assert np.array_equal(a[7:8], b)
