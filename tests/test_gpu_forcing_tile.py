"""The forcing in parity blocks where its column tile is halved to keep more CTAs on
an SM: fewer modes per tile, and shorter member runs (odd member counts leave a
ragged last run).  A member of the ensemble against the same member alone, whose
tile is not halved: every column is computed the same way whatever tile holds it."""
import numpy as np
import pytest

import dns_synth

pytestmark = pytest.mark.gpu
dns = pytest.importorskip("paper_2306_12739_gb300")


@pytest.mark.parametrize("mx,my,mz,E", [(64, 97, 64, 20), (32, 96, 32, 33), (64, 65, 64, 33), (128, 97, 128, 4)])
def test_members_do_not_depend_on_the_forcing_tile(mx, my, mz, E):
    st = dns_synth.make_state(mx, my, mz, 2 * np.pi, np.pi, "couette", E, 150, 5e-2)

    def run(members, s):
        g = dict(flow="couette", mx=mx, my=my, mz=mz, lx=2 * np.pi, lz=np.pi, re=500.0, dt=0.002, members=members,
                 member_block=members)
        ens = dns.Ensemble([g], precision="mixed", plane="lines", ygemm="simt_eo", helm="simt_eo")
        try:
            ens.set_state(0, *(s[k] for k in ("v", "eta", "U", "W")))
            ens.step(2)
            return ens.get_state(0)
        finally:
            ens.close()

    whole = run(E, st)
    for e in (0, E - 1):
        one = run(1, {k: st[k][e:e + 1] for k in st})
        for a, b in zip(whole, one):
            assert np.array_equal(a[e:e + 1], b)
