"""The FP64 per-wavenumber kernels in parity blocks against the oracle: odd and
even Ny from the smallest grid to the largest, member counts off the tiles (1,
3, 5, and one over the members of an apply CTA), a linearised group."""
import numpy as np
import pytest

import dns_synth
import oracle.dns as oracle
import oracle.linear as oracle_linear

pytestmark = pytest.mark.gpu
dns = pytest.importorskip("paper_2306_12739_gb300")


@pytest.mark.parametrize("mx,my,mz,E", [(16, 5, 16, 1), (16, 6, 32, 3), (32, 34, 16, 5), (16, 33, 16, 9), (32, 129, 16, 1)])
def test_fp64_step_matches_oracle(mx, my, mz, E):
    g = dict(flow="poiseuille", mx=mx, my=my, mz=mz, lx=2 * np.pi, lz=np.pi, re=1650.0, dt=0.004, members=E,
             member_block=E)
    st = dns_synth.make_state(mx, my, mz, g["lx"], g["lz"], g["flow"], E, 95, 5e-2)
    ref = oracle.Channel(mx, my, mz, g["lx"], g["lz"], g["re"], g["dt"], g["flow"]).step(
        tuple(st[k] for k in ("v", "eta", "U", "W")), 2)
    ens = dns.Ensemble([g], precision="fp64")
    ens.set_state(0, st["v"], st["eta"], st["U"], st["W"])
    ens.step(2)
    got = ens.get_state(0)
    ens.close()
    for a, b in zip(got, ref):
        assert np.abs(a - b).max() < 1e-12 * np.abs(b).max()


def test_fp64_linear_step_matches_oracle():
    my, mz, E = 22, 16, 11
    g = dict(flow="couette", mx=0, my=my, mz=mz, lx=2 * np.pi, lz=np.pi, re=3000.0, dt=0.04, members=E, linear=True,
             kx_index=2)
    b = dns_synth.make_base_flow(my, mz, g["lz"], "couette", 3)
    st = dns_synth.make_disturbances(my, mz, g["lz"], E, 96)
    ref = oracle_linear.Linear(my, mz, g["lx"], g["lz"], g["re"], g["dt"], 2, b["U"], b["V"], b["W"]).step(
        (st["v"], st["eta"]), 3)
    ens = dns.Ensemble([g], precision="fp64")
    ens.set_base_flow(0, b["U"], b["V"], b["W"])
    ens.set_state(0, st["v"], st["eta"])
    ens.step(3)
    got = ens.get_state(0)
    ens.close()
    for a, r in zip(got[:2], ref):
        assert np.abs(a[..., 0] - r).max() < 1e-11 * np.abs(r).max()
