"""The fused stage's tensor-instruction products may not be further from 64 bits than the
single-precision multiply-adds of the natural-order stage."""
import numpy as np
import pytest

import dns_synth

pytestmark = pytest.mark.gpu
dns = pytest.importorskip("paper_2306_12739_gb300")


def _run(g, st, n, precision, **kw):
    ens = dns.Ensemble([g], precision=precision, use_graph=True, **kw)
    ens.set_state(0, *(st[k] for k in ("v", "eta", "U", "W")))
    ens.step(n)
    got = ens.get_state(0)[:2]
    ens.close()
    return got


@pytest.mark.parametrize("flow,mx,my,mz,E,n,dt,re,form", [
    ("couette", 64, 28, 16, 4, 40, 0.01, 500.0, "advective"),
    ("poiseuille", 32, 24, 32, 4, 40, 0.01, 1650.0, "rotational"),
    ("couette", 48, 36, 32, 3, 20, 0.01, 500.0, "advective"),
    ("couette", 16, 53, 32, 4, 10, 0.01, 500.0, "rotational"),
    ("poiseuille", 16, 106, 16, 1, 20, 0.01, 1650.0, "advective")])
def test_error_is_at_most_the_fp32_stages(flow, mx, my, mz, E, n, dt, re, form):
    """Relative error of v and eta after n steps (root of the sum of squares over the
    fields, as one vector; the mean of three ensembles), kernels bitwise reproducible."""
    lx, lz = (1.75 * np.pi, 1.2 * np.pi) if flow == "couette" else (2 * np.pi, np.pi)
    g = dict(flow=flow, mx=mx, my=my, mz=mz, lx=lx, lz=lz, re=re, dt=dt, members=E, member_block=E, form=form)
    err = {"fused": 0.0, "fused_eo_ff": 0.0}
    for seed in (0, 1000, 2000):
        st = dns_synth.make_state(mx, my, mz, lx, lz, flow, E, seed, 5e-2, spectrum="kolmogorov")
        ref = _run(g, st, n, "fp64")
        for helm in err:
            got = _run(g, st, n, "mixed", helm=helm, plane="lines")
            err[helm] += np.hypot(*(np.linalg.norm(a - r) / np.linalg.norm(r) for a, r in zip(got, ref)))
    assert err["fused_eo_ff"] <= err["fused"]
