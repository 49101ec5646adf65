"""The plane stage as three launches (z inverse, x with the products, z forward)
against the oracle in FP64 and against FP64 in the mixed path: every transform
length, ragged column tiles and line-pair counts, both nonlinear forms, the
smallest wall-normal grid; the cluster and single-CTA kernels stay on request."""
import numpy as np
import pytest

import dns_synth
import oracle.dns as oracle

pytestmark = pytest.mark.gpu
dns = pytest.importorskip("paper_2306_12739_gb300")

SIZES = [(16, 7, 16, 3, "advective"), (16, 6, 48, 1, "rotational"), (48, 7, 16, 2, "advective"),
         (32, 9, 32, 3, "advective"), (32, 6, 128, 1, "advective"), (48, 11, 32, 2, "rotational"),
         (48, 5, 64, 1, "advective"), (64, 8, 48, 3, "advective"), (64, 9, 64, 2, "rotational"),
         (64, 6, 128, 2, "advective"), (128, 7, 64, 1, "advective"), (128, 9, 128, 2, "advective")]


def _group(mx, my, mz, E, form):
    return dict(flow="poiseuille", mx=mx, my=my, mz=mz, lx=2 * np.pi, lz=np.pi, re=1650.0, dt=0.004, members=E,
                form=form)


def _run(g, st, n, precision, plane):
    ens = dns.Ensemble([g], precision=precision, plane=plane)
    kind = dns.dns_kernel_choice(ens.h, 0, "plane")
    ens.set_state(0, st["v"], st["eta"], st["U"], st["W"])
    ens.step(n)
    got = ens.get_state(0)
    ens.close()
    return got, kind


def _rel(a, b):
    return np.abs(a - b).max() / np.abs(b).max()


@pytest.mark.parametrize("mx,my,mz,E,form", SIZES)
def test_split_plane_stage(mx, my, mz, E, form):
    g = _group(mx, my, mz, E, form)
    if (mx, mz) == (32, 128):        # a length pair the library has no plane stage for stays refused
        with pytest.raises(dns.DnsError):
            dns.Ensemble([g], precision="fp64", plane="split")
        return
    st = dns_synth.make_state(mx, my, mz, g["lx"], g["lz"], g["flow"], E, 90, 5e-2)
    ref = oracle.Channel(mx, my, mz, g["lx"], g["lz"], g["re"], g["dt"], g["flow"], form=form).step(
        tuple(st[k] for k in ("v", "eta", "U", "W")), 2)
    fp64, kind = _run(g, st, 2, "fp64", "default")
    assert kind == "split"
    for a, b in zip(fp64, ref):
        assert _rel(a, b) < 1e-12
    mixed, kind = _run(g, st, 2, "mixed", "split")
    assert kind == "split"
    # the mixed path's budget: 1e-6 per field, the mean flow as one field
    assert _rel(mixed[0], ref[0]) < 1e-6 and _rel(mixed[1], ref[1]) < 1e-6
    assert _rel(np.stack(mixed[2:]), np.stack(ref[2:])) < 1e-6


@pytest.mark.parametrize("mx,plane", [(128, "cluster"), (64, "cta")])
def test_fp64_plane_kernels_on_request(mx, plane):
    g = _group(mx, 9, mx, 1, "advective")
    st = dns_synth.make_state(mx, 9, mx, g["lx"], g["lz"], g["flow"], 1, 91, 5e-2)
    a, kind = _run(g, st, 2, "fp64", plane)
    assert kind == plane
    b, _ = _run(g, st, 2, "fp64", "split")
    for x, y in zip(a, b):
        assert _rel(x, y) < 1e-12
