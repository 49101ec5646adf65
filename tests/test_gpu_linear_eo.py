"""Linearised groups on the forcing and apply in parity blocks (the autotuner's
choice, forced here through a cache file) against FP64, and Gram-Schmidt of
vector counts around a gather tile (1, 8, 9) and of vectors longer than one
batch of a cluster, against the oracle."""
import numpy as np
import pytest

import dns_synth
import oracle.linear as oracle_linear

pytestmark = pytest.mark.gpu
dns = pytest.importorskip("paper_2306_12739_gb300")


def _case(my, mz, E, n=1):
    g = dict(flow="couette", mx=0, my=my, mz=mz, lx=2 * np.pi, lz=np.pi, re=1000.0, dt=0.04, members=E, linear=True,
             kx_index=n)
    b = dns_synth.make_base_flow(my, mz, g["lz"], "couette", 21)
    return g, b, dns_synth.make_disturbances(my, mz, g["lz"], E, 22)


def _ens(g, b, st, precision, **kw):
    ens = dns.Ensemble([g], precision=precision, **kw)
    ens.set_base_flow(0, b["U"], b["V"], b["W"])
    ens.set_state(0, st["v"], st["eta"])
    return ens


@pytest.mark.parametrize("my,mz,E", [(5, 16, 1), (22, 32, 7), (65, 16, 33)])
def test_parity_blocks_match_fp64(my, mz, E, tmp_path):
    g, b, st = _case(my, mz, E)
    cache = tmp_path / "tune.txt"
    cache.write_text("helm 0 %d %d %d 8\n" % (my, mz, E))
    out = {}
    for precision, kw in (("fp64", {}), ("mixed", dict(autotune_cache=str(cache)))):
        ens = _ens(g, b, st, precision, **kw)
        if precision == "mixed":
            assert dns.dns_kernel_choice(ens.h, 0, "helm") == "simt_eo"
        ens.step(20)
        ens.set_direction(True)
        ens.step(20)
        out[precision] = ens.get_state(0)[:2]
        ens.close()
    for a, r in zip(out["mixed"], out["fp64"]):
        assert np.abs(a - r).max() < 1e-5 * np.abs(r).max()


@pytest.mark.parametrize("my,mz,E", [(7, 16, 1), (17, 32, 8), (33, 16, 9), (65, 64, 3)])
def test_gram_schmidt_matches_oracle(my, mz, E):
    g, b, st = _case(my, mz, E)
    ref = oracle_linear.Linear(my, mz, g["lx"], g["lz"], g["re"], g["dt"], 1, b["U"], b["V"], b["W"])
    (rv, re), norms = ref.orthonormalize((st["v"], st["eta"]))
    ens = _ens(g, b, st, "fp64")
    got = ens.orthonormalize(0)
    v, eta = ens.get_state(0)[:2]
    ens.close()
    assert np.abs(got - norms).max() < 1e-12 * norms.max()
    for a, r in ((v, rv), (eta, re)):
        assert np.abs(a[..., 0] - r).max() < 1e-11 * np.abs(r).max()
