"""Gram-Schmidt of vectors so small that their squared norms are subnormal."""
import numpy as np
import pytest

import dns_synth

pytestmark = pytest.mark.gpu
dns = pytest.importorskip("paper_2306_12739_gb300")


def test_tiny_vectors_orthonormalise_as_their_multiples():
    """Vectors scaled by a power of two that puts their squared norms near 2^-1029, whose
    reciprocal overflows.  A term of the sums is then known to half a quantum, 2^-1075;
    fewer than 2^12 terms leave each norm and coefficient 2^12 2^-1075 / 2^-1030 = 2^-33
    = 1.2e-10 off, two projections and a normalisation stay far below 1e-8."""
    my, mz, E = 17, 32, 3
    b = dns_synth.make_base_flow(my, mz, np.pi, "couette", 21)
    st = dns_synth.make_disturbances(my, mz, np.pi, E, 22)
    g = dict(flow="couette", mx=0, my=my, mz=mz, lx=2 * np.pi, lz=np.pi, re=1000.0, dt=0.04, members=E, linear=True,
             kx_index=1)
    ens = dns.Ensemble([g], precision="fp64")
    ens.set_base_flow(0, b["U"], b["V"], b["W"])
    # one norm for all: the orthogonal parts stay within a factor of a few of it
    ens.set_state(0, st["v"], st["eta"])
    norms = ens.orthonormalize(0)
    want = ens.get_state(0)[:2]
    scale = 2.0 ** np.floor(np.log2(2.0 ** -515.5 / norms.min()))
    sq = 4 * (norms * scale) ** 2            # the energy norm holds a factor 1/4
    assert sq.max() < 2.0 ** -1024 and sq.min() > 2.0 ** -1034
    ens.set_state(0, st["v"] * scale, st["eta"] * scale)
    tiny = ens.orthonormalize(0)
    got = ens.get_state(0)[:2]
    ens.close()
    assert np.abs(tiny / (norms * scale) - 1).max() < 1e-8
    for a, r in zip(got, want):
        assert np.abs(a - r).max() < 1e-8 * np.abs(r).max()
