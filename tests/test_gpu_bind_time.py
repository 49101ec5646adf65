"""Binding a workspace times whole steps of every candidate: a handle whose steps take
milliseconds must not pay for as many of them as one of 50-microsecond steps."""
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
dns = pytest.importorskip("paper_2306_12739_gb300")


def test_bind_of_a_large_batch_takes_few_steps_per_candidate():
    """Three groups, seven candidates each, at most 25 steps a candidate (two visits of
    a capture, two warm-up steps and three windows), and a quarter of a second for
    everything else (the tunings of single kernels, graphs)."""
    groups = [dict(flow=f, mx=mx, my=my, mz=mx, lx=2 * np.pi, lz=np.pi, re=re, dt=0.005, members=E)
              for f, mx, my, E, re in (("couette", 32, 33, 64, 400.0), ("couette", 48, 49, 32, 800.0),
                                       ("poiseuille", 64, 65, 32, 1650.0))]
    make = lambda: dns.Ensemble(groups, precision="mixed", use_graph=True)
    make().close()                           # loads the kernels
    cfg = dns.make_config(groups, "mixed", use_graph=True)
    t0 = time.perf_counter()
    dns.dns_destroy(dns.dns_create(cfg, 0))
    t1 = time.perf_counter()
    ens = make()
    t2 = time.perf_counter()
    ens.step(20)
    ens.stream.synchronize()
    t3 = time.perf_counter()
    ens.step(20)
    ens.stream.synchronize()
    step = (time.perf_counter() - t3) / 20
    ens.close()
    bind = (t2 - t1) - (t1 - t0)
    assert bind < 0.25 + 3 * 7 * 25 * step, (bind, step)
