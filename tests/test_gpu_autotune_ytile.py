"""The column-tile cap of the register-tiled y-derivatives in the autotuner's cache is
timed on that kernel, whichever y-derivatives the handle that stores it runs: a handle
with the others (which have no such tile) leaves a line that one with them can take."""
import re

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
dns = pytest.importorskip("paper_2306_12739_gb300")


def _caps(tmp_path, ygemm):
    cache = tmp_path / (ygemm + ".txt")
    g = dict(flow="couette", mx=32, my=97, mz=32, lx=2 * np.pi, lz=np.pi, re=500.0, dt=0.01, members=4, member_block=4)
    dns.Ensemble([g], precision="mixed", ygemm=ygemm, helm="simt", plane="lines", autotune_cache=str(cache)).close()
    (line,) = [ln for ln in cache.read_text().splitlines() if ln.startswith("ytile 32 97 32 4 ")]
    return {int(c): float(t) for c, t in re.findall(r" value (\d+) ([0-9.]+) ms", line)}


def test_cached_cap_is_the_register_tiled_kernels(tmp_path):
    own, other = _caps(tmp_path, "simt"), _caps(tmp_path, "simt_eo")
    assert sorted(own) == sorted(other) and len(own) == 3
    # the tensor-instruction y-derivatives take a third of the time at this size
    assert all(other[c] > 0.7 * own[c] for c in own)
