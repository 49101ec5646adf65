"""Every form of the fused stage on mma.sync (one to four 16-row tiles, one and two
warps per tile, both register budgets): the group runs it, it matches FP64, and a
member's bits do not depend on the form."""
import numpy as np
import pytest

import dns_synth

pytestmark = pytest.mark.gpu
dns = pytest.importorskip("paper_2306_12739_gb300")


def _group(mx, my, mz, E):
    return dict(flow="poiseuille", mx=mx, my=my, mz=mz, lx=2 * np.pi, lz=np.pi, re=1650.0, dt=0.004, members=E,
                member_block=E)


def _run(g, st, n, precision, stage=None, **kw):
    ens = dns.Ensemble([g], precision=precision, **kw)
    try:
        if stage:
            assert dns.dns_kernel_choice(ens.h, 0, "helm") == stage
        ens.set_state(0, *(st[k] for k in ("v", "eta", "U", "W")))
        ens.step(n)
        return ens.get_state(0)
    finally:
        ens.close()


def _state(g, seed):
    return dns_synth.make_state(g["mx"], g["my"], g["mz"], g["lx"], g["lz"], g["flow"], g["members"], seed, 5e-2)


# two warps a tile while all of them fit 152 SMs; the last four grids run one
@pytest.mark.parametrize("mx,my,mz,E", [(16, 33, 16, 2), (16, 66, 16, 3), (16, 89, 16, 8), (16, 99, 16, 3), (16, 106, 16, 1),
                                        (48, 33, 48, 16), (48, 65, 48, 5), (32, 89, 32, 8), (48, 99, 32, 3)])
def test_forms_match_fp64(mx, my, mz, E):
    g = _group(mx, my, mz, E)
    st = _state(g, 140)
    ref = _run(g, st, 5, "fp64")
    got = _run(g, st, 5, "mixed", "fused_eo_ff", helm="fused_eo_ff", plane="lines")
    # the mixed path's budget: 1e-6 per field and member, the mean flow as one field
    for e in range(E):
        for a, r in ((got[0], ref[0]), (got[1], ref[1]), (np.stack(got[2:], 1), np.stack(ref[2:], 1))):
            assert np.abs(a[e] - r[e]).max() < 1e-6 * np.abs(r[e]).max()


@pytest.mark.parametrize("my,E", [(33, 4), (65, 4), (97, 2), (106, 1)])
def test_register_budgets_agree_bitwise(my, E, tmp_path):
    g = _group(16, my, 16, E)
    st = _state(g, 141)
    got = []
    for ctas in (2, 3):
        cache = tmp_path / ("tune%d.txt" % ctas)
        cache.write_text("spec_cta 16 %d 16 %d %d\n" % (my, E, ctas))
        got.append(_run(g, st, 3, "mixed", "fused_eo_ff", helm="fused_eo_ff", plane="lines", autotune_cache=str(cache)))
    for a, b in zip(*got):
        assert np.array_equal(a, b)
