"""D2 v of a newly set state in the fused stage in parity blocks (k_mma_derivs), read
from the handle's workspace and held against 64 bits: nothing but the rounding to
single precision may show, at every height of the grid and at any magnitude of the
state."""
import numpy as np
import pytest

import dns_synth

pytestmark = pytest.mark.gpu
dns = pytest.importorskip("paper_2306_12739_gb300")


def _fields(ens, v):
    """The per-plane fields v, Dv, D2v, eta, D eta of a mixed group, [y][e][m][n]: they lie
    one after the other from where the workspace holds v in single precision."""
    raw = ens.ws.cpu().numpy()[ens.ws_ptr - ens.ws.data_ptr():]
    raw = raw[:len(raw) // 256 * 256]
    single = np.ascontiguousarray(v).view(np.float64)
    # (the conversion flushes what is below the normal range to a signed zero)
    single = np.where(np.abs(single) < 2.0 ** -126, np.copysign(0.0, single), single).astype(np.float32)
    pat = single.reshape(-1).view(np.uint8)
    for i in np.nonzero((raw.reshape(-1, 256) == pat[:256]).all(1))[0]:
        if np.array_equal(raw[256 * i:256 * i + len(pat)], pat):
            return raw[256 * i:256 * i + 5 * len(pat)].view(np.complex64).reshape((5,) + v.shape)
    raise AssertionError("v is not in the workspace")


@pytest.mark.parametrize("my,E,scale", [(17, 1, 0), (34, 3, 0), (49, 2, 0), (65, 2, 0), (66, 1, 0), (98, 2, 0),
                                        (106, 1, 0), (65, 1, -100), (106, 1, -95), (33, 1, 40)])
def test_d2v_is_the_rounded_product(my, E, scale):
    """The even and the odd output row e, o = r0 +- r1 of a pair of rows are rounded to
    single precision, then their half sum and difference: at most 2^-24 (|e| + |o|) / 2 +
    2^-24 |r| <= 2 2^-24 max(|r0|, |r1|).  What the product itself leaves (below 1e-10 of
    the column's largest value) and the reference's own rounding (1e-16 times the row
    sums of |D2| |v|, below 1e-9) fit in 2e-9 of the largest.  The conversion of the state
    to pairs of single-precision values drops what is below 2^-126, which a row of D2
    carries on as 2^-126 times the sum of its entries: the small states."""
    mx = mz = 16
    g = dict(flow="couette", mx=mx, my=my, mz=mz, lx=2 * np.pi, lz=np.pi, re=1000.0, dt=0.005, members=E, member_block=E)
    st = dns_synth.make_state(mx, my, mz, g["lx"], g["lz"], "couette", E, 310, 1.0)
    ens = dns.Ensemble([g], precision="mixed", helm="fused_eo_ff")
    try:
        assert dns.dns_kernel_choice(ens.h, 0, "helm") == "fused_eo_ff"
        ens.set_state(0, st["v"] * 2.0 ** scale, st["eta"] * 2.0 ** scale, st["U"], st["W"])
        v = np.ascontiguousarray(ens.get_state(0)[0].transpose(1, 0, 2, 3))
        got = _fields(ens, v)[2].astype(np.complex128)
        D2 = dns.dns_export_grid(ens.h, 0, my)[2][1:-1, 1:-1]
    finally:
        ens.close()
    # (mode (0, 0) has no v; the real and imaginary parts are separate columns)
    want = np.einsum("ij,j...->i...", D2, v)
    flush = (np.abs(D2).sum(1) * 2.0 ** -126).reshape(-1, 1, 1, 1)
    for part in (np.real, np.imag):
        w, d = np.abs(part(want)), np.abs(part(got) - part(want))
        pair = np.maximum(w, w[::-1])
        assert np.all(d <= 2 * 2.0 ** -24 * pair + 2e-9 * w.max(0) + np.maximum(flush, flush[::-1]))
