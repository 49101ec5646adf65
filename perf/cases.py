"""Performance cases of the ensemble channel DNS library.

One pass is what a simulation program does between two snapshots: a state that
is in device memory goes into the handle, n time steps run, and the new state
comes back as a snapshot in device memory.  The handle (operators, workspace,
kernel choices) is made once and kept, as a program keeps it.  Snapshots of the
mixed path, which computes its increments in single precision, are kept in
single precision; those of the FP64 path in double.

A case names its groups as "flow:MxxMyxMz:members:Re", joined by ";" for a
batch of several groups; a linearised group is "linear:nxMyxMz:vectors:Re" with
n the streamwise wavenumber index.
"""
import collections
import math

import numpy as np
import torch

import paper_2306_12739_gb300 as dns

_HANDLES_KEPT = 16
_handles = collections.OrderedDict()

# (Lx, Lz) in units of pi
_BOX = {"couette": (1.75, 1.2), "poiseuille": (2.0, 1.0), "linear": (2.0, 1.0)}


def _case(name, groups, steps, dt, precision="mixed", form="advective", shared=False):
    return {"name": name, "groups": groups, "steps": steps, "dt": dt, "precision": precision, "form": form,
            "shared": shared}


def listed():
    return [
        # a single realisation on the smallest grid: launches and latency
        _case("single", "couette:16x33x16:1:400", 50, 0.01),
        # a few realisations on a ragged grid (odd member count, even Ny)
        _case("ragged", "couette:48x36x32:3:500", 20, 0.01),
        # the minimal-box ensemble: many members of a small grid
        _case("minimal-box", "couette:32x49x32:64:500", 10, 0.01),
        # the standard turbulent-channel ensemble, and the same in the rotational form
        _case("channel", "poiseuille:64x65x64:8:1650", 20, 0.005),
        _case("rotational", "poiseuille:64x65x64:8:1650", 20, 0.005, form="rotational"),
        # statistical-state dynamics: the members share their streamwise mean
        _case("shared-mean", "couette:64x63x64:5:1000", 20, 0.01, shared=True),
        # an uneven batch: three grids in one step
        _case("batch", "couette:32x33x32:64:400;couette:48x49x48:32:800;poiseuille:64x65x64:32:1650", 4, 0.005),
        # the largest benchmarked grid
        _case("large", "poiseuille:128x97x128:16:3250", 2, 0.002),
        # optimal-growth iterations: forward, adjoint, Gram-Schmidt
        _case("optimal", "linear:1x63x64:45:3000;linear:2x63x64:45:3000;linear:3x63x64:45:3000", 20, 0.04),
        # double precision: a small ensemble, the standard one, a 128-point grid
        _case("small-fp64", "couette:16x33x16:4:400", 10, 0.01, precision="fp64"),
        _case("channel-fp64", "poiseuille:64x65x64:8:1650", 2, 0.005, precision="fp64"),
        _case("large-fp64", "poiseuille:128x97x128:1:3250", 1, 0.002, precision="fp64"),
    ]


def _loguniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("mixed", "mixed", "mixed", "mixed", "rotational", "shared", "linear", "fp64"))
    precision = "fp64" if kind == "fp64" else "mixed"
    my = _loguniform(rng, 17, 129)
    steps = rng.randint(2, 20)
    if kind == "linear":
        mz = rng.choice((16, 32, 48, 64, 128))
        vectors = _loguniform(rng, 3, 64)
        groups = ";".join("linear:%dx%dx%d:%d:3000" % (n, my, mz, vectors) for n in range(1, rng.randint(1, 3) + 1))
        return {k: v for k, v in _case("", groups, steps, 0.04).items() if k != "name"}
    mx = rng.choice((16, 32, 48, 64) if kind == "rotational" else (16, 32, 48, 64, 64, 128))
    # the 128-point plane kernels pair 128 with 64 and 128
    mz = rng.choice((64, 128)) if mx == 128 else rng.choice((16, 32, 48, 64))
    members = _loguniform(rng, 1, 64)
    # grid points advanced in a pass, at most those of the largest listed case of the precision
    cap = 2 * 64 * 65 * 64 * 8 if precision == "fp64" else 2 * 128 * 97 * 128 * 16
    while steps > 1 and members * mx * my * mz * steps > cap:
        steps -= 1
    members = max(1, min(members, cap // (mx * my * mz * steps)))
    flow, re = rng.choice((("couette", 500), ("poiseuille", 1650)))
    dt = 0.01 if mx <= 32 else 0.005 if mx <= 64 else 0.002
    c = _case("", "%s:%dx%dx%d:%d:%d" % (flow, mx, my, mz, members, re), steps, dt, precision,
              "rotational" if kind == "rotational" else "advective", kind == "shared")
    return {k: v for k, v in c.items() if k != "name"}


def _groups(case):
    out = []
    for text in case["groups"].split(";"):
        flow, size, members, re = text.split(":")
        mx, my, mz = (int(x) for x in size.split("x"))
        lx, lz = (math.pi * x for x in _BOX[flow])
        g = dict(flow=flow, mx=mx, my=my, mz=mz, lx=lx, lz=lz, re=float(re), dt=case["dt"], members=int(members))
        if flow == "linear":
            g.update(flow="couette", linear=True, kx_index=mx, mx=0)
        else:
            g.update(form=case["form"], shared_mean=case["shared"])
        out.append(g)
    return out


def _nodes(my):
    y = -np.cos(np.pi * np.arange(my) / (my - 1))
    y[0], y[-1] = -1.0, 1.0
    return y


def _kept(g):
    """Kept wavenumber indices (n of the columns, m of the rows): the 2/3 rule."""
    kz = (g["mz"] - 1) // 3
    n = np.array([g["kx_index"]]) if g.get("linear") else np.arange((g["mx"] - 1) // 3 + 1)
    return n, np.arange(-kz, kz + 1)


def _state(g, seed, device):
    """A seeded state: every kept mode a low-order polynomial in y that meets the
    wall conditions, with a decaying energy spectrum, rms 5e-2 about the laminar
    mean flow; a linearised group gets disturbance vectors of rms 1."""
    rng = np.random.RandomState(seed % (1 << 31))
    n, m = _kept(g)
    y = _nodes(g["my"])
    E, lin, linear = g["members"], 1.0 - y[1:-1] ** 2, bool(g.get("linear"))
    cheb = np.polynomial.chebyshev.chebvander(y[1:-1], 4).T                              # [p, j]
    k = np.hypot(n[None, :] * 2 * np.pi / g["lx"], m[:, None] * 2 * np.pi / g["lz"])
    weight = (1.0 + k * g["lx"] / (2 * np.pi)) ** (-4.0 / 3.0)
    if not linear:
        weight[m == 0, 0] = 0.0
    fields = []
    for wall in (lin ** 2, lin):
        c = rng.standard_normal((E, 5, len(m), len(n), 2)) @ np.array([1.0, 1.0j]) * weight
        if not linear:
            # a real field: the n = 0 column is Hermitian in m
            c[:, :, :, 0] = (c[:, :, :, 0] + np.conj(c[:, :, ::-1, 0])) / 2
            if g["shared_mean"]:
                c[:, :, :, 0] = c[:1, :, :, 0]
        p = torch.from_numpy(cheb * wall).to(device).to(torch.complex128)
        fields.append(torch.einsum("pj,epmn->ejmn", p, torch.from_numpy(np.ascontiguousarray(c)).to(device)))
    ms = sum((f.abs() ** 2).sum(dim=(2, 3)).mean(dim=1) for f in fields)
    scale = (1.0 if linear else 5e-2) / torch.sqrt(ms.mean() if not linear and g["shared_mean"] else ms)
    v, eta = (f * scale.reshape(-1, 1, 1, 1) for f in fields)
    if linear:
        return [v.contiguous(), eta.contiguous()]
    lam = y if g["flow"] == "couette" else 1.0 - y ** 2
    U = torch.from_numpy(np.tile(lam, (E, 1))).to(device)
    return [v.contiguous(), eta.contiguous(), U, torch.zeros_like(U)]


def _base(g):
    """Streak-and-roll base flow of a linearised group on the (My, Mz) grid."""
    y, z = _nodes(g["my"])[:, None], np.arange(g["mz"])[None, :] * (2 * np.pi / g["mz"])
    b, q = 2 * np.pi / g["lz"], 1.0 - y ** 2
    U = y + 0.3 * q * (np.cos(z) - 0.4 * np.sin(2 * z))
    # stream function 0.03 q^2 (sin z + 0.5 cos 2z): divergence-free, no slip
    V = 0.03 * q ** 2 * b * (np.cos(z) - np.sin(2 * z))
    W = 0.12 * y * q * (np.sin(z) + 0.5 * np.cos(2 * z))
    return [f + np.zeros((g["my"], g["mz"])) for f in (U, V, W)]


def _handle(case):
    key = tuple(sorted((k, v) for k, v in case.items() if k != "name"))
    if key not in _handles:
        while len(_handles) >= _HANDLES_KEPT:
            _handles.popitem(last=False)[1].close()
        groups = _groups(case)
        ens = dns.Ensemble(groups, precision=case["precision"], use_graph=True)
        for i, g in enumerate(groups):
            if g.get("linear"):
                ens.set_base_flow(i, *_base(g))
        _handles[key] = ens
    _handles.move_to_end(key)
    return _handles[key]


def prepare(case, seed):
    ens = _handle(case)
    ins = [_state(g, seed * 16 + i, ens.device) for i, g in enumerate(_groups(case))]
    outs = [[torch.empty_like(t) for t in st] for st in ins]
    torch.cuda.synchronize()
    return {"ens": ens, "steps": case["steps"], "mixed": case["precision"] == "mixed", "in": ins, "out": outs}


def _addresses(st):
    return [t.data_ptr() for t in st] + [None] * (4 - len(st))


def run(state):
    ens = state["ens"]
    for i, st in enumerate(state["in"]):
        dns.dns_set_state(ens.h, i, 0, st[0].shape[0], *_addresses(st), 1)
    linear = len(state["in"][0]) == 2
    gains = ens.optimal_sweep(state["steps"]) if linear else ens.step(state["steps"])
    for i, st in enumerate(state["out"]):
        dns.dns_get_state(ens.h, i, 0, st[0].shape[0], *_addresses(st), 1)
    # the snapshot; the mean flow is one velocity field
    res = {}
    with torch.cuda.stream(ens.stream):
        for i, st in enumerate(state["out"]):
            snap = {"v": st[0], "eta": st[1]}
            if not linear:
                snap["mean"] = torch.stack(st[2:])
            if state["mixed"]:
                snap = {k: t.to(torch.complex64 if t.is_complex() else torch.float32) for k, t in snap.items()}
            if linear:
                snap["gains"] = gains[i].astype(np.float32 if state["mixed"] else np.float64)
            res["group%d" % i] = snap
    return res


def work(case):
    """State in and out, the per-wavenumber operators of both step lengths once
    (their even and odd halves), and the arithmetic of the sub-steps."""
    mixed = case["precision"] == "mixed"
    nbytes = flops = 0.0
    for g in _groups(case):
        n, m = _kept(g)
        ny, E = g["my"] - 2, g["members"]
        modes, pairs = len(n) * len(m), len(n) * ((len(m) + 1) // 2)
        field = E * ny * modes
        nbytes += 2 * field * (16 + (8 if mixed else 16)) + pairs * 2 * 4 * ny * ny / 2 * (4 if mixed else 8)
        columns = 8 * field * 4 * ny / 2                                     # 3 derivatives, D1 phi, M and P twice
        if g.get("linear"):
            plane = E * ny * (12 * 5 * g["mz"] * math.log2(g["mz"]) + 60 * g["mz"])
            flops += 2 * case["steps"] * 3 * (columns + plane) + 8.0 * E * E * ny * modes * 3
        else:
            pts = g["mx"] * g["mz"]
            transforms, products = (9, 15) if g["form"] == "rotational" else (15, 22)
            plane = E * ny * (transforms * 2.5 * pts * math.log2(pts) + products * pts)
            flops += case["steps"] * 3 * (columns + plane)
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------ the same in 64 bits, by torch


def _diff_matrix(x):
    """First-derivative matrix of the interpolant on the nodes x (barycentric)."""
    d = x[:, None] - x[None, :]
    np.fill_diagonal(d, 1.0)
    c = np.prod(d, axis=1)
    D = c[:, None] / c[None, :] / d
    np.fill_diagonal(D, 0.0)
    np.fill_diagonal(D, -D.sum(axis=1))
    return D


def _y_operators(my):
    """D1, D2 on all nodes, the clamped fourth derivative on the interior ones,
    and the Clenshaw-Curtis weights; formed in extended precision."""
    one = np.longdouble(1)
    pi = np.arctan(one) * 4
    y = -np.cos(pi * np.arange(my) / (my - 1) * one)
    y = (y - y[::-1]) / 2
    D1 = _diff_matrix(y)
    t = y[1:-1]
    T1 = _diff_matrix(t)
    T2 = T1 @ T1
    T3, T4 = T2 @ T1, T2 @ T2
    w, col = (1 - t * t) ** 2, lambda f: f[:, None]
    D4 = col(w) * T4 + col(16 * t ** 3 - 16 * t) * T3 + col(72 * t * t - 24) * T2 + col(96 * t) * T1
    D4 = (D4 + 24 * np.eye(my - 2)) / w[None, :]
    N, k = my - 1, np.arange(0, my, 2)
    cc = np.cos(pi * np.outer(k, np.arange(my)) / N * one)
    half = np.where((k == 0) | (k == N), 0.5, 1.0)
    weights = (2.0 / N) * ((half * 2.0 / (1.0 - k * k))[:, None] * cc).sum(axis=0)
    weights[0] /= 2
    weights[-1] /= 2
    return [np.asarray(a, dtype=np.float64) for a in (D1, D1 @ D1, D4, weights)]


class _Exact:
    """The time step of one group in 64 bits: CN/RK3 in increment form,
    A d = 2 g B x + h dt F per wavenumber pair, library FFTs and products."""

    def __init__(self, g, device):
        self.g, self.device = g, device
        put = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(device)
        D1, D2, D4, w = _y_operators(g["my"])
        self.D1, self.D2, self.w = put(D1).to(torch.complex128), put(D2).to(torch.complex128), put(w)
        self.D1r = put(D1)
        n, m = _kept(g)
        self.kz_max, self.columns = len(m) // 2, len(n)
        kx, kz = n * 2 * np.pi / g["lx"], m * 2 * np.pi / g["lz"]
        self.ikx, self.ikz = put(1j * kx)[None, None, None, :], put(1j * kz)[None, None, :, None]
        k2 = kx[None, :] ** 2 + kz[:, None] ** 2
        self.k2 = put(k2)[None, None]
        self.k2s = torch.where(self.k2 == 0, torch.ones_like(self.k2), self.k2)
        self.absm = put(np.abs(m))
        self.sub = {}
        eye = torch.eye(g["my"] - 2, dtype=torch.float64, device=device)
        D2i, D4i = put(D2[1:-1, 1:-1].copy()), put(D4)
        kk = put(k2[self.kz_max:].copy())[:, :, None, None]
        lap, bilap = D2i - kk * eye, D4i - 2 * kk * D2i + kk * kk * eye
        for h in (0.5, 1.0):
            c = h * g["dt"] / (2 * g["re"])
            fac = [torch.linalg.lu_factor(a) for a in (lap - c * bilap, eye - c * lap, eye - c * D2i)]
            self.sub[h] = (c, fac)
        self.lap, self.bilap, self.D2i, self.D2w = lap, bilap, D2i, put(D2[1:-1][:, [0, -1]].copy())

    def _solve(self, fac, op, x, f, c, hdt):
        """x + A^-1 (2 c B x + s h dt f) for every mode; x, f [e, j, m, n]."""
        def apply(M, z):
            return torch.einsum("mnij,ejmn->eimn", M[self.absm].to(torch.complex128), z)
        rhs = 2 * c * apply(op, x) + hdt * f
        E, ny, nm, nn = rhs.shape
        cols = torch.view_as_real(rhs.permute(2, 3, 1, 0).contiguous()).reshape(nm, nn, ny, 2 * E)
        d = torch.linalg.lu_solve(fac[0][self.absm], fac[1][self.absm], cols)
        return x + torch.view_as_complex(d.reshape(nm, nn, ny, E, 2).contiguous()).permute(3, 2, 0, 1)

    def _velocity(self, v, eta, U=None, W=None):
        pad = lambda f: torch.nn.functional.pad(f, (0, 0, 0, 0, 1, 1))
        dy = lambda D, f: torch.einsum("ij,ejmn->eimn", D, f)
        v, eta = pad(v), pad(eta)
        dv, d2v, de = dy(self.D1, v), dy(self.D2, v), dy(self.D1, eta)
        u, w = (self.ikx * dv - self.ikz * eta) / self.k2s, (self.ikz * dv + self.ikx * eta) / self.k2s
        uy, wy = (self.ikx * d2v - self.ikz * de) / self.k2s, (self.ikz * d2v + self.ikx * de) / self.k2s
        if U is not None:
            for f, F in ((u, U), (w, W), (uy, U @ self.D1r.T), (wy, W @ self.D1r.T)):
                f[:, :, self.kz_max, 0] = F.to(f.dtype)
        return [[u, uy], [v, dv], [w, wy]]

    def _forcing(self, x):
        Nu, Nv, Nw, means = self._terms(x)
        phi = self.ikx * Nu + self.ikz * Nw
        F = -self.k2 * Nv - torch.einsum("ij,ejmn->eimn", self.D1[1:-1, 1:-1], phi)
        return [F, self.ikz * Nu - self.ikx * Nw] + [(a @ self.D1r.T)[:, 1:-1] for a in means]

    def _update(self, x, F, h):
        c, fac = self.sub[h]
        hdt = h * self.g["dt"]
        # the equations carry -F: d(lap v)/dt = F + bilap v / Re with N on the left
        v = self._solve(fac[0], self.bilap, x[0], F[0], c, self.sign * hdt)
        eta = self._solve(fac[1], self.lap, x[1], F[1], c, self.sign * hdt)
        out = [v, eta]
        for U, f in zip(x[2:], F[2:]):
            walls = U[:, [0, -1]] @ self.D2w.T
            rhs = 2 * c * (U[:, 1:-1] @ self.D2i.T + walls) - hdt * f
            out.append(U + torch.nn.functional.pad(torch.linalg.lu_solve(*fac[2], rhs.T).T, (1, 1)))
        if len(x) == 4:
            for a in (v, eta):
                a[:, :, self.kz_max, 0] = 0
            if self.g["flow"] == "poiseuille":
                unit = torch.linalg.lu_solve(*fac[2], torch.full((len(self.D2i), 1), hdt, dtype=torch.float64,
                                                                 device=self.device))[:, 0]
                gamma = (4.0 / 3.0 - out[2] @ self.w) / (unit @ self.w[1:-1])
                out[2][:, 1:-1] += gamma[:, None] * unit
        return out

    sign = -1.0

    def step(self, x):
        F0 = self._forcing(x)
        a = self._update(x, F0, 0.5)
        F1 = self._forcing(a)
        b = self._update(x, [2 * q - p for p, q in zip(F0, F1)], 1.0)
        F2 = self._forcing(b)
        return self._update(x, [(p + 4 * q + r) / 6 for p, q, r in zip(F0, F1, F2)], 1.0)

    # ---- full nonlinear groups
    def _grid(self, c):
        mx, mz, K = self.g["mx"], self.g["mz"], self.kz_max
        Z = torch.zeros(c.shape[:-2] + (mz, mx // 2 + 1), dtype=c.dtype, device=self.device)
        Z[..., :K + 1, :self.columns] = c[..., K:, :]
        Z[..., mz - K:, :self.columns] = c[..., :K, :]
        return torch.fft.irfft2(Z, s=(mz, mx), norm="forward")

    def _kept_of(self, f):
        K = self.kz_max
        F = torch.fft.rfft2(f, norm="forward")
        return torch.cat([F[..., self.g["mz"] - K:, :self.columns], F[..., :K + 1, :self.columns]], dim=-2)

    def _terms(self, x):
        vel = [[f[:, 1:-1] for f in pair] for pair in self._velocity(*x)]
        u, v, w = (self._grid(p[0]) for p in vel)
        N = [self._kept_of(u * self._grid(self.ikx * f) + v * self._grid(fy) + w * self._grid(self.ikz * f))
             for f, fy in vel] if self.g["form"] == "advective" else self._rotational(vel, u, v, w)
        means = [torch.nn.functional.pad((a * v).mean(dim=(-2, -1)), (1, 1)) for a in (u, w)]
        if self.g["shared_mean"]:
            for a in N:
                a[..., 0] = a[..., 0].mean(dim=0, keepdim=True)
            means = [a.mean(dim=0, keepdim=True).expand_as(a) for a in means]
        return N[0], N[1], N[2], means

    def _rotational(self, vel, u, v, w):
        (us, uy), (vs, _), (ws, wy) = vel
        ox = self._grid(wy - self.ikz * vs)
        oy = self._grid(self.ikz * us - self.ikx * ws)
        oz = self._grid(self.ikx * vs - uy)
        return [self._kept_of(a) for a in (oy * w - oz * v, oz * u - ox * w, ox * v - oy * u)]


class _ExactLinear(_Exact):
    """A linearised group: forward or adjoint terms about the base flow."""

    def __init__(self, g, device):
        super().__init__(g, device)
        spec = [self._kept_of(torch.from_numpy(f).to(device).to(torch.complex128)) for f in _base(g)]
        ikz = self.ikz.reshape(1, -1)
        self.base = [[self._grid(c).real, self.D1r @ self._grid(c).real, self._grid(ikz * c).real] for c in spec]
        self.base = [[f[1:-1][None, :, :] for f in row] for row in self.base]
        self.adjoint = False

    def _grid(self, c):
        Z = torch.zeros(c.shape[:-1] + (self.g["mz"],), dtype=c.dtype, device=self.device)
        Z[..., :self.kz_max + 1] = c[..., self.kz_max:]
        Z[..., self.g["mz"] - self.kz_max:] = c[..., :self.kz_max]
        return torch.fft.ifft(Z, norm="forward")

    def _kept_of(self, f):
        F = torch.fft.fft(f, norm="forward")
        return torch.cat([F[..., self.g["mz"] - self.kz_max:], F[..., :self.kz_max + 1]], dim=-1)

    def _terms(self, x):
        vel = [[f[:, 1:-1, :, 0] for f in pair] for pair in self._velocity(*x)]
        kx, ikz = self.ikx.reshape(()), self.ikz[..., 0]
        B = self.base
        p = [[self._grid(f), self._grid(fy), self._grid(ikz * f)] for f, fy in vel]
        adv = [kx * B[0][0] * f + B[1][0] * fy + B[2][0] * fz for f, fy, fz in p]
        if not self.adjoint:
            N = [a + p[1][0] * b[1] + p[2][0] * b[2] for a, b in zip(adv, B)]
        else:
            N = [-adv[0]] + [-adv[d] + sum(p[c][0] * B[c][d] for c in range(3)) for d in (1, 2)]
        return [self._kept_of(a)[..., None] for a in N] + [[]]

    def sweep(self, x, steps):
        for self.adjoint in (False, True):
            for _ in range(steps):
                x = self.step(x)
        # energy coordinates: v, Dv / k, eta / k weighted by the quadrature
        v, eta = x
        s = torch.sqrt(self.w[1:-1] / 4)[None, :, None, None]
        k = torch.sqrt(self.k2)
        dv = torch.einsum("ij,ejmn->eimn", self.D1[1:-1, 1:-1], v)
        A = torch.cat([(s * f).reshape(len(v), -1) for f in (v, dv / k, eta / k)], dim=1).T
        R = torch.linalg.qr(A, mode="r").R
        R = R * (torch.conj(torch.diagonal(R)) / torch.diagonal(R).abs())[:, None]
        T = torch.linalg.inv(R)
        v, eta = (torch.einsum("ek,ejmn->kjmn", T, f) for f in (v, eta))
        return [v, eta], torch.diagonal(R).real


def exact(case, seed):
    device = torch.device("cuda:0" if torch.cuda.is_available() else "cpu")
    res = {}
    for i, g in enumerate(_groups(case)):
        x = _state(g, seed * 16 + i, device)
        if g.get("linear"):
            x, gains = _ExactLinear(g, device).sweep(x, case["steps"])
            res["group%d" % i] = {"v": x[0], "eta": x[1], "gains": gains.cpu().numpy()}
        else:
            e = _Exact(g, device)
            for _ in range(case["steps"]):
                x = e.step(x)
            res["group%d" % i] = {"v": x[0], "eta": x[1], "mean": torch.stack(x[2:])}
    return res
