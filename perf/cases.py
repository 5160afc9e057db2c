"""Performance cases: what a user of the framework has it compute, over its real range.

A case is a scan description plus what is done with it: one operator pair (a forward and
an adjoint application, the body of every iterative reconstruction), a calibration step,
a solve, or a burst of served requests. Sizes are those of phantoms/configs.py (tiny,
phantom and in-vivo scale, the serving mix) and ragged ones between them.

prepare() builds the handle a program keeps, with its path and precision selected, and
seeded inputs on the GPU. exact() evaluates the same operator in 64 bits with plain torch.
"""

import math

import torch

from paper_2511_06627_gb300 import PREC_TF32, FFLOperator
from paper_2511_06627_gb300.autograd import apply_a
from paper_2511_06627_gb300.serving import ReconServer, Request

TINY = dict(nx=32, nz=16, n_angles=8, S=64, P=128, fwhm=2.0, k_max=8, half_width=2)
PHANTOM = dict(nx=128, nz=64, n_angles=24, S=64, P=256, fwhm=3.0, k_max=12, half_width=3)
INVIVO = dict(nx=256, nz=128, n_angles=36, S=128, P=512, fwhm=3.0, k_max=16, half_width=4)
MIDDLE = dict(nx=192, nz=96, n_angles=21, S=64, P=384, fwhm=3.0, k_max=12, half_width=3)
RAGGED = dict(nx=101, nz=37, n_angles=21, S=50, P=202, fwhm=2.5, k_max=10, half_width=2)
GEOMETRY = ("nx", "nz", "n_angles", "S", "P", "fwhm", "k_max", "half_width")


def listed():
    return [
        # the smallest scan: a pair is a handful of short kernels, so launches and latency count
        dict(TINY, name="pair_tiny_full_gemm", kind="pair", path="full_gemm"),
        # a new handle's default path (plain FP32) at the three scales, one of them ragged: odd
        # detector, odd slice count, a period that is not a multiple of four samples
        dict(RAGGED, name="pair_ragged_staged", kind="pair", path="staged"),
        dict(PHANTOM, name="pair_phantom_staged", kind="pair", path="staged"),
        dict(INVIVO, name="pair_invivo_staged", kind="pair", path="staged"),
        # the tensor-core paths of production reconstructions, at the serving mix's middle size in
        # the more precise split and at in-vivo scale in the default one
        dict(MIDDLE, name="pair_middle_full_gemm_tf32", kind="pair", path="full_gemm", tf32=True),
        dict(INVIVO, name="pair_invivo_full_gemm", kind="pair", path="full_gemm"),
        # the second drive axis of the dual-drive scan
        dict(INVIVO, name="pair_invivo_zdrive", kind="zdrive", path="staged"),
        # the in-plane tensor PSF, which couples every slice
        dict(INVIVO, name="pair_invivo_tensor_psf", kind="tensor", path="full_gemm"),
        # two iterations of the joint volume and calibration fit: forward and all gradients, at
        # two sets of gains and PSF widths
        dict(PHANTOM, name="fit_phantom_line_gemm", kind="fit", path="line_gemm"),
        # whole reconstructions: power iteration and Eq. (26), from one scan and from both
        dict(PHANTOM, name="solve_phantom_full_gemm", kind="solve", path="full_gemm", scans="x", iters=100, n_power=50),
        dict(PHANTOM, name="solve_phantom_both_scans", kind="solve", path="full_gemm", scans="xz", iters=20,
             n_power=10),
        # four requests of mixed sizes that arrive together at the reconstruction server
        dict(name="serve_burst", kind="serve", path="full_gemm", iters=40, n_power=20),
    ]


def draw(rng):
    """One more case: the listed kinds, paths and options over the range of sizes between
    the tiny and the in-vivo scale, ragged sizes among them."""
    kind = rng.choice(["pair"] * 5 + ["zdrive", "zdrive", "tensor", "fit", "solve"])
    path = {"zdrive": "staged", "fit": "line_gemm"}.get(kind) or "full_gemm"
    if kind == "pair":
        path = rng.choice(["staged", "staged", "line_gemm", "full_gemm", "full_gemm"])
    top_n, top_z = (256, 128) if kind in ("pair", "zdrive") else (128, 64)
    nx = int(round(math.exp(rng.uniform(math.log(32), math.log(top_n)))))
    nz = int(round(math.exp(rng.uniform(math.log(8), math.log(min(top_z, nx))))))
    if rng.random() < 0.5:
        nx -= nx % 4
    S = rng.choice([40, 50, 64, 64, 128])
    P = max(64, int(2 * nx * rng.uniform(0.8, 1.0)))
    P += P % 2 if S % 4 else 0  # a whole number of four-sample groups a line
    k_max = rng.randint(6, min(16, S // 2 - 2))
    case = dict(kind=kind, path=path, nx=nx, nz=nz, n_angles=rng.randint(8, 36), S=S, P=P,
                fwhm=round(rng.uniform(2.0, 4.0), 2), k_max=k_max, half_width=rng.randint(1, 4))
    if path in ("line_gemm", "full_gemm") and rng.random() < 0.4:
        case["tf32"] = True
    if kind == "solve":
        case.update(scans=rng.choice(["x", "x", "xz"]), iters=rng.randint(10, 40), n_power=10)
    return case


def serve_requests():
    """The burst's scans: the smaller sizes of the serving mix."""
    def scan(nx, nz, m, k):
        return dict(nx=nx, nz=nz, n_angles=m, S=64, P=2 * nx, fwhm=3.0, k_max=k, half_width=max(1, k // 4))
    return [scan(64, 64, 12, 8), scan(128, 64, 24, 12), scan(64, 64, 30, 15), scan(128, 64, 10, 9)]


def _operator(case):
    op = FFLOperator(**{k: case[k] for k in GEOMETRY}, path=case["path"])
    if case.get("tf32"):
        op.set_precision(PREC_TF32)
    return op


def _phantom(case, gen):
    """A volume of a few random ellipsoids and point sources on a weak background inside
    the scanner's cylinder, as phantoms/generators.py draws them (zero outside)."""
    nz, n = case["nz"], case["nx"]
    dev = gen.device
    z = torch.arange(nz, device=dev, dtype=torch.float32).view(-1, 1, 1)
    y = torch.arange(n, device=dev, dtype=torch.float32).view(1, -1, 1)
    x = torch.arange(n, device=dev, dtype=torch.float32).view(1, 1, -1)
    c = (n - 1) / 2
    inside = (x - c) ** 2 + (y - c) ** 2 <= (n / 2 - 2) ** 2
    vol = 1e-4 * inside.expand(nz, n, n).float()
    u = torch.rand(16, 7, generator=gen, device=dev).cpu().tolist()
    for a in u:
        r = a[0] * 0.3 * n
        cy, cx = c + r * math.sin(6.283 * a[1]), c + r * math.cos(6.283 * a[1])
        cz = (0.15 + 0.7 * a[2]) * (nz - 1)
        semi = [max(1.0, (0.03 + 0.1 * a[3]) * nz), 1.0 + (0.02 + 0.1 * a[4]) * n, 1.0 + (0.02 + 0.1 * a[5]) * n]
        d = ((z - cz) / semi[0]) ** 2 + ((y - cy) / semi[1]) ** 2 + ((x - cx) / semi[2]) ** 2
        vol = vol + 10 ** (3 * a[6] - 3) * ((d <= 1) & inside)
    return vol.contiguous()


def _inputs(case, seed):
    """What every kind needs, from the seed alone: a phantom and a data vector of noise, as
    the residual of a reconstruction is."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    x = _phantom(case, gen)
    nb = case["k_max"] * (2 * case["half_width"] + 1)
    y = torch.randn(case["n_angles"], case["nz"], nb, 2, generator=gen, device="cuda")
    return x, y


def _scan_data(case, x, noise):
    """Compressed data of x with noise of half a percent of the largest value."""
    m = _Model(case)
    b = [m.forward(x.double())] if case.get("scans", "x") in ("x", "xz") else []
    if "z" in case.get("scans", "x"):
        b.append(m.forward_z(x.double()))
    b = torch.cat(b)
    scale = 0.005 * float(b.abs().max())
    noise = noise.repeat(b.shape[0] // noise.shape[0], 1, 1, 1)
    return (b + scale * noise.double()).float()


def _fit_inputs(case, seed):
    """Two parameter sets (gains, width) and, for each, the data misfit of the fit against
    a scan whose gains and width are others."""
    x, _ = _inputs(case, seed)
    gen = torch.Generator(device="cuda").manual_seed(seed + 1)
    M = case["n_angles"]
    draw_gains = lambda: 1 + 0.1 * (torch.rand(M, generator=gen, device="cuda") - 0.5)  # noqa: E731
    target = _Model(dict(case, fwhm=1.1 * case["fwhm"]), draw_gains().double()).forward(x.double())
    sets = []
    for k in range(2):
        g = draw_gains()
        w = torch.tensor([case["fwhm"] * (1 + 0.02 * k)], device="cuda")
        misfit = _Model(dict(case, fwhm=float(w.item())), g.double()).forward(x.double()) - target
        sets.append((g, w, misfit.float()))
    return x, sets


def prepare(case, seed):
    kind = case["kind"]
    if kind == "serve":
        reqs = []
        for k, g in enumerate(serve_requests()):
            x, noise = _inputs(g, seed + 100 * k)
            reqs.append((g, _scan_data(g, x, noise)))
        return dict(case=case, server=ReconServer(path=case["path"]), reqs=reqs)
    op = _operator(case)
    if kind == "fit":
        x, sets = _fit_inputs(case, seed)
        sets = [(g.requires_grad_(True), w.requires_grad_(True), y) for g, w, y in sets]
        return dict(case=case, op=op, x=x.requires_grad_(True), sets=sets)
    x, y = _inputs(case, seed)
    if kind == "tensor":
        op.set_psf_model("tensor")
    if kind == "solve":
        op.set_scans(case["scans"])
        return dict(case=case, op=op, b=_scan_data(case, x, y))
    return dict(case=case, op=op, x=x, y=y)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "serve":
        reqs = [Request(geometry=dict(g, k_min=1), data=b, iters=case["iters"], n_power=case["n_power"], name=str(k))
                for k, (g, b) in enumerate(state["reqs"])]
        state["server"].run(reqs)
        return [r.result for r in reqs]
    op = state["op"]
    if kind == "fit":
        out = []
        for gains, width, misfit in state["sets"]:
            b = apply_a(op, state["x"], gains, width)
            out += [b.detach(), *torch.autograd.grad(b, (state["x"], gains, width), misfit)]
        return out
    if kind == "solve":
        x, rep = op.solve(state["b"], iters=case["iters"], n_power=case["n_power"])
        return [x, torch.tensor([rep["residual_first"], rep["residual_last"], rep["ata_norm"]], dtype=torch.float32)]
    if kind == "zdrive":
        return [op.forward_zdrive(state["x"]), op.adjoint_zdrive(state["y"])]
    return [op.forward(state["x"]), op.adjoint(state["y"])]


def _pair_work(case):
    """(bytes, flops) of one forward and one adjoint: volume and data read once and written
    once; two taps a ray and march step, and the line operator as one matrix of the kept
    bins (real and imaginary parts) by the detector bins, per line (per line and slice with
    the tensor PSF; along z, per line and phase through the detector's columns)."""
    n, nz, m = case["nx"], case["nz"], case["n_angles"]
    nb = case["k_max"] * (2 * case["half_width"] + 1)
    vox, lines = nz * n * n, m * nz
    nbytes = 8 * vox + 2 * 8 * lines * nb
    projector = 2 * 4 * m * vox
    line = 2 * 2 * lines * 2 * nb * n
    if case["kind"] == "tensor":
        line *= nz
    if case["kind"] == "zdrive":
        line = 2 * 2 * lines * (case["S"] * n * (2 * case["half_width"] + 1) + 2 * nb * case["S"])
    return nbytes, projector + line


def work(case):
    if case["kind"] == "serve":
        total = [0, 0]
        for g in serve_requests():
            b, f = _pair_work(dict(g, kind="pair"))
            for k, v in enumerate((b, f)):
                total[k] += (case["iters"] + case["n_power"]) * v
        return dict(bytes=total[0], flops=total[1])
    b, f = _pair_work(case)
    if case["kind"] == "solve":
        pairs = case["iters"] + case["n_power"]
        if case["scans"] == "xz":
            bz, fz = _pair_work(dict(case, kind="zdrive"))
            b, f = b + bz, f + fz
        return dict(bytes=pairs * b, flops=pairs * f)
    if case["kind"] == "fit":
        # two steps, each a pair and the two parameter gradients' line operators
        nb = case["k_max"] * (2 * case["half_width"] + 1)
        lines = case["n_angles"] * case["nz"]
        return dict(bytes=2 * (b + 2 * 8 * lines * nb), flops=2 * (f + 2 * 2 * lines * 2 * nb * case["nx"]))
    return dict(bytes=b, flops=f)


# ------------------------------------------------------------------ the operator in 64 bits

def _d1(x):
    """L'(x) = 1/x^2 - 1/sinh(x)^2 of the Langevin function."""
    ax = x.abs()
    x2 = x * x
    series = 1 / 3 - x2 / 15 + 2 * x2**2 / 189 - x2**3 / 675
    safe = torch.where(ax < 0.05, torch.ones_like(x), ax)
    return torch.where(ax < 0.05, series, 1 / safe**2 - 1 / torch.sinh(safe) ** 2)


def _d2(x):
    """L''(x)."""
    ax = x.abs()
    series = -2 * x / 15 + 8 * x**3 / 189 - 6 * x**5 / 675
    safe = torch.where(ax < 0.05, torch.ones_like(x), ax)
    big = safe > 200  # sinh^3 would overflow; its term is zero there
    s = torch.where(big, torch.ones_like(x), safe)
    val = -2 / safe**3 + torch.where(big, torch.zeros_like(x), 2 * torch.cosh(s) / torch.sinh(s) ** 3)
    return torch.where(ax < 0.05, series, torch.sign(x) * val)


def _l_over_x(x):
    """L(x) / x, x >= 0."""
    x2 = x * x
    series = 1 / 3 - x2 / 45 + 2 * x2**2 / 945 - x2**3 / 4725
    safe = torch.where(x < 0.05, torch.ones_like(x), x)
    return torch.where(x < 0.05, series, (1 / torch.tanh(safe) - 1 / safe) / safe)


def _half_point():
    lo, hi = 0.5, 5.0
    for _ in range(200):
        mid = (lo + hi) / 2
        if 1 / mid**2 - 1 / math.sinh(mid) ** 2 > 1 / 6:
            lo = mid
        else:
            hi = mid
    return (lo + hi) / 2


class _Model:
    """A, A_z and their transposes in 64 bits on the GPU: Joseph projection, Langevin PSF on
    a grid Q times finer than the bins, linear interpolation along the FFL trajectory times
    its velocity, and the unitary DFT on the kept bins, the line stages as one matrix."""

    A, Q = 6.0, 8

    def __init__(self, case, gains=None):
        self.case = case
        self.N, self.Nz, self.M = case["nx"], case["nz"], case["n_angles"]
        self.S, self.L = case["S"], case["S"] * case["P"]
        self.nb = case["k_max"] * (2 * case["half_width"] + 1)
        self.a = case["fwhm"] / (2 * _half_point())
        self.D = math.ceil(self.A * self.Q - 1e-9)
        self.g = torch.ones(self.M, device="cuda", dtype=torch.float64) if gains is None else gains
        self._rays, self._lines, self._dft = None, {}, None

    def _range(self, n):
        return torch.arange(n, device="cuda", dtype=torch.float64)

    # -- projection: per angle, the flat voxel index and weight of both taps of [step][ray]
    def _taps(self):
        if self._rays is None:
            n, self._rays = self.N, []
            c = (n - 1) / 2
            s, i = self._range(n)[:, None], self._range(n)[None]
            for m in range(self.M):
                cs, sn = math.cos(m * math.pi / self.M), math.sin(m * math.pi / self.M)
                rows = abs(cs) >= abs(sn) - 1e-9
                f = (i - c) / cs + (s - c) * (sn / cs) + c if rows else -(i - c) / sn + (s - c) * (cs / sn) + c
                k = f.floor()
                taps = []
                for kk, w in ((k, 1 - (f - k)), (k + 1, f - k)):
                    w = torch.where((kk >= 0) & (kk < n), w, torch.zeros_like(w))
                    kk = kk.clamp(0, n - 1)
                    taps.append(((s * n + kk if rows else kk * n + s).long().reshape(-1), w.reshape(-1, 1)))
                self._rays.append((taps, 1 / abs(cs) if rows else 1 / abs(sn)))
        return self._rays

    def project(self, x):
        v = x.reshape(self.Nz, -1).T.contiguous()
        out = torch.empty(self.M, self.Nz, self.N, device="cuda", dtype=torch.float64)
        for m, (taps, scale) in enumerate(self._taps()):
            rays = sum((w * v[k]).view(self.N, self.N, self.Nz).sum(0) for k, w in taps)
            out[m] = scale * rays.T
        return out

    def backproject(self, p):
        v = torch.zeros(self.N * self.N, self.Nz, device="cuda", dtype=torch.float64)
        for m, (taps, scale) in enumerate(self._taps()):
            rays = (scale * p[m].T).repeat(self.N, 1)
            for k, w in taps:
                v.index_add_(0, k, w * rays)
        return v.T.reshape(self.Nz, self.N, self.N).contiguous()

    # -- the line operator per trajectory
    def _fine(self, n):
        return (n - 1) * self.Q + 2 * self.D + 1

    def _offsets(self, n):
        return (self._range(self._fine(n))[:, None] - self.D) / self.Q - self._range(n)[None]

    def dft(self):
        """[2 nb][L]: rows Re, Im of L^-1/2 exp(2 pi i omega j / L)."""
        if self._dft is None:
            c = self.case
            hw = c["half_width"]
            om = torch.tensor([k * c["P"] + d for k in range(1, c["k_max"] + 1) for d in range(-hw, hw + 1)],
                              device="cuda")
            ang = (om[:, None] * torch.arange(self.L, device="cuda")[None] % self.L).double() * (2 * math.pi / self.L)
            self._dft = torch.stack([ang.cos(), ang.sin()], 1).reshape(2 * self.nb, self.L) / math.sqrt(self.L)
        return self._dft

    def slow(self, par):
        c = self._range(self.L) * ((self.N - 1) / (self.L - 1))
        return (self.N - 1) - c if par else c

    def w(self, par):
        """[2 nb][N_e]: the DFT of the samples' interpolation from the fine grid."""
        if par not in self._lines:
            j = self._range(self.L)
            ph = 2 * math.pi * (j % self.S) / self.S
            slope = (self.N - 1) / (self.L - 1) * (-1 if par else 1)
            v = slope + self.A * (2 * math.pi / self.S) * ph.cos()
            t = self.Q * (self.slow(par) + self.A * ph.sin()) + self.D
            ne = self._fine(self.N)
            n = t.floor().clamp(max=ne - 2)
            f = t - n
            n, d = n.long(), self.dft()
            out = torch.zeros(ne, 2 * self.nb, device="cuda", dtype=torch.float64)
            out.index_add_(0, n, ((1 - f) * v)[:, None] * d.T)
            out.index_add_(0, n + 1, (f * v)[:, None] * d.T)
            self._lines[par] = out.T.contiguous()
        return self._lines[par]

    def line(self, par, width_gradient=False):
        u = self._offsets(self.N) / self.a
        h = -3 * _d2(u) * u / self.case["fwhm"] if width_gradient else 3 * _d1(u)
        return self.w(par) @ h

    def lines_forward(self, p, gains=None, width_gradient=False):
        out = torch.empty(self.M, self.Nz, 2 * self.nb, device="cuda", dtype=torch.float64)
        for par in range(2):
            out[:, par::2] = p[:, par::2] @ self.line(par, width_gradient).T
        g = self.g if gains is None else gains
        return (out * g[:, None, None]).view(self.M, self.Nz, self.nb, 2)

    def lines_adjoint(self, y):
        y = y.reshape(self.M, self.Nz, -1) * self.g[:, None, None]
        out = torch.empty(self.M, self.Nz, self.N, device="cuda", dtype=torch.float64)
        for par in range(2):
            out[:, par::2] = y[:, par::2] @ self.line(par)
        return out

    def forward(self, x):
        return self.lines_forward(self.project(x))

    def adjoint(self, y):
        return self.backproject(self.lines_adjoint(y))

    # -- tensor PSF: one matrix per trajectory and slice offset
    def _offset_lines(self):
        u = self._offsets(self.N)
        out = [[], []]
        for d in range(self.Nz):
            rho2 = u * u + d * d
            xi = rho2.sqrt() / self.a
            safe = torch.where(rho2 == 0, torch.ones_like(rho2), rho2)
            h = 3 * (_d1(xi) * u * u + _l_over_x(xi) * d * d) / safe
            h = torch.where(rho2 == 0, torch.ones_like(h), h)
            for par in range(2):
                out[par].append(self.w(par) @ h)
        return [torch.stack(o) for o in out]  # [offset][2 nb][N]

    def forward_tensor(self, x):
        p, t = self.project(x), self._offset_lines()
        out = torch.empty(self.M, self.Nz, 2 * self.nb, device="cuda", dtype=torch.float64)
        z = torch.arange(self.Nz, device="cuda")
        for l in range(self.Nz):
            full = t[l % 2][(z - l).abs()].permute(1, 0, 2).reshape(2 * self.nb, -1)
            out[:, l] = p.reshape(self.M, -1) @ full.T
        return out.view(self.M, self.Nz, self.nb, 2)

    def adjoint_tensor(self, y):
        t, y = self._offset_lines(), y.reshape(self.M, self.Nz, -1)
        p = torch.zeros(self.M, self.Nz * self.N, device="cuda", dtype=torch.float64)
        z = torch.arange(self.Nz, device="cuda")
        for l in range(self.Nz):
            p += y[:, l] @ t[l % 2][(z - l).abs()].permute(1, 0, 2).reshape(2 * self.nb, -1)
        return self.backproject(p.view(self.M, self.Nz, self.N))

    # -- the z-drive scan: the drive and the PSF along z, the raster along the detector
    def _z_reads(self, par):
        """Flat indices into [N + 1][N_ez] and weights of the four taps of [line][sample]."""
        nez = self._fine(self.Nz)
        j = self._range(self.L)
        ph = 2 * math.pi * (j % self.S) / self.S
        v = self.A * (2 * math.pi / self.S) * ph.cos()
        c = self.slow(par)
        u = c.floor().clamp(0, self.N - 1)
        a = c - u
        lines = self._range(self.Nz)[par::2, None]
        t = self.Q * (lines + self.A * ph.sin()) + self.D
        n = t.floor().clamp(max=nez - 2)
        f = t - n
        base = (u * nez + n).long()
        return [(base + off, v * wu * wz) for off, wu, wz in
                ((0, 1 - a, 1 - f), (1, 1 - a, f), (nez, a, 1 - f), (nez + 1, a, f))]

    def forward_z(self, x):
        p, d = self.project(x), self.dft()
        h = 3 * _d1(self._offsets(self.Nz) / self.a)
        out = torch.empty(self.M, self.Nz, 2 * self.nb, device="cuda", dtype=torch.float64)
        for par in range(min(2, self.Nz)):
            reads = self._z_reads(par)
            for m in range(self.M):
                cz = torch.nn.functional.pad((h @ p[m]).T, (0, 0, 0, 1)).reshape(-1)
                out[m, par::2] = self.g[m] * sum(w * cz[k] for k, w in reads) @ d.T
        return out.view(self.M, self.Nz, self.nb, 2)

    def adjoint_z(self, y):
        y, d = y.reshape(self.M, self.Nz, -1), self.dft()
        h = 3 * _d1(self._offsets(self.Nz) / self.a)
        cz = torch.zeros(self.M, (self.N + 1) * self._fine(self.Nz), device="cuda", dtype=torch.float64)
        for par in range(min(2, self.Nz)):
            reads = self._z_reads(par)
            for m in range(self.M):
                s = self.g[m] * (y[m, par::2] @ d)
                for k, w in reads:
                    cz[m].index_add_(0, k.reshape(-1), (w * s).reshape(-1))
        p = torch.stack([(c.view(self.N + 1, -1)[: self.N] @ h).T for c in cz])
        return self.backproject(p)

    # -- Eq. (26)
    def scans(self, which):
        """(apply, transpose) of the selected scans' operator."""
        def fwd(x):
            return torch.cat(([self.forward(x)] if "x" in which else []) + ([self.forward_z(x)] if "z" in which else []))

        def adj(r):
            x = torch.zeros(self.Nz, self.N, self.N, device="cuda", dtype=torch.float64)
            if "x" in which:
                x, r = x + self.adjoint(r[: self.M]), r[self.M:]
            return x + self.adjoint_z(r) if "z" in which else x
        return fwd, adj

    def solve(self, b, iters, n_power, which="x"):
        fwd, adj = self.scans(which)
        shape = (self.Nz, self.N, self.N)
        v = _splitmix(1234, math.prod(shape)).view(shape)
        v = v / v.norm()
        for _ in range(n_power):
            w = adj(fwd(v))
            ata = float((v * w).sum())
            v = w / w.norm()
        tn = sum(4 * math.sin(math.pi * (n - 1) / (2 * n)) ** 2 for n in shape)
        lam = 1e-3 * ata / tn
        tau = 1 / (ata + lam * tn)
        x = torch.zeros(shape, device="cuda", dtype=torch.float64)
        xp, hist = x, []
        for k in range(1, iters + 1):
            y = x + (k - 1) / (k + 2) * (x - xp)
            r = fwd(y) - b
            hist.append(float(r.norm()))
            g = adj(r)
            for ax in range(3):
                d = torch.diff(y, dim=ax)
                pad = [0] * 6
                pad[2 * (2 - ax)] = 1
                lo = torch.nn.functional.pad(d, pad)
                pad[2 * (2 - ax)], pad[2 * (2 - ax) + 1] = 0, 1
                g = g + lam * (lo - torch.nn.functional.pad(d, pad))
            xp, x = x, (y - tau * g).clamp(min=0)
        return x, torch.tensor([hist[0], hist[-1], ata], dtype=torch.float64)


def _splitmix(seed, n):
    """SplitMix64 (Steele, Lea, Flood 2014) at counters 1..n as uniforms in [-1, 1)."""
    import numpy as np

    with np.errstate(over="ignore"):
        z = np.uint64(seed) + np.arange(1, n + 1, dtype=np.uint64) * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        z = z ^ (z >> np.uint64(31))
    return torch.from_numpy((z >> np.uint64(11)).astype(np.float64) * 2.0**-52 - 1.0).cuda()


def exact(case, seed):
    kind = case["kind"]
    if kind == "serve":
        out = []
        for k, g in enumerate(serve_requests()):
            x, noise = _inputs(g, seed + 100 * k)
            out.append(_Model(g).solve(_scan_data(g, x, noise).double(), case["iters"], case["n_power"])[0])
        return out
    if kind == "fit":
        x, sets = _fit_inputs(case, seed)
        out = []
        for g, w, y in sets:
            m = _Model(dict(case, fwhm=float(w.item())), g.double())
            y, p = y.double(), m.project(x.double())
            gg = (y * m.lines_forward(p, torch.ones_like(m.g))).sum((1, 2, 3))
            gw = (y * m.lines_forward(p, width_gradient=True)).sum().view(1)
            out += [m.lines_forward(p), m.adjoint(y), gg, gw]
        return out
    x, y = _inputs(case, seed)
    m = _Model(case)
    if kind == "solve":
        b = _scan_data(case, x, y).double()
        samples = case["S"] * case["P"] * case["nz"] * case["n_angles"] * (case["iters"] + case["n_power"])
        if "z" in case["scans"] and samples > 1e9:
            return None  # the sample-by-sample z-drive products would take minutes
        return list(m.solve(b, case["iters"], case["n_power"], case["scans"]))
    if kind == "tensor":
        return [m.forward_tensor(x.double()), m.adjoint_tensor(y.double())]
    if kind == "zdrive":
        return [m.forward_z(x.double()), m.adjoint_z(y.double())]
    return [m.forward(x.double()), m.adjoint(y.double())]
