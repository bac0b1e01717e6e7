"""The work that users of this library have it do, as measurable cases.

A case is a dict of plain values.  Kinds:
  step      tc_step of one case: the time marching itself, in its three
            arithmetic forms, from the smallest grids to the largest
  batch     tc_batch_step of an ensemble of independent small cases
  restart   a new velocity field into a handle (device buffers), then the
            diagnostics of it: the start of a run and of each loaded snapshot
  physical  spectral -> physical output of one field without allocation

Sizes are those of the library's workloads, tests and benchmark: the smallest
grid of the smoke run, Taylor-vortex grids, 129x128x128, the paper's
129x512x170 (an axial length with prime factors 5 and 17) and the benchmark's
257x512x512; the ensemble is drawn as the benchmark draws its own.
`exact` restates the method in float64 torch, without the library.
"""
import math

import numpy as np
import torch

import paper_0711_1429_gb300 as tc

PREC = {"fp64": tc.TC_PREC_FP64, "mixed": tc.TC_PREC_MIXED, "df64": tc.TC_PREC_DF64}


def _step(name, Nr, Nt, Nz, prec, steps, **kw):
    c = dict(name=name, kind="step", Nr=Nr, Nt=Nt, Nz=Nz, prec=prec, steps=steps, zeta=0.883, Re=3000.0,
             Re_o=0.0, dt=1e-3, Theta=0.0, Lz=0.0, stretch=0.0, amp=0.05, spectrum="k2", autotune=1)
    c.update(kw)
    return c


def listed():
    return [
        # one step of the smallest grid: launches and latency only
        _step("step-33x16x16-fp64", 33, 16, 16, "fp64", 1, Re=200.0, amp=1e-3, spectrum="box", autotune=0),
        # Taylor- and wavy-vortex marching between two samples
        _step("step-64x32x64-fp64", 64, 32, 64, "fp64", 10, zeta=0.5, Re=250.0, dt=1e-2, Theta=math.pi, Lz=4.0,
              amp=1e-2, spectrum="box", autotune=0),
        # the ordinary turbulent grid, in the default and the mixed form
        _step("step-129x128x128-fp64", 129, 128, 128, "fp64", 3),
        _step("step-129x128x128-mixed", 129, 128, 128, "mixed", 5),
        # the paper's production grid, in the default and the double-float form
        _step("step-129x512x170-fp64", 129, 512, 170, "fp64", 3, zeta=0.882, Re=10500.0, dt=0.012, amp=1e-4),
        _step("step-129x512x170-df64", 129, 512, 170, "df64", 5, zeta=0.882, Re=10500.0, dt=0.012, amp=1e-4),
        # the largest grid of the benchmark
        _step("step-257x512x512-fp64", 257, 512, 512, "fp64", 3),
        _step("step-257x512x512-mixed", 257, 512, 512, "mixed", 5),
        # a parameter study: many small cases advanced together
        dict(name="batch-16-fp64", kind="batch", ncases=16, pick=1000, prec="fp64", steps=1),
        # loading a snapshot and reading its diagnostics
        dict(_step("restart-129x128x128-fp64", 129, 128, 128, "fp64", 0, autotune=0), kind="restart"),
        # a field for output or visualisation
        dict(name="physical-257x512x512", kind="physical", Nr=257, Nt=512, Nz=512),
    ]


_NT = [8, 12, 16, 24, 32, 36, 48, 64, 72, 96, 108, 128, 144, 192, 216, 256, 288, 324, 384, 432, 512]
_NZ = [8, 10, 12, 14, 16, 18, 20, 22, 24, 26, 28, 32, 34, 36, 40, 48, 50, 54, 60, 64, 66, 72, 78, 80, 90, 96, 102,
       108, 120, 128, 130, 140, 144, 150, 160, 162, 168, 170, 180, 192, 200, 216, 240, 256, 288, 300, 320, 360, 384,
       400, 432, 448, 480, 512]


def draw(rng):
    def logint(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    kind = rng.choice(["step", "step", "step", "step", "batch", "restart", "physical"])
    if kind == "batch":
        return dict(kind="batch", ncases=rng.randint(4, 16), pick=rng.randrange(1 << 20),
                    prec=rng.choice(["fp64", "fp64", "mixed", "df64"]), steps=rng.randint(1, 2))
    while True:
        Nr, Nt, Nz = logint(17, 257), rng.choice(_NT), rng.choice(_NZ)
        if Nr * Nt * Nz <= 257 * 512 * 512 // 2:
            break
    if kind == "physical":
        return dict(kind="physical", Nr=Nr, Nt=Nt, Nz=Nz)
    c = _step("", Nr, Nt, Nz, rng.choice(["fp64", "fp64", "mixed", "df64"]), rng.randint(1, 5),
              zeta=rng.choice([0.5, 0.75, 0.883, 0.95]), Re=round(rng.uniform(200.0, 3000.0), 1),
              Re_o=round(rng.choice([0.0, 0.0, -100.0, 150.0]), 1), stretch=rng.choice([0.0, 0.0, 1.5]),
              amp=10.0 ** rng.uniform(-4.0, -1.4), spectrum=rng.choice(["k2", "k2", "box"]),
              autotune=rng.choice([0, 1]))
    c["amp"] = float("%.3g" % c["amp"])
    del c["name"]
    if kind == "restart":
        c.update(kind="restart", steps=0, autotune=0)
    return c


# ---- inputs ---------------------------------------------------------------------
def _box(c):
    Ri = 2.0 * c["zeta"] / (1.0 - c["zeta"])
    rc = Ri + 1.0
    Theta = c["Theta"] if c["Theta"] > 0 else 10.0 * math.pi / rc
    Lz = c["Lz"] if c["Lz"] > 0 else 5.0
    return 2.0 * math.pi / Theta, 2.0 * math.pi / Lz, rc


def _fields(c, seed):
    """Random-phase disturbances that satisfy the wall conditions: complex128
    v and eta, [Nr][Nz][Ntheta/2], on the GPU."""
    Nr, Nz, Nh = c["Nr"], c["Nz"], c["Nt"] // 2
    m0, a0, rc = _box(c)
    dev = torch.device("cuda")
    g = torch.Generator(device=dev)
    g.manual_seed(seed)
    xi = torch.view_as_complex(torch.randn(2, 2, Nz, Nh, 2, dtype=torch.float64, device=dev, generator=g))
    n = torch.fft.fftfreq(Nz, d=1.0 / Nz, device=dev, dtype=torch.float64).reshape(Nz, 1)
    j = torch.arange(Nh, device=dev, dtype=torch.float64).reshape(1, Nh)
    if c["spectrum"] == "box":
        a = ((j <= 4) & (n.abs() <= 4)).double() * c["amp"]
        b = a
    else:
        kh = torch.sqrt((j * m0 / rc) ** 2 + (n * a0) ** 2)
        kh[0, 0] = 1.0
        a = kh ** -1.5
        b = a * kh
    keep = torch.ones(Nz, Nh, dtype=torch.float64, device=dev)
    keep[Nz // 2] = 0.0
    keep[Nz // 2:, 0] = 0.0
    keep[0, 0] = 0.0
    x = torch.linspace(-1.0, 1.0, Nr, dtype=torch.float64, device=dev).reshape(Nr, 1, 1)
    bump = 1.0 - x * x
    v = a * keep * (xi[0, 0] * bump ** 2 + xi[0, 1] * (x * bump ** 2))
    e = b * keep * (xi[1, 0] * bump + xi[1, 1] * (x * bump))
    for F in (v, e):
        F[:, Nz // 2 + 1:, 0] = torch.conj(F[:, 1:Nz // 2, 0]).flip(1)
    if c["spectrum"] == "k2":
        w = torch.full((Nh,), 2.0, dtype=torch.float64, device=dev)
        w[0] = 1.0
        s = c["amp"] / math.sqrt(float(((v.abs() ** 2) * w).sum()) / Nr)
        v *= s
        e *= s
    return v, e


def _params(c):
    return tc.make_params(c["Nr"], c["Nt"], c["Nz"], c["zeta"], c["Re"], c["Re_o"], c["dt"], Theta=c["Theta"],
                          Lz=c["Lz"], precision=PREC[c["prec"]], autotune=c["autotune"], stretch=c["stretch"])


def _ensemble(c):
    """The cases of a batch: Nr 33..129, 32, 64 or 128 modes each way."""
    rng = np.random.default_rng(c["pick"])
    out = []
    for _ in range(c["ncases"]):
        Nr = int(rng.integers(33, 130))
        Nt, Nz = (int(x) for x in rng.choice([32, 64, 128], size=2))
        out.append(_step("", Nr, Nt, Nz, c["prec"], c["steps"], zeta=float(rng.uniform(0.7, 0.95)),
                         Re=float(rng.uniform(500.0, 3000.0))))
    return out


class _Owner:
    """Frees a handle or a batch when the last tensor that shows its memory is gone."""

    def __init__(self, handle, destroy):
        self.handle, self.destroy = handle, destroy

    def __del__(self):
        torch.cuda.synchronize()
        self.destroy(self.handle)


class _Array:
    """A resident array of a handle, as torch sees one (no copy); the tensor
    made of it keeps it, and with it the handle."""

    def __init__(self, owner, ptr, shape):
        self.owner = owner
        self.__cuda_array_interface__ = {"shape": shape, "typestr": "<c16", "data": (ptr, False), "version": 3}


def _views(owner, h, c, which):
    shape = (c["Nr"], c["Nz"], c["Nt"] // 2)
    return [torch.as_tensor(_Array(owner, tc.tc_device_array(h, w), shape), device="cuda") for w in which]


def _load(h, v, e):
    tc.tc_set_field_async(h, tc.TC_FIELD_V, v.data_ptr(), v.numel() * 16)
    tc.tc_set_field_async(h, tc.TC_FIELD_ETA, e.data_ptr(), e.numel() * 16)


_VEUW = (tc.TC_ARRAY_V, tc.TC_ARRAY_ETA, tc.TC_ARRAY_U, tc.TC_ARRAY_W)


class _State:
    """What a user's program holds: the handle and its inputs."""

    def __init__(self, c, seed):
        self.c, self.h, self.b = c, None, None
        kind = c["kind"]
        if kind == "batch":
            cases = _ensemble(c)
            self.b = tc.tc_batch_create([_params(k) for k in cases])
            self.owner = _Owner(self.b, tc.tc_batch_destroy)
            self.out = []
            for i, k in enumerate(cases):
                h = tc.tc_batch_case(self.b, i)
                _load(h, *_fields(k, seed + 7919 * i))
                self.out += _views(self.owner, h, k, _VEUW[:2])
        elif kind == "physical":
            g = torch.Generator(device="cuda")
            g.manual_seed(seed)
            Nr, Nz, Nh = c["Nr"], c["Nz"], c["Nt"] // 2
            k = torch.sqrt(torch.fft.fftfreq(Nz, d=1.0 / Nz, device="cuda").double().reshape(Nz, 1) ** 2
                           + torch.arange(Nh, device="cuda").double() ** 2)
            self.spec = torch.view_as_complex(
                torch.randn(Nr, Nz, Nh, 2, dtype=torch.float64, device="cuda", generator=g)) * (1.0 + k) ** -1.5
            self.spec[:, Nz // 2] = 0.0
            self.spec[:, Nz // 2 + 1:, 0] = torch.conj(self.spec[:, 1:Nz // 2, 0]).flip(1)
            self.spec[:, 0, 0] = self.spec[:, 0, 0].real.to(torch.complex128)
            self.phys = torch.empty(Nr, 3 * Nz // 2, 3 * (2 * Nh) // 2, dtype=torch.float64, device="cuda")
        else:
            p = _params(c)
            self.h = tc.tc_create_ex(c["Nr"], c["Nt"], c["Nz"], c["zeta"], c["Re"], c["Re_o"], c["dt"],
                                     Theta=p.Theta, Lz=p.Lz, precision=p.precision, autotune=p.autotune,
                                     stretch=p.stretch)
            self.owner = _Owner(self.h, tc.tc_destroy)
            self.v, self.e = _fields(c, seed)
            self.out = _views(self.owner, self.h, c, _VEUW)
            if kind == "step":
                _load(self.h, self.v, self.e)
                torch.cuda.synchronize()
                self.v = self.e = None


def prepare(case, seed):
    return _State(case, seed)


def run(s):
    c = s.c
    if c["kind"] == "step":
        tc.tc_step(s.h, c["steps"])
        return dict(zip(("v", "eta", "u", "w"), s.out))
    if c["kind"] == "batch":
        tc.tc_batch_step(s.b, c["steps"])
        return s.out
    if c["kind"] == "restart":
        _load(s.h, s.v, s.e)
        d = tc.tc_torque_stats(s.h)
        d.update(u=s.out[2], w=s.out[3])
        return d
    tc.tc_to_physical_noalloc(c["Nr"], c["Nt"], c["Nz"], s.spec.data_ptr(), s.phys.data_ptr(),
                              torch.cuda.current_stream().cuda_stream)
    return s.phys


# ---- the work of one pass -----------------------------------------------------------
def _transform_flops(Nr, Nt, Nz, back, fwd):
    Mt, Mz, Nh = 3 * Nt // 2, 3 * Nz // 2, Nt // 2
    return Nr * (back + fwd) * (Nh * 5.0 * Mz * math.log2(Mz) + Mz * 2.5 * Mt * math.log2(Mt))


def _step_work(c):
    P = c["Nr"] * c["Nz"] * (c["Nt"] // 2)
    sub = _transform_flops(c["Nr"], c["Nt"], c["Nz"], 3, 5) + 9.0 * c["Nr"] * 2.25 * c["Nt"] * c["Nz"] + 600.0 * P
    return {"bytes": 6 * 16 * P, "flops": 3 * c["steps"] * sub}     # v, eta in; v, eta, u, w out


def work(case):
    if case["kind"] == "batch":
        w = [_step_work(k) for k in _ensemble(case)]
        return {"bytes": sum(x["bytes"] for x in w), "flops": sum(x["flops"] for x in w)}
    if case["kind"] == "step":
        return _step_work(case)
    P = case["Nr"] * case["Nz"] * (case["Nt"] // 2)
    if case["kind"] == "restart":
        return {"bytes": 4 * 16 * P, "flops": 200.0 * P}
    return {"bytes": 16 * P + 8 * case["Nr"] * 2.25 * case["Nt"] * case["Nz"],
            "flops": _transform_flops(case["Nr"], case["Nt"], case["Nz"], 1, 0)}


# ---- the method in float64 torch ------------------------------------------------------
# v-eta equations per Fourier pair with five-point compact rows in r, products
# with the 3/2 rule, three-substep Runge-Kutta with Crank-Nicolson; lengths in
# the half gap, velocities in the inner wall's, nu = 2/Re.
_GAMMA, _ZETA, _BETA = (8 / 15, 5 / 12, 3 / 4), (0.0, -17 / 60, -5 / 12), (4 / 15, 1 / 15, 1 / 6)


def _gauss(A, b):
    """Batched elimination with row exchanges, in long double: A (n,k,k), b (n,k)."""
    A, b = A.copy(), b.copy()
    n, k = b.shape
    at = np.arange(n)
    for c in range(k):
        p = c + np.argmax(np.abs(A[:, c:, c]), axis=1)
        rows, piv = A[at, c].copy(), A[at, p].copy()
        A[at, c], A[at, p] = piv, rows
        x, y = b[at, c].copy(), b[at, p].copy()
        b[at, c], b[at, p] = y, x
        for i in range(c + 1, k):
            f = A[:, i, c] / A[:, c, c]
            A[:, i] -= f[:, None] * A[:, c]
            b[:, i] -= f * b[:, c]
    out = np.zeros_like(b)
    for i in range(k - 1, -1, -1):
        out[:, i] = (b[:, i] - np.sum(A[:, i, i + 1:] * out[:, i + 1:], axis=1)) / A[:, i, i]
    return out


def _chain(which, q, x, h):
    """h^n times D, D D_*, D D_* D D_* (n = 1, 2, 4) of ((r - rc)/h)^q at
    r - rc = x[0], r = x[1]."""
    t, y = x[0] / h, h / x[1]

    def der(k):
        return np.zeros_like(t) if k > q else np.longdouble(math.perm(q, k)) * t ** (q - k)

    if which == 0:
        return der(0)
    if which == 1:
        return der(1)
    if which == 2:
        return der(2) + y * der(1) - y * y * der(0)
    return der(4) + 2 * y * der(3) - 3 * y ** 2 * der(2) + 3 * y ** 3 * der(1) - 3 * y ** 4 * der(0)


class _Rows:
    """Radial grid and the five-point rows of I, D, D D_*, D D_* D D_*."""

    def __init__(self, c):
        N = self.N = c["Nr"]
        Ri = 2.0 * c["zeta"] / (1.0 - c["zeta"])
        s = -1.0 + 2.0 * np.arange(N) / (N - 1)
        if c["stretch"] == 0.0:
            self.r, self.jac = Ri + 2.0 * np.arange(N) / (N - 1), np.ones(N)
        else:
            t = np.array([math.tanh(c["stretch"] * x) for x in s])
            self.r = (Ri + 1.0) + t / math.tanh(c["stretch"])
            self.jac = c["stretch"] * (1.0 - t * t) / math.tanh(c["stretch"])
        R = self.r.astype(np.longdouble)
        start = np.clip(np.arange(N) - 2, 0, N - 5)
        pts = R[start[:, None] + np.arange(5)]
        h = ((pts[:, 4] - pts[:, 0]) / 4)[:, None]
        w = np.zeros((4, N, 5), dtype=np.longdouble)             # I, D, DD_*, DD_*DD_*
        ev = {(k, q): _chain(k, q, (pts - R[:, None], pts), h) for k in range(4) for q in range(9)}
        A, b = np.zeros((N, 10, 10), dtype=np.longdouble), np.zeros((N, 10), dtype=np.longdouble)
        for q in range(9):
            A[:, q, :5], A[:, q, 5:] = -ev[3, q], ev[0, q]
        A[:, 9, :5] = 1.0
        b[:, 9] = 1.0
        i = slice(2, N - 2)
        x = _gauss(A[i], b[i])
        w[0, i], w[3, i] = x[:, :5], x[:, 5:] / h[i] ** 4
        V = np.stack([ev[0, q] for q in range(5)], axis=1)
        for k in (1, 2):
            rhs = np.stack([np.sum(w[0] * ev[k, q], axis=1) for q in range(5)], axis=1)
            w[k, i] = _gauss(V[i], rhs[i]) / h[i] ** k
            own = np.stack([_chain(k, q, (0 * R[:, None], R[:, None]), h)[:, 0] for q in range(5)], axis=1)
            one = [1, N - 2] + ([0, N - 1] if k == 1 else [])     # one-sided rows; D at the walls
            w[k, one] = _gauss(V[one], own[one]) / h[one] ** k
        w[0, 1, 1] = w[0, N - 2, 3] = 1.0
        w = w.astype(np.float64)
        self.wall = w[1, 0].copy(), w[1, N - 1].copy()
        w[1, 0] = w[1, N - 1] = 0.0
        self.l = [torch.from_numpy(a).cuda() for a in w]
        self.rt = torch.from_numpy(self.r).cuda().reshape(N, 1)

    def apply(self, k, g):
        N, w = self.N, self.l[k]
        out = torch.zeros_like(g)
        for s in range(5):
            out[2:N - 2] += w[2:N - 2, s, None] * g[s:N - 4 + s]
            out[1] += w[1, s] * g[s]
            out[N - 2] += w[N - 2, s] * g[N - 5 + s]
        return out

    def band(self, terms, P):
        """Sum of rows on (coefficient x unknown), as seven diagonals (N, 7, P)
        about the main one; the one-sided rows 1 and N-2 reach three off it."""
        N = self.N
        out = torch.zeros(N, 7, P, dtype=torch.float64, device="cuda")
        for k, f in terms:
            f, w = f.expand(N, P), self.l[k]
            for s in range(5):
                out[2:N - 2, 1 + s] += w[2:N - 2, s, None] * f[s:N - 4 + s]
                out[1, 2 + s] += w[1, s] * f[s]
                out[N - 2, s] += w[N - 2, s] * f[N - 5 + s]
        return out

    def dense(self, k):
        """Rows of one operator as a matrix (rows 0, N-1 empty)."""
        D = torch.zeros(self.N, self.N, dtype=torch.float64, device="cuda")
        for j in range(1, self.N - 1):
            st = min(max(j - 2, 0), self.N - 5)
            D[j, st:st + 5] = self.l[k][j]
        return D


def _band_mul(B, x):
    N = x.shape[0]
    out = torch.zeros_like(x)
    for d in range(-3, 4):
        a, b = max(0, -d), min(N, N - d)
        out[a:b] += B[a:b, 3 + d] * x[a + d:b + d]
    return out


def _band_solve(B, rhs):
    """Seven-diagonal systems, one per column, by elimination in row order."""
    B, y = B.clone(), rhs.clone()
    N = y.shape[0]
    for j in range(N - 1):
        for i in range(1, min(4, N - j)):
            f = B[j + i, 3 - i] / B[j, 3]
            B[j + i, 4 - i:7 - i] -= f * B[j, 4:7]
            y[j + i] -= f * y[j]
    for j in range(N - 1, -1, -1):
        for i in range(1, min(4, N - j)):
            y[j] -= B[j, 3 + i] * y[j + i]
        y[j] /= B[j, 3]
    return y


class _Method:
    def __init__(self, c, seed):
        self.c, self.R = c, _Rows(c)
        N, Nz, Nh = c["Nr"], c["Nz"], c["Nt"] // 2
        m0, a0, _ = _box(c)
        n = torch.fft.fftfreq(Nz, d=1.0 / Nz, dtype=torch.float64, device="cuda")
        keep = torch.ones(Nz, Nh, dtype=torch.bool, device="cuda")
        keep[Nz // 2] = False
        keep[Nz // 2:, 0] = False
        keep[0, 0] = False
        self.at = torch.nonzero(keep.reshape(-1)).reshape(-1)
        self.m = (torch.arange(Nh, device="cuda").double() * m0).expand(Nz, Nh).reshape(-1)[self.at]
        self.al = (n * a0).reshape(Nz, 1).expand(Nz, Nh).reshape(-1)[self.at]
        v, e = _fields(c, seed)
        self.v, self.e = v.reshape(N, -1)[:, self.at], e.reshape(N, -1)[:, self.at]
        Wo, r = c["Re_o"] / c["Re"], self.R.r
        a = (Wo * r[-1] - r[0]) / (r[-1] ** 2 - r[0] ** 2)
        self.W = torch.from_numpy(a * r + (r[0] - a * r[0] ** 2) / r).cuda()
        self.U = torch.zeros_like(self.W)
        D0 = self.R.dense(0)
        D0[0, 0] = D0[N - 1, N - 1] = 1.0
        self.D0 = torch.linalg.lu_factor(D0)

    def full(self, x, mean=None):
        c = self.c
        N, Nz, Nh = c["Nr"], c["Nz"], c["Nt"] // 2
        F = torch.zeros(N, Nz * Nh, dtype=torch.complex128, device="cuda")
        F[:, self.at] = x
        F = F.reshape(N, Nz, Nh)
        F[:, Nz // 2 + 1:, 0] = torch.conj(F[:, 1:Nz // 2, 0]).flip(1)
        if mean is not None:
            F[:, 0, 0] = mean.to(torch.complex128)
        return F

    def compact_D(self, f, walls=None):
        rhs = self.R.apply(1, f)
        if walls is not None:
            rhs[0], rhs[-1] = walls
        x = torch.linalg.lu_solve(*self.D0, torch.view_as_real(rhs.contiguous()).reshape(f.shape[0], -1))
        return torch.view_as_complex(x.reshape(f.shape + (2,)).contiguous())

    def velocity(self):
        r, m, al = self.R.rt, self.m, self.al
        c = 1.0 / (al ** 2 + m ** 2 / r ** 2)
        Ds = self.compact_D(self.v) + self.v / r
        return c * (1j * al * Ds - 1j * m / r * self.e), c * (1j * m / r * Ds + 1j * al * self.e)

    def products(self, u, w):
        c = self.c
        Nz, Nh, Mt, Mz = c["Nz"], c["Nt"] // 2, 3 * c["Nt"] // 2, 3 * c["Nz"] // 2
        h = Nz // 2
        phys = [_physical(F) for F in (self.full(u, self.U), self.full(self.v), self.full(w, self.W))]
        out = {}
        for a, b in ("uu", "uv", "uw", "vv", "vw", "ww"):
            S = torch.fft.rfft2(phys["uvw".index(a)] * phys["uvw".index(b)], dim=(1, 2))[:, :, :Nh] / (Mt * Mz)
            F = torch.zeros(c["Nr"], Nz, Nh, dtype=torch.complex128, device="cuda")
            F[:, :h], F[:, h + 1:] = S[:, :h], S[:, Mz - h + 1:]
            out[a + b] = F
        return out

    def step(self):
        c, R, N = self.c, self.R, self.c["Nr"]
        r, m, al, nu, dt, P = R.rt, self.m, self.al, 2.0 / c["Re"], c["dt"], self.at.numel()
        g = al ** 2 * r ** 2 + m ** 2
        c0, c1 = r ** 2 / g, 2 * r * m ** 2 / g ** 2
        c2 = 2 * m ** 2 * (m ** 2 - 3 * al ** 2 * r ** 2) / g ** 3
        c3 = -24 * m ** 2 * al ** 2 * r * (m ** 2 - al ** 2 * r ** 2) / g ** 4
        k2 = al ** 2 + m ** 2 / r ** 2
        one = torch.ones_like(r)
        Mv = R.band([(0, one), (2, -c0), (1, c1)], P)
        Lv = nu * R.band([(2, 2 * one), (3, -c0), (2, -2 * c1 / r), (0, -k2),
                          (1, c2 / r + c3 - c1 / r ** 2 - 2 * m ** 2 * c0 / r ** 3)], P)
        Me, Le = R.band([(0, one)], P), nu * R.band([(2, one), (0, -k2)], P)
        M0, L2 = R.dense(0), nu * R.dense(2)
        LU = L2 + nu * R.dense(0) / r.reshape(1, N) ** 2
        Eo = None
        for k in range(3):
            u, w = self.velocity()
            p = self.products(u, w)
            uv0, vw0 = p["uv"][:, 0, 0].real, p["vw"][:, 0, 0].real
            p = {q: F.reshape(N, -1)[:, self.at] for q, F in p.items()}
            A = R.apply
            Ev = (nu * (-3 * A(2, c1 * (1j * al * u + 1j * m / r * w))
                        + 2j * m * (A(2, c0 / r ** 2 * w) - A(1, c1 / r ** 2 * w) - A(0, w / r ** 2)))
                  - 1j * al * (A(2, c0 * p["uv"]) - A(1, c1 * p["uv"]) + A(0, p["uv"]))
                  - 1j * m * (A(2, c0 * p["vw"] / r) + A(1, (2 * c0 / r ** 2 - c1 / r) * p["vw"]) + A(0, p["vw"] / r))
                  + A(1, c0 * (al ** 2 * p["uu"] + 2 * al * m / r * p["uw"] + m ** 2 / r ** 2 * p["ww"]) - p["vv"])
                  + A(0, (p["ww"] - p["vv"]) / r))
            Ee = (nu * 2j * m * (A(1, u / r ** 2) + 2 * A(0, u / r ** 3) - 1j * al * A(0, self.v / r ** 2))
                  - 1j * m * (A(1, p["uv"] / r) + A(0, 1j * al * p["uu"] / r + 2 * p["uv"] / r ** 2
                                                     + 1j * m * p["uw"] / r ** 2))
                  + 1j * al * (A(1, p["vw"]) + A(0, 1j * al * p["uw"] + 1j * m * p["ww"] / r + 2 * p["vw"] / r)))
            r1 = r.reshape(N)
            EU = -A(1, uv0[:, None])[:, 0] - A(0, (uv0 / r1)[:, None])[:, 0]
            EW = -A(1, vw0[:, None])[:, 0] - 2 * A(0, (vw0 / r1)[:, None])[:, 0]
            E = (Ev, Ee, EU, EW)
            Eo = Eo or E
            x = [dt * (_GAMMA[k] * a + _ZETA[k] * b) for a, b in zip(E, Eo)]
            b = _BETA[k] * dt
            rv = _band_mul(Mv, self.v) + b * _band_mul(Lv, self.v) + x[0]
            re = _band_mul(Me, self.e) + b * _band_mul(Le, self.e) + x[1]
            rU = M0 @ self.U + b * (LU @ self.U) + x[2]
            rW = M0 @ self.W + b * (L2 @ self.W) + x[3]
            for a in (rv, re, rU):
                a[0] = a[N - 1] = 0.0
            rv[1] = rv[N - 2] = 0.0
            rW[0], rW[N - 1] = 1.0, c["Re_o"] / c["Re"]
            Sv, Se = Mv - b * Lv, Me - b * Le
            Sv[1] = Sv[N - 2] = 0.0
            for s in range(5):                                   # Dv = 0 at the walls
                Sv[1, 2 + s], Sv[N - 2, s] = R.wall[0][s], R.wall[1][s]
            for S in (Sv, Se):
                S[0, 3] = S[N - 1, 3] = 1.0
            SU, SW = M0 - b * LU, M0 - b * L2
            for S in (SU, SW):
                S[0, 0] = S[N - 1, N - 1] = 1.0
            self.v, self.e = _band_solve(Sv, rv), _band_solve(Se, re)
            self.U, self.W = torch.linalg.solve(SU, rU), torch.linalg.solve(SW, rW)
            Eo = E

    def stats(self):
        c, R, N = self.c, self.R, self.c["Nr"]
        nu, r, W = 2.0 / c["Re"], R.r, self.W.cpu().numpy()
        si, so = R.wall[0] @ W[:5] - W[0] / r[0], R.wall[1] @ W[-5:] - W[-1] / r[-1]
        u, w = self.velocity()
        u, v, w = self.full(u, self.U), self.full(self.v), self.full(w, self.W)
        m0, a0, _ = _box(c)
        Nz, Nh = c["Nz"], c["Nt"] // 2
        n = torch.fft.fftfreq(Nz, d=1.0 / Nz, dtype=torch.float64, device="cuda")
        m, al = (torch.arange(Nh, device="cuda").double() * m0).reshape(1, 1, Nh), (n * a0).reshape(1, Nz, 1)
        rr = R.rt.reshape(N, 1, 1)
        walls = [torch.from_numpy(x).cuda().to(torch.complex128) for x in R.wall]

        def D(F):
            f = F.reshape(N, -1)
            return self.compact_D(f, (walls[0] @ f[:5], walls[1] @ f[N - 5:])).reshape(F.shape)

        wt = torch.full((Nh,), 2.0, dtype=torch.float64, device="cuda")
        wt[0] = 1.0

        def prof(F):
            return (F.abs() ** 2 * wt).sum(dim=(1, 2)).cpu().numpy()

        S2 = (2 * (prof(D(v)) + prof(1j * m / rr * w + v / rr) + prof(1j * al * u))
              + prof(D(w) - w / rr + 1j * m / rr * v) + prof(1j * al * v + D(u)) + prof(1j * m / rr * u + 1j * al * w))
        q = np.ones(N)
        for k, x in enumerate((3 / 8, 7 / 6, 23 / 24)):
            q[k] = q[N - 1 - k] = x
        q = q * R.jac * r
        return {"t": 0.0, "step": None, "G_inner": 2 * math.pi * r[0] * abs(si),
                "G_outer": 2 * math.pi * r[-1] ** 2 / r[0] * abs(so),
                "Re_tau_inner": math.sqrt(abs(si) / nu), "Re_tau_outer": math.sqrt(abs(so) / nu),
                "energy": 0.5 * float(q @ (prof(u) + prof(v) + prof(w)) / q.sum()),
                "dissipation": nu * float(q @ S2 / q.sum()),
                "power_in": nu * float(r[-1] * W[-1] * so - r[0] * W[0] * si) / (0.5 * (r[-1] ** 2 - r[0] ** 2)),
                "u": u, "w": w}


def _physical(F):
    """Half spectrum [Nr][Nz][Nh] -> values on the 3/2 grid [Nr][Mz][Mt]."""
    Nr, Nz, Nh = F.shape
    Mz, Mt, h = 3 * Nz // 2, 3 * Nh, Nz // 2
    pad = torch.zeros(Nr, Mz, Mt // 2 + 1, dtype=torch.complex128, device="cuda")
    pad[:, :h, :Nh], pad[:, Mz - h + 1:, :Nh] = F[:, :h], F[:, h + 1:]
    return torch.fft.irfft2(pad, s=(Mz, Mt), dim=(1, 2)) * (Mz * Mt)


def exact(case, seed):
    if case["kind"] == "physical":
        return _physical(_State(case, seed).spec)
    if case["kind"] == "restart":
        return _Method(case, seed).stats()
    out = []
    cases = _ensemble(case) if case["kind"] == "batch" else [case]
    for i, c in enumerate(cases):
        s = _Method(c, seed + 7919 * i)
        for _ in range(c["steps"]):
            s.step()
        if case["kind"] == "batch":
            out += [s.full(s.v), s.full(s.e)]
        else:
            u, w = s.velocity()
            out = {"v": s.full(s.v), "eta": s.full(s.e), "u": s.full(u, s.U), "w": s.full(w, s.W)}
    return out
