"""The time steps this library is used for, as measurable cases.

A pass is one CFL-limited step of a simulation, as ``run.advance`` and a user's own loop take it: ``max_dt`` on the
device, then ``step_devdt`` in place on the device state (or, for many small problems, one ``ader_batch_advance``).
Solvers with FP64 arithmetic give the FP64 state, the face field and dt.  FP32-bulk solvers keep an FP64 state of FP32
accuracy; their programs take the frame they write out from it in FP32, and that frame is their output.

``exact`` is the same step in plain torch FP64: the paper's scheme (arXiv:1006.2146) in matrix form.  Node values are
the basis evaluated at the nodes, every flux-mode rule is a matrix, the predictor matches du/dtau = -div F mode by
mode, and the face and edge averages are weights of the facial polynomial's modes.
"""
import functools
import math

import numpy as np
import torch

import paper_1006_2146_gb300 as ader
from paper_1006_2146_gb300 import _lib, inputs

CFL = 0.4
FOUR_PI = 4.0 * math.pi


def _case(name, ic, shape, order, form="modal", solver="hll", fp32=False):
    nz, ny, nx = shape
    return {"name": name, "ic": ic, "nz": nz, "ny": ny, "nx": nx, "order": order, "form": form, "solver": solver,
            "fp32": fp32}


def listed():
    return [
        # an interactive or test-sized run with the default solver: launches and one wave of blocks decide
        _case("euler_fp64_o3_small", "smooth", (16, 16, 16), 3),
        # the benchmark's planar shock tube at production size, FP64
        _case("euler_fp64_o3_sod", "sod", (256, 256, 256), 3, "nodal"),
        # second order with the linearized solver on a ragged box (no axis a multiple of a tile)
        _case("euler_fp64_o2_ragged", "smooth", (93, 75, 110), 2, "modal", "linearized"),
        # the paper's 96^3 hydrodynamic mesh at its highest order
        _case("euler_fp64_o4", "smooth", (96, 96, 96), 4),
        # a shock tube in a closed box: reflecting walls along x, outflow along y
        _case("euler_fp64_o3_walls", "walls", (64, 64, 100), 3, "nodal"),
        # the 2-D vortex of the paper's accuracy tables, run as a slab one zone deep
        _case("euler_fp64_o3_slab", "vortex", (1, 512, 512), 3),
        # the paper's 97^3 MHD mesh, divergence-free FP64
        _case("mhd_fp64_o3", "mhd", (97, 97, 97), 3),
        # the same shock tube as a production run in FP32 bulk precision
        _case("euler_fp32_o3_sod", "sod", (256, 256, 256), 3, "nodal", fp32=True),
        # highest order in FP32 bulk
        _case("euler_fp32_o4", "smooth", (128, 128, 128), 4, fp32=True),
        # second order in FP32 bulk on a ragged box
        _case("euler_fp32_o2_ragged", "smooth", (99, 150, 203), 2, "modal", "linearized", fp32=True),
        # magnetised flow in FP32 bulk with the seven-wave solver
        _case("mhd_fp32_o3_linearized", "mhd", (128, 128, 128), 3, "modal", "linearized", fp32=True),
        # a parameter study: many small problems of mixed physics, order, form and solver in one batched step
        {"name": "batch_fp32", "ic": "batch", "count": 32, "smallest": 16, "largest": 48},
    ]


# measured cost of a step per zone in ns, to keep a drawn case below the largest listed one (about 150 ms)
_COST = {("euler", False): {2: 3.2, 3: 9.5, 4: 36.0}, ("mhd", False): {2: 11.0, 3: 30.0, 4: 110.0},
         ("euler", True): {2: 0.2, 3: 0.4, 4: 2.4}, ("mhd", True): {2: 1.0, 3: 2.3, 4: 8.0}}


def draw(rng):
    kind = rng.random()
    if kind < 0.1:
        smallest = rng.choice((16, 20, 24))
        return {"ic": "batch", "count": rng.randint(4, 40), "smallest": smallest,
                "largest": smallest + 4 * rng.randint(1, 6)}
    fp32 = rng.random() < 0.5
    order = rng.choice((2, 3, 3, 4))
    ic = "mhd" if kind > 0.65 else rng.choice(("smooth", "smooth", "sod", "walls", "vortex"))
    cost = _COST["mhd" if ic == "mhd" else "euler", fp32][order]
    most = min(120e6 / cost, 256 ** 3 if order < 4 else 160 ** 3, 128 ** 3 if ic == "mhd" else 1 << 62)
    zones = math.exp(rng.uniform(math.log(10 ** 3), math.log(most)))
    if ic == "vortex":
        n = max(32, min(1024, int(zones ** 0.5)))
        shape = (1, n, n)
    else:
        # sides around the cube root, each up to 1.5 times longer or shorter, whatever remainder that leaves
        side = zones ** (1.0 / 3.0)
        a, b = (math.exp(rng.uniform(-0.4, 0.4)) for _ in range(2))
        shape = tuple(max(6, int(side * f)) for f in (a, b, 1.0 / (a * b)))
    form, solver = rng.choice(("modal", "nodal")), rng.choice(("hll", "linearized"))
    case = _case("", ic, shape, order, form, solver, fp32)
    del case["name"]
    return case


# ----------------------------------------------------------------------------- initial states
def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _centres(shape, dev):
    nz, ny, nx = shape
    ax = [(torch.arange(m, dtype=torch.float64, device=dev) + 0.5) / m for m in (nz, ny, nx)]
    return ax[0][:, None, None], ax[1][None, :, None], ax[2][None, None, :]


def _conserved(rho, v, P, gamma):
    ke = 0.5 * rho * (v[0] ** 2 + v[1] ** 2 + v[2] ** 2)
    return torch.stack([rho, rho * v[0], rho * v[1], rho * v[2], P / (gamma - 1.0) + ke]).contiguous()


def _waves(rng, shape, dev, amp, modes=10):
    """A periodic field of a few random plane waves, at most `amp` in size."""
    z, y, x = _centres(shape, dev)
    out = torch.zeros(shape, dtype=torch.float64, device=dev)
    weights = []
    for _ in range(modes):
        k = rng.integers(-3, 4, 3)
        w = 1.0 / (1.0 + float(np.sqrt((k ** 2).sum())))
        weights.append(w)
        out += w * torch.cos(2 * math.pi * (k[0] * x + k[1] * y + k[2] * z) + rng.uniform(0, 2 * math.pi))
    return out * (amp / sum(weights))


def _smooth(rng, shape, dev, gamma, amp=0.6):
    rho = 1.0 + _waves(rng, shape, dev, amp)
    P = 1.0 + _waves(rng, shape, dev, amp)
    return _conserved(rho, [_waves(rng, shape, dev, amp) for _ in range(3)], P, gamma)


def _sod(rng, shape, dev, gamma, periodic=True):
    """A planar shock tube: normal, position and jump from the seed; the fronts' zones hold sub-sampled averages."""
    nz, ny, nx = shape
    normal = [(1, 0), (1, 1), (2, 1)][int(rng.integers(0, 3))] if periodic else (1, 0)
    shift, rr, pr = rng.uniform(0, 1), rng.uniform(4, 10), rng.uniform(5, 12)
    sub = 8
    x = (torch.arange(nx * sub, dtype=torch.float64, device=dev) + 0.5) / (nx * sub)
    y = (torch.arange(ny * sub, dtype=torch.float64, device=dev) + 0.5) / (ny * sub)
    s = normal[0] * x[None, :] + normal[1] * y[:, None]
    left = (torch.remainder(s + shift, 1.0) < 0.5) if periodic else (s < 0.3 + 0.4 * shift)
    left = left.double().reshape(ny, sub, nx, sub).mean(dim=(1, 3)).expand(nz, ny, nx)
    zero = torch.zeros(shape, dtype=torch.float64, device=dev)
    return _conserved(left + (1 - left) / rr, [zero, zero, zero], left + (1 - left) / pr, gamma)


def _vortex(rng, shape, dev, gamma):
    """The isentropic vortex of the paper's Sec. VI.1 on [-5, 5]^2, its centre and strength from the seed."""
    z, y, x = _centres(shape, dev)
    cx, cy, eps = rng.uniform(-1, 1), rng.uniform(-1, 1), rng.uniform(4, 5.5)
    X, Y = 10 * x - 5 - cx, 10 * y - 5 - cy
    e = torch.exp(0.5 * (1 - X * X - Y * Y)) + 0 * z
    T = 1.0 - (gamma - 1.0) * eps ** 2 / (8 * gamma * math.pi ** 2) * e * e
    rho = T ** (1.0 / (gamma - 1.0))
    a = eps / (2 * math.pi) * e
    return _conserved(rho, [1.0 - a * Y, 1.0 + a * X, torch.zeros_like(rho)], rho * T, gamma)


def _magnetised(rng, shape, dev, gamma):
    """A smooth random flow threaded by a uniform field plus the curl of random plane waves (div B = 0)."""
    U = _smooth(rng, shape, dev, gamma, amp=0.5)
    nz, ny, nx = shape
    h = (1.0 / nx, 1.0 / ny, 1.0 / nz)
    A = [_waves(rng, shape, dev, 0.15) for _ in range(3)]       # its values serve as the edge averages
    up = lambda a, d: torch.roll(a, -1, 2 - d) - a
    mean = rng.normal(size=3)
    mean *= 1.5 / np.linalg.norm(mean)
    B = torch.stack([up(A[2], 1) / h[1] - up(A[1], 2) / h[2] + mean[0],
                     up(A[0], 2) / h[2] - up(A[2], 0) / h[0] + mean[1],
                     up(A[1], 0) / h[0] - up(A[0], 1) / h[1] + mean[2]]).contiguous()
    zb = [0.5 * (B[d] + torch.roll(B[d], -1, 2 - d)) for d in range(3)]
    U[4] += (zb[0] ** 2 + zb[1] ** 2 + zb[2] ** 2) / (2 * FOUR_PI)
    return U, B


def _problems(case):
    """The cases a batched case stands for: sizes, physics and schemes spread over the set, whatever the seed."""
    if case["ic"] != "batch":
        return [case]
    sizes = range(case["smallest"], case["largest"] + 1, 4)
    out = []
    for p in range(case["count"]):
        n = sizes[(5 * p) % len(sizes)]
        ic = ("smooth", "mhd", "sod", "mhd")[p % 4]
        out.append(dict(_case("", ic, (n, n + p % 3, n), 2 + (p // 2) % 3, ("modal", "nodal")[p // 3 % 2],
                              "hll" if ic == "mhd" else ("hll", "linearized")[p // 4 % 2], True)))
    return out


def _gamma(case):
    return 5.0 / 3.0 if case["ic"] == "mhd" else 1.4


def _lengths(case):
    return inputs.slab_lengths(10.0) if case["ic"] == "vortex" else (1.0, 1.0, 1.0)


def _states(case, seed):
    """[(U, Bface or None)] of every problem of the case."""
    dev = _device()
    rng = np.random.default_rng((2 * seed + 1) & 0x7FFFFFFF)
    out = []
    for c in _problems(case):
        shape, gamma = (c["nz"], c["ny"], c["nx"]), _gamma(c)
        if c["ic"] == "mhd":
            out.append(_magnetised(rng, shape, dev, gamma))
        elif c["ic"] in ("sod", "walls"):
            out.append((_sod(rng, shape, dev, gamma, c["ic"] == "sod"), None))
        else:
            out.append(({"smooth": _smooth, "vortex": _vortex}[c["ic"]](rng, shape, dev, gamma), None))
    return out


WALLS = ("reflective", "reflective", "outflow", "outflow", "periodic", "periodic")


# ----------------------------------------------------------------------------- the measured pass
class _Batch:
    """A batched handle and the buffers a program keeps with it."""

    def __init__(self, problems, states):
        flag = lambda c: (_lib.ADER_FP32_BULK | (_lib.ADER_NODAL if c["form"] == "nodal" else 0)
                          | (_lib.ADER_MHD if c["ic"] == "mhd" else 0))
        self.h = _lib.ader_batch_create([(c["nx"], c["ny"], c["nz"], 1 / c["nx"], 1 / c["ny"], 1 / c["nz"])
                                         for c in problems],
                                        [c["order"] for c in problems], [_gamma(c) for c in problems],
                                        [_lib.ADER_HLL if c["solver"] == "hll" else _lib.ADER_LINEARIZED
                                         for c in problems], [flag(c) for c in problems])
        self.U, self.B = [s[0] for s in states], [s[1] for s in states]
        self.dt = torch.zeros(len(problems), dtype=torch.float64, device="cuda")

    def step(self):
        _lib.ader_batch_advance(self.h, self.U, self.B, CFL, self.dt)
        return {"U": [u.float() for u in self.U], "B": [b.float() for b in self.B if b is not None],
                "dt": self.dt.float()}

    def __del__(self):
        _lib.ader_batch_destroy(self.h)


class _Single:
    """A solver, its state and the device time step."""

    def __init__(self, case, state):
        mhd = case["ic"] == "mhd"
        self.solver = ader.Solver((case["nz"], case["ny"], case["nx"]), order=case["order"], form=case["form"],
                                  solver=case["solver"], gamma=_gamma(case), fp32=case["fp32"],
                                  lengths=_lengths(case), mhd=mhd)
        if case["ic"] == "walls":
            self.solver.set_boundary(WALLS)
        self.U, self.B = state
        self.fp32 = case["fp32"]
        self.dt = torch.zeros(1, dtype=torch.float64, device="cuda")

    def step(self):
        self.solver.max_dt(self.U, CFL, self.dt, Bface=self.B)
        self.solver.step_devdt(self.U, self.dt, Bface=self.B)
        out = {"U": self.U, "dt": self.dt}
        if self.B is not None:
            out["B"] = self.B
        return {k: v.float() for k, v in out.items()} if self.fp32 else out


def prepare(case, seed):
    states = _states(case, seed)
    _lib.ader_trim_local_memory()          # a program of its own starts with no other kernel's stack
    return _Batch(_problems(case), states) if case["ic"] == "batch" else _Single(case, states[0])


def run(state):
    return state.step()


# FLOPs per zone of the scheme's own arithmetic (Euler; MHD's eight variables and edge fields cost about 2.5 times)
_FLOPS = {2: 2100, 3: 6600, 4: 26500}


def work(case):
    out = {"bytes": 0.0, "flops": 0.0}
    for c in _problems(case):
        zones, mhd = c["nz"] * c["ny"] * c["nx"], c["ic"] == "mhd"
        # the FP64 state (and face field) read and written once; an FP32 frame written where there is one
        out["bytes"] += zones * (8 if mhd else 5) * (20 if c["fp32"] else 16)
        out["flops"] += zones * _FLOPS[c["order"]] * (2.5 if mhd else 1.0)
    return out


# ----------------------------------------------------------------------------- the same step in plain FP64 torch
_P = ((1.0,), (0.0, 1.0), (-1 / 12, 0.0, 1.0), (0.0, -3 / 20, 0.0, 1.0))      # Eq. 9
_T = 1 / 3


def _p(a, x):
    return sum(c * x ** i for i, c in enumerate(_P[a]))


def _p_mean(a):
    return 1.0 if a == 0 else 0.0


_MODES2 = [(0, 0, 0, 0), (1, 0, 0, 0), (0, 1, 0, 0), (0, 0, 1, 0), (0, 0, 0, 1)]
_SPACE3 = _MODES2[:4] + [(2, 0, 0, 0), (0, 2, 0, 0), (0, 0, 2, 0), (1, 1, 0, 0), (0, 1, 1, 0), (1, 0, 1, 0)]
_SPACE4 = _SPACE3 + [(3, 0, 0, 0), (0, 3, 0, 0), (0, 0, 3, 0), (2, 1, 0, 0), (2, 0, 1, 0), (1, 2, 0, 0), (0, 2, 1, 0),
                     (1, 0, 2, 0), (0, 1, 2, 0), (1, 1, 1, 0)]
_MODES = {2: _MODES2,                                                          # Eqs. 14-16
          3: _SPACE3 + [(0, 0, 0, 1), (0, 0, 0, 2), (1, 0, 0, 1), (0, 1, 0, 1), (0, 0, 1, 1)],
          4: _SPACE4 + [(0, 0, 0, 1), (0, 0, 0, 2), (0, 0, 0, 3), (1, 0, 0, 1), (0, 1, 0, 1), (0, 0, 1, 1),
                        (1, 0, 0, 2), (0, 1, 0, 2), (0, 0, 1, 2), (2, 0, 0, 1), (0, 2, 0, 1), (0, 0, 2, 1),
                        (1, 1, 0, 1), (0, 1, 1, 1), (1, 0, 1, 1)]}
_FACE_MODES = {2: [(0, 0, 0), (1, 0, 0), (0, 1, 0), (0, 0, 1)],                # Eqs. D.2, D.7, D.12
               3: [(0, 0, 0), (1, 0, 0), (0, 1, 0), (2, 0, 0), (0, 2, 0), (1, 1, 0), (0, 0, 1), (0, 0, 2), (1, 0, 1),
                   (0, 1, 1)],
               4: [(0, 0, 0), (1, 0, 0), (0, 1, 0), (2, 0, 0), (0, 2, 0), (1, 1, 0), (3, 0, 0), (0, 3, 0), (2, 1, 0),
                   (1, 2, 0), (0, 0, 1), (0, 0, 2), (0, 0, 3), (1, 0, 1), (0, 1, 1), (1, 0, 2), (0, 1, 2), (2, 0, 1),
                   (0, 2, 1), (1, 1, 1)]}


def _points(text):
    """Node coordinates from a compact list: + and - are +-1/2, p and n are +-1/4, t 1/3, T 2/3, 0 and 1 themselves."""
    value = {"+": 0.5, "-": -0.5, "p": 0.25, "n": -0.25, "t": _T, "T": 2 * _T, "0": 0.0, "1": 1.0, "h": 0.5}
    return np.array([[value[ch] for ch in word] for word in text.split()])


_NODES = {                                                                     # Eqs. 31, 37, 46 and A.1, B.1, C.1
    (2, "modal"): _points("+000 -000 0+00 0-00 00+0 00-0"),
    (3, "modal"): _points("0000 ++00 +-00 +0+0 +0-0 -+00 --00 -0+0 -0-0 0++0 0-+0 0+-0 0--0 "
                          "+00h -00h 0+0h 0-0h 00+h 00-h"),
    (4, "modal"): _points("0000 +000 p000 n000 -000 0+00 0p00 0n00 0-00 00+0 00p0 00n0 00-0 "
                          "+++0 +-+0 ++-0 +--0 -++0 --+0 -+-0 ---0 "
                          "000t ++0t +-0t +0+t +0-t -+0t --0t -0+t -0-t 0++t 0-+t 0+-t 0--t "
                          "000T +00T -00T 0+0T 0-0T 00+T 00-T"),
    (2, "nodal"): _points("0000 +000 0+00 00+0 0001"),
    (3, "nodal"): _points("0000 +000 -000 0+00 0-00 00+0 00-0 0++0 +0+0 ++00 000h +00h 0+0h 00+h 0001"),
    (4, "nodal"): _points("0000 +++0 +000 -000 0+00 0-00 00+0 00-0 0++0 -0+0 +0+0 +-00 ++00 0+-0 n--0 p--0 -n-0 -p-0 "
                          "--n0 --p0 000t +00t -00t 0+0t 0-0t 00+t 00-t 0++t +0+t ++0t 000T +00T 0+0T 00+T 0001")}
_FACE_NODES = {2: _points("+0h -0h 0+h 0-h 001"),                              # Eqs. D.1, D.6, D.11
               3: _points("000 ++0 -+0 +-0 --0 +0h -0h 0+h 0-h 001"),
               4: _points("000 +00 p00 n00 -00 0+0 0p0 0n0 0-0 ++0 -+0 +-0 --0 00t ++t -+t +-t --t 00T +0T -0T 0+T "
                          "0-T 001")}


def _basis(order, pts):
    return np.array([[_p(a, x) * _p(b, y) * _p(c, z) * t ** d for a, b, c, d in _MODES[order]] for x, y, z, t in pts])


def _x_flux_rule(order):
    """Modal form: {mode: row over the nodes} of the x-flux modes (Eqs. 33, 40, 49)."""
    I = np.eye(len(_NODES[order, "modal"]))
    X = lambda n: I[n - 1]
    if order == 2:
        return {2: X(1) - X(2)}
    m = {}
    if order == 3:
        q1, q2, q3 = X(2) + X(3) + X(4) + X(5), X(6) + X(7) + X(8) + X(9), X(10) + X(11) + X(12) + X(13)
        m[2] = 0.25 * (q1 - q2)
        m[5] = 0.5 * (q1 + q2 - q3) - 2 * X(1)
        m[8] = X(2) - X(3) - X(6) + X(7)
        m[10] = X(4) - X(5) - X(8) + X(9)
        m[13] = 2 * (X(14) - X(15) - m[2])
        return m
    q1, q2 = X(14) + X(15) + X(16) + X(17), X(18) + X(19) + X(20) + X(21)
    q3, q4 = X(14) + X(16) + X(18) + X(20), X(15) + X(17) + X(19) + X(21)
    q5, q6 = X(14) + X(15) + X(18) + X(19), X(16) + X(17) + X(20) + X(21)
    q7 = X(23) + X(24) - X(25) - X(26) - X(27) - X(28) + X(29) + X(30)
    q8 = X(23) + X(27) - X(24) - X(28) - X(31) - X(33) + X(32) + X(34)
    q9 = X(25) + X(29) - X(26) - X(30) - X(31) - X(32) + X(33) + X(34)
    q10 = X(23) + X(24) + X(25) + X(26) - X(27) - X(28) - X(29) - X(30)
    m[5] = 2 * (X(2) - 2 * X(1) + X(5))
    m[8] = 0.5 * (X(14) - X(15) + X(16) - X(17) - X(18) + X(19) - X(20) + X(21))
    m[10] = 0.5 * (X(14) + X(15) - X(16) - X(17) - X(18) - X(19) + X(20) + X(21))
    m[11] = 16 / 3 * (X(2) - 2 * X(3) + 2 * X(4) - X(5))
    m[2] = 2 / 3 * (X(2) - X(5)) - 0.1 * m[11] + (q1 - q2) / 12
    m[14] = q8 + 0.5 * (q3 - q4) - 2 * (X(6) - X(9))
    m[15] = q9 + 0.5 * (q5 - q6) - 2 * (X(10) - X(13))
    m[16] = q7 + 0.5 * (q1 - q2) - 2 * (X(2) - X(5))
    m[18] = m[16] - 2 * q7
    m[20] = X(14) - X(15) - X(16) + X(17) - X(18) + X(19) + X(20) - X(21)
    m[27] = 1.125 * (q1 - q2) + 4.5 * (X(36) - X(37)) - 2.25 * q10
    m[24] = 3 * (X(36) - X(37)) - 0.75 * q10 + 0.375 * (m[16] + m[18]) - m[27]
    m[30] = 3 * (X(36) - 2 * X(35) + X(37)) - 1.5 * m[5]
    m[33] = 3 * (X(23) - X(27) - X(24) + X(28)) - 3 * m[8]
    m[35] = 3 * (X(25) - X(29) - X(26) + X(30)) - 3 * m[10]
    return m


def _face_rule(order):
    """Matrix (facial modes x facial nodes) of App. D: Eqs. D.4 and D.14, interpolation at order 3 (Eq. D.9)."""
    pts = _FACE_NODES[order]
    if order == 3:
        return np.linalg.inv(np.array([[_p(a, y) * _p(b, z) * t ** d for a, b, d in _FACE_MODES[3]]
                                       for y, z, t in pts]))
    I = np.eye(len(pts))
    X = lambda n: I[n - 1]
    if order == 2:
        m4 = 2 * X(5) - 0.5 * (X(1) + X(2) + X(3) + X(4))
        return np.stack([X(5) - m4, X(1) - X(2), X(3) - X(4), m4])
    m = {}
    q1 = 3 * (X(20) - X(21)) - 1.5 * (X(15) - X(16) + X(17) - X(18))
    q2 = 1.5 * (X(20) - X(21) - X(2) + X(5))
    q3 = 3 * (X(22) - X(23)) - 1.5 * (X(15) + X(16) - X(17) - X(18))
    q4 = 1.5 * (X(22) - X(23) - X(6) + X(9))
    m[1] = (2 * X(1) + X(2) + X(5) + X(6) + X(9)) / 6
    m[4] = 2 * (X(2) - 2 * X(1) + X(5))
    m[5] = 2 * (X(6) - 2 * X(1) + X(9))
    m[6] = X(10) - X(11) - X(12) + X(13)
    m[7] = 16 / 3 * (X(2) - 2 * X(3) + 2 * X(4) - X(5))
    m[8] = 16 / 3 * (X(6) - 2 * X(7) + 2 * X(8) - X(9))
    m[9] = 2 * (X(10) - 2 * X(6) + X(11) - X(12) + 2 * X(9) - X(13))
    m[10] = 2 * (X(10) - 2 * X(2) + X(12) - X(11) + 2 * X(5) - X(13))
    m[2] = X(2) - X(5) + m[10] / 12 - 0.1 * m[7]
    m[3] = X(6) - X(9) + m[9] / 12 - 0.1 * m[8]
    m[13] = 4.5 * (X(24) - X(1)) - 13.5 * (X(19) - X(14))
    m[12] = 2.25 * (X(24) - X(19) - X(14) + X(1) - 2 / 3 * m[13])
    m[11] = (1.5 * X(24) - 2.5 * X(14) + 0.25 * (X(15) + X(16) + X(17) + X(18)) - 0.25 * m[4] - 0.25 * m[5]
             - 4 / 3 * m[12] - 13 / 9 * m[13])
    m[14] = 3 * q2 - 2 * q1 - 1.5 * m[10]
    m[16] = 3 * (q1 - q2) + 2.25 * m[10]
    m[15] = 3 * q4 - 2 * q3 - 1.5 * m[9]
    m[17] = 3 * (q3 - q4) + 2.25 * m[9]
    m[18] = 3 * (X(20) - 2 * X(19) + X(21)) - 1.5 * m[4]
    m[19] = 3 * (X(22) - 2 * X(19) + X(23)) - 1.5 * m[5]
    m[20] = 3 * (X(15) - X(16) - X(17) + X(18)) - 3 * m[6]
    return np.stack([m[k] for k in range(1, 21)])


def _swapped(e, d):
    """Exponents or coordinates with axis 0 and axis d exchanged."""
    e = list(e)
    e[0], e[d] = e[d], e[0]
    return tuple(e)


@functools.lru_cache(maxsize=None)
def _predictor_tables(order, form):
    """(V, [A_x, A_y, A_z]): node values V m, and new evolutionary modes sum_d c_d A_d F_d from the node fluxes."""
    modes, pts = _MODES[order], _NODES[order, form]
    at = {m: i for i, m in enumerate(modes)}
    V = _basis(order, pts)
    evo = [i for i, m in enumerate(modes) if m[3] > 0]
    A = []
    for d in range(3):
        E = np.zeros((len(modes), len(pts)))                    # flux modes from node fluxes
        if form == "nodal":
            E = np.linalg.inv(V)
        else:
            where = {tuple(p): n for n, p in enumerate(pts.tolist())}
            to = [where[_swapped(p, d)] for p in pts.tolist()]  # the x-rule's nodes seen along axis d
            for k, row in _x_flux_rule(order).items():
                E[at[_swapped(modes[k - 1], d)], to] += row
        D = np.zeros((len(modes), len(modes)))                  # d/d(axis d), in the basis of Eq. 9
        for k, m in enumerate(modes):
            for a, c in {0: {}, 1: {0: 1.0}, 2: {1: 2.0}, 3: {2: 3.0, 0: 0.1}}[m[d]].items():
                D[at[m[:d] + (a,) + m[d + 1:]], k] += c
        R = -(D @ E)
        A.append(np.stack([R[at[modes[k][:3] + (modes[k][3] - 1,)]] / modes[k][3] for k in evo]))
    return V, A


@functools.lru_cache(maxsize=None)
def _face_tables(order, d, s):
    """(u_b weights, <u> weights, facial node matrix, <F> weights, {(t, side): (<u>_e, <F>_e weights)}) of a face."""
    modes, x = _MODES[order], 0.5 * s
    t = [a for a in range(3) if a != d]
    ub = _basis(order, [[x if a == d else 0.0 for a in range(3)] + [0.5]])[0]

    def mean(fixed):
        w = [_p(m[d], x) / (m[3] + 1) for m in modes]
        for a in t:
            w = [v * (_p(m[a], fixed[a]) if a in fixed else _p_mean(m[a])) for v, m in zip(w, modes)]
        return np.array(w)

    def face_mean(slot, at):
        w = []
        for m in _FACE_MODES[order]:
            v = 1.0 / (m[2] + 1)
            for q in range(2):
                v *= _p(m[q], at) if q == slot else _p_mean(m[q])
            w.append(v)
        return np.array(w)

    pts = np.zeros((len(_FACE_NODES[order]), 4))
    pts[:, d], pts[:, t[0]], pts[:, t[1]], pts[:, 3] = (x, *_FACE_NODES[order].T)
    rule = _face_rule(order)
    edges = {(a, e): (mean({a: 0.5 * e}), face_mean(q, 0.5 * e) @ rule)
             for q, a in enumerate(t) for e in (1, -1)}
    return ub, mean({}), _basis(order, pts), face_mean(None, 0.0) @ rule, edges


def _dot(M, X):
    """A matrix (or row) over the first axis of X, without the zero entries' work."""
    M = np.asarray(M)
    rows = M[None] if M.ndim == 1 else M
    out = torch.tensordot(torch.tensor(rows, dtype=X.dtype, device=X.device), X, dims=1)
    return out[0] if M.ndim == 1 else out


def _at(a, d, k):
    """The value k zones up along direction d (periodic)."""
    return torch.roll(a, -k, -1 - d)


def _weighted(candidates, smooth, linear):
    w = [g / (1e-12 + s) ** 2 for g, s in zip(linear, smooth)]
    total = sum(w)
    return [sum(a * c[r] for a, c in zip(w, candidates)) / total for r in range(len(candidates[0]))]


def _weno3(a, d):
    """The quadratic zone WENO along d: the P1 and P2 moments."""
    m2, m1, p1, p2 = (_at(a, d, k) for k in (-2, -1, 1, 2))
    cand = [((3 * a - 4 * m1 + m2) / 2, (a - 2 * m1 + m2) / 2), ((p1 - m1) / 2, (p1 - 2 * a + m1) / 2),
            ((4 * p1 - 3 * a - p2) / 2, (p2 - 2 * p1 + a) / 2)]
    return _weighted(cand, [b * b + 13 / 3 * c * c for b, c in cand], (1, 10, 1))


def _weno4(a, d):
    """The cubic zone WENO along d: the P1, P2 and P3 moments."""
    out = []
    for lo in (-3, -2, -1, 0):
        # zone averages of P1, P2, P3 over zone k: k, k^2, k^3 + k/10
        ks = [k for k in range(lo, lo + 4) if k]
        M = np.linalg.inv(np.array([[k, k * k, k ** 3 + k / 10] for k in ks]))
        diff = torch.stack([_at(a, d, k) - a for k in ks])
        out.append(tuple(_dot(M, diff)))
    return _weighted(out, [(b + e / 10) ** 2 + 13 / 3 * c * c + 781 / 20 * e * e for b, c, e in out], (1, 10, 10, 1))


def _face_b(b, d, order):
    """Sec. III: zone average and normal moments of the field from its face values (face i at i - 1/2)."""
    m, p = b, _at(b, d, 1)
    if order == 2:
        return [0.5 * (m + p), p - m]
    mm, pp = _at(b, d, -1), _at(b, d, 2)
    if order == 3:
        cand = [((8 * m - mm + 5 * p) / 12, p - m, (p + mm - 2 * m) / 2),
                ((8 * p - pp + 5 * m) / 12, p - m, (m + pp - 2 * p) / 2)]
        return _weighted(cand, [c[1] ** 2 + 13 / 3 * c[2] ** 2 for c in cand], (1, 1))
    mmm, ppp = _at(b, d, -2), _at(b, d, 3)
    cand = [((9 * p + 19 * m - 5 * mm + mmm) / 24, (59 * p - 57 * m - 3 * mm + mmm) / 60,
             (3 * p - 7 * m + 5 * mm - mmm) / 4, (p - 3 * m + 3 * mm - mmm) / 6),
            ((13 * p + 13 * m - pp - mm) / 24, (63 * p - 63 * m - pp + mm) / 60, (pp - p - m + mm) / 4,
             (pp - 3 * p + 3 * m - mm) / 6),
            ((ppp - 5 * pp + 19 * p + 9 * m) / 24, (3 * pp - ppp + 57 * p - 59 * m) / 60,
             (5 * pp - ppp - 7 * p + 3 * m) / 4, (ppp - 3 * pp + 3 * p - m) / 6)]
    return _weighted(cand, [(c[1] + c[3] / 10) ** 2 + 13 / 3 * c[2] ** 2 + 781 / 20 * c[3] ** 2 for c in cand],
                     (1, 2, 1))


def _zone_modes(u, order, normal=None):
    """Spatial modes of one zone-averaged variable; normal = (direction, its moments) where a face field gives them."""
    line = {2: lambda d: _weno3(u, d)[:1], 3: lambda d: _weno3(u, d), 4: lambda d: _weno4(u, d)}[order]
    m = [normal[1] if normal and normal[0] == d else line(d) for d in range(3)]
    W = [u] + [m[d][0] for d in range(3)]
    if order > 2:
        slope = lambda a, d: _weno3(a, d)[0]
        W += [m[d][1] for d in range(3)]
        W += [0.5 * (slope(W[1], 1) + slope(W[2], 0)), 0.5 * (slope(W[2], 2) + slope(W[3], 1)),
              0.5 * (slope(W[1], 2) + slope(W[3], 0))]
    if order == 4:
        W += [m[d][2] for d in range(3)]
        W += [slope(W[4 + a], d) for a in range(3) for d in range(3) if d != a]
        W.append((slope(W[7], 2) + slope(W[8], 0) + slope(W[9], 1)) / 3)
    return torch.stack(W)


def _pressure(u, gamma):
    e = u[4] - 0.5 * (u[1] ** 2 + u[2] ** 2 + u[3] ** 2) / u[0]
    if len(u) == 8:
        e = e - (u[5] ** 2 + u[6] ** 2 + u[7] ** 2) / (2 * FOUR_PI)
    return (gamma - 1) * e


def _flux(u, gamma, d):
    """Eq. 3, direction d, for states with the variable on the first axis."""
    v, P = [u[1 + c] / u[0] for c in range(3)], _pressure(u, gamma)
    if len(u) == 5:
        f = [u[1 + d]] + [u[1 + c] * v[d] + (P if c == d else 0.0) for c in range(3)] + [(u[4] + P) * v[d]]
        return torch.stack(f)
    B = u[5:]
    P = P + (B[0] ** 2 + B[1] ** 2 + B[2] ** 2) / (2 * FOUR_PI)
    vB = v[0] * B[0] + v[1] * B[1] + v[2] * B[2]
    f = [u[1 + d]] + [u[1 + c] * v[d] - B[d] * B[c] / FOUR_PI + (P if c == d else 0.0) for c in range(3)]
    f.append((u[4] + P) * v[d] - B[d] * vB / FOUR_PI)
    return torch.stack(f + [v[d] * B[c] - v[c] * B[d] for c in range(3)])


def _speed(u, gamma, d):
    a2 = gamma * _pressure(u, gamma) / u[0]
    if len(u) == 5:
        return torch.sqrt(a2)
    s = a2 + (u[5] ** 2 + u[6] ** 2 + u[7] ** 2) / (FOUR_PI * u[0])
    n2 = u[5 + d] ** 2 / (FOUR_PI * u[0])
    return torch.sqrt(0.5 * (s + torch.sqrt(torch.clamp(s * s - 4 * a2 * n2, min=0.0))))


def _abs_jacobian(mean, gamma, d):
    """|A| of direction d at the primitive state `mean` = (rho, v, P[, B]), as a function of a jump of states."""
    rho, v, P = mean[0], mean[1:4], mean[4]
    a2 = gamma * P / rho
    a = torch.sqrt(a2)
    t = [c for c in range(3) if c != d]
    u, q2 = v[d], v[0] ** 2 + v[1] ** 2 + v[2] ** 2
    B = [b / math.sqrt(FOUR_PI) for b in mean[5:]] if len(mean) == 8 else [torch.zeros_like(rho)] * 3
    bn2, bt2 = B[d] ** 2 / rho, (B[t[0]] ** 2 + B[t[1]] ** 2) / rho
    total = a2 + bn2 + bt2
    root = torch.sqrt(torch.clamp(total ** 2 - 4 * a2 * bn2, min=0.0))
    cf2, cs2 = 0.5 * (total + root), torch.clamp(0.5 * (total - root), min=0.0)
    cf, cs, ca = torch.sqrt(cf2), torch.sqrt(cs2), torch.sqrt(bn2)
    apart = cf2 - cs2 > 1e-12 * cf2
    af = torch.where(apart, torch.sqrt(torch.clamp(a2 - cs2, min=0.0)), torch.ones_like(a))
    as_ = torch.where(apart, torch.sqrt(torch.clamp(cf2 - a2, min=0.0)), torch.zeros_like(a))
    n = torch.sqrt(af ** 2 + as_ ** 2)
    af, as_ = af / n, as_ / n
    bt = torch.sqrt(B[t[0]] ** 2 + B[t[1]] ** 2)
    some = bt > 1e-12 * torch.sqrt(rho * total)
    safe, half = torch.where(some, bt, torch.ones_like(bt)), torch.full_like(bt, math.sqrt(0.5))
    e1, e2 = torch.where(some, B[t[0]] / safe, half), torch.where(some, B[t[1]] / safe, half)
    sg, sr = torch.where(B[d] >= 0, 1.0, -1.0), torch.sqrt(rho)
    fc, sc = af * cf, as_ * cs
    det = fc ** 2 + sc ** 2

    def apply(dU):
        dr = dU[0]
        dv = [(dU[1 + c] - v[c] * dr) / rho for c in range(3)]
        k = 1 / math.sqrt(FOUR_PI)
        db = [dU[5 + c] * k if len(dU) == 8 and c != d else torch.zeros_like(dr) for c in range(3)]
        dP = (gamma - 1) * (dU[4] - 0.5 * q2 * dr - rho * sum(v[c] * dv[c] for c in range(3))
                            - sum(B[c] * db[c] for c in t))
        vp, vq = e1 * dv[t[0]] + e2 * dv[t[1]], e1 * dv[t[1]] - e2 * dv[t[0]]
        bp, bq = e1 * db[t[0]] + e2 * db[t[1]], e1 * db[t[1]] - e2 * db[t[0]]
        alf = [0.5 * (vq - s * sg * bq / sr) * torch.abs(u + s * ca) for s in (1, -1)]
        fd, sd = (fc * dv[d] - sc * sg * vp) / det, (sc * dv[d] + fc * sg * vp) / det
        X, Y = dP / (rho * a2), bp / (sr * a)
        fs, ss = af * X + as_ * Y, as_ * X - af * Y
        fast = [torch.abs(u + s * cf) * 0.5 * (fs + s * fd) for s in (1, -1)]
        slow = [torch.abs(u + s * cs) * 0.5 * (ss + s * sd) for s in (1, -1)]
        F, S, Fd, Sd = fast[0] + fast[1], slow[0] + slow[1], fast[0] - fast[1], slow[0] - slow[1]
        r = torch.abs(u) * (dr - dP / a2) + rho * (af * F + as_ * S)
        vp, vq = sg * (fc * Sd - sc * Fd), alf[0] + alf[1]
        bp, bq = a * sr * (as_ * F - af * S), -sg * sr * (alf[0] - alf[1])
        w, b = [None] * 3, [torch.zeros_like(r)] * 3
        w[d], w[t[0]], w[t[1]] = fc * Fd + sc * Sd, e1 * vp - e2 * vq, e2 * vp + e1 * vq
        b[t[0]], b[t[1]] = e1 * bp - e2 * bq, e2 * bp + e1 * bq
        out = [r] + [v[c] * r + rho * w[c] for c in range(3)]
        out.append(0.5 * q2 * r + rho * sum(v[c] * w[c] for c in range(3)) + rho * a2 * (af * F + as_ * S) / (gamma - 1)
                   + sum(B[c] * b[c] for c in t))
        return torch.stack(out + ([x / k for x in b] if len(dU) == 8 else []))
    return apply


def _riemann(solver, gamma, d, ubL, ubR):
    """The face solver with its speeds or eigen-structure frozen at the barycentre states: f(uL, uR, FL, FR)."""
    if solver == "hll":
        vL, vR, cL, cR = ubL[1 + d] / ubL[0], ubR[1 + d] / ubR[0], _speed(ubL, gamma, d), _speed(ubR, gamma, d)
        lo = torch.clamp(torch.minimum(vL - cL, vR - cR), max=0.0)
        hi = torch.clamp(torch.maximum(vL + cL, vR + cR), min=0.0)
        return lambda uL, uR, FL, FR: (hi * FL - lo * FR + hi * lo * (uR - uL)) / (hi - lo)       # Eq. 56
    prim = lambda u: [u[0]] + [u[1 + c] / u[0] for c in range(3)] + [_pressure(u, gamma)] + list(u[5:])
    A = _abs_jacobian([0.5 * (x + y) for x, y in zip(prim(ubL), prim(ubR))], gamma, d)
    return lambda uL, uR, FL, FR: 0.5 * (FL + FR) - 0.5 * A(uR - uL)


def _exact_step(U, B, case, dx, dt):
    """(U, Bface) after one ADER-WENO step of size dt on the periodic box (Eqs. 6 and 8)."""
    order, form, solver, gamma = case["order"], case["form"], case["solver"], _gamma(case)
    modes = [_zone_modes(U[v], order) for v in range(5)]
    for d in range(3 if B is not None else 0):
        first, *normal = _face_b(B[d], d, order)
        modes.append(_zone_modes(first, order, (d, normal)))
    W = torch.stack(modes, 1)
    del modes
    V, A = _predictor_tables(order, form)
    m = torch.cat([W, torch.zeros((V.shape[1] - len(W),) + W.shape[1:], dtype=W.dtype, device=W.device)])
    for _ in range(order - 1):
        nodes = _dot(V, m)
        new = 0.0
        for d in range(3):
            used = np.flatnonzero(np.abs(A[d]).max(axis=0) > 1e-13)
            f = torch.stack([_flux(nodes[n], gamma, d) for n in used])
            new = new + (dt / dx[d]) * _dot(A[d][:, used], f)
        m[len(W):] = new
        del nodes, f, new
    mean = W[0]
    out, edge = U.clone(), {}
    for d in range(3):
        side = {}
        for s in (1, -1):
            wb, wa, N, wf, we = _face_tables(order, d, s)
            ub = _dot(wb, m)
            ok = (ub[0] > 0) & (_pressure(ub, gamma) > 0)
            f = torch.stack([_flux(_dot(row, m), gamma, d) for row in N])
            side[s] = (torch.where(ok, ub, mean), _dot(wa, m), _dot(wf, f),
                       {key: (_dot(u, m), _dot(w, f)) for key, (u, w) in we.items()} if B is not None else {})
            del f
        L, R = side[1], [_at(x, d, 1) for x in side[-1][:3]]        # face i + 1/2: zone i below, zone i + 1 above
        solve = _riemann(solver, gamma, d, L[0], R[0])
        F = solve(L[1], R[1], L[2], R[2])[:5]
        out -= (dt / dx[d]) * (F - _at(F, d, -1))
        for key, (u, f) in L[3].items():
            edge[(d,) + key] = solve(u, _at(side[-1][3][key][0], d, 1), f, _at(side[-1][3][key][1], d, 1))
    if B is None:
        return out, None
    # Eq. 7: E_c on the edges along c, the mean of the four adjacent faces' fluxes with their signs
    E = []
    for c in range(3):
        a, b = (c + 1) % 3, (c + 2) % 3
        # E_c = -(flux of B_b along a) = +(flux of B_a along b)
        E.append(0.25 * (edge[b, a, 1][5 + a] + _at(edge[b, a, -1][5 + a], a, 1)
                         - edge[a, b, 1][5 + b] - _at(edge[a, b, -1][5 + b], b, 1)))
    newB = B.clone()
    for d in range(3):                                              # Eq. 8; the face i - 1/2 lies one zone lower
        a, b = (d + 1) % 3, (d + 2) % 3
        Ea, Eb = _at(E[a], d, -1), _at(E[b], d, -1)
        newB[d] -= dt * ((Eb - _at(Eb, a, -1)) / dx[a] - (Ea - _at(Ea, b, -1)) / dx[b])
    return out, newB


def _exact_walls(U, case, dx, dt):
    """The same step in the box of WALLS, on the state extended by ghost zones."""
    G = 4 if case["order"] == 4 else 3
    nz, ny, nx = U.shape[1:]
    x = torch.arange(-G, nx + G, device=U.device)
    mirror = torch.where(x < 0, -1 - x, torch.where(x >= nx, 2 * nx - 1 - x, x))
    W = U[..., mirror].clone()
    W[1] = torch.where((x < 0) | (x >= nx), -W[1], W[1])
    W = W[:, :, torch.arange(-G, ny + G, device=U.device).clamp(0, ny - 1)]
    return _exact_step(W, None, case, dx, dt)[0][:, :, G:-G, G:-G].contiguous()


def _exact_dt(U, B, gamma, dx):
    state = U
    if B is not None:
        state = torch.cat([U, torch.stack([0.5 * (B[d] + _at(B[d], d, 1)) for d in range(3)])])
    return CFL / sum((torch.abs(U[1 + d] / U[0]) + _speed(state, gamma, d)) / dx[d] for d in range(3)).max()


def exact(case, seed):
    problems = _problems(case)
    for c in problems:          # the modes, node values and fluxes of the plain form have to fit the card
        if c["nz"] * c["ny"] * c["nx"] * len(_MODES[c["order"]]) * (8 if c["ic"] == "mhd" else 5) * 8 * 6 > 150e9:
            return None
    got = []
    for c, (U, B) in zip(problems, _states(case, seed)):
        length = _lengths(c)
        dx = [length[0] / c["nx"], length[1] / c["ny"], length[2] / c["nz"]]
        dt = _exact_dt(U, B, _gamma(c), dx)
        if c["ic"] == "walls":
            U = _exact_walls(U, c, dx, dt)
        else:
            U, B = _exact_step(U, B, c, dx, dt)
        got.append((U, B, dt))
    if case["ic"] == "batch":
        return {"U": [g[0] for g in got], "B": [g[1] for g in got if g[1] is not None],
                "dt": torch.stack([g[2] for g in got])}
    out = {"U": got[0][0], "dt": got[0][2].reshape(1)}
    if got[0][1] is not None:
        out["B"] = got[0][1]
    return out
