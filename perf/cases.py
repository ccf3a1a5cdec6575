"""The measured workloads of the solver: what a program does with it once its plan stands.

Every case goes through the public binding (`flups.Solver`, the `flups_server_*` calls).  Kinds:

- ``solve``   one solve on device arrays with a plan the program keeps (a time step of a flow solver);
- ``host``    the same through pinned host arrays (a CPU code that hands its right-hand side over);
- ``plan``    a new plan, one solve with it, and its release (a problem that is met once: most
              requests of the served stream start with this);
- ``served``  a burst of requests to a running server that holds their plans.

A case names its faces per direction as two letters or PER / UNB (E even, O odd, U unbounded), its
grid cells per direction (`nx`, ...; the stored count is one more in a node-centred direction) and its
arithmetic: f32, f64, or f64e (FP64 arrays, FP64-class tolerance).  Sizes are the ones of the bench and
of the served stream, and products 2^a 3^b between them.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2211_07777_gb300 import flups as F
from paper_2211_07777_gb300 import serve as S
from paper_2211_07777_gb300 import workloads as W

FACE = {"E": F.EVEN, "O": F.ODD, "U": F.UNB}
PREC = {"f32": F.F32, "f64": F.F64, "f64e": F.F64E}
DEV = "cuda"


def _case(name, n, bc, prec, center="cell", kind="solve", op="poisson"):
    return {"name": name, "kind": kind, "nx": n[0], "ny": n[1], "nz": n[2], "x": bc[0], "y": bc[1], "z": bc[2],
            "center": center, "prec": prec, "op": op}


def listed():
    return [
        # the smallest call: a coarse periodic box (a multigrid bottom, a unit test, a large batch of small problems)
        _case("per32_f64", (32, 32, 32), ("PER", "PER", "PER"), "f64"),
        # a small ragged box with wall, inflow and open faces
        _case("semi48_f32", (48, 32, 36), ("EU", "EO", "UNB"), "f32"),
        # free-space potential of a compact source, FP64: the method's validation workload
        _case("unb128_f64", (128, 128, 128), ("UNB", "UNB", "UNB"), "f64"),
        # the same at a size with a factor 3, FP64-class arithmetic
        _case("unb192_f64e", (192, 192, 192), ("UNB", "UNB", "UNB"), "f64e"),
        # node-centred channel: walls in x, periodic in y (stored without its duplicate node), open in z
        _case("mixed256_f32", (256, 256, 256), ("EE", "PER", "UNB"), "f32", center="node"),
        # the largest single-precision free-space solve
        _case("unb512_f32", (512, 512, 512), ("UNB", "UNB", "UNB"), "f32"),
        # a large periodic box in double precision (spectral turbulence)
        _case("per1024_f64", (1024, 1024, 1024), ("PER", "PER", "PER"), "f64"),
        # walls on every side but one direction, FP64, factor 3: all real-to-real transforms
        _case("sym192_f64", (192, 192, 192), ("EO", "OO", "EE"), "f64"),
        # velocity of a vortex ring over a wall (Biot-Savart), the served stream's vector request
        _case("ring128_f32", (128, 128, 128), ("UNB", "UNB", "EE"), "f32", op="biot"),
        # a CPU code's field, pinned host memory in and out
        _case("host256_f32", (256, 256, 256), ("UNB", "UNB", "PER"), "f32", kind="host"),
        # a problem met once: plan, solve, release
        _case("plan96_f64", (96, 96, 96), ("UNB", "UO", "PER"), "f64", kind="plan"),
        # eight requests of mixed size, operator and precision to a warm server
        {"name": "served8", "kind": "served", "count": 8, "stream": 4, "nmax": 128},
    ]


def _size(rng, lo, hi):
    """A product 2^a 3^b in [lo, hi], uniform in its logarithm."""
    want = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    best = min((2 ** a * 3 ** b for a in range(0, 11) for b in range(0, 6) if lo <= 2 ** a * 3 ** b <= hi),
               key=lambda v: abs(math.log(v / want)))
    return best


PERIOD = {"PER": 1, "UNB": 2, "EE": 2, "OO": 2}  # extension length over cells; every other type 4


def _ext(case):
    return [case["n" + d] * PERIOD.get(case[d], 4) for d in "xyz"]


def draw(rng):
    kind = rng.choice(["solve"] * 8 + ["host", "plan"] * 2 + ["served"])
    if kind == "served":
        return {"kind": "served", "count": rng.randint(4, 16), "stream": rng.randrange(1 << 20),
                "nmax": rng.choice([64, 96, 128])}
    while True:
        faces = []
        for _ in range(3):
            t = rng.random()
            faces.append("PER" if t < 0.25 else ("UNB" if t < 0.55 else rng.choice("EOU") + rng.choice("EOU")))
        faces = ["UNB" if f == "UU" else f for f in faces]
        op = "biot" if rng.random() < 0.3 else "poisson"
        base = _size(rng, 24, 192 if kind == "plan" else 512)
        n = [base if rng.random() < 0.5 else _size(rng, max(16, base // 2), min(512, base * 2)) for _ in range(3)]
        c = _case("", n, faces, rng.choice(["f32", "f64", "f64e"]), rng.choice(["cell", "cell", "node"]), kind, op)
        del c["name"]
        ext = _ext(c)
        total = ext[0] * ext[1] * ext[2] * (3 if op == "biot" else 1)
        # no dearer than the largest listed case, and a period the solver takes; host arrays and new
        # plans at the sizes where programs use them
        if max(ext) > 2048 or total > (1 << (28 if kind != "solve" else 29)):
            continue
        if op == "biot" and max(ext) > 1024:
            continue
        return c


# --------------------------------------------------------------------------------------------------
# Inputs.
# --------------------------------------------------------------------------------------------------
def _geom(case):
    """Stored counts, spacings and lengths: unit spacing ratio 1 / max cells, so a box of mixed sizes keeps cubic cells."""
    cells = [case["nx"], case["ny"], case["nz"]]
    h = 1.0 / max(cells)
    node = case["center"] == "node"
    # a node-centred periodic direction is stored without its duplicate node
    n = [c + (1 if node and case[d] != "PER" else 0) for c, d in zip(cells, "xyz")]
    return n, (h, h, h), tuple(c * h for c in cells)


def _axes(case):
    n, h, _ = _geom(case)
    off = 0.0 if case["center"] == "node" else 0.5
    return [(torch.arange(n[d], device=DEV, dtype=torch.float64) + off) * h[d] for d in range(3)]


def _field(case, seed):
    """Gaussian blobs in the middle of the box plus resolved small scales (1%): a vorticity or charge density."""
    rng = np.random.default_rng(int(seed))
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    x, y, z = _axes(case)
    _, _, L = _geom(case)
    dt = torch.float32 if case["prec"] == "f32" else torch.float64
    out = []
    for _ in range(3 if case["op"] == "biot" else 1):
        f = torch.zeros((len(z), len(y), len(x)), device=DEV, dtype=dt)
        for _ in range(3):
            c = rng.uniform(0.35, 0.65, 3) * L
            s = rng.uniform(0.06, 0.12) * min(L)
            a = float(rng.uniform(0.5, 2.0) * rng.choice([-1.0, 1.0]))
            gx, gy, gz = (torch.exp(-(v - float(m)) ** 2 / (2 * s * s)).to(dt) for v, m in zip((x, y, z), c))
            f.add_((a * gz)[:, None, None] * gy[None, :, None] * gx[None, None, :])
        f.add_(torch.randn(f.shape, device=DEV, dtype=dt, generator=g), alpha=0.01)
        out.append(f)
    return torch.stack(out) if case["op"] == "biot" else out[0]


def _faces(case):
    return tuple((F.PER, F.PER) if case[d] == "PER" else (F.UNB, F.UNB) if case[d] == "UNB" else
                 tuple(FACE[c] for c in case[d]) for d in "xyz")


def _unbounded(case):
    return any("U" in case[d] for d in "xyz")


def _solver(case):
    n, h, L = _geom(case)
    bc = _faces(case)
    biot = case["op"] == "biot"
    return F.Solver(n, S.vector_bc(bc) if biot else bc, L=L, h=h, prec=PREC[case["prec"]],
                    center=F.NODE if case["center"] == "node" else F.CELL,
                    green="hej2" if _unbounded(case) else "spectral", op=F.BIOT_SAVART if biot else F.POISSON)


class _Burst:
    """A server and a fixed list of requests with their pinned arrays."""

    def __init__(self, case, seed):
        self.server = None
        self.reqs = _requests(case)
        self.rhs = [_request_input(r, seed).cpu().pin_memory() for r in self.reqs]
        self.phi = [torch.empty_like(f).pin_memory() for f in self.rhs]
        self.c = [S.c_request(r) for r in self.reqs]
        self.server = F.flups_server_create(8 << 30, 8)

    def __del__(self):
        if self.server is not None:
            F.flups_server_destroy(self.server)


def _requests(case):
    sizes = [s for s in (32, 48, 64, 96, 128) if s <= case["nmax"]]
    return W.served_stream(nreq=case["count"], seed=case["stream"], sizes=sizes)


def _request_case(r):
    def name(f):
        if f[0] == F.PER:
            return "PER"
        s = "".join({F.EVEN: "E", F.ODD: "O", F.UNB: "U"}[v] for v in f)
        return "UNB" if s == "UU" else s
    c = _case("", r.n, tuple(name(f) for f in r.bc), "f32" if r.prec == F.F32 else "f64",
              op="biot" if r.op == F.BIOT_SAVART else "poisson")
    del c["name"]
    return c


def _request_input(r, seed):
    return _field(_request_case(r), int(seed) * 1009 + r.rid)


def prepare(case, seed):
    if case["kind"] == "served":
        return _Burst(case, seed)
    rhs = _field(case, seed)
    st = {"case": case, "rhs": rhs}
    if case["kind"] == "host":
        st["rhs"] = rhs.cpu().pin_memory()
        st["phi"] = torch.empty_like(st["rhs"]).pin_memory()
    else:
        st["phi"] = torch.empty_like(rhs)
    if case["kind"] != "plan":
        st["solver"] = _solver(case)
    return st


def run(state):
    if isinstance(state, _Burst):
        left = {F.flups_server_submit(state.server, c, f, p)
                for c, f, p in zip(state.c, state.rhs, state.phi)}
        while left:
            for ticket, _, status in F.flups_server_wait(state.server):
                if status != 0:
                    raise RuntimeError(f"request failed: {status}")
                left.discard(ticket)
        return state.phi
    kind = state["case"]["kind"]
    if kind == "host":
        state["solver"].solve_host(state["phi"], state["rhs"])
    elif kind == "plan":
        s = _solver(state["case"])
        s.solve(state["phi"], state["rhs"])
        torch.cuda.current_stream().synchronize()  # a plan is released when its solve is over
        s.close()
    else:
        state["solver"].solve(state["phi"], state["rhs"])
    return state["phi"]


# --------------------------------------------------------------------------------------------------
# What a pass cannot do without, and how close another correct solver comes.
# --------------------------------------------------------------------------------------------------
def work(case):
    """Right-hand side read and solution written once; a real FFT forward and back (2.5 M log2 M each) on the
    smallest periodic domain: N points in periodic and wall-bounded directions, 2 N in directions with an open face."""
    if case["kind"] == "served":
        parts = [work(dict(_request_case(r), kind="solve")) for r in _requests(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    n, _, _ = _geom(case)
    nc = 3 if case["op"] == "biot" else 1
    m = 1.0
    for d in "xyz":
        m *= case["n" + d] * (2 if "U" in case[d] else 1)
    return {"bytes": 2.0 * nc * n[0] * n[1] * n[2] * (4 if case["prec"] == "f32" else 8),
            "flops": nc * 2 * 2.5 * m * math.log2(m)}


def tolerance(case):
    # four times the largest error against exact() over listed and drawn cases: f32 2.7e-7, f64 1.8e-15,
    # f64e 7.9e-15
    if case["kind"] == "served" or case["prec"] == "f32":
        return {"rel": 1.2e-6}
    return {"rel": 3.2e-14} if case["prec"] == "f64e" else {"rel": 8e-15}


# --------------------------------------------------------------------------------------------------
# The same solve in plain torch, 64 bits: explicit periodic extensions, FFTs over the extended box.
# --------------------------------------------------------------------------------------------------
SWAP = {"E": "O", "O": "E", "U": "U"}


def _extend(f, ax, t, node):
    """Periodic extension of f along ax for face letters t (or PER / UNB)."""
    if t in ("UE", "UO"):
        return _extend(f.flip(ax), ax, t[::-1], node)
    cat = lambda *p: torch.cat(p, dim=ax)  # noqa: E731
    N = f.shape[ax] - (1 if node and t != "PER" else 0)
    sl = lambda a, b: f.narrow(ax, a, b - a)  # noqa: E731
    if t == "PER":
        return f
    if not node:
        if t == "UNB":
            return cat(f, torch.zeros_like(f))
        r = f.flip(ax)
        if t in ("EE", "OO"):
            return cat(f, r if t == "EE" else -r)
        if t in ("EO", "OE"):
            half = cat(f, -r if t == "EO" else r)
            return cat(half, -half)
        z = torch.zeros_like(f)
        return cat(f, z, z, r if t == "EU" else -r)
    if t == "UNB":
        return cat(f, torch.zeros_like(sl(1, N)))
    f = f.clone()
    if t[0] == "O":
        f.narrow(ax, 0, 1).zero_()
    if t[1] == "O":
        f.narrow(ax, N, 1).zero_()
    sl = lambda a, b: f.narrow(ax, a, b - a)  # noqa: E731
    r = sl(1, N).flip(ax)
    if t in ("EE", "OO"):
        return cat(f, r if t == "EE" else -r)
    if t in ("EO", "OE"):
        half = cat(f, -r if t == "EO" else r)
        return cat(half, -half)
    pad = torch.zeros_like(f.narrow(ax, 0, 1)).expand(*[2 * N - 1 if d == ax else s for d, s in enumerate(f.shape)])
    back = sl(1, N + 1).flip(ax)
    return cat(f, pad, back if t == "EU" else -back)


def _restrict(e, ax, t, node, n):
    o = e.narrow(ax, 0, n)
    if t in ("UE", "UO"):
        o = o.flip(ax)
    o = o.clone()
    if node and t != "PER" and t != "UNB":
        if t[0] == "O":
            o.narrow(ax, 0, 1).zero_()
        if t[1] == "O":
            o.narrow(ax, n - 1, 1).zero_()
    return o


def _e1(s):
    """Exponential integral E1(s), s > 0: int_0^inf exp(-s e^u) du over 60 panels of 16 Gauss-Legendre nodes."""
    x, w = np.polynomial.legendre.leggauss(16)
    umax = torch.log(60.0 / s.clamp(max=30.0) + 1.0)
    acc = torch.zeros_like(s)
    for p in range(60):
        for xi, wi in zip(x, w):
            u = umax * ((p + 0.5 * (float(xi) + 1.0)) / 60)
            acc += float(wi) * 0.5 * umax / 60 * torch.exp(-s * torch.exp(u))
    return acc


def _green(types, P, h):
    """Spectrum of the smoothed Green's function on folded modes [z, y, x] (P/2 + 1 each), eps = 2 h."""
    half = [torch.arange(p // 2 + 1, device=DEV, dtype=torch.float64) for p in P]
    unb = ["U" in t for t in types]
    shape = lambda v, d: v.reshape([-1 if 2 - d == a else 1 for a in range(3)])  # noqa: E731
    k2 = sum((shape((2 * math.pi * half[d] / (P[d] * h)) ** 2, d) for d in range(3) if not unb[d]),
             torch.zeros(1, 1, 1, device=DEV, dtype=torch.float64))
    du = sum(unb)
    if du == 0:
        return torch.where(k2 > 0, -1.0 / k2.clamp(min=1e-300), torch.zeros_like(k2))
    r2 = sum(shape((half[d] * h) ** 2, d) for d in range(3) if unb[d])
    eps = 2.0 * h
    if du == 3:
        r = r2.sqrt()
        g = torch.where(r > 0, -torch.erf(r / (math.sqrt(2) * eps)) / (4 * math.pi * r.clamp(min=1e-300)),
                        torch.full_like(r, -1.0 / ((2 * math.pi) ** 1.5 * eps)))
    elif du == 1:
        k, z = torch.broadcast_tensors(k2.sqrt(), r2.sqrt())
        a, b = k * eps / math.sqrt(2), z / (math.sqrt(2) * eps)
        gauss = torch.exp(-a * a - b * b)
        minus = torch.where(a >= b, torch.special.erfcx((a - b).clamp(min=0)) * gauss,
                            torch.exp(-k * z) * torch.erfc((a - b).clamp(max=0)))
        g = -(minus + torch.special.erfcx(a + b) * gauss) / (4 * k.clamp(min=1e-300))
        g0 = 0.5 * z * torch.erf(b) + eps / math.sqrt(2 * math.pi) * torch.exp(-b * b)
        g = torch.where(k > 0, g, g0)
    else:
        # -(1/4 pi) int_0^inf exp(-a e^s - b e^-s) ds over each wavenumber's own range
        d0 = [d for d in range(3) if not unb[d]][0]
        plane = r2.squeeze()
        ks = k2.reshape(-1)
        b = plane / (2 * eps * eps)
        x, w = np.polynomial.legendre.leggauss(24)
        out = []
        for k in ks.tolist():
            if k == 0.0:
                rr = plane.sqrt()
                g = (torch.log(rr.clamp(min=1e-300)) + 0.5 * _e1(b.clamp(min=1e-300))) / (2 * math.pi)
                out.append(torch.where(rr > 0, g, torch.full_like(rr, (math.log(2 * eps * eps) - 0.57721566490153286061) /
                                                                 (4 * math.pi))))
                continue
            a = k * eps * eps / 2
            smax = math.log(max(60.0 / a, math.e))
            npan = max(1, math.ceil(smax / 0.5))
            acc = torch.zeros_like(b)
            for p in range(npan):
                for xi, wi in zip(x, w):
                    s = (p + 0.5 * (float(xi) + 1)) * smax / npan
                    acc.add_(torch.exp(-a * math.exp(s) - b * math.exp(-s)), alpha=float(wi) * 0.5 * smax / npan)
            out.append(acc / (-4 * math.pi))
        g = torch.stack(out, dim=2 - d0)
    for d in range(3):
        if unb[d]:
            idx = torch.arange(P[d], device=DEV)
            idx = torch.minimum(idx, P[d] - idx)
            g = h * torch.fft.rfft(g.index_select(2 - d, idx), dim=2 - d).real
    return g


def _exact_solve(case, f):
    n, hs, _ = _geom(case)
    h, node, biot = hs[0], case["center"] == "node", case["op"] == "biot"
    types = [case[d] for d in "xyz"]
    comps = [f] if not biot else list(f)

    def source(c, d):  # faces of source component c: the normal component takes the other parity at a wall
        t = types[d]
        return "".join(SWAP[x] for x in t) if biot and c == d and t not in ("PER", "UNB") else t

    def result(c, d):  # faces of the curl's component c: d_a f_b, a = c + 1, b = c + 2
        a, b = (c + 1) % 3, (c + 2) % 3
        t = source(b, d)
        return "".join(SWAP[x] for x in t) if d == a and t not in ("PER", "UNB") else t

    spec = []
    for c, e in enumerate(comps):
        e = e.double()
        for d in range(3):
            e = _extend(e, 2 - d, source(c, d), node)
        P = [e.shape[2], e.shape[1], e.shape[0]]
        spec.append(torch.fft.rfftn(e))
        del e
    G = _green(types, P, h)
    for d in (1, 2):
        idx = torch.arange(P[d], device=DEV)
        G = G.index_select(2 - d, torch.minimum(idx, P[d] - idx)) if G.shape[2 - d] > 1 else G
    if biot:
        ik = []
        for d in range(3):
            m = torch.arange(P[d] if d else P[0] // 2 + 1, device=DEV, dtype=torch.float64)
            m = torch.where(2 * m > P[d], m - P[d], m)
            m = torch.where(2 * m.abs() == P[d], torch.zeros_like(m), m)
            w = (2j * math.pi / (P[d] * h)) * m
            ik.append(w.reshape([-1 if 2 - d == a else 1 for a in range(3)]))
        spec = [ik[(c + 1) % 3] * spec[(c + 2) % 3] - ik[(c + 2) % 3] * spec[(c + 1) % 3] for c in range(3)]
    out = []
    while spec:
        u = torch.fft.irfftn(spec.pop(0).mul_(G), s=(P[2], P[1], P[0]))
        for d in range(3):
            u = _restrict(u, 2 - d, result(len(out), d) if biot else types[d], node, n[d])
        out.append(u)
    return torch.stack(out) if biot else out[0]


def exact(case, seed):
    if case["kind"] == "served":
        return [_exact_solve(_request_case(r), _request_input(r, seed)).cpu() for r in _requests(case)]
    u = _exact_solve(case, _field(case, seed))
    return u.cpu() if case["kind"] == "host" else u
