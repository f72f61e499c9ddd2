"""The workloads a user runs, as timed cases: the fields of one scene at its
receivers (FP32 and FP64), the path lists, a batch of moving frames, a
gradient step, and the large office from its ray launch on.

`prepare` makes the inputs of a case on the GPU, `run` is one pass through the
public calls of `paper_2310_10578_gb300.creep`, `exact` the same outputs in 64
bits from the method's formulas (image method, Fermat reflection points,
creeping geodesics, Fock--Pekeris functions), written with torch and numpy
only.  Scenes come from `scenes.py` at the sizes of the benchmark, of the
tests, or between them.
"""
import functools
import math

import numpy as np
import torch

from paper_2310_10578_gb300 import creep, scenes

C0 = 299792458.0
WALLS = (5.0, 0.3)          # permittivity of the dielectric walls (eps', eps'')
FLOOR = (4.0, 0.2)
BAND3 = (2.4e9, 5.8e9, 28e9)


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # the analytic-sphere validation: one body, no walls, a short call
        dict(name="ring", kind="field", scene="ring", n_rx=4096, freqs=1),
        # a few probe points in a furnished room: latency and launches
        dict(name="probe", kind="field", scene="room", cyl=20, n_rx=97, freqs=3),
        # the headline workload: the signal map of a room with people
        dict(name="room", kind="field", scene="room", cyl=20, nx=256, ny=256, freqs=3),
        # a fine map of a sparser room at one frequency, odd grid
        dict(name="map", kind="field", scene="room", cyl=7, nx=811, ny=643, freqs=1),
        # the room in FP64, as a reference solution is computed
        dict(name="room_fp64", kind="field", scene="room", cyl=20, nx=173, ny=139, freqs=3, fp64=True),
        # dielectric walls, creeping rays with extra turns and off the walls
        dict(name="extended", kind="field", scene="room", cyl=20, nx=131, ny=127, freqs=3, ext=True, enc=2),
        # which paths reach each receiver (canonical lists)
        dict(name="paths", kind="paths", scene="room", cyl=20, nx=122, ny=94, freqs=1),
        # one gradient step of a dense crowd (FP64 adjoint, the default)
        dict(name="grad_dense", kind="grad", scene="room", cyl=200, nx=64, ny=64, freqs=1),
        # a gradient step of a small room over a band, FP32 adjoint
        dict(name="grad_band", kind="grad", scene="room", cyl=12, nx=61, ny=47, freqs=3, grad32=True),
        # walking people: frames with their own bodies, band and receivers
        dict(name="crowd", kind="batch", frames=24, cyl=50, freqs=16, rx_lo=1000, rx_hi=65536),
        # one floor section: ray launch, then reflections to order 3
        dict(name="office_floor", kind="office", rx=4, ry=3, furn=600, cyl=4, sph=1, nx=250, ny=160),
        # the whole building, one transmitter
        dict(name="office", kind="office", rx=20, ry=15, furn=15000, cyl=100, sph=10, nx=1250, ny=800),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["ring", "room", "room", "room", "points", "fp64", "ext", "paths", "grad", "batch", "office"])
    if kind == "ring":
        return dict(kind="field", scene="ring", n_rx=_log(rng, 200, 60000), freqs=_log(rng, 1, 8),
                    fp64=rng.random() < 0.3)
    if kind == "points":
        return dict(kind="field", scene="room", cyl=_log(rng, 1, 60), n_rx=_log(rng, 1, 4000), freqs=_log(rng, 1, 16))
    if kind == "room":
        nx = _log(rng, 40, 800)
        return dict(kind="field", scene="room", cyl=_log(rng, 1, 60), nx=nx, ny=max(1, int(nx * rng.uniform(0.5, 0.9))),
                    freqs=_log(rng, 1, 16))
    if kind == "fp64":
        nx = _log(rng, 10, 180)
        return dict(kind="field", scene="room", cyl=_log(rng, 1, 30), nx=nx, ny=max(1, int(nx * rng.uniform(0.5, 0.9))),
                    freqs=_log(rng, 1, 8), fp64=True)
    if kind == "ext":
        nx = _log(rng, 20, 140)
        return dict(kind="field", scene="room", cyl=_log(rng, 1, 20), nx=nx, ny=max(1, int(nx * rng.uniform(0.5, 0.9))),
                    freqs=_log(rng, 1, 6), ext=True, enc=rng.randrange(3))
    if kind == "paths":
        nx = _log(rng, 10, 250)
        return dict(kind="paths", scene="room", cyl=_log(rng, 1, 60), nx=nx, ny=max(1, int(nx * rng.uniform(0.5, 0.9))),
                    freqs=1)
    if kind == "grad":
        nx = _log(rng, 12, 90)
        return dict(kind="grad", scene="room", cyl=_log(rng, 4, 200), nx=nx, ny=max(1, int(nx * rng.uniform(0.5, 0.9))),
                    freqs=_log(rng, 1, 4), grad32=rng.random() < 0.3)
    if kind == "batch":
        lo = _log(rng, 30, 3000)
        return dict(kind="batch", frames=_log(rng, 2, 30), cyl=_log(rng, 3, 60), freqs=_log(rng, 1, 16), rx_lo=lo,
                    rx_hi=_log(rng, lo, 60000))
    rx, ry = rng.randint(2, 8), rng.randint(2, 6)
    cells = rx * ry
    return dict(kind="office", rx=rx, ry=ry, furn=int(cells * rng.uniform(10, 50)), cyl=max(2, cells // 3),
                sph=max(1, cells // 30), nx=int(rx * rng.uniform(16, 60)), ny=int(ry * rng.uniform(16, 50)))


# ------------------------------------------------------------------ inputs
def _freqs(n, rng):
    if n <= 3:
        return np.asarray(BAND3[1:2] if n == 1 else BAND3[:n])
    return np.sort(rng.uniform(2.4e9, 28e9, n))


def _frame_rx(case):
    """Receivers per frame of a batch, log-uniform: part of its shape, the same for every seed."""
    rng = np.random.default_rng(case["frames"])
    lo, hi = math.log(case["rx_lo"]), math.log(case["rx_hi"])
    return [int(round(math.exp(x))) for x in rng.uniform(lo, hi, case["frames"])]


def _scene(case, seed):
    """The scene of a case (a scenes.Scene, or a scenes.Crowd for a batch)."""
    rng = np.random.default_rng([seed, 77])
    if case["kind"] == "batch":
        cw = scenes.crowd(n_frames=case["frames"], n_cyl=case["cyl"], n_freq=case["freqs"],
                          rx_range=(case["rx_hi"], case["rx_hi"]), seed=seed)
        cw.rx = [r[:n] for r, n in zip(cw.rx, _frame_rx(case))]
        return cw
    if case["kind"] == "office":
        return scenes.office(n_rooms=(case["rx"], case["ry"]), n_furn=case["furn"], n_cyl=case["cyl"],
                             n_sph=case["sph"], n_tx=1, nx=case["nx"], ny=case["ny"], seed=seed)
    f = _freqs(case["freqs"], rng)
    if case["scene"] == "ring":
        n = case["n_rx"]
        sc = scenes.sphere_ring(n_rx=n, radius=float(rng.uniform(0.3, 0.6)))
        # receivers off the axis through the source, where a creeping ray has its caustic
        phi = 2.0 * np.pi * (np.arange(n) + rng.uniform(0.2, 0.8)) / n
        sc.rx = np.stack([2.0 * np.cos(phi), 2.0 * np.sin(phi), np.zeros(n)], axis=1).astype(np.float32)
        sc.freqs = np.sort(rng.uniform(2.0e9, 8.0e9, case["freqs"]))
        return sc
    eps = [FLOOR, None, WALLS, WALLS, WALLS, WALLS] if case.get("ext") else None
    sc = scenes.room(n_cyl=case["cyl"], nx=case.get("nx", 1), ny=case.get("ny", 1), freqs=f, seed=seed, face_eps=eps)
    if "n_rx" in case:
        n = case["n_rx"]
        sc.rx = np.stack([rng.uniform(0.1, 9.9, n), rng.uniform(0.1, 7.9, n), rng.uniform(0.8, 1.6, n)],
                         axis=1).astype(np.float32)
    if case["kind"] == "grad":
        # off the grid: a path point on a face's edge has a one-sided derivative
        sc.rx = (sc.rx + rng.uniform(-0.02, 0.02, sc.rx.shape)).astype(np.float32)
    sc.max_enc = case.get("enc", 0)
    sc.wall_creep = bool(case.get("ext"))
    return sc


def _cotangent(case, seed, n_f, n_rx):
    """dLoss/dE of a gradient step: a weighted zone."""
    g = np.random.default_rng([seed, 5]).standard_normal((n_f, 3, n_rx, 2))
    return g.astype(np.float32)


def _options(case, sc):
    enable = creep.RT_EN_ALL | (creep.RT_EN_WALL_CREEP if getattr(sc, "wall_creep", False) else 0)
    return creep.options(max_order=sc.max_order, enable=enable, max_encirclements=getattr(sc, "max_enc", 0),
                         precision=creep.RT_PREC_FP64 if case.get("fp64") else creep.RT_PREC_FP32)


def prepare(case, seed):
    sc = _scene(case, seed)
    st = {"kind": case["kind"], "opts": _options(case, sc)}
    if case["kind"] == "batch":
        S = creep.Scene(sc.tri, sc.tri_face, np.zeros((0, 6)))
        S.set_tx(sc.tx, sc.pol)
        S.set_freqs(sc.freqs[0])
        B = creep.Batch(S, sc.n_rx, case["freqs"], case["cyl"])
        for i in range(sc.n_frames):
            B.set_frame(i, sc.bodies[i], sc.freqs[i])
        rx = torch.from_numpy(B.rx_pack([np.ascontiguousarray(r.T) for r in sc.rx])).cuda()
        st.update(scene=S, batch=B, rx=rx, out=torch.empty(6 * case["freqs"] * B.total_rx, device="cuda"))
        # a program that evaluates the frames again and again replays them
        side = torch.cuda.Stream()
        B.evaluate(rx, st["out"], opts=st["opts"])
        torch.cuda.synchronize()
        B.capture(rx, st["out"], opts=st["opts"], stream=side)
        torch.cuda.synchronize()
        return st
    S = creep.Scene.from_scene(sc)
    st.update(scene=S, rx=torch.from_numpy(sc.rx_soa()).cuda(),
              out=torch.empty((S.n_f, 3, sc.n_rx, 2), device="cuda"))
    if case["kind"] == "grad":
        st["gE"] = torch.from_numpy(_cotangent(case, seed, S.n_f, sc.n_rx)).cuda()
        st["gopts"] = creep.options(max_order=2, precision=creep.RT_PREC_FP32 if case.get("grad32")
                                    else creep.RT_PREC_FP64)
    return st


def run(st):
    S = st["scene"]
    if st["kind"] == "batch":
        st["batch"].replay()
        return st["out"]
    if st["kind"] == "office":
        S.candidates_device(4096, 3)
        return S.evaluate(st["rx"], st["out"], opts=st["opts"])
    if st["kind"] == "paths":
        return S.paths(st["rx"], opts=st["opts"])
    if st["kind"] == "grad":
        E, codes, counts, _ = S.evaluate_with_paths(st["rx"], out=st["out"], opts=st["opts"])
        return (E, counts) + S.backward(st["rx"], codes, counts, st["gE"], opts=st["gopts"])
    return S.evaluate(st["rx"], st["out"], opts=st["opts"])


def work(case):
    """Receivers in, fields (or path codes) out; each candidate path's geometry
    once per receiver (60 flops an image path, 150 a body's ray, each with one
    segment test), one phase (30) a direct ray and frequency."""
    if case["kind"] == "batch":
        n, bodies, faces = sum(_frame_rx(case)), case["cyl"], 6
    elif case["kind"] == "office":
        n, bodies, faces = case["nx"] * case["ny"], case["cyl"] + case["sph"], 12
    elif case["scene"] == "ring":
        n, bodies, faces = case["n_rx"], 1, 0
    else:
        n, bodies, faces = case.get("n_rx", case.get("nx", 0) * case.get("ny", 0)), case["cyl"], 6
    nf = case.get("freqs", 1)
    image = 1 + faces * faces
    rays = 1 + 2 * (1 + case.get("enc", 0)) * (1 + (faces if case.get("ext") else 0))
    flops = n * (image * 85 + bodies * rays * 175 + nf * 30)
    out = 8 * 256 + 8 if case["kind"] == "paths" else 24 * nf
    if case["kind"] == "grad":
        flops *= 9                      # a path's field with its eight derivatives
        out += 24 * nf
    return {"bytes": n * (12 + out) + bodies * 64 + faces * 150, "flops": flops}


# ------------------------------------------------------------------ 64-bit values
def exact(case, seed):
    if case["kind"] == "paths":
        return None
    sc = _scene(case, seed)
    if case["kind"] == "batch":
        parts = []
        for i in range(sc.n_frames):
            with torch.no_grad():
                parts.append(_real(_Field(sc.frame(i)).total()).reshape(-1))
        return torch.cat(parts)
    if case["kind"] == "office":
        if sc.n_rx * len(sc.tri) > 4e8:
            return None
        with torch.no_grad():
            F = _Field(sc)
            return _real(F.total(F.launch(4096, 3)))
    F = _Field(sc)
    if case["kind"] != "grad":
        with torch.no_grad():
            return _real(F.total())
    for t in (F.body, F.tx, F.freq):
        t.requires_grad_(True)
    E = _real(F.total())
    g = torch.from_numpy(_cotangent(case, seed, E.shape[0], E.shape[2])).to(E)
    gb, gt, gf = torch.autograd.grad((E * g).sum(), (F.body, F.tx, F.freq))
    return E.detach(), None, gb, gt, gf


def _real(E):
    return torch.view_as_real(E.resolve_conj().contiguous())


def _airy(z):
    """Ai and Ai' of complex z, |arg z| < 2 pi / 3: Maclaurin series to |z| = 7, the asymptotic series beyond."""
    z = np.asarray(z, dtype=complex)
    a0, b0 = 0.35502805388781723926, 0.25881940379280679841
    f, g, df, dg = np.ones_like(z), z.copy(), np.zeros_like(z), np.ones_like(z)
    s = np.where(np.abs(z) <= 7.0, z, 0.0)
    z3, tf, tg = s ** 3, np.ones_like(z), s.copy()
    g = s.copy()
    for k in range(1, 90):
        tdf = tf * s * s / (3 * k - 1)
        tdg = tg * s * s / (3 * k)
        tf, tg = tf * z3 / ((3 * k - 1) * (3 * k)), tg * z3 / ((3 * k) * (3 * k + 1))
        f, g, df, dg = f + tf, g + tg, df + tdf, dg + tdg
    ai, dai = a0 * f - b0 * g, a0 * df - b0 * dg
    l = np.where(np.abs(z) > 7.0, z, 8.0)
    ze = 2.0 / 3.0 * l ** 1.5
    u, su, sv = 1.0, np.ones_like(l), np.ones_like(l)
    for k in range(1, 22):
        u *= (6 * k - 5) * (6 * k - 3) * (6 * k - 1) / (216.0 * k * (2 * k - 1))
        t = (-1) ** k * u / ze ** k
        su, sv = su + t, sv - t * (6 * k + 1) / (6 * k - 1)
    h = np.exp(-ze) / (2.0 * math.sqrt(math.pi))
    big = np.abs(z) > 7.0
    return np.where(big, h * su / l ** 0.25, ai), np.where(big, -h * sv * l ** 0.25, dai)


def _airy_neg(x):
    """Ai(-x), Ai'(-x) for real x > 0, from the two turned arguments."""
    w = np.exp(1j * np.pi / 3)
    (p, dp), (q, dq) = _airy(x * w), _airy(x / w)
    return (w * p + q / w).real, -(w * w * dp + dq / (w * w)).real


@functools.lru_cache(maxsize=None)
def _fock():
    """Chebyshev pieces (width 1/4) of the regular Fock--Pekeris functions on
    [-10, 1.5], and the creeping-mode constants of the residue series above."""
    om, pref = np.exp(2j * np.pi / 3), np.exp(-1j * np.pi / 4) / math.sqrt(math.pi)
    gx, gw = np.polynomial.legendre.leggauss(16)

    def rule(a, b):
        m = max(1, int(math.ceil((b - a) / 0.25)))
        e = np.linspace(a, b, m + 1)
        h = (e[1:] - e[:-1]) / 2
        return ((e[1:] + e[:-1])[:, None] / 2 + h[:, None] * gx).ravel(), (h[:, None] * gw).ravel()

    def left(x, dx):                       # W1/(2j W2) at tau = -x, both kinds
        (p, dp), (q, dq) = _airy(-x * om), _airy(-x / om)
        r = np.exp(1j * np.pi / 3)
        return -x, dx * r * p / q / 2j, dx * r * om * om * dp / dq / 2j

    n = 24
    t = np.cos(np.pi * (np.arange(n) + 0.5) / n)
    coef = []
    for piece in range(46):
        xi = -10.0 + 0.25 * (piece + 0.5 + 0.5 * t)
        u, w = rule(0.0, 14.0)
        r = np.exp(1j * np.pi / 6)
        (p, dp), (q, dq) = _airy(u * r), _airy(u * r / om)
        parts = [(u * r, w * r * p / q * np.exp(1j * np.pi / 6) / 2.0,
                  w * r * dp / dq * om * np.exp(1j * np.pi / 6) / 2.0)]
        x0 = min(xi.min(), 0.0) ** 2 / 4.0
        if x0 > 0.0:
            x, w = rule(0.0, x0)
            parts.append(left(x.astype(complex), w))
        u, w = rule(0.0, 12.0)
        r = np.exp(1j * np.pi / 4)
        parts.append(left(x0 + u * r, w * r))
        val = sum(np.exp(-1j * xi[:, None] * tau) @ np.stack([a, b], 1) for tau, a, b in parts) * pref
        k = np.arange(n)
        T = np.cos(np.pi * k[:, None] * (np.arange(n) + 0.5) / n)
        cf = 2.0 / n * T @ val
        cf[0] /= 2.0
        coef.append(cf)
    zs, cs = [], []
    for hard in (False, True):
        i = np.arange(1, 17)
        x = (3.0 * np.pi * (4 * i - (3 if hard else 1)) / 8.0) ** (2.0 / 3.0)
        for _ in range(8):
            a, d = _airy_neg(x)
            x = x + (d / (-x * a) if hard else a / d)
        a, d = _airy_neg(x)
        zs.append(x)
        cs.append(1.0 / (x * a * a) if hard else 1.0 / (d * d))
    return np.stack(coef), np.stack(zs), np.stack(cs)


def _faddeeva(z):
    """w(z), Im z > 0 (Weideman's rational approximation, 48 terms)."""
    a, L = _weideman(48)
    den = L - 1j * z
    Z = (L + 1j * z) / den
    p = torch.full_like(z, a[-1])
    for c in a[-2::-1]:
        p = p * Z + c
    return 2.0 * p / den ** 2 + (1.0 / math.sqrt(math.pi)) / den


@functools.lru_cache(maxsize=None)
def _weideman(N):
    M, L = 2 * N, math.sqrt(N / math.sqrt(2.0))
    t = L * np.tan(np.arange(-M + 1, M) * np.pi / (2 * M))
    f = np.exp(-t * t) * (L * L + t * t)
    k = np.arange(-M + 1, M)
    return [float(np.sum(f * np.cos(n * k * np.pi / M)) / (2 * M)) for n in range(1, N + 1)], L


def _bracket(xi, K):
    """P + (c/xi)(1 - F(X)), X = (K xi)^2, soft and hard."""
    coef, zs, cs = _fock()
    dev = xi.device
    c = complex(np.exp(-1j * np.pi / 4) / (2.0 * math.sqrt(math.pi)))
    low = xi <= 1.5
    x = torch.where(low, xi, torch.full_like(xi, 1.0))
    j = ((x.detach() + 10.0) * 4.0).floor().clamp(0, 45).long()
    t = 2.0 * ((x + 10.0) * 4.0 - j) - 1.0
    C = torch.from_numpy(coef).to(dev)[j]                           # [..., n, 2]
    b1 = b2 = torch.zeros_like(C[..., 0, :])
    for k in range(coef.shape[1] - 1, 0, -1):
        b1, b2 = 2.0 * t[..., None] * b1 - b2 + C[..., k, :], b1
    reg = t[..., None] * b1 - b2 + C[..., 0, :]                     # P + c/xi
    y = torch.where(low, torch.full_like(xi, 2.0), xi)
    e = complex(np.exp(1j * np.pi / 6))
    pre = complex(-np.exp(-1j * np.pi / 12) / (2.0 * math.sqrt(math.pi)))
    res = pre * torch.stack([sum(float(cs[h, i]) * torch.exp(-y * (float(zs[h, i]) * e)) for i in range(zs.shape[1]))
                             for h in (0, 1)], dim=-1)              # P
    s = K * xi.abs()
    near = s * s <= 4.0
    sn = torch.where(near, s, torch.full_like(s, 1.0))
    w = _faddeeva(sn * complex(np.exp(3j * np.pi / 4)))
    f_xi = torch.sign(xi) * math.sqrt(math.pi) * K * complex(np.exp(1j * np.pi / 4)) * w
    f_near = (torch.where(low[..., None], reg, res + (c / y)[..., None])) - (c * f_xi)[..., None]
    sf = torch.where(near, torch.full_like(s, 3.0), s)
    mid = sf * sf <= 36.0
    sm = torch.where(mid, sf, torch.full_like(s, 3.0))
    F = math.sqrt(math.pi) * sm * complex(np.exp(1j * np.pi / 4)) * _faddeeva(sm * complex(np.exp(3j * np.pi / 4)))
    u = 0.5 / torch.where(mid, torch.full_like(s, 40.0), sf * sf)
    acc = torch.ones_like(u) + 0j
    for n in range(16, 1, -1):
        acc = 1.0 + (2 * n - 1) * u * 1j * acc
    omf = torch.where(mid, 1.0 - F, -1j * u * acc)
    xs = torch.where(near, torch.full_like(xi, 1.0), xi)
    P = torch.where(low[..., None], reg - (c / torch.where(low, xs, x))[..., None], res)
    f_far = P + (c / xs * omf)[..., None]
    out = torch.where(near[..., None], f_near, f_far)
    return out[..., 0], out[..., 1]


def _dot(a, b):
    return (a * b).sum(-1)


def _unit(a):
    return a / a.norm(dim=-1, keepdim=True)


class _Field:
    """The coherent field of a scene at its receivers in 64 bits.  Candidates are
    decided on the values; the field of the valid ones is differentiable in
    body [n, 4] (centre, radius), tx and freq."""

    def __init__(self, sc):
        dev = "cuda" if torch.cuda.is_available() else "cpu"
        d = functools.partial(torch.tensor, dtype=torch.float64, device=dev)
        self.tri = d(np.asarray(sc.tri, dtype=np.float64).reshape(-1, 3, 3))
        self.face = torch.tensor(np.asarray(sc.tri_face, dtype=np.int64).reshape(-1), device=dev)
        b = np.asarray(sc.bodies, dtype=np.float64).reshape(-1, 6)
        self.body, self.tall = d(b[:, 1:5]), d(b[:, 5])
        self.cyl = torch.tensor(b[:, 0] == 1, device=dev)
        self.tx, self.pol, self.freq = d(sc.tx), d(sc.pol), d(sc.freqs)
        self.P = d(sc.rx)
        self.order, self.enc, self.wall = sc.max_order, getattr(sc, "max_enc", 0), getattr(sc, "wall_creep", False)
        fe = getattr(sc, "face_eps", None)
        self.eps = [None if fe is None or fe[f][0] == 0 else complex(fe[f][1], -fe[f][2])
                    for f in range(0 if fe is None else len(fe))]
        self.n_face = int(self.face.max()) + 1 if len(self.face) else 0
        first = torch.full((self.n_face,), -1, dtype=torch.long, device=dev)
        for t in range(len(self.face) - 1, -1, -1) if len(self.face) < 2000 else ():
            first[self.face[t]] = t
        if len(self.face) >= 2000:
            first = torch.tensor(np.unique(self.face.cpu().numpy(), return_index=True)[1], device=dev)
        v = self.tri[first]
        self.nrm = _unit(torch.cross(v[:, 1] - v[:, 0], v[:, 2] - v[:, 0], dim=-1)) if self.n_face else v[:, 0]
        self.off = _dot(self.nrm, v[:, 0])
        self.lists = [torch.nonzero(self.face == f)[:, 0] for f in range(self.n_face)] if self.n_face <= 64 else None
        self.ok = torch.nonzero(~self.inside())[:, 0]
        n = len(self.P)
        self.E = torch.zeros((len(self.freq), 3, n), dtype=torch.complex128, device=dev)

    # ---- decisions
    def inside(self):
        c, a = self.body[:, :3].detach(), self.body[:, 3].detach()
        out = torch.zeros(len(self.P), dtype=torch.bool, device=self.P.device)
        for i in range(len(c)):
            w = self.P - c[i]
            if self.cyl[i]:
                out |= (w[:, 0] ** 2 + w[:, 1] ** 2 <= a[i] ** 2) & (w[:, 2] >= 0) & (w[:, 2] <= self.tall[i])
            else:
                out |= _dot(w, w) <= a[i] ** 2
        return out

    @torch.no_grad()
    def clear(self, A, B, skip=(), skip_body=None):
        """The open segments A -> B free of every triangle (but those of the faces
        in skip) and body (but skip_body)."""
        out = torch.ones(len(A), dtype=torch.bool, device=A.device)
        step = max(1, int(4e6 // max(1, len(self.tri), len(self.body))))
        for i in range(0, len(A), step):
            s = slice(i, i + step)
            out[s] = self._clear(A[s], B[s], [f[s] if torch.is_tensor(f) else f for f in skip],
                                 None if skip_body is None else skip_body[s])
        return out

    def _clear(self, A, B, skip, skip_body):
        eps = 1e-6
        hit = torch.zeros(len(A), dtype=torch.bool, device=A.device)
        D = B - A
        if len(self.tri):
            v0 = self.tri[:, 0]
            e1, e2 = self.tri[:, 1] - v0, self.tri[:, 2] - v0
            T, Dn = A[:, None] - v0, D[:, None].expand(-1, len(v0), -1)
            p = torch.cross(Dn, e2.expand_as(T), dim=-1)
            det = (p * e1).sum(-1)
            inv = 1.0 / torch.where(det == 0, torch.ones_like(det), det)
            q = torch.cross(T, e1.expand_as(T), dim=-1)
            u, v, t = (T * p).sum(-1) * inv, (Dn * q).sum(-1) * inv, (q * e2).sum(-1) * inv
            h = (det != 0) & (u >= 0) & (v >= 0) & (u + v <= 1) & (t >= eps) & (t <= 1 - eps)
            for f in skip:
                h &= self.face[None] != (f[:, None] if torch.is_tensor(f) else f)
            hit |= h.any(1)
        if len(self.body):
            c, a = self.body[:, :3].detach(), self.body[:, 3].detach()
            W = A[:, None] - c
            Dn = D[:, None].expand_as(W)
            t = (-_dot(W, Dn) / _dot(Dn, Dn)).clamp(eps, 1 - eps)
            q = W + Dn * t[..., None]
            sph = _dot(q, q) < a * a
            qa = (Dn[..., :2] ** 2).sum(-1)
            qb = 2.0 * (W[..., :2] * Dn[..., :2]).sum(-1)
            qc = (W[..., :2] ** 2).sum(-1) - a * a
            disc = qb * qb - 4.0 * qa * qc
            sq = disc.clamp(min=0).sqrt()
            qs = torch.where(qa > 0, qa, torch.ones_like(qa))
            inf = torch.full_like(qa, math.inf)
            t1 = torch.where(qa > 0, (-qb - sq) / (2 * qs), torch.where(qc < 0, -inf, inf))
            t2 = torch.where(qa > 0, (-qb + sq) / (2 * qs), torch.where(qc < 0, inf, -inf))
            dz = Dn[..., 2]
            ds = torch.where(dz != 0, dz, torch.ones_like(dz))
            ta, tb = -W[..., 2] / ds, (self.tall - W[..., 2]) / ds
            zin = (W[..., 2] > 0) & (W[..., 2] < self.tall)
            t3 = torch.where(dz != 0, torch.minimum(ta, tb), torch.where(zin, -inf, inf))
            t4 = torch.where(dz != 0, torch.maximum(ta, tb), torch.where(zin, inf, -inf))
            lo, hi = torch.maximum(t1, t3), torch.minimum(t2, t4)
            cy = ((disc > 0) | (qa == 0)) & (lo < hi) & (lo < 1 - eps) & (hi > eps)
            h = torch.where(self.cyl, cy, sph)
            if skip_body is not None:
                h &= torch.arange(len(c), device=A.device) != skip_body[:, None]
            hit |= h.any(1)
        return ~hit

    def in_face(self, f, Q):
        ids = self.lists[f] if self.lists is not None else torch.nonzero(self.face == f)[:, 0]
        out = torch.zeros(len(Q), dtype=torch.bool, device=Q.device)
        for t in ids.tolist():
            v = self.tri[t]
            n = torch.cross(v[1] - v[0], v[2] - v[0], dim=-1)
            m = torch.ones_like(out)
            for k in range(3):
                e = v[(k + 1) % 3] - v[k]
                m &= torch.cross(e.expand_as(Q), Q - v[k], dim=-1) @ n >= 0
            out |= m
        return out

    def mirror(self, X, f):
        return X - self.nrm[f] * (2.0 * (_dot(X, self.nrm[f]) - self.off[f]))[..., None]

    def dist(self, X, f):
        return X @ self.nrm[f] - self.off[f]

    # ---- polarisation
    def launch_pol(self, d):
        p = self.pol - d * _dot(d, self.pol)[:, None]
        return _unit(p) + 0j

    def bounce(self, f, E, si, sr):
        n = self.nrm[f]
        eps = self.eps[f] if f < len(self.eps) else None
        if eps is None:
            return 2.0 * (E @ (n + 0j))[:, None] * n - E
        cth = (si @ n).abs()
        r = torch.sqrt(eps - (1.0 - cth * cth) + 0j)
        gs, gp = (cth - r) / (cth + r), (eps * cth - r) / (eps * cth + r)
        ep = _unit(torch.cross(n.expand_as(si), si, dim=-1))
        a = gs * _dot(E, ep + 0j)
        b = gp * _dot(E, torch.cross(ep, si, dim=-1) + 0j)
        return a[:, None] * ep + b[:, None] * torch.cross(ep, sr, dim=-1)

    def add(self, idx, e, amp, length):
        """Rays of polarisation e [m, 3] (per frequency: [n_f, m, 3]), amplitude, length."""
        k = 2.0 * math.pi * self.freq / C0
        cyc = length[None] * (self.freq / C0)[:, None]
        ph = torch.exp(-2j * math.pi * (cyc - cyc.detach().floor()))
        e = e if e.dim() == 3 else e[None]
        con = (e * (ph * amp)[..., None]).transpose(1, 2)
        self.E = self.E.index_add(2, idx, con)

    # ---- planar paths
    def planar(self, seq):
        k = len(seq)
        X, imgs = self.tx, []
        for f in seq:
            X = self.mirror(X, f)
            imgs.append(X)
        idx, P = self.ok, self.P[self.ok]
        with torch.no_grad():
            keep, Y, Q = torch.ones(len(idx), dtype=torch.bool, device=P.device), P, [None] * k
            for m in range(k - 1, -1, -1):
                di, dy = self.dist(imgs[m], seq[m]), self.dist(Y, seq[m])
                keep &= di * dy < 0
                Q[m] = imgs[m] + (Y - imgs[m]) * (di / (di - dy))[:, None]
                Y = Q[m]
            sel = torch.nonzero(keep)[:, 0]
            for m in range(k):
                if len(sel):
                    sel = sel[self.in_face(seq[m], Q[m][sel])]
            pts = [self.tx.expand_as(P)] + Q + [P]
            for m in range(k + 1):
                if len(sel):
                    skip = [seq[i] for i in (m - 1, m) if 0 <= i < k]
                    sel = sel[self.clear(pts[m][sel], pts[m + 1][sel], skip)]
        if not len(sel):
            return
        idx, P = idx[sel], P[sel]
        Y, Q = P, [None] * k
        for m in range(k - 1, -1, -1):
            di, dy = self.dist(imgs[m], seq[m]), self.dist(Y, seq[m])
            Q[m] = imgs[m] + (Y - imgs[m]) * (di / (di - dy))[:, None]
            Y = Q[m]
        pts = [self.tx.expand_as(P)] + Q + [P]
        L = (P - (imgs[-1] if k else self.tx)).norm(dim=-1)
        s = _unit(pts[1] - pts[0])
        e = self.launch_pol(s)
        for m in range(k):
            t = _unit(pts[m + 2] - pts[m + 1])
            e = self.bounce(seq[m], e, s, t)
            s = t
        self.add(idx, e, 1.0 / L, L)

    # ---- bodies: pairs (receiver r, body b)
    def frame(self, S, P, b):
        c, a, cyl = self.body[b, :3], self.body[b, 3], self.cyl[b]
        flat = torch.where(cyl, 0.0, 1.0).to(P)[:, None] * torch.tensor([0.0, 0.0, 1.0]).to(P) \
            + torch.tensor([1.0, 1.0, 0.0]).to(P)
        ws, wp = (S - c) * flat, (P - c) * flat
        ds, dp = ws.norm(dim=-1), wp.norm(dim=-1)
        u = ws / ds[:, None]
        pu = _dot(wp, u)
        vp = wp - u * pu[:, None]
        pv = vp.norm(dim=-1)
        v = vp / pv[:, None]
        gam = torch.atan2(pv, pu)
        sps, sqp = (ds * ds - a * a).sqrt(), (dp * dp - a * a).sqrt()
        return dict(c=c, a=a, cyl=cyl, ds=ds, dp=dp, u=u, v=v, pu=pu, pv=pv, gam=gam, sps=sps, sqp=sqp,
                    bs=torch.atan2(sps, a), bp=torch.atan2(sqp, a), h=self.tall[b])

    @staticmethod
    def take(F, s):
        return {k: x[s] for k, x in F.items()}

    def slope(self, F, psi):
        """dL/dpsi and d2L/dpsi2 of the two-leg length at the circle point psi."""
        a, c, s = F["a"], torch.cos(psi), torch.sin(psi)
        g = h = 0.0
        for x, y in ((F["ds"], torch.zeros_like(psi)), (F["pu"], F["pv"])):
            l = ((a * c - x) ** 2 + (a * s - y) ** 2).sqrt()
            t = a * (x * s - y * c) / l
            g = g + t
            h = h + (a * (x * c + y * s) - t * t) / l
        return g, h

    def refl_point(self, F, S, P, psi):
        a, cs, sn = F["a"], torch.cos(psi), torch.sin(psi)
        n = F["u"] * cs[:, None] + F["v"] * sn[:, None]
        l1 = ((a * cs - F["ds"]) ** 2 + (a * sn) ** 2).sqrt()
        l2 = ((a * cs - F["pu"]) ** 2 + (a * sn - F["pv"]) ** 2).sqrt()
        z = torch.where(F["cyl"], S[2] + (P[:, 2] - S[2]) * l1 / (l1 + l2), F["c"][:, 2] + a * n[:, 2])
        return n, torch.cat([F["c"][:, :2] + a[:, None] * n[:, :2], z[:, None]], 1)

    def pairs(self, S, chunk):
        """Pairs of receivers chunk with bodies whose frame exists."""
        B = len(self.body)
        r = chunk[:, None].expand(-1, B).reshape(-1)
        b = torch.arange(B, device=r.device)[None].expand(len(chunk), -1).reshape(-1)
        c, a = self.body[b, :3].detach(), self.body[b, 3].detach()
        w = torch.where(self.cyl[b], 0.0, 1.0).to(a)
        ws, wp = S.detach() - c, self.P[r] - c
        ok = (ws[:, 0] ** 2 + ws[:, 1] ** 2 + w * ws[:, 2] ** 2 > a * a) & \
             (wp[:, 0] ** 2 + wp[:, 1] ** 2 + w * wp[:, 2] ** 2 > a * a)
        return r[ok], b[ok]

    def reflections(self, r, b):
        S = self.tx
        with torch.no_grad():
            F = self.frame(S, self.P[r], b)
            lit = F["gam"] < F["bs"] + F["bp"]
            r, b, F = r[lit], b[lit], self.take(F, lit)
            lo, hi = torch.zeros_like(F["gam"]), F["gam"].clone()
            for _ in range(54):
                mid = 0.5 * (lo + hi)
                up = self.slope(F, mid)[0] >= 0
                lo, hi = torch.where(up, lo, mid), torch.where(up, mid, hi)
            psi = 0.5 * (lo + hi)
            n, Q = self.refl_point(F, S, self.P[r], psi)
            z = Q[:, 2] - F["c"][:, 2]
            s = torch.nonzero(~F["cyl"] | ((z >= 0) & (z <= F["h"])))[:, 0]
            s = s[self.clear(S.expand_as(Q[s]), Q[s], skip_body=b[s])]
            s = s[self.clear(Q[s], self.P[r[s]], skip_body=b[s])]
        if not len(s):
            return
        r, b, psi = r[s], b[s], psi[s]
        P = self.P[r]
        F = self.frame(S, P, b)
        g, h = self.slope(F, psi)
        psi = psi - (g - g.detach()) / h.detach()
        n, Q = self.refl_point(F, S, P, psi)
        a, cyl = F["a"], F["cyl"]
        si, sr = (Q - S).norm(dim=-1), (P - Q).norm(dim=-1)
        shi = (Q - S) / si[:, None]
        cth = (-_dot(shi, n)).clamp(min=1e-30)
        shr = _unit(shi + n * (2.0 * cth)[:, None])
        f1 = torch.where(cyl, 2.0 * (1.0 - shi[:, 2] ** 2) / (a * cth), 2.0 / (a * cth))
        f2 = torch.where(cyl, torch.zeros_like(a), 2.0 * cth / a)
        sphi = -shi[:, 0] * n[:, 1] + shi[:, 1] * n[:, 0]
        rho = torch.where(cyl, a * (1.0 - cth * cth) / torch.where(cyl, sphi * sphi, torch.ones_like(a)), a)
        r1, r2 = 1.0 / (1.0 / si + f1), 1.0 / (1.0 / si + f2)
        A = (r1 * r2 / ((r1 + sr) * (r2 + sr))).sqrt() / si
        ep = _unit(torch.cross(n, shi, dim=-1))
        e0 = self.launch_pol(shi)
        Es, Eh = _dot(e0, ep + 0j), _dot(e0, torch.cross(ep, shi, dim=-1) + 0j)
        k = (2.0 * math.pi * self.freq / C0)[:, None]
        m = (k / 2.0) ** (1.0 / 3.0) * rho ** (1.0 / 3.0)
        xi = -2.0 * m * cth
        go = xi < -10.0
        xs = torch.where(go, torch.full_like(xi, -1.0), xi)
        Bs, Bh = _bracket(xs, (k * si * sr / (si + sr) / (2.0 * m * m)).sqrt())
        pre = -(-4.0 / xs).sqrt() * torch.exp(-1j * xs ** 3 / 12.0)
        Rs = torch.where(go, -torch.ones_like(Bs), pre * Bs)
        Rh = torch.where(go, torch.ones_like(Bh), pre * Bh)
        e = (Rs * Es)[..., None] * ep + (Rh * Eh)[..., None] * torch.cross(ep, shr, dim=-1)
        self.add(r, e, A[None], si + sr)

    def geodesic(self, S, P, b, way, turns):
        F = self.frame(S, P, b)
        a, cyl = F["a"], F["cyl"]
        arc = (F["gam"] if way == 0 else 2.0 * math.pi - F["gam"]) - F["bs"] - F["bp"]
        sg = 1.0 if way == 0 else -1.0
        p1, p2 = sg * F["bs"], F["gam"] - sg * F["bp"]
        n1 = F["u"] * torch.cos(p1)[:, None] + F["v"] * torch.sin(p1)[:, None]
        n2 = F["u"] * torch.cos(p2)[:, None] + F["v"] * torch.sin(p2)[:, None]
        exists = arc > 0
        arc = arc + 2.0 * math.pi * turns
        H = F["sps"] + a * arc + F["sqp"]
        dz = P[:, 2] - S[2]
        sin0 = torch.where(cyl, H / (H * H + dz * dz).sqrt(), torch.ones_like(H))
        z1 = torch.where(cyl, S[2] + dz * F["sps"] / H, F["c"][:, 2] + a * n1[:, 2])
        z2 = torch.where(cyl, S[2] + dz * (F["sps"] + a * arc) / H, F["c"][:, 2] + a * n2[:, 2])
        for z in (z1, z2):
            exists = exists & (~cyl | ((z >= F["c"][:, 2]) & (z <= F["c"][:, 2] + F["h"])))
        Q1 = torch.cat([F["c"][:, :2] + a[:, None] * n1[:, :2], z1[:, None]], 1)
        Q2 = torch.cat([F["c"][:, :2] + a[:, None] * n2[:, :2], z2[:, None]], 1)
        sp, t, sq = F["sps"] / sin0, a * arc / sin0, F["sqp"] / sin0
        rho = a / sin0 ** 2
        perp = torch.where(cyl, torch.ones_like(a), F["pv"])
        amp = torch.where(cyl, 1.0 / (sp * sq * (sp + t + sq)).sqrt(),
                          (-1.0) ** turns * (a * F["sps"] / F["ds"] / perp).sqrt() / sq.sqrt() / sp)
        caus = torch.where(cyl, 1.0, 1j if way else 1.0).to(torch.complex128)
        return dict(n1=n1, n2=n2, Q1=Q1, Q2=Q2, sp=sp, t=t, sq=sq, rho=rho, amp=amp * caus, ok=exists)

    def creeping(self, r, b, way, turns, wall=None):
        S = self.tx if wall is None else self.mirror(self.tx, wall)
        with torch.no_grad():
            G = self.geodesic(S, self.P[r], b, way, turns)
            s = torch.nonzero(G["ok"])[:, 0]
            if wall is None:
                s = s[self.clear(S.expand_as(G["Q1"][s]), G["Q1"][s], skip_body=b[s])]
            s = s[self.clear(G["Q2"][s], self.P[r[s]], skip_body=b[s])]
            if wall is not None:
                dS, dQ = self.dist(self.tx, wall), self.dist(G["Q1"], wall)
                s = s[(dS * dQ > 0)[s]]
                Q = S + (G["Q1"] - S) * (-dS / (-dS - dQ))[:, None]
                s = s[self.in_face(wall, Q[s])]
                s = s[self.clear(self.tx.expand_as(Q[s]), Q[s], [wall])]
                s = s[self.clear(Q[s], G["Q1"][s], [wall], b[s])]
        if not len(s):
            return
        r, b = r[s], b[s]
        P = self.P[r]
        G = self.geodesic(S, P, b, way, turns)
        t1, t2 = _unit(G["Q1"] - S), _unit(P - G["Q2"])
        if wall is None:
            e0 = self.launch_pol(t1)
        else:
            dI, dQ = self.dist(S, wall), self.dist(G["Q1"], wall)
            Q = S + (G["Q1"] - S) * (dI / (dI - dQ))[:, None]
            si = _unit(Q - self.tx)
            e0 = self.bounce(wall, self.launch_pol(si), si, t1)
        Es, Eh = _dot(e0, torch.cross(t1, G["n1"], dim=-1) + 0j), _dot(e0, G["n1"] + 0j)
        k = (2.0 * math.pi * self.freq / C0)[:, None]
        m = (k / 2.0) ** (1.0 / 3.0) * G["rho"] ** (1.0 / 3.0)
        Lp = G["sp"] * G["sq"] / (G["sp"] + G["sq"])
        Bs, Bh = _bracket(m * G["t"] / G["rho"], (k * Lp / (2.0 * m * m)).sqrt())
        pre = -m * (2.0 / k).sqrt() * G["amp"]
        e = (Bs * Es * pre)[..., None] * torch.cross(t2, G["n2"], dim=-1) + (Bh * Eh * pre)[..., None] * G["n2"]
        self.add(r, e, 1.0, G["sp"] + G["t"] + G["sq"])

    def total(self, seqs=None):
        if seqs is None:
            f = range(self.n_face)
            seqs = [(i,) for i in f if self.order >= 1] + [(i, j) for i in f for j in f
                                                           if i != j and self.order >= 2]
        for q in [()] + list(seqs):
            self.planar(q)
        if len(self.body) and len(self.ok):
            for chunk in self.ok.split(max(1, int(2e6 // len(self.body)))):
                r, b = self.pairs(self.tx, chunk)
                self.reflections(r, b)
                for turns in range(self.enc + 1):
                    for way in (0, 1):
                        self.creeping(r, b, way, turns)
                for f in range(self.n_face if self.wall else 0):
                    r, b = self.pairs(self.mirror(self.tx, f), chunk)
                    for turns in range(self.enc + 1):
                        for way in (0, 1):
                            self.creeping(r, b, way, turns, f)
        return self.E

    @torch.no_grad()
    def launch(self, n_rays, order):
        """Face sequences of rays from the transmitter (spherical Fibonacci
        lattice, specular bounces at the nearest triangle), every prefix once."""
        i = np.arange(n_rays)
        z = 1.0 - (2.0 * i + 1.0) / n_rays
        ph = i * (np.pi * (3.0 - math.sqrt(5.0)))
        rho = np.sqrt(np.maximum(0.0, 1.0 - z * z))
        D = torch.from_numpy(np.stack([rho * np.cos(ph), rho * np.sin(ph), z], 1)).to(self.P)
        O = self.tx.expand_as(D).clone()
        v0 = self.tri[:, 0]
        e1, e2 = self.tri[:, 1] - v0, self.tri[:, 2] - v0
        seq = torch.full((n_rays, 3), -1, dtype=torch.long, device=D.device)
        live, out = torch.ones(n_rays, dtype=torch.bool, device=D.device), set()
        for k in range(order):
            best = torch.full((n_rays,), math.inf, dtype=torch.float64, device=D.device)
            tid = torch.zeros(n_rays, dtype=torch.long, device=D.device)
            for s in torch.arange(n_rays, device=D.device).split(max(1, int(8e6 // len(v0)))):
                T, d = O[s][:, None] - v0, D[s][:, None].expand(-1, len(v0), -1)
                p = torch.cross(d, e2.expand_as(d), dim=-1)
                det = (p * e1).sum(-1)
                inv = 1.0 / torch.where(det.abs() < 1e-14, torch.ones_like(det), det)
                q = torch.cross(T, e1.expand_as(T), dim=-1)
                u, v, t = (T * p).sum(-1) * inv, (d * q).sum(-1) * inv, (q * e2).sum(-1) * inv
                hit = (det.abs() >= 1e-14) & (u >= 0) & (u <= 1) & (v >= 0) & (u + v <= 1) & (t > 1e-9)
                if k:
                    hit &= self.face[None] != seq[s, k - 1][:, None]
                best[s], tid[s] = torch.where(hit, t, math.inf).min(1)
            live &= torch.isfinite(best)
            f = self.face[tid]
            seq[:, k] = torch.where(live, f, -1)
            out.update(tuple(x[:k + 1]) for x in seq[live].tolist())
            t = torch.where(live, best, 0.0)[:, None]
            O = O + D * t
            n = self.nrm[f]
            D = D - n * (2.0 * _dot(D, n))[:, None]
        return sorted(out, key=lambda q: (len(q), q))
