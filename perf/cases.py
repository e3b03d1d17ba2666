"""The measured workloads of the acoustic FWI framework.

Each case is one call (or one loop iteration) of the public API on inputs
shaped like the framework's own workloads (``inputs.py``, ``bench.py``): the
paper's accuracy set-up, single requests of the serving stream, the breast and
skull gradients, one iteration of the imaging loop, an uneven batch, and the
extended schemes of Sec. 2.4 (fourth order in time, sinc points, PML,
attenuation).  Models are drawn on the GPU from the seed; observed data are
the direct arrivals through water, as a user's measured traces would mostly
be.  Time axes are cut so that a state stays within about 30 GB.

``exact`` computes the same discrete scheme in 64 bits with plain torch.
"""
import math

import numpy as np
import torch

from paper_2110_03345_gb300 import binding, inputs, invert

DEV = "cuda:0"
SPONGE = 20
BUDGET = 60 << 30          # bytes a plan may hold: a serving process shares the card
F0 = 500e3                 # centre frequency of the transducers
SEED = 1009


# --------------------------------------------------------------------------
# the cases
# --------------------------------------------------------------------------

def _case(name, call, shape, nt, shots, nrec, order=8, density=True, scheme="leapfrog", sinc=False):
    nz, ny, nx = ((0,) + tuple(shape)) if len(shape) == 2 else tuple(shape)
    c = dict(call=call, nz=nz, ny=ny, nx=nx, nt=nt, shots=shots, nrec=nrec, order=order,
             density=density, scheme=scheme, sinc=sinc)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the accuracy set-up of Sec. 3.1: one source in a 256^2 box, the
        # smallest call, where each time step is a few microseconds
        _case("forward2d_accuracy", "forward", (256, 256), 1000, 1, 64, density=False),
        # a forward request of the serving stream: one shot, ragged grid
        _case("forward2d_request", "forward", (700, 748), 1500, 1, 64),
        # a gradient request with high-order off-grid points, 10th order in space
        _case("gradient2d_sinc", "gradient", (897, 1012), 800, 1, 64, order=10, sinc=True),
        # a batch of shots of the breast gradient (the default benchmark's grid and batch)
        _case("gradient2d_breast", "gradient", (1024, 1024), 400, 15, 256),
        # one iteration of the imaging loop of Sec. 3.2: low-pass, gradient of
        # 16 shots, model update (constant density)
        _case("iteration2d", "iteration", (456, 485), 1200, 16, 128, density=False),
        # uneven independent forward problems in one CUDA graph
        _case("batch2d_uneven", "batch", (1024, 1024), 1200, 8, 64),
        # the breast gradient with the fourth-order time scheme, twice the step
        _case("gradient2d_time4", "gradient", (800, 872), 300, 6, 128, scheme="time4"),
        # the breast gradient with the perfectly matched layer
        _case("gradient2d_pml", "gradient", (1024, 1024), 250, 6, 128, scheme="pml"),
        # a 3D forward request of the serving stream
        _case("forward3d_request", "forward", (152, 160, 176), 500, 1, 128, order=10),
        # one shot of the skull gradient (Sec. 3.3), the largest grid
        _case("gradient3d_skull", "gradient", (256, 256, 256), 220, 1, 512, order=10),
        # the skull gradient with soft-tissue attenuation, y = 2
        _case("gradient3d_att2", "gradient", (192, 180, 200), 160, 1, 256, order=10, scheme="att2"),
        # the skull gradient with the perfectly matched layer
        _case("gradient3d_pml", "gradient", (160, 144, 168), 160, 1, 128, order=10, scheme="pml"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges: every kind above, other sizes."""
    k = rng.randrange(12)
    side = lambda lo, hi: rng.randint(lo, hi)  # noqa: E731
    order = rng.choice((8, 10))
    if k == 0:
        return _case(None, "forward", (side(160, 400), side(160, 400)), side(600, 1200), 1, side(16, 128),
                     order=order, density=rng.random() < 0.5)
    if k == 1:
        return _case(None, "forward", (side(512, 1024), side(512, 1024)), side(1000, 1600), 1, side(32, 128),
                     order=order)
    if k == 2:
        return _case(None, "gradient", (side(512, 1024), side(512, 1024)), side(400, 1000), 1, side(32, 128),
                     order=order, sinc=rng.random() < 0.7)
    if k == 3:
        return _case(None, "gradient", (side(600, 1024), side(600, 1024)), side(200, 400), _log(rng, 2, 15),
                     side(64, 256))
    if k == 4:
        return _case(None, "iteration", (side(300, 500), side(300, 500)), side(600, 1200), side(4, 16),
                     side(64, 128), density=False)
    if k == 5:
        n = 4 * side(128, 256)
        return _case(None, "batch", (n, n), side(600, 1200), side(3, 8), side(32, 64))
    if k == 6:
        return _case(None, "gradient", (side(500, 900), side(500, 900)), side(150, 300), side(1, 6),
                     side(64, 128), density=rng.random() < 0.7, scheme="time4")
    if k == 7:
        return _case(None, "gradient", (side(500, 1024), side(500, 1024)), side(100, 250), side(1, 6),
                     side(64, 128), density=rng.random() < 0.7, scheme="pml")
    if k == 8:
        return _case(None, "forward", (side(128, 192), side(128, 192), side(128, 192)), side(200, 400), 1,
                     side(32, 128), order=10, density=rng.random() < 0.7)
    if k == 9:
        return _case(None, "gradient", (side(128, 240), side(128, 240), side(128, 240)), side(80, 200), 1,
                     side(64, 512), order=order, density=rng.random() < 0.7)
    if k == 10:
        return _case(None, "gradient", (side(128, 192), side(128, 192), side(128, 192)), side(80, 150), 1,
                     side(64, 256), order=10, scheme="att2")
    return _case(None, "gradient", (side(128, 160), side(128, 160), side(128, 168)), side(80, 150), 1,
                 side(64, 128), order=10, density=rng.random() < 0.7, scheme="pml")


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------

def _coords(shape):
    ax = [(torch.arange(n, device=DEV, dtype=torch.float32) + 0.5 - n / 2) for n in shape]
    return torch.meshgrid(*ax, indexing="ij")


def _ellipse(Y, X, cy, cx, ay, ax, th):
    c, s = math.cos(th), math.sin(th)
    u, v = c * (X - cx) + s * (Y - cy), -s * (X - cx) + c * (Y - cy)
    return (u / ax) ** 2 + (v / ay) ** 2 <= 1.0


def _noise(shape, rng, cells):
    low = rng.standard_normal([1, 1] + [cells] * len(shape)).astype(np.float32)
    mode = "bicubic" if len(shape) == 2 else "trilinear"
    f = torch.nn.functional.interpolate(torch.from_numpy(low).to(DEV), size=tuple(shape), mode=mode,
                                        align_corners=True)[0, 0]
    return f / f.std()


def _breast(shape, rng):
    """Water, an ellipse of fatty tissue with 20-40 inclusions, smooth noise in
    the speed of sound; the density is constant within each tissue."""
    Y, X = _coords(shape)
    m = min(shape)
    vp = torch.full(shape, 1500.0, device=DEV)
    rho = torch.full(shape, 1000.0, device=DEV)
    ay, ax = rng.uniform(0.342, 0.39, 2) * m
    breast = _ellipse(Y, X, 0.0, 0.0, ay, ax, rng.uniform(0, math.pi))
    vp[breast] = float(rng.uniform(1430, 1470))
    rho[breast] = float(rng.uniform(950, 980))
    for _ in range(int(rng.integers(20, 41))):
        r, ang = math.sqrt(rng.uniform(0, 1)) * 0.8, rng.uniform(0, 2 * math.pi)
        sy, sx = rng.uniform(0.02, 0.146, 2) * m
        e = _ellipse(Y, X, r * ay * math.sin(ang), r * ax * math.cos(ang), sy, sx,
                     rng.uniform(0, math.pi)) & breast
        vp[e] = float(rng.uniform(1400, 1600))
        rho[e] = float(rng.uniform(950, 1100))
    vp = torch.where(breast, vp + 5.0 * _noise(shape, rng, 96), vp)
    return vp.clamp_(1400.0, 1600.0).contiguous(), rho.contiguous()


def _skull(shape, rng):
    """Water, an ellipsoidal skull shell, soft tissue inside (smooth variations
    of the speed); the density is constant within each."""
    Z, Y, X = _coords(shape)
    m = min(shape)
    a = np.array([20.0, 23.0, 19.0]) / 64.0 * m * rng.uniform(0.94, 1.0, 3)
    t = 6.0 / 64.0 * m
    outer = (Z / a[0]) ** 2 + (Y / a[1]) ** 2 + (X / a[2]) ** 2 <= 1.0
    inner = (Z / (a[0] - t)) ** 2 + (Y / (a[1] - t)) ** 2 + (X / (a[2] - t)) ** 2 <= 1.0
    vp = torch.full(shape, 1500.0, device=DEV)
    rho = torch.full(shape, 1000.0, device=DEV)
    vp[outer], rho[outer] = 2800.0, 1900.0
    vp = torch.where(inner, 1540.0 + 10.0 * _noise(shape, rng, 12), vp)
    rho[inner] = 1040.0
    return vp.contiguous(), rho.contiguous()


def _setting(case):
    """Spacing, step, largest speed and layer width of a case."""
    three = case["nz"] > 0
    c_max = 2800.0 if three else 1600.0
    dx = 0.25e-3 if three else (0.5e-3 if case["call"] == "iteration" else 0.1e-3)
    cfl = 0.8 if case["scheme"] == "time4" else 0.4
    dt = 0.08e-6 if case["call"] == "iteration" else cfl * dx / c_max
    nb = 16 if three and max(case["nz"], case["ny"], case["nx"]) < 200 else SPONGE
    return dx, dt, c_max, nb


def _problem(case, seed, shape, nt, shots):
    """Host geometry and device arrays of one problem."""
    rng = np.random.default_rng([SEED, seed])
    dx, dt, c_max, nb = _setting(case)
    nd, nrec = len(shape), case["nrec"]
    vp, rho = (_breast if nd == 2 else _skull)(shape, rng)
    ctr = tuple(n / 2 * dx for n in shape)
    rad = (0.4395 if nd == 2 else 25.0 / 64.0) * min(shape) * dx
    if case["call"] == "forward" and shots == 1 and case["name_source"] == "centre":
        src = np.array([[[shape[0] // 2 * dx, shape[1] // 2 * dx]]])
        rec = inputs.ring(nrec, ctr, 0.39 * min(shape) * dx, rotation=float(rng.uniform()))
    elif nd == 2:
        rec = inputs.ring(nrec, ctr, rad, rotation=float(rng.uniform()))
        fire = (np.arange(shots) * max(1, nrec // shots) + int(rng.integers(nrec))) % nrec
        src = rec[fire][:, None, :]
    else:
        rec = inputs.fibonacci_sphere(nrec, ctr, rad)
        src = rec[rng.choice(nrec, shots, replace=False)][:, None, :]
    if case["call"] == "iteration":
        w = inputs.tone_burst(F0, dt, nt, t0=3.0 / 300e3)
    else:
        w = inputs.ricker(F0, dt, nt, amp=float(rng.uniform(0.8, 1.2)))
    wav = torch.as_tensor(np.broadcast_to(w, (shots, 1, nt)).astype(np.float32).copy(), device=DEV)
    if not case["density"]:
        rho = None
    return dict(shape=shape, nt=nt, dx=dx, dt=dt, c_max=c_max, nb=nb, vp=vp, rho=rho, src=src, rec=rec,
                wav=wav, wavelet=w)


def _direct_arrivals(p):
    """Measured traces: the wavelet delayed by the water path, with the
    geometric decay, and 2% of noise."""
    src = torch.as_tensor(p["src"][:, 0, :], device=DEV, dtype=torch.float32)
    rec = torch.as_tensor(p["rec"], device=DEV, dtype=torch.float32)
    d = torch.cdist(src, rec).clamp_min(2 * p["dx"])
    w = torch.as_tensor(p["wavelet"], device=DEV, dtype=torch.float32)
    nt, nd = p["nt"], len(p["shape"])
    t = torch.arange(nt, device=DEV, dtype=torch.float32)
    # amplitude of the solver's point source: 1 / (4 pi r) in 3D, about
    # sqrt(c / (8 pi w0 r)) c0 in 2D
    if nd == 3:
        amp = 1.0 / (4.0 * math.pi * d)
    else:
        amp = torch.sqrt(1500.0 / (8.0 * math.pi * 2.0 * math.pi * F0 * d))
    at = t[None, None, :] - (d / 1500.0 / p["dt"])[:, :, None]
    i0 = at.floor()
    f = at - i0
    i0 = i0.long()
    pick = lambda i: torch.where((i >= 0) & (i < nt), w[i.clamp(0, nt - 1)], 0.0 * f)  # noqa: E731
    obs = amp[:, :, None] * ((1 - f) * pick(i0) + f * pick(i0 + 1))
    g = torch.Generator(device=DEV)
    g.manual_seed(int(abs(hash((nt, float(p["rec"][0, 0])))) % (1 << 31)))
    obs += 0.02 * obs.square().mean().sqrt() * torch.randn(obs.shape, generator=g, device=DEV)
    return obs.contiguous()


def _batch_sizes(case, seed):
    """Sides, time axes and shot counts of an uneven batch."""
    rng = np.random.default_rng([SEED, 4, case["ny"], case["nt"], case["shots"]])
    out = []
    for i in range(case["shots"]):
        f = 1.0 if i == 0 else rng.uniform(0.25, 1.0)
        n = max(256, 4 * int(case["ny"] * f / 4))
        out.append((n, case["nt"] if i == 0 else int(rng.integers(case["nt"] // 4, case["nt"])),
                    int(rng.integers(1, 9))))
    return out


def _parts(case, seed):
    case = dict(case)
    case["name_source"] = "centre" if (case["call"] == "forward" and not case["density"]
                                       and case["nz"] == 0) else "ring"
    shape = (case["ny"], case["nx"]) if case["nz"] == 0 else (case["nz"], case["ny"], case["nx"])
    if case["call"] == "batch":
        return [_problem(case, 100 * seed + i, (n, n), nt, ns)
                for i, (n, nt, ns) in enumerate(_batch_sizes(case, seed))]
    p = _problem(case, seed, shape, case["nt"], case["shots"])
    if case["call"] in ("gradient", "iteration"):
        p["obs"] = _direct_arrivals(p)
    if case["scheme"] == "att2":
        # 0.5 dB/cm at 1 MHz in tissue, none in water: nepers/m per (rad/s)^2
        p["alpha0"] = torch.where(p["rho"] != 1000.0, 5.756 / (2 * math.pi * 1e6) ** 2, 0.0).to(torch.float32)
    return [p]


def _step_ms(case):
    return 5.0


def _ids(case, p):
    """The shots of the iteration: every shot, in a drawn order."""
    return np.random.default_rng([SEED, 7, p["nt"]]).permutation(p["src"].shape[0])


def _mask(p):
    ctr = tuple(n / 2 * p["dx"] for n in p["shape"])
    rad = 0.4395 * min(p["shape"]) * p["dx"] - 5 * p["dx"]
    return inputs.disk_mask(p["shape"], p["dx"], ctr, rad)


def prepare(case, seed):
    parts = _parts(case, seed)
    if case["call"] == "batch":
        entries = [dict(shape=p["shape"], spacing=p["dx"], nt=p["nt"], dt=p["dt"], order=case["order"],
                        sponge=p["nb"], c_ref=p["c_max"], vp=p["vp"], rho=p["rho"],
                        geometry=binding.Geometry(p["src"], p["rec"]), wavelet=p["wav"]) for p in parts]
        return dict(case=case, batch=binding.Batch(entries, budget=BUDGET), keep=parts)
    p = parts[0]
    plan = binding.Plan(p["shape"], p["dx"], p["nt"], p["dt"], order=case["order"], sponge=p["nb"],
                        c_ref=p["c_max"], budget=BUDGET)
    opts = dict(time4=dict(time_order=4), pml=dict(boundary=binding.BOUNDARY_PML)).get(case["scheme"], {})
    if case["sinc"]:
        opts["interp"] = binding.INTERP_SINC
    if opts:
        plan.set_options(**opts)
    if case["scheme"] == "att2":
        plan.set_attenuation(p["alpha0"], 2)
    s = dict(case=case, plan=plan, p=p, geo=binding.Geometry(p["src"], p["rec"]))
    if case["call"] == "iteration":
        vp0 = torch.full(p["shape"], 1500.0, device=DEV)
        p["vp"] = (0.5 * (vp0 + p["vp"])).contiguous()   # a model half way to the true one
        mask = torch.as_tensor(_mask(p), device=DEV, dtype=torch.float32)
        s["inv"] = invert.Inversion(plan, p["src"], p["rec"], p["wav"], p["obs"], mask=mask,
                                    bounds=(1400.0, 1600.0), max_shots=case["shots"])
        s["ids"] = _ids(case, p)
    return s


def run(state):
    case = state["case"]
    if case["call"] == "batch":
        return state["batch"].run()
    p, plan = state["p"], state["plan"]
    if case["call"] == "forward":
        return plan.forward(p["vp"], p["rho"], state["geo"], p["wav"])
    if case["call"] == "iteration":
        vp = p["vp"].clone()                             # the loop updates its model in place
        J = state["inv"].iterate(vp, state["ids"], 400e3, _step_ms(case))
        return {"misfit": J, "vp": vp, "gradient": state["inv"].grad}
    J, g, _ = plan.gradient(p["vp"], p["rho"], state["geo"], p["wav"], p["obs"])
    return {"misfit": J, "gradient": g}


def work(case):
    """Inputs read once and outputs written once; operations of the stencil
    updates (symmetric sums counted once per tap pair)."""
    R, nd = case["order"] // 2, 2 if case["nz"] == 0 else 3
    lap = nd * 3 * R + 8                  # add, multiply-add per tap pair; the update
    grad = nd * (3 * R + 2) if case["density"] else 0
    if case["call"] == "batch":
        b = f = 0.0
        for n, nt, ns in _batch_sizes(case, 0):
            b += 4.0 * (2 * n * n + ns * nt + ns * case["nrec"] * nt)
            f += float(n) * n * ns * (nt - 1) * (lap + grad)
        return {"bytes": b, "flops": f}
    n = case["ny"] * case["nx"] * max(1, case["nz"])
    ns, nt, nrec = case["shots"], case["nt"], case["nrec"]
    per = {"time4": 2 * (lap + grad), "pml": lap + grad + 2, "att2": lap + grad + 6}.get(case["scheme"], lap + grad)
    fields = 1 + int(case["density"]) + int(case["scheme"] == "att2")
    b = 4.0 * (fields * n + ns * nt + ns * nrec * nt)
    sweeps = 1
    if case["call"] != "forward":
        b += 4.0 * n
        sweeps = 2
    if case["call"] == "iteration":
        b += 4.0 * 2 * n
    return {"bytes": b, "flops": float(n) * ns * (nt - 1) * (per * sweeps + 2 * (sweeps - 1))}


# --------------------------------------------------------------------------
# the same in 64 bits
# --------------------------------------------------------------------------

_W2 = {8: (-205 / 72, 8 / 5, -1 / 5, 8 / 315, -1 / 560),
       10: (-5269 / 1800, 5 / 3, -5 / 21, 5 / 126, -5 / 1008, 1 / 3150)}
_W1 = {8: (0.0, 4 / 5, -1 / 5, 4 / 105, -1 / 280),
       10: (0.0, 5 / 6, -5 / 21, 5 / 84, -5 / 504, 1 / 1260)}


class _Exact:
    """The discrete schemes in float64, fields [shot][axes]."""

    def __init__(self, case, p, shots):
        self.case, self.p, self.nd = case, p, len(p["shape"])
        self.dx, self.dt, self.nt = p["dx"], p["dt"], p["nt"]
        self.w2 = [w / self.dx ** 2 for w in _W2[case["order"]]]
        self.w1 = [w / self.dx for w in _W1[case["order"]]]
        self.shots = shots
        vp = p["vp"].double()
        self.vp, self.k = vp, (vp * self.dt) ** 2
        self.b = None
        if p["rho"] is not None:
            lr = p["rho"].double().log()
            self.b = [self._d1_edge(lr, a) for a in range(self.nd)]
        nb = p["nb"]
        self.A = []
        for a, n in enumerate(p["shape"]):
            i = torch.arange(n, device=DEV, dtype=torch.float64)
            delta = torch.clamp(torch.maximum(nb - i, i - (n - 1 - nb)), min=0.0)
            smax = 3.0 * p["c_max"] * math.log(1000.0) / (2.0 * nb * self.dx)
            v = smax * (delta / nb) ** 2 * self.dt * 0.5
            self.A.append(v.reshape([-1 if q == a else 1 for q in range(self.nd)]))
        self.a = sum(self.A)
        self.src = self._points(p["src"][shots, 0, :])
        self.rec = self._points(p["rec"])
        self.q = p["wav"][shots, 0, :].double() / self.dx ** self.nd

    # ---- stencils
    def _tap(self, out, u, ax, j, w):
        n = u.shape[ax]
        out.narrow(ax, 0, n - j).add_(u.narrow(ax, j, n - j), alpha=w)

    def _tapm(self, out, u, ax, j, w):
        n = u.shape[ax]
        out.narrow(ax, j, n - j).add_(u.narrow(ax, 0, n - j), alpha=w)

    def lap(self, u):
        out = u * (self.nd * self.w2[0])
        for a in range(self.nd):
            ax = u.dim() - self.nd + a
            for j in range(1, len(self.w2)):
                self._tap(out, u, ax, j, self.w2[j])
                self._tapm(out, u, ax, j, self.w2[j])
        return out

    def d1(self, u, a, out=None):
        out = torch.zeros_like(u) if out is None else out
        ax = u.dim() - self.nd + a
        for j in range(1, len(self.w1)):
            self._tap(out, u, ax, j, self.w1[j])
            self._tapm(out, u, ax, j, -self.w1[j])
        return out

    def _d1_edge(self, f, a):
        n, R = f.shape[a], len(self.w1) - 1
        idx = torch.arange(n, device=DEV)
        out = torch.zeros_like(f)
        for j in range(1, R + 1):
            out += self.w1[j] * (f.index_select(a, (idx + j).clamp(max=n - 1))
                                 - f.index_select(a, (idx - j).clamp(min=0)))
        return out

    def L(self, u):
        out = self.lap(u)
        if self.b is not None:
            for a in range(self.nd):
                out.addcmul_(self.b[a].expand_as(u), self.d1(u, a), value=-1.0)
        return out

    def LT(self, v):
        out = self.lap(v)
        if self.b is not None:
            for a in range(self.nd):
                self.d1(self.b[a] * v, a, out)
        return out

    # ---- points
    def _axis(self, x, n):
        if not self.case["sinc"]:
            i0 = min(max(int(math.floor(x)), 0), n - 2)
            return [(i0, 1.0 - (x - i0)), (i0 + 1, x - i0)]
        r, b, f = 4, 6.31, int(math.floor(x))
        out = []
        for j in range(2 * r):
            d = f - r + 1 + j - x
            win = float(np.i0(b * math.sqrt(max(0.0, 1.0 - (d / r) ** 2)))) / float(np.i0(b)) if abs(d) <= r else 0.0
            out.append((f - r + 1 + j, win * float(np.sinc(d))))
        return out

    def _points(self, xyz):
        """(flat node index, weight) of each point, [point][corner]."""
        node, wt = [], []
        for x in np.asarray(xyz):
            pts = [(0, 1.0)]
            for a, n in enumerate(self.p["shape"]):
                ax = self._axis(float(x[a]) / self.dx, n)
                pts = [(i * n + j, w * v) for i, w in pts for j, v in ax]
            node.append([i for i, _ in pts])
            wt.append([w for _, w in pts])
        return torch.tensor(node, device=DEV), torch.tensor(wt, device=DEV, dtype=torch.float64)

    def add_sources(self, f, val):
        node, wt = self.src
        f.view(f.shape[0], -1).scatter_add_(1, node, wt * val[:, None])

    def add_receivers(self, f, r):
        node, wt = self.rec
        flat = f.view(f.shape[0], -1)
        flat.index_add_(1, node.reshape(-1), (r[:, :, None] * wt).reshape(f.shape[0], -1))

    def sample(self, u):
        node, wt = self.rec
        return (u.view(u.shape[0], -1)[:, node] * wt).sum(-1)

    # ---- sweeps
    def qn(self, n):
        return self.q[:, n] if 0 <= n < self.nt else torch.zeros_like(self.q[:, 0])

    def forward(self, keep):
        sh = (len(self.shots),) + self.p["shape"]
        z = lambda: torch.zeros(sh, device=DEV, dtype=torch.float64)  # noqa: E731
        u, um = z(), z()
        d = torch.zeros(sh[0], self.rec[0].shape[0], self.nt, device=DEV, dtype=torch.float64)
        hist = []
        sc, inv = self.case["scheme"], 1.0 / (1.0 + self.a)
        one = 1.0 - self.a
        if sc == "att2":
            att = 2.0 * self.p["alpha0"].double() * self.vp / self.dt
            lold = z()
        if sc == "pml":
            phi = [z() for _ in range(self.nd)]
            qq = z() if self.nd == 3 else None
            co = self.pml()
        for n in range(self.nt - 1):
            d[:, :, n] = self.sample(u)
            acc = self.L(u)
            self.add_sources(acc, self.qn(n))
            if sc == "time4":
                kw = self.k * acc
                acc2 = self.L(kw)
                self.add_sources(acc2, self.qn(n + 1) - 2 * self.qn(n) + self.qn(n - 1))
                h = kw + self.k * acc2 / 12.0
                keepit = (h, kw)
            elif sc == "att2":
                lu = self.lap(u)
                dl = lu - lold
                lold = lu
                h = self.k * (acc + att * dl)
                keepit = (h + 0.5 * self.k * att * dl,)
            elif sc == "pml":
                for a in range(self.nd):
                    self.d1(phi[a], a, acc)
                h = self.k * acc
                keepit = (h,)
                h = h - co["e"] * u
                if qq is not None:
                    h = h - co["f"] * qq
            else:
                h = self.k * acc
                keepit = (h,)
            up = (2.0 * u - one * um + h) * inv
            um, u = u, up
            if sc == "pml":
                if qq is not None:
                    qq = qq + self.dt * u
                for a in range(self.nd):
                    phi[a] = co["p"][a] * phi[a] + co["b"][a] * self.d1(u, a)
                    if qq is not None:
                        phi[a] += co["g"][a] * self.d1(qq, a)
            if keep:
                hist.append(keepit)
        d[:, :, self.nt - 1] = self.sample(u)
        return d, hist

    def pml(self):
        A, e, f = self.A, 0.0, 0.0
        for i in range(self.nd):
            for j in range(i + 1, self.nd):
                e = e + 4.0 * A[i] * A[j]
        if self.nd == 3:
            f = 8.0 * A[0] * A[1] * A[2] / self.dt
        p, b, g = [], [], []
        for i in range(self.nd):
            o = [A[j] for j in range(self.nd) if j != i]
            p.append((1 - A[i]) / (1 + A[i]))
            b.append(2.0 * (sum(o) - A[i]) / (1 + A[i]))
            g.append(4.0 * o[0] * o[1] / (self.dt * (1 + A[i])) if self.nd == 3 else None)
        return dict(e=e, f=f, p=p, b=b, g=g)

    def adjoint(self, r, hist):
        """dJ/dm of residual traces r (summed over the shots)."""
        sh = (len(self.shots),) + self.p["shape"]
        z = lambda: torch.zeros(sh, device=DEV, dtype=torch.float64)  # noqa: E731
        g = torch.zeros(self.p["shape"], device=DEV, dtype=torch.float64)
        sc, inv, one = self.case["scheme"], 1.0 / (1.0 + self.a), 1.0 - self.a
        if sc == "pml":
            return self.adjoint_pml(r, hist, g, z)
        lam, lamp = z(), z()
        if sc == "att2":
            att = 2.0 * self.p["alpha0"].double() * self.vp / self.dt
            qa = z()

        def image(n, lam, ky):
            g.sub_((lam * hist[n][0]).sum(0))
            if sc == "time4":
                g.sub_((ky * hist[n][1]).sum(0) / 12.0)
        for k in range(self.nt - 1, 0, -1):
            ky = None
            acc = self.LT(lam)
            if sc == "time4":
                ky = self.k * acc
                acc2 = self.LT(ky)
                self.add_receivers(acc2, 12.0 * r[:, :, k])
                F = ky + self.k * acc2 / 12.0
            else:
                self.add_receivers(acc, r[:, :, k])
                if sc == "att2":
                    lc = self.lap(att * lam)
                    acc = acc + (lc - qa)
                    qa = lc
                F = self.k * acc
            if k <= self.nt - 2:
                image(k, lam, ky)
                hist[k] = None
            lam, lamp = (2.0 * lam - one * lamp + F) * inv, lam
        image(0, lam, self.k * self.LT(lam) if sc == "time4" else None)
        return g / self.dt ** 2

    def adjoint_pml(self, r, hist, g, z):
        co, inv, one = self.pml(), 1.0 / (1.0 + self.a), 1.0 - self.a
        ph = [z() for _ in range(self.nd)]
        qb = z() if self.nd == 3 else None
        xn, xc = z(), z()
        self.add_receivers(xn, r[:, :, self.nt - 1])
        self.add_receivers(xc, r[:, :, self.nt - 2])
        for n in range(self.nt - 2, -1, -1):
            ub = xn
            for a in range(self.nd):
                ub = ub - self.d1(co["b"][a] * ph[a], a)
            if qb is not None:
                for a in range(self.nd):
                    qb = qb - self.d1(co["g"][a] * ph[a], a)
                ub = ub + self.dt * qb
            c = ub * inv
            if qb is not None:
                qb = qb - co["f"] * c
            kc = self.k * c
            g.sub_((kc * hist[n][0]).sum(0))
            hist[n] = None
            prev = -one * c
            if n >= 1:
                self.add_receivers(prev, r[:, :, n - 1])
            xc = xc + (2.0 - co["e"]) * c + self.LT(kc)
            for a in range(self.nd):
                ph[a] = co["p"][a] * ph[a] - self.d1(kc, a)
            xn, xc = xc, prev
        return g / self.dt ** 2


def _lowpass64(x, f_max, dt, M):
    j = np.arange(-M, M + 1)
    h = np.sinc(2.0 * f_max * dt * j) * 0.5 * (1.0 + np.cos(np.pi * j / (M + 1)))
    h = torch.as_tensor(h / h.sum(), device=DEV)
    n = x.shape[-1]
    L = n + 2 * M
    F = torch.fft.rfft(x, L) * torch.fft.rfft(h, L)
    return torch.fft.irfft(F, L)[..., M:M + n]


def exact(case, seed):
    parts = _parts(case, seed)
    if case["call"] == "batch":
        return [_Exact(case, p, list(range(p["src"].shape[0]))).forward(False)[0] for p in parts]
    p = parts[0]
    if case["call"] == "forward":
        return _Exact(case, p, [0]).forward(False)[0]
    extra = {}
    if case["call"] == "iteration":
        p["vp"] = (0.5 * (torch.full(p["shape"], 1500.0, device=DEV) + p["vp"])).contiguous()
        ids = _ids(case, p)
        M = int(math.ceil(3.0 / (400e3 * p["dt"])))
        p["src"] = p["src"][ids]
        p["wav"] = _lowpass64(p["wav"][ids].double(), 400e3, p["dt"], M)
        p["obs"] = _lowpass64(p["obs"][ids].double(), 400e3, p["dt"], M)
    fields = (2 if case["scheme"] == "time4" else 1) * p["nt"] * 8.0 * float(np.prod(p["shape"]))
    group = max(1, int(48e9 / fields))
    J, g, ns = 0.0, 0.0, p["src"].shape[0]
    for s0 in range(0, ns, group):
        shots = list(range(s0, min(ns, s0 + group)))
        E = _Exact(case, p, shots)
        d, hist = E.forward(True)
        r = d - p["obs"][shots].double()
        J += 0.5 * float((r * r).sum())
        g = g + E.adjoint(r, hist)
        del hist, E
    if case["call"] == "iteration":
        vp = p["vp"].double()
        dv = torch.as_tensor(_mask(p), device=DEV) * (-2.0 * g / vp ** 3)
        extra["vp"] = (vp - _step_ms(case) * dv / dv.abs().max()).clamp(1400.0, 1600.0)
    return {"misfit": J, "gradient": g, **extra}
