"""Performance cases: the work that users of the library have it do, through its public calls.

Films (2D, state g) and bulk bodies (3D, state h) of the sizes, laws and tolerances of this
repository's workloads, tests and benchmark, from the smallest calls, where launches and
barriers count, to the largest grids; FP64 transforms ("f64") and the precision form with FP32
transforms over an FP64 state ("f32").  Kinds of a case:

  film_rhs       one right-hand side with a fixed number of outside iterations (an external
                 integrator's call; the first pass starts the outside iteration cold, later
                 passes from the previous one)
  film_step      a solver resumed from a checkpoint that lies on the device makes a number of
                 BS23 step attempts with warm-started outside iterations: the FP64 solver's
                 converged by the stop test, the precision form's a fixed number of them
                 (iter_tol = 0), so that a pass is the same work wherever its sums are rounded
  film_batch     a sweep of independent films resumed and advanced together
  film_gradient  loss and gradient (jc map, h_e knots) of a film solve with frozen steps
  film_readout   h_z of a given state
  bulk_rhs, bulk_step, bulk_readout   the same of bulk bodies (readout: j = curl h)

A right-hand side or a readout of the "f32" form holds single-precision values widened to FP64;
run() returns them as the single-precision tensors that they are.  Likewise what depends on an
"f32" solve as a whole (states, gradients).
"""
import math

import numpy as np
import torch

from paper_1801_04869_gb300 import native

DEV = "cuda"


# ------------------------------------------------------------------------------------------
# cases
# ------------------------------------------------------------------------------------------
def listed():
    return [
        # the smallest call: a right-hand side on a lock-step test grid, latency alone
        dict(name="film_rhs_64_f64", kind="film_rhs", nx=64, ny=64, prec=0, shape="rect", side=32,
             n=19.0, amp=0.5, iters=4, jcmap=False, gamma=1.0),
        # the square film of 64 x 64 cells in 128 x 128, FP64: four attempts of its ramp
        dict(name="film_step_128_f64", kind="film_step", nx=128, ny=128, prec=0, shape="rect",
             side=64, n=19.0, amp=0.3, attempts=4, count_iters=0),
        # a disk with a filled hole, a jc map and the elliptic law, sides that are no powers of two
        dict(name="film_rhs_512_hole_f32", kind="film_rhs", nx=512, ny=512, prec=1, shape="hole",
             side=201, n=30.0, amp=0.4, iters=6, jcmap=True, gamma=1.5),
        # the strip of the paper's Figure 2 (1024 x 256 cells), the precision form
        dict(name="film_rhs_1024x256_f32", kind="film_rhs", nx=1024, ny=256, prec=1, shape="rect",
             side=511, n=30.0, amp=0.8, iters=5, jcmap=False, gamma=1.0),
        # the plain FP64 solver on a large film
        dict(name="film_rhs_1024_f64", kind="film_rhs", nx=1024, ny=1024, prec=0, shape="disk",
             side=487, n=30.0, amp=0.85, iters=5, jcmap=False, gamma=1.0),
        # the benchmark's film: 1024 x 512 cells in 2048 x 2048, two step attempts
        dict(name="film_step_2048_f32", kind="film_step", nx=2048, ny=2048, prec=1, shape="rect",
             side=1024, n=30.0, amp=0.3, attempts=2, count_iters=11),
        # a sweep of small films advanced by one call
        dict(name="film_batch_24_f32", kind="film_batch", count=24, prec=1, max_side=128, attempts=2,
             count_iters=8),
        # gradient of a short frozen solve, the gradient workload's film at half its grid
        dict(name="film_gradient_512_f32", kind="film_gradient", nx=512, ny=512, prec=1,
             shape="rect", side=256, n=30.0, amp=0.4, steps=3, ckpt=2),
        # the field map of an ordinary film, as a ramp records it at every output time
        dict(name="film_readout_256_f32", kind="film_readout", nx=256, ny=256, prec=1,
             shape="disk", side=117, n=30.0, amp=0.5),
        # a small bulk body in FP64: a ball with odd diameter
        dict(name="bulk_rhs_32_f64", kind="bulk_rhs", nx=32, ny=32, nz=32, prec=0, shape="ball",
             side=17, n=25.0, iters=4, b0=0.0),
        # the cube of 64^3 cells in 128^3: two step attempts of its ramp
        dict(name="bulk_step_128_f32", kind="bulk_step", nx=128, ny=128, nz=128, prec=1,
             shape="box", side=64, n=25.0, attempts=2),
        # the largest: the cube of 128^3 cells in 256^3
        dict(name="bulk_rhs_256_f32", kind="bulk_rhs", nx=256, ny=256, nz=256, prec=1, shape="box",
             side=128, n=25.0, iters=5, b0=0.0),
    ]


def _phases(c):
    """Rough cost of a pass: cells x transforms x relative cost of the precision."""
    k = c["kind"]
    if k == "film_batch":
        side = 256 if c["max_side"] <= 128 else 512
        return c["count"] * side * side * c["attempts"] * 3 * (5 + 4 * c["count_iters"]) * (60 if c["prec"] == 0 else 12)
    cells = c["nx"] * c["ny"] * c.get("nz", 1)
    it = c.get("iters", c.get("count_iters") or 6)
    if k == "film_gradient":
        rounds = 3 * c["steps"] * 3 * (5 + 4 * 6)
    elif k.startswith("film"):
        rounds = 3 if k == "film_readout" else (5 + 4 * it) * (3 * c["attempts"] if "attempts" in c else 1)
    else:
        rounds = 15 if k == "bulk_readout" else 30 * (1 + it) * (3 * c["attempts"] if "attempts" in c else 1)
    return cells * rounds * ((20 if k.startswith("film") else 11) if c["prec"] == 0 else 1)


def draw(rng):
    top = max(_phases(c) for c in listed())
    while True:
        kind = rng.choice(["film_rhs", "film_rhs", "film_step", "film_batch", "film_gradient",
                           "film_readout", "bulk_rhs", "bulk_rhs", "bulk_step", "bulk_readout"])
        prec = rng.choice([0, 1])
        if kind == "film_batch":
            c = dict(kind=kind, count=rng.randint(3, 40), prec=prec, max_side=rng.choice([96, 128, 250]),
                     attempts=rng.randint(1, 2), count_iters=rng.randint(4, 12))
        elif kind.startswith("film"):
            lx = rng.randint(6, 11)
            ly = min(11, max(6, lx + rng.choice([-2, -1, 0, 0, 0, 1, 2])))
            if kind in ("film_gradient", "film_step"):      # square grids in the workloads
                ly = lx
            if kind == "film_gradient":
                lx = ly = min(lx, 9 if prec == 1 else 10)
            if kind == "film_readout" and prec == 1:
                lx, ly = min(lx, 9), min(ly, 9)
            nx, ny = 1 << lx, 1 << ly
            side = rng.randint(min(nx, 2 * ny) * 5 // 16, min(nx, 2 * ny) // 2 + 1)
            c = dict(kind=kind, nx=nx, ny=ny, prec=prec, shape=rng.choice(["rect", "disk", "hole"]),
                     side=side, n=rng.choice([19.0, 30.0, 50.0]))
            if kind == "film_rhs":
                jcmap = rng.random() < 0.4
                top_amp = 0.4 if jcmap else 0.85 if prec == 0 else 0.7 if c["n"] > 30.0 or max(nx, ny) > 1024 else 0.8
                c.update(amp=round(rng.uniform(0.5, 1.0) * top_amp, 3),
                         iters=rng.randint(1, 9), jcmap=jcmap, gamma=rng.choice([1.0, 1.0, 1.5]))
            elif kind == "film_step":
                c.update(amp=round(rng.uniform(0.2, 0.5), 3), attempts=rng.randint(1, 4 if prec == 0 else 2),
                         count_iters=0 if prec == 0 else rng.randint(4, 14))
            elif kind == "film_gradient":
                c.update(amp=round(rng.uniform(0.2, 0.4), 3), steps=rng.randint(1, 5),
                         ckpt=rng.randint(1, 3), shape="rect", n=rng.choice([19.0, 30.0]))
            else:
                c.update(amp=round(rng.uniform(0.3, 0.85), 3))
        else:
            l0 = rng.randint(4, 8)
            e = [1 << min(8, max(4, l0 + rng.choice([-1, 0, 0, 0, 1]))) for _ in range(3)]
            if kind == "bulk_step":
                e = [1 << l0] * 3
            side = rng.randint(min(e) * 6 // 16, min(e) // 2 + 1)
            c = dict(kind=kind, nx=e[0], ny=e[1], nz=e[2], prec=prec, side=side,
                     shape=rng.choice(["box", "ball", "layer"]), n=rng.choice([19.0, 25.0, 30.0]))
            if kind == "bulk_rhs":
                c.update(iters=rng.randint(1, 6), b0=rng.choice([0.0, 0.0, 0.3]))
            elif kind == "bulk_step":
                c.update(attempts=rng.randint(1, 2))
        if _phases(c) <= 0.9 * top:
            return c


# ------------------------------------------------------------------------------------------
# inputs
# ------------------------------------------------------------------------------------------
T0 = 0.05            # time of the given states
FILM_KNOTS = ((0.0, 1.0), (0.0, 0.5))
BULK_KNOTS = ((0.0, 0.5, 1.0), (0.0, 0.25, 0.25))
STEP_H = 2e-5        # first step of the solves
T_CKPT = T0 + 1e-4   # the output time at which they are checkpointed
T_END = 1.0


def _half(c):
    """Half extents of D: the conductor's long side spans [-1, 1] (film) or [-1/2, 1/2] (bulk)
    with `side` cells; square cells."""
    cell = (2.0 if "nz" not in c else 1.0) / c["side"]
    return [0.5 * cell * c[a] for a in ("nx", "ny", "nz") if a in c], cell


def _centres(count, cell, device=None):
    return (torch.arange(count, dtype=torch.float64, device=device) + (0.5 - 0.5 * count)) * cell


def _film_geometry(c, device="cpu"):
    """uint8 mask and the distance from the film's edge (0 outside), [y, x]."""
    (Lx, Ly), cell = _half(c)
    x, y = _centres(c["nx"], cell, device)[None, :], _centres(c["ny"], cell, device)[:, None]
    ay = 0.5 if c["shape"] == "rect" else 1.0
    ay = min(ay, 0.75 * Ly)
    if c["shape"] == "rect":
        dist = torch.minimum(1.0 - x.abs(), ay - y.abs())
    else:
        r = torch.sqrt(x * x + y * y)
        dist = min(1.0, ay) - r
    dist = dist + 0.5 * cell
    mask = (dist > 0.5 * cell).to(torch.uint8)
    if c["shape"] == "hole":
        hx = 0.1
        mask[(x - hx) ** 2 + y * y <= 0.0625 * min(1.0, ay) ** 2] = 2
    return mask, torch.where(mask != 0, dist.clamp(min=0.0), torch.zeros_like(dist))


def _smooth(shape, g, device):
    """A sum of four low-frequency cosines, at most 1 in magnitude."""
    out = torch.zeros(shape, dtype=torch.float64, device=device)
    for _ in range(4):
        arg = torch.zeros((1,) * len(shape), dtype=torch.float64, device=device)
        for a, s in enumerate(shape):
            v = torch.arange(s, dtype=torch.float64, device=device) / s
            v = v.reshape([s if b == a else 1 for b in range(len(shape))])
            arg = arg + 2 * math.pi * int(g.integers(1, 4)) * v
        out = out + float(g.uniform(-1, 1)) * torch.cos(arg + float(g.uniform(0, 2 * math.pi)))
    return out / max(1.0, float(out.abs().max()))


def _film_state(c, seed):
    """A critical-state sand pile with a smooth disturbance."""
    _, dist = _film_geometry(c, DEV)
    g = np.random.default_rng([seed, 11])
    depth = float(g.uniform(0.2, 0.3))
    return (c["amp"] * dist.clamp(max=depth) * (1.0 + 0.1 * _smooth(dist.shape, g, DEV))).contiguous()


def _jc_map(c, seed):
    z = np.random.default_rng([seed, 12]).standard_normal((c["ny"], c["nx"]))
    return np.exp(0.2 * np.clip(z, -3.5, 3.5) - 0.02)


def _bulk_geometry(c, device="cpu"):
    L, cell = _half(c)
    x = _centres(c["nx"], cell, device)[None, None, :]
    y = _centres(c["ny"], cell, device)[None, :, None]
    z = _centres(c["nz"], cell, device)[:, None, None]
    if c["shape"] == "ball":
        dist = 0.5 - torch.sqrt(x * x + y * y + z * z)
    else:
        dist = torch.minimum(torch.minimum(0.5 - x.abs(), 0.5 - y.abs()), 0.5 - z.abs())
    dist = dist + 0.5 * cell
    mask = (dist > 0.5 * cell).to(torch.uint8)
    if c["shape"] == "layer":            # a cutting layer across the body
        mask = torch.where((mask != 0) & (x.abs() < 1.1 * cell) & (y > 0), torch.full_like(mask, 2), mask)
    return mask, torch.where(mask != 0, dist.clamp(min=0.0), torch.zeros_like(dist))


def _bulk_state(c, seed):
    """A shielding profile |grad h_z| ~ jc with smooth disturbances of every component (half of
    that where the Kim law lowers jc)."""
    mask, dist = _bulk_geometry(c, DEV)
    g = np.random.default_rng([seed, 13])
    h = torch.zeros((3,) + tuple(mask.shape), dtype=torch.float64, device=DEV)
    h[2] = 0.2 - (0.5 if c.get("b0", 0.0) > 0 else 1.0) * dist.clamp(max=float(g.uniform(0.1, 0.15)))
    for k in range(3):
        h[k] += 0.03 * _smooth(mask.shape, g, DEV)
    return h


def _film_problem(c, seed, **over):
    (Lx, Ly), _ = _half(c)
    jc = _jc_map(c, seed) if c.get("jcmap") or c["kind"] == "film_gradient" else None
    fixed = c.get("count_iters", 0)
    kw = dict(dim=2, nx=c["nx"], ny=c["ny"], Lx=Lx, Ly=Ly, mask=_film_geometry(c)[0].numpy(),
              n=c["n"], rho_out=1.0, precision=c["prec"], iter_tol=0.0 if fixed else 2e-4,
              iter_max=fixed or 3000, rtol=1e-6, atol=1e-6, he_knots=FILM_KNOTS, gamma=c.get("gamma", 1.0), jc_map=jc)
    kw.update(over)
    return native.Problem(**kw)


def _bulk_problem(c, **over):
    L, _ = _half(c)
    kw = dict(dim=3, nx=c["nx"], ny=c["ny"], nz=c["nz"], Lx=L[0], Ly=L[1], Lz=L[2],
              mask=_bulk_geometry(c)[0].numpy(), n=c["n"], rho_out=5.0, precision=c["prec"],
              iter_tol=1e-4, iter_max=3000, rtol=1e-6, atol=1e-6, he_knots=BULK_KNOTS,
              b0=c.get("b0", 0.0))
    kw.update(over)
    return native.Problem(**kw)


def _films(c):
    """The films of a sweep: shape, side, power law and ramp amplitude vary."""
    g = np.random.default_rng([c["count"], c["max_side"], 14])
    out = []
    for i in range(c["count"]):
        side = int(g.integers(64, c["max_side"] + 1))
        n = 1 << math.ceil(math.log2(2 * side))
        out.append(dict(kind="film_step", nx=n, ny=n, prec=c["prec"], side=side, amp=0.3,
                        shape=("rect", "disk")[int(g.integers(0, 2))], n=(19.0, 30.0, 50.0)[int(g.integers(0, 3))],
                        ramp=float(g.uniform(0.2, 1.0)), count_iters=c["count_iters"]))
    return out


def _ramp(f):
    return ((0.0, 1.0), (0.0, f["ramp"]))


def _gradient_plan(c, seed):
    """Frozen steps, outside-iteration counts and the target of a short solve."""
    g = np.random.default_rng([seed, 15])
    steps = [(T0 + 1e-4 * i, 1e-4) for i in range(c["steps"])]
    counts = [int(g.integers(3, 8)) for _ in range(3 * c["steps"])]
    return steps, counts


def prepare(case, seed):
    c = case
    k = c["kind"]
    s = {"case": c}
    if k == "film_batch":
        films = _films(c)
        s["ps"] = [_film_problem(f, seed, he_knots=_ramp(f)) for f in films]
        for i, (p, f) in enumerate(zip(s["ps"], films)):
            p.mf_set_state(T0, _film_state(f, seed + i), h=STEP_H)
        native.advance_batch(s["ps"], [T_CKPT] * len(films))
        s["blobs"] = [p.mf_checkpoint_save() for p in s["ps"]]
        s["y"] = [p.state_tensor() for p in s["ps"]]
        return s
    film = k.startswith("film")
    s["p"] = _film_problem(c, seed) if film else _bulk_problem(c)
    y = _film_state(c, seed) if film else _bulk_state(c, seed)
    if k.endswith("_step"):
        s["p"].mf_set_state(T0, y, h=STEP_H)
        s["p"].mf_advance(T_CKPT)
        s["blob"] = s["p"].mf_checkpoint_save()
        s["y"] = y
    else:
        s["y"] = y
        s["out"] = torch.zeros_like(y)
    if k == "film_gradient":
        s["steps"], s["counts"] = _gradient_plan(c, seed)
        s["target"] = 0.05 * _smooth((c["ny"], c["nx"]), np.random.default_rng([seed, 16]), DEV)
    return s


# ------------------------------------------------------------------------------------------
# one pass
# ------------------------------------------------------------------------------------------
def _shown(c, t):
    return t.float() if c["prec"] == 1 else t


def run(state):
    s, c = state, state["case"]
    k = c["kind"]
    if k.endswith("_rhs"):
        s["p"].mf_rhs(T0, s["y"], s["out"], force_iters=c["iters"], allow_noconv=True)
        return _shown(c, s["out"])
    if k.endswith("_step"):
        p = s["p"]
        p.mf_checkpoint_restore(s["blob"])
        p.mf_advance(T_END, max_attempts=c["attempts"])
        t, _ = p.mf_get_state(s["y"])
        return {"t": t, "y": _shown(c, s["y"])}
    if k == "film_batch":
        for p, b in zip(s["ps"], s["blobs"]):
            p.mf_checkpoint_restore(b)
        native.advance_batch(s["ps"], [T_END] * len(s["ps"]), max_attempts=c["attempts"])
        for p, y in zip(s["ps"], s["y"]):
            p.mf_get_state(y)
        return [_shown(c, y) for y in s["y"]]
    if k == "film_gradient":
        loss, jcbar, knots, _ = s["p"].mf_film_solve_gradient(s["y"], s["target"], s["steps"], s["counts"],
                                                              ckpt_every=c["ckpt"])
        return {"loss": loss, "jcbar": _shown(c, jcbar),
                "knots": np.array(knots, dtype=np.float32 if c["prec"] == 1 else np.float64)}
    s["p"].mf_readout(native.MF_READ_HZ if k == "film_readout" else native.MF_READ_J, out=s["out"], t=T0, y=s["y"])
    return _shown(c, s["out"])


def work(case):
    """Inputs read once, outputs written once; the transforms (2.5 N log2 N each for N real
    values) that the method takes, plus the power laws (one transcendental, counted as 20)."""
    c = case
    if c["kind"] == "film_batch":
        w = [work(dict(kind="film_step", nx=n, ny=n, prec=c["prec"], attempts=c["attempts"],
                       iters=c["count_iters"]))
             for n in [256 if c["max_side"] > 64 else 128] * c["count"]]
        return {"bytes": sum(x["bytes"] for x in w), "flops": sum(x["flops"] for x in w)}
    cells = c["nx"] * c["ny"] * c.get("nz", 1)
    fields = 3 if "nz" in c else 1
    byts = cells * (16 * fields + 1)
    per = 2.5 * cells * math.log2(cells)
    film = "nz" not in c
    it = c.get("iters", c.get("count_iters") or (6 if film else 4))
    # film: g, g_x, g_y, e_x, e_y, h_in and two round trips per iteration (the last one is half);
    # bulk: a round trip of three components for j, -curl e and two per iteration
    rhs = (6 + 4 * it - 2) * per if film else (12 + 12 * it) * per
    rhs += cells * 20
    n = 3 * c["attempts"] if "attempts" in c else 1
    if c["kind"].endswith("_readout"):
        return {"bytes": byts, "flops": (2 if film else 6) * per}
    if c["kind"] == "film_gradient":
        # forward, the segment recomputed from its checkpoint, and the product of each call
        return {"bytes": cells * 33, "flops": 3 * c["steps"] * 3 * (6 + 4 * 5) * per}
    return {"bytes": byts, "flops": n * rhs}


# ------------------------------------------------------------------------------------------
# the same in 64 bits with torch alone
# ------------------------------------------------------------------------------------------
def _k(n, L):
    m = torch.fft.fftfreq(n, d=1.0 / n, dtype=torch.float64, device=DEV)
    k = math.pi * m / L
    odd = k.clone()
    odd[n // 2] = 0.0
    return k, odd


class _Film:
    def __init__(self, c, seed, knots=FILM_KNOTS):
        (Lx, Ly), cell = _half(c)
        self.c, self.cell = c, cell
        self.mask = _film_geometry(c)[0].to(DEV)
        self.out, self.sc = self.mask == 0, self.mask == 1
        kx, kxo = _k(c["nx"], Lx)
        ky, kyo = _k(c["ny"], Ly)
        k2 = kx[None, :] ** 2 + ky[:, None] ** 2
        G = torch.exp(-k2 * cell * cell)              # sigma^2 = 2 cell^2
        ka = torch.sqrt(k2)
        self.Dx, self.Dy = 1j * kxo[None, :] * G, 1j * kyo[:, None] * G
        self.K1 = torch.where(ka > 0, 2.0 / torch.where(ka > 0, ka, torch.ones_like(ka)), torch.zeros_like(ka))
        self.K2, self.Kh = 0.35 * ka * G, 0.5 * ka
        jc = _jc_map(c, seed) if c.get("jcmap") or c["kind"] == "film_gradient" else np.ones((c["ny"], c["nx"]))
        self.jc = torch.as_tensor(jc, device=DEV)
        self.knots = knots
        self.n_out = int(self.out.sum())
        self.warm = self.committed = None
        self.first = False

    def hed(self, t):
        (t0, t1), (v0, v1) = self.knots
        return (v1 - v0) / (t1 - t0)

    @staticmethod
    def ap(m, f):
        return torch.fft.ifft2(m * torch.fft.fft2(f)).real

    def e(self, g):
        gh = torch.fft.fft2(g)
        jx, jy = torch.fft.ifft2(self.Dy * gh).real, -torch.fft.ifft2(self.Dx * gh).real
        ig2 = torch.where(self.sc, 1.0 / self.c.get("gamma", 1.0) ** 2, 1.0)
        j2 = jx * jx + jy * jy * ig2
        tiny = torch.where(j2 > 0, j2, torch.ones_like(j2))
        p = torch.where(j2 > 0, (tiny / self.jc ** 2) ** (0.5 * (self.c["n"] - 1.0)), torch.zeros_like(j2))
        rho = torch.where(self.sc, p / self.jc, torch.ones_like(p))
        return rho * jx, rho * jy * ig2

    def outside(self, h_in, hed, start, iters, tol):
        """(g_dot, last iterate, converged) from the given free-space start."""
        N = h_in.numel()
        zero = torch.zeros_like(h_in)
        hd = torch.where(self.out, start, h_in)
        hd = torch.where(self.out, hd - (hd.sum() - N * hed) / self.n_out, hd)
        for i in range(iters):
            u = self.ap(self.K1, hd)
            gd = u - torch.where(self.out, u, zero).sum() / self.n_out
            if tol is not None:
                r = float(torch.where(self.out, gd.abs(), zero).sum() / self.n_out)
                if r < tol:
                    return torch.where(self.out, zero, gd), hd, True, r
            if i == iters - 1:
                break
            w = self.ap(self.K2, torch.where(self.out, gd, zero))
            hd = torch.where(self.out, hd - w, hd)
            hd = torch.where(self.out, hd - (hd.sum() - N * hed) / self.n_out, hd)
        return torch.where(self.out, zero, gd), hd, tol is None, (r if tol is not None else 0.0)

    def rhs(self, t, g, iters=None):
        ex, ey = self.e(g)
        curl = torch.fft.ifft2(self.Dx * torch.fft.fft2(ey) - self.Dy * torch.fft.fft2(ex)).real
        hed = self.hed(t)
        first, self.first = self.first, False
        start = self.committed if first and self.committed is not None else self.warm
        if start is None:
            start = torch.full_like(g, 1.0) * hed
        iters = iters or self.c.get("count_iters", 0)
        gd, hd, ok, r = self.outside(-curl, hed, start, iters or 3000, None if iters else 2e-4)
        self.warm = hd if ok or r < 0.2 else None
        return gd, ok

    def accept(self):
        self.committed = self.warm

    def begin(self):
        self.first = True


class _Bulk:
    def __init__(self, c):
        L, cell = _half(c)
        self.c = c
        self.mask = _bulk_geometry(c)[0].to(DEV)
        self.out, self.sc = self.mask == 0, self.mask == 1
        kx, kxo = _k(c["nx"], L[0])
        ky, kyo = _k(c["ny"], L[1])
        kz, kzo = _k(c["nz"], L[2])
        k2 = kx[None, None, :] ** 2 + ky[None, :, None] ** 2 + kz[:, None, None] ** 2
        self.G = torch.exp(-k2 * 1.5 * cell * cell)   # sigma^2 = 3 cell^2
        self.ik2 = torch.where(k2 > 0, 1.0 / torch.where(k2 > 0, k2, torch.ones_like(k2)), torch.zeros_like(k2))
        self.k = (kxo[None, None, :], kyo[None, :, None], kzo[:, None, None])
        self.warm = None

    def cross(self, f, v):
        a = [torch.fft.fftn(x) for x in v]
        kx, ky, kz = self.k
        h = (ky * a[2] - kz * a[1], kz * a[0] - kx * a[2], kx * a[1] - ky * a[0])
        return torch.stack([torch.fft.ifftn(1j * f * x).real for x in h])

    def curl(self, v):
        return self.cross(self.G, v)

    def hed(self, t):
        return 0.5 if t < 0.5 else 0.0

    def rhs(self, t, h, iters=None):
        j = self.curl(h)
        jc = 1.0
        if self.c.get("b0", 0.0) > 0:
            jc = 1.0 / (1.0 + torch.sqrt((h * h).sum(0)) / self.c["b0"])
        jn = torch.sqrt((j * j).sum(0))
        rho = torch.where(self.sc, (jn / jc) ** (self.c["n"] - 1.0) / jc, torch.full_like(jn, 5.0))
        h_in = -self.curl(rho * j)
        hed = torch.zeros(3, 1, 1, 1, dtype=torch.float64, device=DEV)
        hed[2] = self.hed(t)
        hd = torch.where(self.out, self.warm if self.warm is not None else hed.expand_as(h), h_in)
        tol, ok = 1e-4 * max(1.0, self.hed(t)), iters is not None
        for _ in range(iters or 3000):
            jd = torch.where(self.out, torch.zeros((), dtype=torch.float64, device=DEV), self.curl(hd))
            new = torch.where(self.out, hed + self.cross(self.ik2, jd), hd)
            if iters is None:
                r = float((torch.sqrt(((new - hd) ** 2).sum(0)) * self.out).sum() / self.out.sum())
                ok = r < tol
            hd = new
            if iters is None and ok:
                break
        self.warm = hd
        return hd, ok

    def accept(self):
        pass

    def begin(self):
        pass


def _integrate(F, y, attempts, t=T0, h=STEP_H, rtol=1e-6, atol=1e-6):
    """BS23 with first-same-as-last and the library's step control, away from knots: to the time of
    the checkpoint, then a number of attempts."""
    k1, failed, left = None, False, attempts
    while t < T_CKPT or left > 0:
        lim = T_CKPT if t < T_CKPT else T_END
        left -= t >= T_CKPT
        proposed, clipped = h, t + 1.1 * h >= lim
        h = lim - t if clipped else h
        F.begin()
        ok, err = True, math.inf
        if k1 is None:
            k1, ok = F.rhs(t, y)
            k1 = k1 if ok else None
        if ok:
            k2, ok = F.rhs(t + 0.5 * h, y + 0.5 * h * k1)
        if ok:
            k3, ok = F.rhs(t + 0.75 * h, y + 0.75 * h * k2)
        if ok:
            yn = y + h * (2.0 / 9.0 * k1 + 1.0 / 3.0 * k2 + 4.0 / 9.0 * k3)
            k4, ok = F.rhs(t + h, yn)
        if ok:
            E = h * (-5.0 / 72.0 * k1 + 1.0 / 12.0 * k2 + 1.0 / 9.0 * k3 - 0.125 * k4)
            err = float((E.abs() / (atol + rtol * torch.maximum(y.abs(), yn.abs()))).max())
        if not ok:
            h, failed = 0.5 * h, True
            continue
        fac = max(0.2, 0.9 * err ** (-1.0 / 3.0)) if err > 0 else 5.0
        if err <= 1.0:
            F.accept()
            t, y, k1 = lim if clipped else t + h, yn, k4
            fac = min(fac, 1.0 if failed else 5.0)
            h = proposed * min(fac, 1.0) if clipped and h < proposed else h * fac
            failed = False
        else:
            h, failed = h * fac, True
    return t, y


def _gradient_exact(c, seed):
    """The frozen solve differentiated by torch's autograd: every call starts its outside iteration
    from the previous call's last iterate, the first from h_e_dot."""
    F = _Film(c, seed)
    F.jc.requires_grad_(True)
    kv = torch.tensor(FILM_KNOTS[1], dtype=torch.float64, device=DEV, requires_grad=True)
    steps, counts = _gradient_plan(c, seed)
    g = _film_state(c, seed)
    target = 0.05 * _smooth((c["ny"], c["nx"]), np.random.default_rng([seed, 16]), DEV)
    hed = kv[1] - kv[0]
    warm, it = None, iter(counts)

    def f(g):
        nonlocal warm
        ex, ey = F.e(g)
        curl = torch.fft.ifft2(F.Dx * torch.fft.fft2(ey) - F.Dy * torch.fft.fft2(ex)).real
        start = warm if warm is not None else torch.ones_like(g) * hed
        gd, warm, _, _ = F.outside(-curl, hed, start, next(it), None)
        return gd

    for t, h in steps:
        k1 = f(g)
        k2 = f(g + 0.5 * h * k1)
        k3 = f(g + 0.75 * h * k2)
        g = g + h * (2.0 / 9.0 * k1 + 1.0 / 3.0 * k2 + 4.0 / 9.0 * k3)
    T = steps[-1][0] + steps[-1][1]
    hz = kv[0] + (kv[1] - kv[0]) * T + F.ap(F.Kh, g)
    loss = 0.5 * F.cell ** 2 * ((hz - target) ** 2).sum()
    loss.backward()
    return {"loss": float(loss), "jcbar": F.jc.grad, "knots": kv.grad.cpu().numpy()}


def exact(case, seed):
    c = case
    k = c["kind"]
    if k == "film_gradient":
        return _gradient_exact(c, seed)
    with torch.no_grad():
        if k == "film_batch":
            if c["count"] > 24 or c["max_side"] > 128:      # many small operations: over the time allowed
                return None
            return [_integrate(_Film(f, seed, _ramp(f)), _film_state(f, seed + i), c["attempts"])[1]
                    for i, f in enumerate(_films(c))]
        film = k.startswith("film")
        F = _Film(c, seed) if film else _Bulk(c)
        y = _film_state(c, seed) if film else _bulk_state(c, seed)
        if k.endswith("_rhs"):
            return F.rhs(T0, y, c["iters"])[0]
        if k.endswith("_step"):
            t, y = _integrate(F, y, c["attempts"])
            return {"t": t, "y": y}
        if film:
            return 0.5 * T0 + F.ap(F.Kh, y)
        return F.curl(y)
