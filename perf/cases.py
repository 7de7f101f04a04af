"""What the solver and its surrogate are measured on.

Every case is work that a program does through the public entry points:

  step   one lattice (Solver): restart from heights on the device, a run of
         time steps, the heights read back to the device, as a program does
         that makes trajectories or continues one film after another;
  host   the same from page-locked host memory, one step at a time: a
         program that couples the film to something on the host;
  batch  many lattices at once (Batch): restart, a run of steps, read-out;
  state  the analysis of a state: diagnostics, free energy, power spectra
         and the ring means around a drop, with the results on the host;
  unet   the surrogate of 64 steps: predictions, and one step of its
         training with the gradients.

Inputs follow the recipes of the solver's own workloads: spinodal films of
flat layers plus Gaussian noise, lenses floating on two flat layers, thin
dewetting films, sweeps over random parameters.
"""
import math

import numpy as np
import torch

from paper_2409_16659_gb300 import mlswlbm as B

DEG = math.pi / 180.0


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # the benchmark film: three layers, a window of 64 steps
        dict(name="film3_1024", kind="step", film="film", lattice=2, n=3, nx=1024, ny=1024,
             steps=64),
        # the largest single lattice: four lenses on two flat layers
        dict(name="lens3_2048", kind="step", film="lens", lattice=2, n=3, nx=2048, ny=2048,
             steps=24),
        # the smallest two-dimensional run: a dewetting film followed for
        # tens of thousands of steps, read every few hundred
        dict(name="dewet2_64", kind="step", film="dewet", lattice=2, n=2, nx=64, ny=64, steps=200),
        # odd sides, relaxation time other than 1, every spreading
        # coefficient set, exponents (4, 3)
        dict(name="general4_501x333", kind="step", film="general", lattice=2, n=4, nx=501, ny=333,
             steps=20, tau=0.8, nw=4, mw=3, pseed=11),
        # the pseudo-two-dimensional film of the long runs
        dict(name="film2_1d_512", kind="step", film="film", lattice=1, n=2, nx=512, ny=1,
             steps=2000),
        # one step between two exchanges of the heights with the host
        dict(name="host_film3_1024", kind="host", film="film", lattice=2, n=3, nx=1024, ny=1024,
             steps=1),
        # a stability sweep: uneven instances, 2 to 5 layers, sides 64 to 512
        dict(name="sweep_48", kind="batch", sweep=True, count=48, steps=16, pseed=3),
        # the audit and training windows of the surrogate: alike instances
        dict(name="windows_256x16", kind="batch", sweep=False, n=3, nx=256, ny=256, count=16,
             steps=64),
        # the analysis of one film
        dict(name="state_film3_1024", kind="state", n=3, nx=1024, ny=1024, nbins=512, rings=300),
        # the surrogate: a full batch, one small sample, a training step
        dict(name="unet_predict_256x32", kind="unet", train=False, nx=256, ny=256, count=32),
        dict(name="unet_predict_128x1", kind="unet", train=False, nx=128, ny=128, count=1),
        dict(name="unet_train_256x16", kind="unet", train=True, nx=256, ny=256, count=16),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "line", "host", "batch", "windows", "state",
                       "predict", "train"])
    if kind == "step":
        film = rng.choice(["film", "dewet", "lens", "general"])
        nx, ny = _log_int(rng, 24, 2000), _log_int(rng, 24, 2000)
        n = {"film": rng.randint(1, 5), "dewet": 2, "lens": 3, "general": rng.randint(1, 5)}[film]
        if film == "lens":
            nx = ny = max(64, nx)
        steps = max(2, min(rng.randint(8, 200), int(1.0e8 / (n * nx * ny))))
        c = dict(kind="step", film=film, lattice=2, n=n, nx=nx, ny=ny, steps=steps)
        if film == "general":
            nw, mw = rng.choice([(3, 2), (4, 3), (9, 3), (6, 2)])
            c.update(tau=rng.choice([1.0, 0.8, 1.3]), nw=nw, mw=mw, pseed=rng.randrange(1000))
        return c
    if kind == "line":
        return dict(kind="step", film="film", lattice=1, n=rng.randint(1, 5),
                    nx=_log_int(rng, 48, 1100), ny=1, steps=rng.randint(200, 2000))
    if kind == "host":
        return dict(kind="host", film="film", lattice=2, n=rng.randint(1, 3),
                    nx=_log_int(rng, 64, 1024), ny=_log_int(rng, 64, 1024),
                    steps=rng.choice([1, 1, 2, 5]))
    if kind == "batch":
        return dict(kind="batch", sweep=True, count=rng.randint(4, 48), steps=rng.randint(4, 16),
                    pseed=rng.randrange(1000))
    if kind == "windows":
        nx = rng.randint(48, 256)
        return dict(kind="batch", sweep=False, n=rng.randint(1, 5), nx=nx, ny=rng.randint(48, 256),
                    count=rng.randint(2, 16), steps=rng.randint(16, 64))
    if kind == "state":
        nx, ny = 2 ** rng.randint(6, 10), 2 ** rng.randint(6, 10)
        return dict(kind="state", n=rng.randint(1, 5), nx=nx, ny=ny, nbins=min(nx, ny) // 2,
                    rings=rng.randint(8, 300))
    if kind == "predict":
        return dict(kind="unet", train=False, nx=rng.choice([128, 256]), ny=rng.choice([128, 256]),
                    count=_log_int(rng, 1, 31))
    return dict(kind="unet", train=True, nx=rng.choice([128, 256]), ny=rng.choice([128, 256]),
                count=_log_int(rng, 1, 15))


# ---------------------------------------------------------------------------
# parameters and initial heights
# ---------------------------------------------------------------------------
def _young(gamma, theta_deg, n):
    c = math.cos(theta_deg * DEG) - 1.0
    return [[gamma[i] * c] + [0.0] * (n - i - 1) for i in range(n)]


def _params(c):
    n, film = int(c["n"]), c.get("film", "film")
    p = dict(n=n, lattice=int(c.get("lattice", 2)), nx=int(c["nx"]), ny=int(c["ny"]),
             tau=float(c.get("tau", 1.0)), beta=[1.0] * n, nw=3, mw=2)
    if film == "film":
        gamma = [0.01, 0.008, 0.006, 0.005, 0.004][:n]
        p.update(gamma=gamma, S=_young(gamma, 20.0, n),
                 mu=[1 / 6, 2 / 6, 4 / 6, 4 / 6, 4 / 6][:n], hstar=0.07)
    elif film == "dewet":
        gamma = [0.01] * n
        p.update(gamma=gamma, S=_young(gamma, 20.0, n), mu=[1 / 6] * n, hstar=0.05)
    elif film == "lens":
        g = 0.125 / _radius(c)
        p.update(gamma=[g, g, g], mu=[1 / 6, 2 / 6, 4 / 6], hstar=0.05,
                 S=[[0.0, 0.0, 0.0], [0.0, 0.0], [2.0 * g * (math.cos(20.0 * DEG) - 1.0)]])
    else:
        r = np.random.default_rng(int(c["pseed"]))
        p.update(gamma=[float(v) for v in np.exp(r.uniform(np.log(2e-3), np.log(2e-2), n))],
                 mu=[float(v) for v in np.exp(r.uniform(np.log(0.03), np.log(0.25), n))],
                 beta=[float(v) for v in r.uniform(0.8, 1.5, n)],
                 S=[[float(v) for v in r.uniform(-1e-3, 5e-4, n - i)] for i in range(n)],
                 nw=int(c["nw"]), mw=int(c["mw"]), hstar=float(r.uniform(0.05, 0.1)))
    return p


def _radius(c):
    return min(int(c["nx"]), int(c["ny"])) * (200.0 / 2048.0)


def _lens_heights(c, seed):
    nx, ny, r = int(c["nx"]), int(c["ny"]), _radius(c)
    rng = np.random.default_rng(seed)
    centres = []
    while len(centres) < 4:
        q = rng.uniform(0.0, 1.0, 2) * (nx, ny)
        d = [np.minimum(np.abs(q - o), (nx, ny) - np.abs(q - o)) for o in centres]
        if all(math.hypot(*v) >= 2.6 * r for v in d):
            centres.append(q)
    th = 20.0 * DEG
    rc = r / math.sin(th)
    x = torch.arange(nx, dtype=torch.float64, device="cuda")[None, :]
    y = torch.arange(ny, dtype=torch.float64, device="cuda")[:, None]
    arc = torch.zeros((ny, nx), dtype=torch.float64, device="cuda")
    for cx, cy in centres:
        dx, dy = (x - cx).abs(), (y - cy).abs()
        dx, dy = torch.minimum(dx, nx - dx), torch.minimum(dy, ny - dy)
        cap = torch.sqrt(torch.clamp(rc * rc - dx * dx - dy * dy, min=0.0)) - rc * math.cos(th)
        arc = torch.maximum(arc, torch.clamp(cap, min=0.0))
    one = torch.ones_like(arc)
    return torch.stack([one, 0.3 * r - arc, 0.05 + 2.0 * arc]).float().contiguous()


def _heights(c, seed, count=None):
    """Heights [n][ny][nx] (or [count][n][ny][nx]) on the device."""
    n, nx, ny, film = int(c["n"]), int(c["nx"]), int(c["ny"]), c.get("film", "film")
    if film == "lens":
        return _lens_heights(c, seed)
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    shape = (n, ny, nx) if count is None else (int(count), n, ny, nx)
    means = [0.25] * n if film == "dewet" else [1.0, 0.8, 0.6, 0.7, 0.9][:n]
    m = torch.tensor(means, device="cuda").view(n, 1, 1)
    return (m + 1e-3 * torch.randn(shape, generator=g, device="cuda")).float().contiguous()


def _instances(c, seed):
    """Parameter sets and device heights of a batch."""
    count = int(c["count"])
    if not c["sweep"]:
        p = _params(c)
        h = _heights(c, seed, count)
        return [p] * count, [h[j] for j in range(count)]
    r = np.random.default_rng(int(c["pseed"]))
    q = np.random.default_rng([int(seed), 5])
    params, heights = [], []
    for _ in range(count):
        n, side = int(r.integers(2, 6)), int(r.choice([64, 128, 256, 512]))
        gamma = [float(v) for v in np.exp(r.uniform(np.log(2e-3), np.log(2e-2), n))]
        mu = [1 / 16] + [float(v / 16) for v in np.exp(r.uniform(np.log(0.25), np.log(4.0), n - 1))]
        params.append(dict(n=n, lattice=2, nx=side, ny=side, tau=1.0, gamma=gamma,
                           S=_young(gamma, 20.0, n), mu=mu, beta=[1.0] * n, nw=3, mw=2,
                           hstar=0.07))
        means, amps = r.uniform(0.6, 1.1, n), q.uniform(-1.0, 1.0, n)
        kx, ky = (int(v) for v in q.integers(1, 9, 2))
        x = torch.arange(side, dtype=torch.float64, device="cuda")
        mode = torch.cos(2.0 * math.pi / side * (kx * x[None, :] + ky * x[:, None]))
        t = lambda v: torch.tensor(v, dtype=torch.float64, device="cuda").view(n, 1, 1)  # noqa: E731
        heights.append((t(means) + 1e-4 * t(amps) * mode).float().contiguous())
    return params, heights


# ---------------------------------------------------------------------------
# prepare and run
# ---------------------------------------------------------------------------
EXTRA = [1.0, 0.8, 0.6, 0.5, 1.0]  # the film's tensions over 0.01, viscosity ratios over 4


def _unet_layers():
    """(channels in, channels out) of the fifteen convolutions."""
    down = [(16, 32), (32, 32), (32, 64), (64, 64), (64, 128), (128, 128), (128, 256), (256, 256)]
    up = [(384, 128), (128, 128), (192, 64), (64, 64), (96, 32), (32, 32), (32, 16)]
    return down + up


def _unet_weights(seed):
    """He-normal weights and small biases, flat, in the library's order."""
    r = np.random.default_rng([int(seed), 9])
    out = []
    for ci, co in _unet_layers():
        out.append(r.standard_normal(co * 9 * ci, dtype=np.float32) * np.float32(math.sqrt(2 / (9 * ci))))
        out.append(r.standard_normal(co, dtype=np.float32) * np.float32(0.01))
    return np.concatenate(out)


def _target(h):
    """A film 64 steps later, nearly: its noise smoothed."""
    m = h.mean(dim=(2, 3), keepdim=True)
    s = sum(torch.roll(h, k, d) for k, d in ((1, 2), (-1, 2), (1, 3), (-1, 3)))
    return (m + (0.5 * (h - m) + 0.125 * (s - 4 * m))).contiguous()


def _populations(c, seed):
    """A state in motion: the film's heights in the rest populations, small
    moving ones; and the shifts of its layers."""
    h = _heights(c, seed)
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) + 1)
    f = 1e-4 * torch.randn((h.shape[0], 9) + tuple(h.shape[1:]), generator=g, device="cuda")
    H = h.mean(dim=(1, 2))
    f[:, 0] = h - H.view(-1, 1, 1)
    return h, H.cpu().numpy(), f.cpu().numpy()


def prepare(case, seed):
    kind, st = case["kind"], torch.cuda.current_stream()
    if kind == "step":
        h = _heights(case, seed)
        return dict(kind=kind, steps=int(case["steps"]), h=h, out=torch.empty_like(h),
                    s=B.Solver(_params(case), h.cpu().numpy(), stream=st))
    if kind == "host":
        h = _heights(case, seed).cpu().pin_memory()
        out = torch.empty_like(h).pin_memory()
        return dict(kind=kind, steps=int(case["steps"]), keep=(h, out), h=h.numpy(),
                    out=out.numpy(), s=B.Solver(_params(case), h.numpy(), stream=st))
    if kind == "batch":
        params, heights = _instances(case, seed)
        flat = torch.cat([x.reshape(-1) for x in heights])
        return dict(kind=kind, steps=int(case["steps"]), h=flat, out=torch.empty_like(flat),
                    ids=list(range(len(params))),
                    b=B.Batch(params, [x.cpu().numpy() for x in heights], stream=st))
    if kind == "state":
        h, H, f = _populations(case, seed)
        s = B.Solver(_params(case), h.cpu().numpy(), stream=st)
        s.load_state(H, f)
        r = np.random.default_rng([int(seed), 7])
        return dict(kind=kind, s=s, nbins=int(case["nbins"]), rings=int(case["rings"]),
                    centre=(float(r.uniform(0, case["nx"])), float(r.uniform(0, case["ny"]))))
    c = dict(n=3, nx=case["nx"], ny=case["ny"])
    h = _heights(c, seed, case["count"])
    u = B.UNet(3, int(case["nx"]), int(case["ny"]), int(case["count"]), extra=EXTRA, seed=1,
               in_scale=1.0, out_scale=4.0, stream=st)
    u.set_params(_unet_weights(seed))
    return dict(kind=kind, train=bool(case["train"]), u=u, h=h,
                target=_target(h) if case["train"] else None, out=torch.empty_like(h))


def run(state):
    kind = state["kind"]
    if kind == "step":
        s = state["s"]
        s.set_heights_device(state["h"])
        s.step(state["steps"])
        return s.get_heights_device(state["out"])
    if kind == "host":
        s = state["s"]
        s.set_heights(state["h"])
        s.step(state["steps"])
        return s.get_heights(state["out"])
    if kind == "batch":
        b = state["b"]
        b.set_heights_device_many(state["ids"], state["h"])
        b.step(state["steps"])
        return b.get_heights_device_many(state["ids"], state["out"])
    if kind == "state":
        s = state["s"]
        mass, ke, hmin = s.get_diagnostics()
        prof, cells = s.radial_profile(state["centre"], state["rings"])
        return dict(mass=mass, kinetic=ke, hmin=hmin, energy=s.free_energy(),
                    spectrum=s.spectrum(state["nbins"]), profile=prof, cells=cells)
    u = state["u"]
    if not state["train"]:
        return u.predict(state["h"], state["out"])
    loss = u.train_step(state["h"], state["target"], 1e-5)
    return dict(loss=loss, gradients=u.param_grads())


# ---------------------------------------------------------------------------
# what one pass cannot do without
# ---------------------------------------------------------------------------
def _step_work(p, steps):
    """Restart, steps and read-out of one lattice. For tau = 1 a step maps
    thickness and flux to the next ones (2 or 3 values a layer-site); for
    another tau the populations carry the state. Each step reads and writes
    it once. About 200 operations a layer-site (80 on a line)."""
    sites = p["n"] * p["nx"] * p["ny"]
    flat = p["lattice"] == 1
    words = (2 if flat else 3) if p["tau"] == 1.0 else (3 if flat else 9)
    return 8.0 * sites + 8.0 * words * sites * steps, (80.0 if flat else 200.0) * sites * steps


def work(case):
    kind = case["kind"]
    if kind in ("step", "host"):
        b, f = _step_work(_params(case), int(case["steps"]))
        return dict(bytes=b, flops=f)
    if kind == "batch":
        if case["sweep"]:
            r = np.random.default_rng(int(case["pseed"]))
            b = f = 0.0
            for _ in range(int(case["count"])):
                n, side = int(r.integers(2, 6)), int(r.choice([64, 128, 256, 512]))
                for k in (n, n - 1, n):  # the draws of an instance's parameters
                    r.uniform(0, 1, k)
                w = _step_work(dict(n=n, nx=side, ny=side, lattice=2, tau=1.0), int(case["steps"]))
                b, f = b + w[0], f + w[1]
            return dict(bytes=b, flops=f)
        b, f = _step_work(_params(case), int(case["steps"]))
        return dict(bytes=b * case["count"], flops=f * case["count"])
    cells = float(case["nx"]) * case["ny"]
    if kind == "state":
        n = int(case["n"])
        fft = 5.0 * math.log2(cells) * cells * n
        return dict(bytes=36.0 * n * cells + 8.0 * n * case["nbins"] + 8.0 * (n + 2) * case["rings"],
                    flops=fft + 60.0 * n * cells)
    flops, level = 0.0, [0, 0, 1, 1, 2, 2, 3, 3, 2, 2, 1, 1, 0, 0, 0]
    for (ci, co), lev in zip(_unet_layers(), level):
        flops += 2.0 * 9 * ci * co * cells / 4 ** lev
    nparam = float(sum(co * 9 * ci + co for ci, co in _unet_layers()))
    count = float(case["count"])
    if case["train"]:
        return dict(bytes=24.0 * cells * count + 28.0 * nparam, flops=3.0 * flops * count)
    return dict(bytes=24.0 * cells * count + 4.0 * nparam, flops=flops * count)


# ---------------------------------------------------------------------------
# the same in 64 bits, from the equations
# ---------------------------------------------------------------------------
C9 = [(0, 0), (1, 0), (1, 1), (0, 1), (-1, 1), (-1, 0), (-1, -1), (0, -1), (1, -1)]
W9 = [4 / 9] + [1 / 9, 1 / 36] * 4
C3 = [(0, 0), (1, 0), (-1, 0)]
W3 = [2 / 3, 1 / 6, 1 / 6]


def _at(a, c):
    """a at x + c, periodic; the last two dimensions are (y, x)."""
    if c[0]:
        a = torch.roll(a, -c[0], -1)
    return torch.roll(a, -c[1], -2) if c[1] else a


def _gradient(a, C, W):
    gx = sum(3 * w * c[0] * (_at(a, c) - a) for c, w in zip(C, W) if c[0])
    gy = sum(3 * w * c[1] * (_at(a, c) - a) for c, w in zip(C, W) if c[1]) if len(C) == 9 else 0 * a
    return gx, gy


def _friction(p, h, jx, jy):
    """2 mu_i h_i a_i: the pressure gradients G that drive the fluxes J
    through Stokes layers with slip, J = L G, times the thicknesses."""
    n = p["n"]
    L = [[None] * n for _ in range(n)]
    for j in range(n):
        ub = 0 * h[0]
        for i in range(n):
            m, b = 1.0 / p["mu"][i], p["beta"][i]
            s = -h[j] if j > i else 0 * h[0]
            g = 1.0 if i == j else 0.0
            ub = ub + b * m * (s - g * (h[i] + 0.5 * b))
            L[i][j] = h[i] * ub + m * h[i] ** 2 * (0.5 * s - g * h[i] / 3)
            ub = ub + m * h[i] * (s - 0.5 * g * h[i])
    bx, by = list(jx), list(jy)
    for c in range(n):
        for r in range(c + 1, n):
            l = L[r][c] / L[c][c]
            for q in range(c + 1, n):
                L[r][q] = L[r][q] - l * L[c][q]
            bx[r], by[r] = bx[r] - l * bx[c], by[r] - l * by[c]
    for c in reversed(range(n)):
        for q in range(c + 1, n):
            bx[c], by[c] = bx[c] - L[c][q] * bx[q], by[c] - L[c][q] * by[q]
        bx[c], by[c] = bx[c] / L[c][c], by[c] / L[c][c]
    return [h[i] * bx[i] for i in range(n)], [h[i] * by[i] for i in range(n)]


def _phi(p, k, d):
    """The wetting potential phi_k and its derivative."""
    nw, mw = p["nw"], p["mw"]
    r = k * p["hstar"] / d
    return ((nw * r ** mw - mw * r ** nw) / (nw - mw),
            nw * mw / (nw - mw) * (r ** nw - r ** mw) / d)


def _exact_steps(p, h, steps):
    """Heights [n][ny][nx] after `steps` steps from rest, in 64 bits."""
    n, C, W = p["n"], (C9, W9)[0] if p["lattice"] == 2 else C3, W9 if p["lattice"] == 2 else W3
    Q, om = len(C), 1.0 / p["tau"]
    h = h.double()
    f = [h] + [torch.zeros_like(h) for _ in range(Q - 1)]
    for _ in range(steps):
        h = sum(f)
        jx = sum(c[0] * v for c, v in zip(C, f) if c[0])
        jy = sum(c[1] * v for c, v in zip(C, f) if c[1]) if Q == 9 else torch.zeros_like(h)
        z = torch.cumsum(h, 0)
        gx, gy = _gradient(z, C, W)
        lap = sum(6 * w * (_at(z, c) - z) for c, w in zip(C[1:], W[1:]))
        slope = 1 + 0.5 * (gx * gx + gy * gy)
        ten = [p["gamma"][i] + 0 * h[0] for i in range(n)]
        dis = [0 * h[0] for _ in range(n)]
        for l in range(n):
            for m in range(l + 1, n + 1):
                s = p["S"][l][m - l - 1]
                if s == 0.0:
                    continue
                phi, dphi = _phi(p, m - l, z[m - 1] - (z[l - 1] if l else 0.0))
                e = s * dphi * (slope[l - 1] if l else 1.0)
                if l:
                    ten[l - 1] = ten[l - 1] + s * phi
                    dis[l - 1] = dis[l - 1] - e
                dis[m - 1] = dis[m - 1] + e
        jump = torch.stack([dis[i] - ten[i] * lap[i] for i in range(n)])
        pr = torch.flip(torch.cumsum(torch.flip(jump, [0]), 0), [0])
        px, py = _gradient(pr, C, W)
        Rx, Ry = _friction(p, h, jx, jy)
        Fx, Fy = -h * px + torch.stack(Rx), -h * py + torch.stack(Ry)
        ux, uy = jx / h, jy / h
        u2 = ux * ux + uy * uy
        eq = [None] + [w * h * (3 * (c[0] * ux + c[1] * uy) + 4.5 * (c[0] * ux + c[1] * uy) ** 2 - 1.5 * u2)
                       for c, w in zip(C[1:], W[1:])]
        eq[0] = h - sum(eq[1:])
        f = [_at(f[k] + om * (eq[k] - f[k]) + 3 * W[k] * (C[k][0] * Fx + C[k][1] * Fy),
                 (-C[k][0], -C[k][1])) for k in range(Q)]
    return sum(f)


def _exact_state(case, seed):
    """Diagnostics, free energy, spectra and ring means of the state."""
    p = _params(case)
    _h, H, f = _populations(case, seed)
    n, nx, ny, nb, rings = p["n"], p["nx"], p["ny"], int(case["nbins"]), int(case["rings"])
    f = torch.from_numpy(f).cuda().double()
    d = f.sum(1)
    h = d + torch.from_numpy(H).cuda().double().view(n, 1, 1)
    jx = sum(c[0] * f[:, k] for k, c in enumerate(C9))
    jy = sum(c[1] * f[:, k] for k, c in enumerate(C9))
    z = torch.cumsum(h, 0)
    gx, gy = _gradient(z, C9, W9)
    slope = 1 + 0.5 * (gx * gx + gy * gy)
    energy = sum(p["gamma"][i] * slope[i].sum() for i in range(n))
    for l in range(n):
        for m in range(l + 1, n + 1):
            s = p["S"][l][m - l - 1]
            if s != 0.0:
                phi = _phi(p, m - l, z[m - 1] - (z[l - 1] if l else 0.0))[0]
                energy = energy + s * (phi * (slope[l - 1] if l else 1.0)).sum()
    F = torch.fft.fft2(d - d.mean(dim=(1, 2), keepdim=True)).abs() ** 2
    k = lambda m: torch.fft.fftfreq(m, 1.0 / m, device="cuda", dtype=torch.float64)  # noqa: E731
    b = torch.round(torch.sqrt(k(nx)[None, :] ** 2 + k(ny)[:, None] ** 2)).long().reshape(-1)
    keep = b < nb
    cnt = torch.bincount(b[keep], minlength=nb)
    spec = torch.stack([torch.bincount(b[keep], weights=F[i].reshape(-1)[keep], minlength=nb)
                        for i in range(n)]) / cnt.clamp(min=1)
    r = np.random.default_rng([int(seed), 7])
    cx, cy = float(r.uniform(0, case["nx"])), float(r.uniform(0, case["ny"]))
    dx = torch.arange(nx, device="cuda", dtype=torch.float64) - cx
    dy = torch.arange(ny, device="cuda", dtype=torch.float64) - cy
    dx, dy = dx - nx * torch.round(dx / nx), dy - ny * torch.round(dy / ny)
    ring = torch.floor(torch.sqrt(dx[None, :] ** 2 + dy[:, None] ** 2)).long().reshape(-1)
    keep = ring < rings
    cells = torch.bincount(ring[keep], minlength=rings)
    zs = torch.cat([torch.zeros_like(z[:1]), z])
    prof = torch.stack([torch.bincount(ring[keep], weights=zs[m].reshape(-1)[keep], minlength=rings)
                        for m in range(n + 1)]) / cells.clamp(min=1)
    return dict(mass=h.sum(dim=(1, 2)).cpu().numpy(), kinetic=float(((jx ** 2 + jy ** 2) / (2 * h)).sum()),
                hmin=float(h.min()), energy=float(energy), spectrum=spec.cpu().numpy(),
                profile=prof.cpu().numpy(), cells=cells.cpu().numpy())


def _conv(x, w, b):
    x = torch.nn.functional.pad(x, (1, 1, 1, 1), mode="circular")
    return torch.nn.functional.conv2d(x, w, b)


def _unet_forward(weights, x):
    """The network on input planes x [1][16][ny][nx]: its 16 output planes."""
    act = lambda l, v: torch.relu(_conv(v, *weights[l]))  # noqa: E731
    pool = lambda v: torch.nn.functional.avg_pool2d(v, 2)  # noqa: E731
    up = lambda v: v.repeat_interleave(2, 2).repeat_interleave(2, 3)  # noqa: E731
    s0 = act(1, act(0, x))
    s1 = act(3, act(2, pool(s0)))
    s2 = act(5, act(4, pool(s1)))
    d = act(7, act(6, pool(s2)))
    for l, s in ((8, s2), (10, s1), (12, s0)):
        d = act(l + 1, act(l, torch.cat([up(d), s], 1)))
    return _conv(d, *weights[14])


def _exact_unet(case, seed):
    n, nx, ny, count = 3, int(case["nx"]), int(case["ny"]), int(case["count"])
    h = _heights(dict(n=n, nx=nx, ny=ny), seed, count)
    target = _target(h).double()
    h = h.double()
    flat, weights, off = torch.from_numpy(_unet_weights(seed)).cuda().double(), [], 0
    for ci, co in _unet_layers():
        w = flat[off:off + co * 9 * ci].view(co, 3, 3, ci).permute(0, 3, 1, 2).contiguous()
        b = flat[off + co * 9 * ci:off + co * 9 * ci + co].clone()
        weights.append((w.requires_grad_(case["train"]), b.requires_grad_(case["train"])))
        off += co * 9 * ci + co
    d = h - h.mean(dim=(2, 3), keepdim=True)
    rms = d.square().mean(dim=(1, 2, 3), keepdim=True).sqrt()
    planes = torch.tensor(EXTRA, dtype=torch.float64, device="cuda").view(1, 5, 1, 1)
    out, loss = torch.empty_like(h), 0.0
    for j in range(count):
        x = torch.zeros((1, 16, ny, nx), dtype=torch.float64, device="cuda")
        x[:, :n] = d[j:j + 1] / rms[j:j + 1]
        x[:, n:n + 5] = planes
        with torch.set_grad_enabled(bool(case["train"])):
            y = _unet_forward(weights, x)[:, :n]
            if case["train"]:
                e = (y - (target[j:j + 1] - h[j:j + 1]) * 4.0 / rms[j:j + 1]).square().sum() / h.numel()
                e.backward()
                loss += float(e.detach())
            else:
                out[j] = h[j] + (y - y.mean(dim=(2, 3), keepdim=True))[0] * rms[j] / 4.0
    if not case["train"]:
        return out
    grads = [v for w, b in weights for v in (w.grad.permute(0, 2, 3, 1).reshape(-1), b.grad)]
    return dict(loss=loss, gradients=torch.cat(grads))


def exact(case, seed):
    kind = case["kind"]
    if kind in ("step", "host"):
        out = _exact_steps(_params(case), _heights(case, seed), int(case["steps"]))
        return out.cpu().numpy() if kind == "host" else out
    if kind == "batch":
        params, heights = _instances(case, seed)
        if not case["sweep"]:  # alike instances: side by side in one array
            h = torch.stack(heights).transpose(0, 1).contiguous()
            return _exact_steps(params[0], h, int(case["steps"])).transpose(0, 1).reshape(-1)
        return torch.cat([_exact_steps(p, h, int(case["steps"])).reshape(-1)
                          for p, h in zip(params, heights)])
    if kind == "state":
        return _exact_state(case, seed)
    return _exact_unet(case, seed)
