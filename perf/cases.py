"""Performance cases of the worm-LBM library: what its users have it do, through its public
entry points, from a 64 x 64 test pulse to grids of gigabytes.

Every case is one job as a program runs it: set the start field, step, read the moments (or
the reductions, the state, or gradients).  Handles, options and device inputs are made in
`prepare` and kept, as a program keeps them.  Sizes are those of the repository's own
workloads and tests (the Gaussian test, the 2048 x 2048 pulses, the 4096 x 256 in-plane
film, films of the 96-film recipe, the 1024 x 1024 adjoint) and generic ones between.

`exact` is the method in torch float64, written out here on its own: directions, weights,
worm paths, the time-adaptive schedule, walls, relaxation, moments; gradients by torch's own
differentiation of it.
"""
import math
import random

import numpy as np
import torch

PER, ISO, DIF, SPE = 0, 1, 2, 3
THETA, TREF = 624.8074248458514, 300.0
# wall sets: kinds of x-, x+, y-, y+; wall temperatures; specularities
WALLS = {
    "periodic": ((PER, PER, PER, PER), (300.0,) * 4, (0.0,) * 4),
    "film": ((ISO, ISO, DIF, DIF), (301.0, 300.0, 300.0, 300.0), (0.0,) * 4),
    "channel": ((ISO, ISO, PER, PER), (300.0,) * 4, (0.0,) * 4),
    "square": ((ISO, ISO, ISO, ISO), (300.0, 300.0, 300.0, 301.0), (0.0,) * 4),
    "rough": ((ISO, SPE, DIF, DIF), (301.0, 300.0, 300.0, 300.0), (0.0, 0.0, 0.5, 0.0)),
    "box": ((DIF, DIF, DIF, DIF), (300.0,) * 4, (0.0,) * 4),
}


def listed():
    return [
        # The paper's Gaussian test at its small size: parameter scans run it hundreds of
        # times; a step of it is over in microseconds, so launches and latency count.
        dict(name="pulse_64_q16", kind="run", nx=64, ny=64, q=16, walls="periodic", mfp=8.0,
             steps=500, bf16=False, field=False, graph=0, speed=1.0, emulate_3d=True),
        # A thin film run to its steady state: the windowed steady-state driver, with a
        # reduction after each of the last ten steps of every check.
        dict(name="steady_film_200x24_q32", kind="steady", nx=200, ny=24, q=32, walls="film",
             mfp=24.0, steps=1200, bf16=False, field=False, graph=0, speed=1.0,
             emulate_3d=True),
        # The throughput workload: 16 pulses on a large periodic grid, float32 storage, steps
        # replayed as graphs on a stream of its own.
        dict(name="pulses_2048_q64", kind="run", nx=2048, ny=2048, q=64, walls="periodic",
             mfp=6.09, steps=480, bf16=False, field=False, graph=48, speed=1.0,
             emulate_3d=False),
        # The same with bfloat16 storage.
        dict(name="pulses_2048_q64_bf16", kind="run", nx=2048, ny=2048, q=64, walls="periodic",
             mfp=6.09, steps=480, bf16=True, field=False, graph=48, speed=1.0,
             emulate_3d=False),
        # The in-plane film of the conductivity study, float32, launched step by step as a
        # program without any option set does.
        dict(name="film_4096x256_q128", kind="run", nx=4096, ny=256, q=128, walls="film",
             mfp=256.0, steps=480, bf16=False, field=False, graph=0, speed=1.0,
             emulate_3d=True),
        # The same with bfloat16 storage and graph replay.
        dict(name="film_4096x256_q128_bf16", kind="run", nx=4096, ny=256, q=128, walls="film",
             mfp=256.0, steps=480, bf16=True, field=False, graph=48, speed=1.0,
             emulate_3d=True),
        # A ragged sample with a per-cell mean-free-path field, one specular and one partly
        # specular wall, restarted from a state and read back as one (coupled solvers).
        dict(name="ragged_777x313_q40", kind="state", nx=777, ny=313, q=40, walls="rough",
             mfp=0.0, steps=200, bf16=False, field=True, graph=0, speed=1.0, emulate_3d=True),
        # Sixteen films of the 96-film recipe stepped together, bfloat16, graph replay.
        dict(name="batch_films_16_bf16", kind="films", count=16, recipe=4, steps=192, bf16=True,
             graph=48),
        # A multigray run: eight bands of different speeds and mean free paths on one
        # periodic grid, stepped as a batch in float32.
        dict(name="bands_8x256_q32", kind="bands", count=8, nx=256, ny=256, q=32,
             walls="periodic", steps=200, bf16=False, graph=0),
        # The adjoint workload: log-normal mean-free-path field, checkpoints every 50 steps,
        # gradients of a probe line's temperature.
        dict(name="adjoint_1024_q64", kind="adjoint", nx=1024, ny=1024, q=64, walls="channel",
             mfp=0.0, steps=200, ckpt=50, field=True, speed=1.0, emulate_3d=True),
        # One iteration of an inversion through the torch function: new field in, gradients of
        # temperature and flux out.
        dict(name="inversion_256_q32", kind="autograd", nx=256, ny=256, q=32, walls="film",
             mfp=0.0, steps=96, ckpt=24, field=True, speed=1.0, emulate_3d=True),
        # Monitoring a running film: moments and the float64 reductions of a state.
        dict(name="monitor_4096x256_q128", kind="monitor", nx=4096, ny=256, q=128, walls="film",
             mfp=64.0, steps=24, bf16=False, field=False, graph=0, speed=1.0,
             emulate_3d=True),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more job of the same ranges; at most the largest listed one's updates."""
    kind = rng.choice(["run"] * 6 + ["steady", "state", "films", "bands", "adjoint", "autograd",
                                     "monitor"])
    q = 8 * rng.choice([1, 2, 3, 4, 5, 8, 8, 12, 16, 16, 32])
    if kind == "films":
        return dict(kind=kind, count=rng.randint(3, 16), recipe=rng.randint(5, 10 ** 6),
                    steps=rng.randint(20, 96), bf16=rng.random() < 0.6, graph=rng.choice([0, 48]))
    if kind == "bands":
        nx, ny = _log(rng, 40, 400), _log(rng, 40, 400)
        return dict(kind=kind, count=rng.randint(2, 8), nx=nx, ny=ny, q=min(q, 64),
                    walls=rng.choice(["periodic", "film", "channel"]), steps=rng.randint(20, 150),
                    bf16=rng.random() < 0.3, graph=rng.choice([0, 48]))
    walls = rng.choice(["periodic", "periodic", "film", "film", "channel", "square", "rough",
                        "box"])
    if kind in ("adjoint", "autograd"):
        nx, ny, q = _log(rng, 60, 500), _log(rng, 60, 500), min(q, 64)
        k = rng.randint(5, 30)
        return dict(kind=kind, nx=nx, ny=ny, q=q, walls=walls, mfp=0.0, steps=k * 3 + rng.randint(0, 7),
                    ckpt=k, field=True, speed=1.0, emulate_3d=True)
    top = 64e6 if kind in ("run", "monitor") else 8e6
    nx = _log(rng, 33, 4200)
    ny = _log(rng, 16, max(17, min(2100, top / q / nx * 4)))
    while nx * ny * q > 4 * top:
        nx = max(33, nx // 2)
    steps = rng.randint(11, 300)
    if kind == "steady":
        steps = 40 * rng.randint(2, 5)
    if kind == "monitor":
        steps = rng.randint(2, 20)
    speed = rng.choice([1.0, 1.0, 1.0, 0.6])
    return dict(kind=kind, nx=nx, ny=ny, q=q, walls=walls, mfp=float(_log(rng, 2, 400)), steps=steps,
                bf16=rng.random() < 0.4, field=rng.random() < 0.3, graph=rng.choice([0, 0, 48]),
                speed=speed, emulate_3d=rng.random() < 0.7)


# ------------------------------------------------------------------------------ inputs
def _pulses(nx, ny, rng, n=16, dev="cuda"):
    """n Gaussian pulses of 1 K at random centres (minimum-image distance), float32."""
    y = torch.arange(ny, device=dev, dtype=torch.float64)[:, None]
    x = torch.arange(nx, device=dev, dtype=torch.float64)[None, :]
    out = torch.zeros(ny, nx, device=dev, dtype=torch.float64)
    for _ in range(n):
        cx, cy = rng.uniform(0, nx), rng.uniform(0, ny)
        s = math.exp(rng.uniform(math.log(4.0), math.log(32.0)))
        dx, dy = x - cx, y - cy
        dx = dx - nx * torch.round(dx / nx)
        dy = dy - ny * torch.round(dy / ny)
        out += torch.exp(-(dx * dx) / (2 * s * s)) * torch.exp(-(dy * dy) / (2 * s * s))
    return out.float()


def _profile(nx, ny, rng, hot, cold, dev="cuda"):
    """A film's linear start profile with a smooth perturbation of a few per cent."""
    x = (torch.arange(nx, device=dev, dtype=torch.float64) + 1.0) / (nx + 1.0)
    y = (torch.arange(ny, device=dev, dtype=torch.float64) + 0.5) / ny
    out = ((hot - TREF) + (cold - hot) * x)[None, :].expand(ny, nx).clone()
    for _ in range(4):
        a, px, py = 0.03 * rng.standard_normal(), rng.integers(1, 6), rng.integers(0, 4)
        out += a * torch.sin(math.pi * int(px) * x)[None, :] * torch.cos(math.pi * int(py) * y)[:, None]
    return out.float()


def _start(case, rng):
    kinds, tw, _ = WALLS[case["walls"]]
    if kinds[0] == ISO and tw[0] != tw[1]:
        return _profile(case["nx"], case["ny"], rng, tw[0], tw[1])
    return _pulses(case["nx"], case["ny"], rng, n=16 if case["nx"] >= 1000 else 1)


def _mfp_field(nx, ny, rng, corr=32.0):
    """Smooth random log-normal mean free path around 8 cells (correlation 32 cells), within
    three standard deviations (shorter than a cell and a half would be refused)."""
    noise = torch.from_numpy(rng.standard_normal((ny, nx))).cuda()
    ky = torch.fft.fftfreq(ny, device="cuda", dtype=torch.float64)[:, None]
    kx = torch.fft.fftfreq(nx, device="cuda", dtype=torch.float64)[None, :]
    corr = min(corr, nx / 8, ny / 8)
    kern = torch.exp(-2.0 * (math.pi * corr) ** 2 * (kx * kx + ky * ky))
    g = torch.fft.ifft2(torch.fft.fft2(noise) * kern).real
    g = (g - g.mean()) / g.std()
    return torch.exp(math.log(8.0) + 0.5 * g.clamp(-3.0, 3.0)).float()


def _specs(case):
    """The instances of a batch case (sizes from the case alone)."""
    if case["kind"] == "films":        # the recipe of the 96-film batch
        r = random.Random(case["recipe"])
        out = []
        for _ in range(case["count"]):
            ny = _log(r, 16, 512)
            nx = int(round(ny * r.uniform(8, 32)))
            kn = math.exp(r.uniform(math.log(0.01), math.log(100.0)))
            q = r.choice((16, 32, 64, 128, 256))
            while nx * ny * q > 3e8:
                nx, ny = nx // 2, ny // 2
            out.append(dict(nx=nx, ny=ny, q=q, mfp=max(1.6, kn * ny), walls="film", speed=1.0))
        return out
    return [dict(nx=case["nx"], ny=case["ny"], q=case["q"], mfp=4.0 * 2.0 ** k,
                 walls=case["walls"], speed=1.0 - 0.09 * k) for k in range(case["count"])]


def _inputs(case, seed):
    """Device inputs of a case, from the seed alone."""
    rng = np.random.default_rng(seed)
    if case["kind"] in ("films", "bands"):
        return dict(dT=[_start(s, rng) for s in _specs(case)])
    got = dict(dT=_start(case, rng))
    if case["field"]:
        got["mfp"] = _mfp_field(case["nx"], case["ny"], rng)
    if case["kind"] == "state":
        # a state out of equilibrium: the start field with per-direction deviations of 10 %
        d = _framed_equilibrium(case, got["dT"])
        g = torch.Generator(device="cuda").manual_seed(seed)
        d *= 1.0 + 0.1 * torch.randn(d.shape, generator=g, device="cuda", dtype=torch.float32)
        got["state"] = d.float()
    if case["kind"] == "adjoint":
        got["gT"] = torch.zeros(case["ny"], case["nx"], device="cuda")
        got["gT"][:, (3 * case["nx"]) // 4] = 1.0 / case["ny"]
    if case["kind"] == "autograd":
        got["wT"] = torch.from_numpy(rng.uniform(0.5, 1.5, (case["ny"], case["nx"]))).cuda().float()
    return got


def _framed_equilibrium(case, dT):
    w = torch.tensor(_Lattice.of(case["q"]).w, device="cuda")
    de = _e_eq(TREF + dT.double()) - _e_eq(TREF)
    de = torch.nn.functional.pad(de[None, None], (1, 1, 1, 1), mode="replicate")[0, 0]
    return (w[:, None, None] * de[None]).float()


def prepare(case, seed):
    import paper_1911_00180_gb300 as wl
    from paper_1911_00180_gb300 import wlbm as api
    got = _inputs(case, seed)
    kind = case["kind"]
    st = dict(case=case, **got)
    if kind == "autograd":
        kinds, tw, sp = WALLS[case["walls"]]
        st["spec"] = dict(nx=case["nx"], ny=case["ny"], q=case["q"], bc=kinds, steps=case["steps"],
                          ckpt=case["ckpt"], emulate_3d=case["emulate_3d"], specularity=sp,
                          speed=case["speed"])
        st["tw"] = torch.tensor(tw, dtype=torch.float64)
        return st
    # graph replay wants a stream of the program's own
    st["stream"] = torch.cuda.Stream() if case.get("graph") else torch.cuda.current_stream()
    st["stream"].wait_stream(torch.cuda.current_stream())
    bf16 = wl.STORE_BF16_DEV if case.get("bf16") else wl.STORE_FP32_DEV
    with torch.cuda.stream(st["stream"]):
        if kind in ("films", "bands"):
            specs = []
            for s in _specs(case):
                kinds, tw, sp = WALLS[s["walls"]]
                specs.append(dict(nx=s["nx"], ny=s["ny"], q=s["q"], bc=kinds, t_wall=tw,
                                  specularity=sp, mfp=s["mfp"], speed=s["speed"]))
            st["h"] = wl.WormLBMBatch(specs, storage=bf16, stream=st["stream"])
            if case["graph"]:
                st["h"].wlbm_batch_set_option(api.OPT_GRAPH_STEPS, case["graph"])
            return st
        kinds, tw, sp = WALLS[case["walls"]]
        st["h"] = wl.WormLBM(case["nx"], case["ny"], case["q"],
                             mfp=None if case["field"] else case["mfp"],
                             mfp_field=got.get("mfp"), bc=kinds, t_wall=tw, specularity=sp,
                             storage=bf16, emulate_3d=case["emulate_3d"], speed=case["speed"],
                             stream=st["stream"])
        if case.get("graph"):
            st["h"].wlbm_set_option(api.OPT_GRAPH_STEPS, case["graph"])
        if kind == "monitor":
            st["h"].wlbm_init_temperature(got["dT"])
            st["h"].wlbm_step(case["steps"])
    return st


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "autograd":
        from paper_1911_00180_gb300 import autograd as ag
        mfp = state["mfp"].clone().requires_grad_(True)
        tw = state["tw"].clone().requires_grad_(True)
        dT0 = state["dT"].clone().requires_grad_(True)
        T, qx, qy = ag.wlbm_run_moments(mfp, tw, dT0, state["spec"])
        loss = (state["wT"] * T).mean() + 50.0 * qx.mean() + 20.0 * (qy * state["wT"]).mean()
        loss.backward()
        return [T.detach(), qx.detach(), qy.detach(), mfp.grad, tw.grad, dT0.grad]
    h = state["h"]
    with torch.cuda.stream(state["stream"]):
        if kind in ("films", "bands"):
            h.wlbm_batch_init_temperature(state["dT"])
            h.wlbm_batch_step(case["steps"])
            return [list(v.wlbm_moments()) for v in h.instances]
        if kind == "run":
            h.wlbm_init_temperature(state["dT"])
            h.wlbm_step(case["steps"])
            return list(h.wlbm_moments())
        if kind == "state":
            h.wlbm_init_temperature(state["dT"])
            h.wlbm_set_state(state["state"])
            h.wlbm_step(case["steps"])
            # the interior is the state; the frame around it holds the walls' own values
            return [h.wlbm_get_state()[:, 1:-1, 1:-1]]
        if kind == "steady":
            h.wlbm_init_temperature(state["dT"])
            steps, conv, r = h.wlbm_run_steady(case["steps"], case["steps"] // 4, 0.0, 10)
            return [steps, int(conv), torch.tensor(r[:8], dtype=torch.float64),
                    *h.wlbm_moments()]
        if kind == "monitor":
            T, qx, qy = h.wlbm_moments()
            return [T, qx, qy, torch.tensor(h.wlbm_reduce()[:8], dtype=torch.float64)]
        h.wlbm_adjoint_forward(state["dT"], case["steps"], case["ckpt"])
        T, qx, qy = h.wlbm_moments()
        g_mfp, g_tw, g_dT0 = h.wlbm_adjoint_backward(state["gT"])
        return [T, qx, qy, g_mfp, torch.tensor(g_tw, dtype=torch.float64), g_dT0]


def work(case):
    """Bytes: fields read and written once and, where a state is kept, that state written
    once and read once.  Operations: 5 per direction, cell and step (relaxation 1 - W and
    source, two products, a sum, the local energy); a reverse step 8."""
    kind = case["kind"]
    if kind in ("films", "bands"):
        cells = [(s["nx"] * s["ny"], s["q"]) for s in _specs(case)]
    else:
        cells = [(case["nx"] * case["ny"], case["q"])]
    el = 2 if case.get("bf16") else 4
    fields = sum(16 * c for c, _ in cells)
    state = sum(c * q * el for c, q in cells)
    upd = sum(c * q for c, q in cells) * case["steps"]
    if kind == "monitor":
        return {"bytes": state + sum(28 * c for c, _ in cells), "flops": 8 * state / el}
    if kind == "state":
        return {"bytes": 2 * state, "flops": 5 * upd}
    if kind in ("adjoint", "autograd"):
        return {"bytes": 3 * fields + 2 * state, "flops": 18 * upd}
    return {"bytes": fields + 2 * state, "flops": 5 * upd}


# ------------------------------------------------------------- the method in float64
HOPS = ((1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1))
NORMAL = ((1, 0), (-1, 0), (0, 1), (0, -1))


class _Lattice:
    """Ring directions, angular weights, worm paths and the mean-hop correction of Q."""
    _made = {}

    @classmethod
    def of(cls, q):
        if q not in cls._made:
            cls._made[q] = cls(q)
        return cls._made[q]

    def __init__(self, q):
        m = q // 8
        ring = [(x, y) for x in range(-m, m + 1) for y in range(-m, m + 1)
                if max(abs(x), abs(y)) == m]
        ring.sort(key=lambda v: math.atan2(v[1], v[0]) % (2 * math.pi))
        self.dirs = ring
        ang = [math.atan2(y, x) for x, y in ring]
        gap = [(ang[(i + 1) % q] - ang[i]) % (2 * math.pi) for i in range(q)]
        self.w = np.array([(gap[i - 1] + gap[i]) / (4 * math.pi) for i in range(q)])
        self.s = np.array([(x / math.hypot(x, y), y / math.hypot(x, y)) for x, y in ring])
        self.worm, mean = [], 0.0
        for a, b in ring:
            px = py = 0
            path, length = [], 0.0
            for n in range(1, m + 1):
                pick, best = -1, m * m
                for k, (hx, hy) in enumerate(HOPS):
                    d2 = (m * (px + hx) - n * a) ** 2 + (m * (py + hy) - n * b) ** 2
                    if d2 <= best:
                        pick, best = k, d2
                path.append(pick)
                px, py = px + HOPS[pick][0], py + HOPS[pick][1]
                length += math.sqrt(2.0) if pick >= 4 else 1.0
            self.worm.append(path)
            mean += length / m
        self.lam = q / mean
        self.q, self.m = q, m


def _schedule(lat, steps, speed):
    """Per step: directions grouped by (hop, paused)."""
    pos = [(0, 0)] * lat.q
    done = [0] * lat.q
    for n in range(1, steps + 1):
        groups = {}
        for i in range(lat.q):
            k = lat.worm[i][done[i] % lat.m]
            x, y = pos[i][0] + HOPS[k][0], pos[i][1] + HOPS[k][1]
            hop = x * x + y * y <= ((n + 1) ** 2 if speed == 1.0 else (speed * n + 1.0) ** 2)
            groups.setdefault((k, not hop), []).append(i)
            if hop:
                pos[i] = (x, y)
                done[i] += 1
        yield groups


def _e_eq(t):
    if isinstance(t, torch.Tensor):
        return 1.0 / torch.expm1(THETA / t)
    return 1.0 / math.expm1(THETA / t)


def _shift(a, c):
    """b(y) = a(y - c) over the last two axes, zero from outside."""
    cx, cy = c
    h, w = a.shape[-2:]
    p = torch.nn.functional.pad(a, (1, 1, 1, 1))
    return p[..., 1 - cy:1 - cy + h, 1 - cx:1 - cx + w]


class _Exact:
    """One grid in float64; walls[k] as in WALLS; mfp a number or an (ny, nx) tensor."""

    def __init__(self, nx, ny, q, walls, mfp, emulate_3d, speed, tw=None):
        self.nx, self.ny, self.lat, self.speed = nx, ny, _Lattice.of(q), speed
        self.kinds, t, sp = WALLS[walls]
        self.tw = [torch.tensor(v, dtype=torch.float64, device="cuda") for v in t] if tw is None else tw
        self.p = [1.0 if k == SPE else s for k, s in zip(self.kinds, sp)]
        W = speed / (mfp.double() if isinstance(mfp, torch.Tensor) else
                     torch.full((ny, nx), float(mfp), dtype=torch.float64, device="cuda"))
        W = (1.5 if emulate_3d else 1.0) * (W * (1.0 - W) + W * W * self.lat.lam)
        f = torch.nn.functional.pad(W, (1, 1, 1, 1))
        self.W = self._links(f[None])[0]
        self.w = torch.tensor(self.lat.w, device="cuda")
        self.s = torch.tensor(self.lat.s, device="cuda")
        d = np.array(self.lat.dirs)
        at = {v: i for i, v in enumerate(self.lat.dirs)}
        self.rule = []
        for n in NORMAL + ((1, 1), (-1, 1), (1, -1), (-1, -1)):
            corner = n[0] != 0 and n[1] != 0
            inward = (d[:, 0] * n[0] > 0) & (d[:, 1] * n[1] > 0) if corner else d @ np.array(n) > 0
            rho = np.where(inward, self.lat.w * (self.lat.s @ (np.array(n) / math.hypot(*n))), 0.0)
            flat = d @ np.array(n) == 0
            mir = [at[(-a, b) if n[0] else (a, -b)] for a, b in self.lat.dirs]
            t64 = lambda v: torch.tensor(v, device="cuda")
            self.rule.append((t64(inward), t64(rho / rho.sum()), t64(flat), t64(mir)))

    def _links(self, a):
        nx, ny = self.nx, self.ny
        if self.kinds[2] == PER:
            xs = slice(1, nx + 1) if self.kinds[0] == PER else slice(0, nx + 2)
            a = a.clone()
            a[:, 0, xs] = a[:, ny, xs].clone()
            a[:, ny + 1, xs] = a[:, 1, xs].clone()
        if self.kinds[0] == PER:
            a = a.clone()
            a[:, :, 0] = a[:, :, nx].clone()
            a[:, :, nx + 1] = a[:, :, 1].clone()
        return a

    def _adiabatic(self, old, rule, p):
        """New values of adiabatic ghost cells (q, cells)."""
        inward, rho, flat, mir = self.rule[rule]
        a = torch.where(inward[:, None], 0.0, old).sum(0)
        out = torch.where(flat[:, None], p * old, 0.0)
        return torch.where(inward[:, None], old + p * old[mir] + (1.0 - p) * rho[:, None] * a, out)

    def bounds(self, d):
        nx, ny, k = self.nx, self.ny, self.kinds
        if all(v == PER for v in k):
            return self._links(d)
        d = d.clone()
        edge = ((slice(1, ny + 1), 0), (slice(1, ny + 1), nx + 1),
                (0, slice(1, nx + 1)), (ny + 1, slice(1, nx + 1)))
        corners = ((0, 0, 0, 2, 4), (0, nx + 1, 1, 2, 5), (ny + 1, 0, 0, 3, 6), (ny + 1, nx + 1, 1, 3, 7))
        for s in range(4):
            if k[s] in (DIF, SPE):
                d[(slice(None),) + edge[s]] = self._adiabatic(d[(slice(None),) + edge[s]].clone(), s, self.p[s])
        for y, x, xw, yw, rule in corners:
            if k[xw] in (DIF, SPE) and k[yw] in (DIF, SPE):
                d[:, y, x] = self._adiabatic(d[:, y, x].clone()[:, None], rule, 0.0)[:, 0]
        de = [_e_eq(t) - _e_eq(TREF) for t in self.tw]
        for s in range(4):
            if k[s] == ISO:
                v = d[(slice(None),) + edge[s]]
                d[(slice(None),) + edge[s]] = (self.w * de[s])[:, None].expand_as(v)
        for y, x, xw, yw, _ in corners:
            if PER not in (k[xw], k[yw]):
                for s in (xw, yw):
                    if k[s] == ISO:
                        d[:, y, x] = self.w * de[s]
                        break
        return self._links(d)

    def update(self, d, groups):
        d = self.bounds(d)
        keep = 1.0 - self.W
        f = self.W * d.sum(0)
        new = torch.empty_like(d)
        for (k, paused), idx in groups.items():
            gain = self.w[idx][:, None, None] * _shift(f, HOPS[k])
            own = keep * d[idx]
            new[idx] = (own if paused else _shift(own, HOPS[k])) + gain
        return new

    def start(self, dT):
        de = _e_eq(TREF + dT.double()) - _e_eq(TREF)
        de = torch.nn.functional.pad(de[None, None], (1, 1, 1, 1), mode="replicate")[0, 0]
        return self.w[:, None, None] * de[None]

    def moments(self, d):
        i = d[:, 1:-1, 1:-1]
        E = i.sum(0)
        e0 = _e_eq(TREF)
        T = THETA / torch.log1p(1.0 / (e0 + E)) - TREF
        qx, qy = (torch.tensordot(self.s[:, a], i, dims=([0], [0])) * self.speed for a in (0, 1))
        return T, qx, qy

    def reduce(self, d):
        """Energies (interior, with the walls') and mean fluxes, band flux, band slope of E."""
        nx, ny = self.nx, self.ny
        E = d[:, 1:-1, 1:-1].sum(0)
        _, qx, qy = self.moments(d)
        full = d.sum(0)
        held = torch.zeros_like(full, dtype=torch.bool)
        held[1:-1, 1:-1] = True
        dif = [k in (DIF, SPE) for k in self.kinds]
        held[1:-1, 0], held[1:-1, -1], held[0, 1:-1], held[-1, 1:-1] = dif
        held[0, 0], held[0, -1] = dif[0] and dif[2], dif[1] and dif[2]
        held[-1, 0], held[-1, -1] = dif[0] and dif[3], dif[1] and dif[3]
        x0, m = nx // 4, nx // 2
        xs = torch.arange(x0, x0 + m, device="cuda", dtype=torch.float64)
        mine = [qx.mean(), qy.mean(), qx[:, x0:x0 + m].mean(),
                ((xs - xs.mean()) * E[:, x0:x0 + m].mean(0)).sum() / ((xs - xs.mean()) ** 2).sum()]
        mine = [float(v) for v in mine]
        return [float(E.sum()), float(full[held].sum())], mine

    def conduct(self, r, mfp, emulate_3d):
        """The six reductions with the apparent and the band conductivity after them."""
        D = self.speed * mfp / (3.0 if emulate_3d else 2.0) if mfp else float("nan")
        de = float(_e_eq(self.tw[0]) - _e_eq(self.tw[1]))
        iso = self.kinds[0] == ISO and self.kinds[1] == ISO and de != 0.0
        return r + [r[2] * self.nx / (D * de) if iso else float("nan"),
                    r[4] / (-D * r[5]) if r[5] != 0.0 else float("nan")]


def _grid(case, got, tw=None):
    mfp = got["mfp"] if case["field"] else case["mfp"]
    return _Exact(case["nx"], case["ny"], case["q"], case["walls"], mfp, case["emulate_3d"],
                  case["speed"], tw)


def _gradients(case, got):
    """The run's moments and gradients in float64 by differentiating it, from checkpoints."""
    from torch.utils.checkpoint import checkpoint
    mfp = got["mfp"].double().requires_grad_(True)
    dT0 = got["dT"].double().requires_grad_(True)
    tw = [torch.tensor(v, dtype=torch.float64, device="cuda", requires_grad=True)
          for v in WALLS[case["walls"]][1]]
    g = _Exact(case["nx"], case["ny"], case["q"], case["walls"], mfp, case["emulate_3d"],
               case["speed"], tw)
    d = g.start(dT0)
    todo = list(_schedule(g.lat, case["steps"], case["speed"]))

    def some(d, W, t0, t1, t2, t3, part):
        g.W, g.tw = W, [t0, t1, t2, t3]
        for groups in part:
            d = g.update(d, groups)
        return d

    W = g.W
    for a in range(0, len(todo), 10):
        d = checkpoint(some, d, W, *tw, todo[a:a + 10], use_reentrant=False)
    T, qx, qy = g.moments(d)
    if case["kind"] == "adjoint":
        loss = (got["gT"].double() * T).sum()
    else:
        wT = got["wT"].double()
        loss = (wT * T).mean() + 50.0 * qx.mean() + 20.0 * (qy * wT).mean()
    loss.backward()
    zero = torch.zeros((), dtype=torch.float64, device="cuda")
    gt = torch.stack([zero if t.grad is None else t.grad for t in tw]).cpu()
    return [T.detach(), qx.detach(), qy.detach(), mfp.grad, gt, dT0.grad]


def exact(case, seed):
    kind = case["kind"]
    got = _inputs(case, seed)
    if kind in ("adjoint", "autograd"):
        return _gradients(case, got)
    with torch.no_grad():
        if kind in ("films", "bands"):
            out = []
            for s, dT in zip(_specs(case), got["dT"]):
                g = _Exact(s["nx"], s["ny"], s["q"], s["walls"], s["mfp"], True, s["speed"])
                d = g.start(dT)
                for groups in _schedule(g.lat, case["steps"], s["speed"]):
                    d = g.update(d, groups)
                out.append(list(g.moments(d)))
            return out
        g = _grid(case, got)
        d = got["state"].double() if kind == "state" else g.start(got["dT"])
        every = case["steps"] // 4 if kind == "steady" else 0
        sums = [0.0] * 4
        for n, groups in enumerate(_schedule(g.lat, case["steps"], case["speed"]), 1):
            d = g.update(d, groups)
            if every and n > 4 * every - 10:
                sums = [a + b / 10.0 for a, b in zip(sums, g.reduce(d)[1])]
        if kind == "run":
            return list(g.moments(d))
        if kind == "state":
            return [d[:, 1:-1, 1:-1]]
        mfp = None if case["field"] else case["mfp"]
        tot, mine = g.reduce(d)
        r = g.conduct(tot + (sums if every else mine), mfp, case["emulate_3d"])
        r = torch.tensor(r, dtype=torch.float64)
        if kind == "steady":
            return [None, None, r, *g.moments(d)]
        return [*g.moments(d), r]
