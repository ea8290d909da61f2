"""The work that a program has this library do, for timing and comparison.

A case is one of seven kinds of calls:
  event        an MV collision from its charges: the initial state, the time
               steps, T^{mu nu}(z) sampled on the way
  steps        two time steps of fields that the caller set
  run          one step of an event too large to begin anew each time
  ensemble     independent events of uneven size advanced as one batch
  observables  the Gauss residual and T^{mu nu} of fields that the caller set
  analysis     the event mean, the local rest frame and its rapidity profiles
  gradient     the mid-rapidity energy and its gradient in the MV charges
`exact` evaluates the same formulas (Ipp & Mueller, Secs. 2 to 4) in plain
64-bit torch.
"""
from __future__ import annotations

import ctypes as C
import math

import numpy as np
import torch

import glasma_inputs as gi
from paper_2009_02044_gb300 import glasma as G


# ---------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------

def _lattice(kind, nc, nz, ny, nx, sigma_l, steps, every, **kw):
    d = dict(kind=kind, nc=nc, nz=nz, ny=ny, nx=nx, a_z=1.0, dt=0.5,
             sigma_l=sigma_l, g2mu=0.1, m_ir=0.2, precision="fp32",
             scheme="leapfrog", steps=steps, every=every)
    d.update(kw)
    return d


def listed():
    improved = dict(a_z=0.25, dt=0.25, g2mu=0.05, m_ir=0.1, scheme="implicit")
    return [
        # the smallest event: many steps of a lattice that does not fill the
        # GPU, the size at which results are checked against a reference
        dict(_lattice("event", 2, 128, 16, 16, 4.0, 100, 20, precision="fp64"),
             name="event_su2_128x16x16_fp64"),
        # the event of the headline benchmark, through the collision
        dict(_lattice("event", 3, 512, 64, 64, 8.0, 100, 50),
             name="event_su3_512x64x64_fp32"),
        # its time step by itself, on a shorter lattice
        dict(_lattice("steps", 3, 128, 64, 64, 4.0, 2, 2),
             name="steps_su3_128x64x64_fp32"),
        # the time step on a lattice that no tile divides
        dict(_lattice("steps", 3, 131, 45, 48, 4.0, 2, 2),
             name="steps_su3_131x45x48_fp32"),
        # a large transverse plane, few operations per byte, sampled often as
        # the study of rapidity profiles does
        dict(_lattice("event", 2, 1024, 128, 128, 8.0, 64, 8),
             name="event_su2_1024x128x128_fp32"),
        # double precision, for checks of the single-precision runs
        dict(_lattice("event", 3, 160, 24, 24, 4.0, 40, 20, precision="fp64"),
             name="event_su3_160x24x24_fp64"),
        # the improved scheme at the size it is made for
        dict(_lattice("run", 3, 2048, 128, 128, 2.0, 1, 1, before=16, **improved),
             name="run_su3_2048x128x128_improved"),
        # and its time step on a lattice for trying out parameters
        dict(_lattice("steps", 3, 160, 32, 32, 1.0, 2, 2, **improved),
             name="steps_su3_160x32x32_improved"),
        # an event average: 24 collisions of three transverse sizes
        dict(_lattice("ensemble", 3, 256, 64, 64, 6.0, 100, 100, events=24),
             name="ensemble_su3_24x256_fp32"),
        # monitoring a run: both observables to the host
        dict(_lattice("observables", 3, 160, 64, 64, 4.0, 0, 0),
             name="observables_su3_160x64x64_fp32"),
        # the rapidity profiles of 8 sampled events
        dict(kind="analysis", events=8, samples=88, nz=768, points=25,
             name="analysis_8x88x768"),
        # one gradient of an optimisation in the initial charges
        dict(_lattice("gradient", 2, 256, 32, 32, 4.0, 200, 20,
                      precision="fp64"),
             name="gradient_su2_256x32x32_fp64"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _fits(case):
    """Whether the nuclei fit the box and stay in it for all the steps."""
    az, n = case["a_z"], case["steps"] + case.get("before", 0)
    reach = 4 * case["sigma_l"] + (math.ceil(4 * case["sigma_l"] / az) + 2) * az
    return reach + case["dt"] * (n + 1) + 3 * az < case["nz"] * az / 2.0


def draw(rng):
    while True:
        kind = rng.choice(["event"] * 5 + ["steps"] * 4 + ["improved"] * 2
                          + ["ensemble", "observables", "analysis", "gradient"])
        if kind == "analysis":
            return dict(kind=kind, events=rng.randint(1, 32),
                        samples=_log_int(rng, 20, 400), nz=_log_int(rng, 128, 1500),
                        points=rng.randint(5, 200))
        nz, ny, nx = _log_int(rng, 64, 1024), _log_int(rng, 6, 128), _log_int(rng, 6, 128)
        if rng.random() < 0.3:      # square planes of whole warps are common
            ny = nx = rng.choice([16, 32, 64, 128])
        nc, prec = rng.choice([2, 3]), rng.choice(["fp32", "fp32", "fp64"])
        sigma = rng.choice([1.0, 2.0, 4.0, 8.0])
        every = rng.choice([2, 8, 20])
        steps = every * rng.randint(1, max(1, 120 // every))
        if kind == "event":
            thin = rng.random() < 0.3
            c = _lattice(kind, nc, nz, ny, nx, sigma, steps, every, precision=prec)
            if thin:
                c.update(a_z=0.125, dt=0.0625, sigma_l=1.0, g2mu=0.4, m_ir=0.1)
        elif kind == "steps":
            c = _lattice(kind, nc, nz, ny, nx, sigma, 2, 2, precision=prec)
        elif kind == "improved":
            kind, steps = rng.choice([("steps", 2), ("event", 2 * rng.randint(1, 10))])
            c = _lattice(kind, nc, nz, ny, nx, min(sigma, 2.0), steps, 2, precision=prec,
                         a_z=0.25, dt=0.25, g2mu=0.05, m_ir=0.1, scheme="implicit")
        elif kind == "ensemble":
            c = _lattice(kind, nc, nz, ny, nx, sigma, steps, steps, precision=prec,
                         events=rng.randint(2, 24))
        elif kind == "observables":
            c = _lattice(kind, nc, nz, ny, nx, sigma, 0, 0, precision=prec)
        else:
            prec = "fp64"
            c = _lattice(kind, 2, nz, ny, nx, sigma, steps, 20, precision=prec)
        sites = nz * ny * nx * c.get("events", 1)
        # bounds that keep a drawn case below the largest listed one
        cost = sites * max(c["steps"], 1) * (1 if nc == 2 else 4)
        cost *= 8 if prec == "fp64" else 1
        cost *= 8 if c["scheme"] == "implicit" else 1
        cost *= 12 if kind == "gradient" else 1
        if not _fits(c) or cost > 5e8 or (kind in ("steps", "observables") and sites > 700000):
            continue
        return c


# ---------------------------------------------------------------------------
# what a program has in hand before the call
# ---------------------------------------------------------------------------

def _cfg(case, **kw):
    keys = ("nc", "nz", "ny", "nx", "a_z", "dt", "sigma_l", "g2mu", "m_ir",
            "precision", "scheme")
    return gi._cfg(**dict({k: case[k] for k in keys}, **kw))


def _rho(case, seed, nx=None, ny=None):
    """MV charges [N][a][y][x], standard deviation g^2 mu per site."""
    shape = (2, case["nc"] ** 2 - 1, ny or case["ny"], nx or case["nx"])
    return case["g2mu"] * np.random.default_rng(seed).standard_normal(shape)


def _events(case):
    """(ny, nx) of the events: a third each at 1/2, 3/4 and the whole size."""
    n = case["events"]
    return [(max(1, case["ny"] * (2 + 3 * k // n) // 4),
             max(1, case["nx"] * (2 + 3 * k // n) // 4)) for k in range(n)]


def _fields(case, seed):
    """Links near the identity, fields and charges of generic values, as
    matrices and components in the order of glasma_set_fields (on the GPU)."""
    g = torch.Generator("cuda").manual_seed(seed)
    na, shape = case["nc"] ** 2 - 1, (case["nz"], case["ny"], case["nx"])

    def normal(*s):
        return torch.randn(*s, generator=g, device="cuda", dtype=torch.float64)

    U = torch.stack([_expi(0.2 * normal(na, *shape), case["nc"]) for _ in range(3)])
    E = 0.05 * normal(3, na, *shape)
    U[2, :, :, -1] = torch.eye(case["nc"], dtype=U.dtype, device="cuda")[:, :, None, None]
    E[2, :, -1] = 0.0
    QA, QB = torch.zeros(2, na, *shape, device="cuda", dtype=torch.float64)
    if case["kind"] == "observables":   # steps go on for ever: charges would leave the box
        w = case["nz"] // 4
        QA[:, 2 * w:3 * w] = 0.1 * normal(na, w, *shape[1:])
        QB[:, w:2 * w] = 0.1 * normal(na, w, *shape[1:])
    return U, E, QA, QB


def _tables(case, seed):
    """T^{mu nu} tables [event][sample x nz][4] of timelike flow: a glasma
    between two receding sheets."""
    rng = np.random.default_rng(seed)
    az, dts, t0 = 0.125, 0.5, 4.0
    t = t0 + dts * np.arange(case["samples"])[:, None]
    z = (np.arange(case["nz"]) - case["nz"] / 2) * az
    z = np.clip(z, -0.98 * t, 0.98 * t)
    tau, eta = np.sqrt(t * t - z * z), np.arctanh(z / t)
    tabs = np.empty((case["events"], case["samples"], case["nz"], 4))
    for e in range(case["events"]):
        a = rng.uniform(0.5, 2.0)
        loc = a / tau * np.exp(-0.5 * ((eta - 0.1 * rng.standard_normal()) / 1.4) ** 2)
        pl = 0.05 * loc * rng.standard_normal(loc.shape)
        ch, sh = np.cosh(eta), np.sinh(eta)
        tabs[e] = np.stack([loc * ch * ch + pl * sh * sh, loc * sh * sh + pl * ch * ch,
                            0.5 * (loc - pl), (loc + pl) * sh * ch], -1)
    return tabs, (t0, dts, -case["nz"] / 2 * az, az)


class _Memory:
    """The device memory of contexts, owned by the program: every block is a
    torch tensor, so results are used where the library left them."""

    def __init__(self):
        self.blocks = {}
        self.order = []

        @G._ALLOC_FN
        def alloc(nbytes, stream, user):
            try:
                b = torch.empty(int(nbytes), dtype=torch.uint8, device="cuda")
            except Exception:
                return None
            self.blocks[b.data_ptr()] = b
            self.order.append(b)
            return b.data_ptr()

        @G._FREE_FN
        def free(ptr, nbytes, stream, user):
            b = self.blocks.pop(ptr, None)
            self.order = [x for x in self.order if x is not b]

        self.table = G.glasma_allocator()
        self.table.alloc, self.table.free, self.table.user = alloc, free, None
        self.keep = (alloc, free)

    def context(self, cfg, rho):
        p, out = G.make_params(cfg), C.c_void_p()
        G._check(G.load_library().glasma_init_mv(
            C.byref(p), rho.ctypes.data_as(C.POINTER(C.c_double)),
            C.c_void_p(torch.cuda.current_stream().cuda_stream),
            C.byref(self.table), C.byref(out)), "glasma_init_mv")
        return G.Handle(out, p, self)

    def state(self, cfg):
        """Links and fields after an even number of leapfrog steps, in the
        library's layout (the links of the improved scheme move from buffer
        to buffer: fields only)."""
        rs = 4 if cfg["precision"] == "fp32" else 8
        dtype = torch.float32 if rs == 4 else torch.float64
        na, V = cfg["nc"] ** 2 - 1, cfg["nz"] * cfg["ny"] * cfg["nx"]
        links = 12 * V if cfg["nc"] == 2 else 54 * 32 * ((V + 31) // 32)
        E = next(b for b in self.order if b.numel() == 3 * na * V * rs)
        if cfg["scheme"] == "implicit":
            return [E.view(dtype)]
        U = next(b for b in self.order if b.numel() == links * rs)
        return [U.view(dtype), E.view(dtype)]


def prepare(case, seed):
    s = dict(case=case)
    kind = case["kind"]
    if kind == "event":
        s.update(cfg=_cfg(case), rho=_rho(case, seed))
    elif kind == "run":
        s.update(cfg=_cfg(case), h=G.glasma_init_mv(_cfg(case), _rho(case, seed)))
        G.glasma_step(s["h"], case["before"])
    elif kind == "ensemble":
        s["events"] = [(_cfg(case, ny=ny, nx=nx), _rho(case, [seed, k], nx, ny))
                       for k, (ny, nx) in enumerate(_events(case))]
    elif kind in ("steps", "observables"):
        U, E, QA, QB = _fields(case, seed)
        # (the context begins as an event of thin nuclei, which the fields replace)
        s.update(cfg=_cfg(case, sigma_l=0.5 * case["a_z"]), memory=_Memory())
        s["h"] = s["memory"].context(s["cfg"], _rho(case, seed))
        G.glasma_set_fields(s["h"], U.permute(0, 3, 4, 5, 1, 2).cpu().numpy(),
                            *(f.movedim(-4, -1).cpu().numpy() for f in (E, QA, QB)))
    elif kind == "analysis":
        tabs, s["grid"] = _tables(case, seed)
        s["tabs"] = torch.from_numpy(tabs).cuda()
        s["eta"] = torch.linspace(-1.2, 1.2, case["points"], dtype=torch.float64,
                                  device="cuda")
        s["taus"] = _taus(case)
    elif kind == "gradient":
        s.update(cfg=_cfg(case), rho=_rho(case, seed))
    torch.cuda.synchronize()
    return s


def _taus(case):
    """Proper times whose profile lies inside the sampled grid."""
    last = 4.0 + 0.5 * (case["samples"] - 1)
    far = min(last, case["nz"] / 2 * 0.125) / math.cosh(1.2)
    return [4.0 + f * max(far - 4.0, 0.0) for f in (0.0, 0.5, 1.0)]


def _kept(tab, cfg):
    """A run's samples are kept in the precision of its state."""
    return tab.float() if cfg["precision"] == "fp32" else tab


def _event(cfg, rho, steps, every):
    """The samples, and in double precision the state: in single precision,
    rounding noise of the fields adds up over many steps, in the pure gauge
    behind the nuclei above all, and the samples are what such a run is for."""
    memory = _Memory()
    h = memory.context(cfg, rho)
    tabs = torch.empty(steps // every, cfg["nz"], 4, dtype=torch.float64, device="cuda")
    for k in range(steps // every):
        G.glasma_step(h, every)
        G.glasma_tmunu_device(h, tabs[k].data_ptr())
    state = memory.state(cfg) if cfg["precision"] == "fp64" else []
    G.glasma_free(h)
    return [_kept(tabs, cfg)] + state


def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind == "event":
        return _event(state["cfg"], state["rho"], case["steps"], case["every"])
    if kind == "steps":
        G.glasma_step(state["h"], case["steps"])
        return state["memory"].state(state["cfg"])
    if kind == "run":
        G.glasma_step(state["h"], case["steps"])
        tab = torch.empty(case["nz"], 4, dtype=torch.float64, device="cuda")
        G.glasma_tmunu_device(state["h"], tab.data_ptr())
        return [_kept(tab, state["cfg"])]
    if kind == "ensemble":
        memory = _Memory()
        hs = [memory.context(cfg, rho) for cfg, rho in state["events"]]
        batch = G.glasma_batch_create(hs)
        G.glasma_batch_step(batch, case["steps"])
        tabs = torch.empty(len(hs), case["nz"], 4, dtype=torch.float64, device="cuda")
        for k, h in enumerate(hs):
            G.glasma_tmunu_device(h, tabs[k].data_ptr())
        G.glasma_batch_free(batch)
        out = _kept(tabs, state["events"][0][0])
        for h in hs:
            G.glasma_free(h)
        return list(out)
    if kind == "observables":
        gauss = G.glasma_gauss_residual(state["h"])
        tab, energy = G.glasma_tmunu(state["h"])
        if case["precision"] == "fp32":
            tab, energy = tab.astype(np.float32), np.float32(energy)
        return [np.array(gauss), tab, energy]
    if kind == "analysis":
        t0, dts, z0, az = state["grid"]
        n_t, nz, eta = case["samples"], case["nz"], state["eta"]
        stream = torch.cuda.current_stream()
        rest = torch.empty(n_t * nz, 8, dtype=torch.float64, device="cuda")
        G.glasma_rest_frame(state["tabs"].data_ptr(), case["events"], n_t * nz,
                            rest.data_ptr(), stream)
        prof = torch.empty(3, case["points"], dtype=torch.float64, device="cuda")
        for k, tau in enumerate(state["taus"]):
            at = torch.full_like(eta, tau)
            G.glasma_sample_grid(rest.data_ptr(), n_t, nz, 8, 4, t0, dts, z0, az,
                                 at.data_ptr(), eta.data_ptr(), case["points"],
                                 prof[k].data_ptr(), stream=stream)
        x, f = eta.cpu().numpy(), prof.cpu().numpy()
        return [rest, prof, np.array(G.glasma_fit_gaussian(x, f[0], 0.1))]
    value, grad = G.glasma_adjoint_energy(state["cfg"], state["rho"], case["steps"],
                                          _half_width(case), case["every"])
    return [value, grad]


def _half_width(case):
    return 0.0625 * case["nz"] * case["a_z"]


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def _site_work(case):
    """Bytes and operations of one step of one site: three links and three
    fields read and written; three plaquettes of two products, with one
    projection and two transports each, and an exponential and a product
    per link."""
    rs = 4 if case["precision"] == "fp32" else 8
    link, field, prod = ((4, 3, 28), (18, 8, 198))[case["nc"] - 2]
    return 2 * 3 * (link + field) * rs, (3 * 5 + 3 * 3) * prod


def work(case):
    kind = case["kind"]
    if kind == "analysis":
        n = case["samples"] * case["nz"]
        return dict(bytes=8 * n * (4 * case["events"] + 8), flops=n * (4 * case["events"] + 30))
    b, f = _site_work(case)
    sites = case["nz"] * case["ny"] * case["nx"]
    if kind == "ensemble":
        sites = case["nz"] * sum(ny * nx for ny, nx in _events(case))
    if kind == "observables":
        return dict(bytes=sites * b // 2, flops=sites * 2 * f)
    if case["scheme"] == "implicit":
        # two further link arrays are read, and the transverse terms are
        # evaluated in three time slots
        b, f = 1.75 * b, 3 * f
    steps = case["steps"]
    if kind == "gradient":      # forward, and backward through every step
        b, f = 3 * b, 3 * f
    samples = steps // case["every"] if kind == "event" else 0 if kind == "steps" else 1
    # every step reads and writes the state, a sample reads it, and an event
    # writes its initial one
    begins = 0 if kind in ("steps", "run") else 1
    return dict(bytes=sites * b * (steps + 0.5 * samples + 0.5 * begins),
                flops=sites * f * (steps + samples))


# ---------------------------------------------------------------------------
# the same formulas in 64 bits; fields are [...][z][y][x], matrices [N][N]
# in front
# ---------------------------------------------------------------------------

def _generators(nc):
    t = np.zeros((nc * nc - 1, nc, nc), complex)
    pairs = [(0, 1)] if nc == 2 else [(0, 1), (0, 2), (1, 2)]
    for k, (i, j) in enumerate(pairs):
        a = (0, 3, 5)[k]
        t[a, i, j] = t[a, j, i] = 0.5
        t[a + 1, i, j], t[a + 1, j, i] = -0.5j, 0.5j
    t[2, 0, 0], t[2, 1, 1] = 0.5, -0.5
    if nc == 3:
        t[7] = np.diag([1, 1, -2]) / (2 * math.sqrt(3))
    return torch.from_numpy(t).cuda()


def _mat(v, nc):
    return torch.einsum("aij,azyx->ijzyx", _generators(nc), v.to(torch.complex128))


def _comp(m):
    """Re tr(2 t^a m), the components of a hermitian m."""
    t = _generators(m.shape[0])
    return torch.stack([2 * sum((t[a, j, i] * m[i, j]).real
                                for i in range(m.shape[0]) for j in range(m.shape[0])
                                if abs(t[a, j, i].item()) > 0) for a in range(len(t))])


def _mm(a, b):
    return (a[:, :, None] * b[None]).sum(1)


def _dag(a):
    return a.transpose(0, 1).conj().resolve_conj()


def _im_proj(m):
    """Im tr(t^a m)."""
    return 0.5 * _comp((m - _dag(m)) / 2j)


def _eye(like):
    return torch.eye(like.shape[0], dtype=like.dtype, device=like.device)[:, :, None, None, None]


def _expi(v, nc, c=1.0):
    """exp(i c v^a t^a) by its series, halved until it converges fast."""
    x = 1j * c * _mat(v, nc)
    n = float(x.detach().abs().max()) * nc
    halvings = max(0, math.ceil(math.log2(max(n, 1e-300) / 0.25)))
    x, n = x / 2 ** halvings, n / 2 ** halvings
    term = total = x
    k = 1
    while k < 18 and n ** (k + 1) / math.factorial(k + 1) > 1e-18:
        k += 1
        term = _mm(term, x) / k
        total = total + term
    for _ in range(halvings):
        total = 2 * total + _mm(total, total)
    return total + _eye(total)


def _log(w):
    """The components of h with exp(i h^a t^a) = w, w near the identity."""
    s = (w - _dag(w)) / 2j
    s2, term, total, c = _mm(s, s), s, s, 1.0
    for k in range(1, 60):
        term = _mm(term, s2)
        c *= (2 * k - 1) / (2 * k)
        total = total + term * (c / (2 * k + 1))
        if float(term.detach().abs().max()) * c < 1e-20:
            break
    return _comp(total)


def _shift(f, d, n):
    return torch.roll(f, -n, dims=(-1, -2, -3)[d])


class _Exact:
    """One event in 64 bits."""

    def __init__(self, cfg, rho=None, fields=None):
        self.c, self.n, self.prev = cfg, 0, None
        nz = cfg["nz"]
        iz = torch.arange(nz, device="cuda")[:, None, None]
        self.up = (iz < nz - 1).double()      # a z link starts here
        self.down = (iz > 0).double()         # and one ends here
        self.a = (1.0, 1.0, cfg["a_z"])
        if fields is not None:
            self.U, self.E = list(fields[0]), list(fields[1])
            self.QA, self.QB = fields[2:]
            self.prev = [_mm(_expi(e, cfg["nc"], -cfg["dt"]), u) for u, e in zip(self.U, self.E)]
        else:
            self._init(rho)

    def _init(self, rho):
        c, nc = self.c, self.c["nc"]
        ny, nx = rho.shape[-2:]
        sy = torch.sin(math.pi * torch.arange(ny, device="cuda", dtype=torch.float64) / ny)
        sx = torch.sin(math.pi * torch.arange(nx, device="cuda", dtype=torch.float64) / nx)
        k2 = 4 * sy[:, None] ** 2 + 4 * sx ** 2
        phi = torch.fft.ifft2(torch.fft.fft2(rho) / (k2 + c["m_ir"] ** 2)).real
        zc, d = c["nz"] * c["a_z"] / 2, (math.ceil(4 * c["sigma_l"] / c["a_z"]) + 2) * c["a_z"]
        e4 = math.erf(4 / math.sqrt(2))

        def lam(centre, behind):
            u = [(k * c["a_z"] - centre) / c["sigma_l"] * behind for k in range(c["nz"])]
            v = [0.0 if x <= -4 else 1.0 if x >= 4 else
                 (math.erf(x / math.sqrt(2)) + e4) / (2 * e4) for x in u]
            return torch.tensor(v, dtype=torch.float64, device="cuda")[:, None, None]

        links = []
        for shift in (0.0, -c["dt"]):
            u = [None, None]
            for N, (centre, behind) in enumerate(((zc + d - shift, 1.0), (zc - d + shift, -1.0))):
                vd = _expi(phi[N][:, None] * lam(centre, behind), nc)
                for i in (0, 1):
                    w = _mm(_dag(vd), _shift(vd, i, 1))
                    u[i] = w if u[i] is None else _mm(u[i], w)
            links.append(u)
        one = _eye(links[0][0]).expand_as(links[0][0])
        self.U, self.prev = links[0] + [one], links[1] + [one]
        self.E = [_log(_mm(links[0][i], _dag(links[1][i]))) / c["dt"] for i in (0, 1)]
        self.E.append(torch.zeros_like(self.E[0]))
        rho3 = self.divergence()
        z = torch.arange(c["nz"], device="cuda", dtype=torch.float64)[:, None, None] * c["a_z"]
        self.QA, self.QB = rho3 * (z > zc), rho3 * (z < zc)

    def divergence(self):
        total = 0.0
        for i in range(3):
            u, e = _shift(self.U[i], i, -1), _shift(_mat(self.E[i], self.c["nc"]), i, -1)
            back = _comp(_mm(_mm(_dag(u), e), u))
            total = total + (self.E[i] - (back * self.down if i == 2 else back)) / self.a[i] ** 2
        return total

    def gauss(self):
        q = self.QA + self.QB
        g = self.divergence() - q
        return torch.stack([g.abs().max(), g.square().mean().sqrt(), q.abs().max()])

    def force(self, slot, i):
        """-sum_j 2/a_j^2 Im tr t^a (U_ij + U_i-j); slot(d, zplane): the links
        of direction d in a plane that does or does not contain z."""
        F = 0.0
        for j in range(3):
            if j == i:
                continue
            ui, uj = slot(i, 2 in (i, j)), slot(j, 2 in (i, j))
            p = _mm(_mm(_mm(ui, _shift(uj, i, 1)), _dag(_shift(ui, j, 1))), _dag(uj))
            um, ujm = _shift(ui, j, -1), _shift(uj, j, -1)
            m = _mm(_mm(_mm(ui, _dag(_shift(ujm, i, 1))), _dag(um)), ujm)
            f, b = _im_proj(p), _im_proj(m)
            if j == 2:
                f, b = f * self.up, b * self.down
            F = F - 2 / self.a[j] ** 2 * (f + b)
        return F * self.up if i == 2 else F

    def _hop(self):
        c = self.c
        r = c["dt"] / c["a_z"]
        return math.floor((self.n + 1) * r + 0.5) > math.floor(self.n * r + 0.5)

    def current(self):
        """Charges after the step's hop and dt J_z."""
        if not self._hop():
            return self.QA, self.QB, torch.zeros_like(self.QA)
        uz, nc = self.U[2], self.c["nc"]
        qb = _comp(_mm(_mm(_dag(uz), _mat(self.QB, nc)), uz))
        qa = _comp(_mm(_mm(uz, _shift(_mat(self.QA, nc), 2, 1)), _dag(uz))) * self.up
        return qa, _shift(qb, 2, -1) * self.down, self.c["a_z"] ** 2 * (qa - self.QB) * self.up

    def e_next(self):
        qa, qb, dj = self.current()
        E = [self.E[i] + self.c["dt"] * self.force(lambda d, z: self.U[d], i) for i in range(3)]
        return E[:2] + [E[2] + dj], qa, qb

    def links(self, E):
        nc, dt = self.c["nc"], self.c["dt"]
        return [_mm(_expi(E[i], nc, dt), self.U[i]) for i in range(3)]

    def step(self):
        E, qa, qb = (self.e_improved if self.c["scheme"] == "implicit" else self.e_next)()
        self.prev, self.U = self.U, self.links(E)
        self.E, self.QA, self.QB, self.n = E, qa, qb, self.n + 1

    def e_improved(self):
        """Plaquette terms averaged over t_{n+1}, t_n, t_{n-1} with weights
        1/4, 1/2, 1/4: every link in the transverse plane, z links only in
        the planes containing z; iterated with relaxation."""
        c = self.c
        qa, qb, dj = self.current()

        def slot(links):
            return lambda d, z: self.U[d] if z and d != 2 else links[d]

        base = [self.E[i] + c["dt"] * (0.5 * self.force(slot(self.U), i)
                                       + 0.25 * self.force(slot(self.prev), i)) for i in range(3)]
        base[2] = base[2] + dj
        rate = 2 * c["dt"] ** 2
        omega, E = 1.0, self.E
        for _ in range(2 + math.ceil(math.log(1e-16) / math.log(rate / (2 + rate)))):
            X = slot(self.links(E))
            E = [(1 - omega) * E[i] + omega * (base[i] + 0.25 * c["dt"] * self.force(X, i))
                 for i in range(3)]
            omega = 2 / (2 + rate)
        return E, qa, qb

    def table(self):
        U, a = self.U, self.a
        En, _, _ = self.e_next()
        e2 = [0.5 * (self.E[i] ** 2 + En[i] ** 2).sum(0) / a[i] ** 2 for i in range(3)]

        def sides(i, j):
            return _mm(U[i], _shift(U[j], i, 1)), _mm(U[j], _shift(U[i], j, 1))

        b, B = {}, {}
        for i, j in ((0, 1), (0, 2), (1, 2)):
            x, y = sides(i, j)
            m = self.up if j == 2 else 1.0
            b[i, j] = (x - y).abs().square().sum((0, 1)) / (a[i] * a[j]) ** 2 * m
            B[i, j] = 2 * _im_proj(_mm(x, _dag(y))) / (a[i] * a[j]) * m
        p_t = 0.5 * e2[2] + b[0, 1]
        p_l = 0.5 * (e2[0] + e2[1]) + b[0, 2] + b[1, 2] - p_t
        s_l = sum((self.E[i] + En[i]) / (2 * a[i]) * B[i, 2] for i in (0, 1)).sum(0)
        return torch.stack([x.mean((-1, -2)) for x in (p_l + 2 * p_t, p_l, p_t, s_l)], -1)

    def state(self):
        """Links and fields in the library's layout: U - 1 in 32 bits."""
        nc = self.c["nc"]
        E = torch.stack(self.E).reshape(-1)
        if self.c["scheme"] == "implicit":
            return [E]
        out = []
        for u in self.U:
            u = u - _eye(u) if self.c["precision"] == "fp32" else u
            if nc == 2:
                out.append(u[0].reshape(2, -1).T.contiguous())
            else:
                u = u.reshape(9, -1)
                u = torch.nn.functional.pad(torch.view_as_real(u.contiguous()),
                                            (0, 0, 0, -u.shape[1] % 32))
                u = u.reshape(9, -1, 32, 2).permute(1, 0, 2, 3).contiguous()
                out.append(torch.view_as_complex(u))
        return [torch.view_as_real(torch.stack(out)).reshape(-1), E]


def _exact_event(cfg, rho, steps, every):
    x, tabs = _Exact(cfg, torch.from_numpy(rho).cuda()), []
    for k in range(steps):
        x.step()
        if (k + 1) % every == 0:
            tabs.append(x.table())
    return x, torch.stack(tabs)


def _exact_gradient(cfg, rho, steps, half_width):
    from torch.utils.checkpoint import checkpoint
    r = torch.from_numpy(rho).cuda().requires_grad_()
    x = _Exact(cfg, r)

    def step(n, *s):
        x.n, x.U, x.E, x.QA, x.QB = n, s[0:3], s[3:6], s[6], s[7]
        x.step()
        return (*x.U, *x.E, x.QA, x.QB)

    s = (*x.U, *x.E, x.QA, x.QB)
    for n in range(steps):
        s = checkpoint(step, n, *s, use_reentrant=False)
    x.n, x.U, x.E, x.QA, x.QB = steps, s[0:3], s[3:6], s[6], s[7]
    z = torch.arange(cfg["nz"], device="cuda", dtype=torch.float64) * cfg["a_z"]
    inside = (z - cfg["nz"] * cfg["a_z"] / 2).abs() < half_width
    value = cfg["a_z"] * (x.table()[:, 0] * inside).sum()
    value.backward()
    return [value.item(), r.grad]


def _exact_analysis(case, seed):
    tabs, (t0, dts, z0, az) = _tables(case, seed)
    m = tabs.mean(0)
    eps, pl, s = m[..., 0], m[..., 1], m[..., 3]
    root = np.sqrt((eps + pl) ** 2 - 4 * s * s)
    rest = np.concatenate([m, np.stack([(eps - pl + root) / 2, (pl - eps + root) / 2,
                                        2 * s / (eps + pl + root), np.ones_like(eps)], -1)], -1)
    eta, prof = np.linspace(-1.2, 1.2, case["points"]), []
    for tau in _taus(case):
        ft, fz = (tau * np.cosh(eta) - t0) / dts, (tau * np.sinh(eta) - z0) / az
        inside = (ft >= 0) & (ft <= case["samples"] - 1) & (fz >= 0) & (fz <= case["nz"] - 1)
        k = np.clip(np.floor(ft).astype(int), 0, case["samples"] - 2)
        j = np.clip(np.floor(fz).astype(int), 0, case["nz"] - 2)
        wt, wz, g = ft - k, fz - j, rest[..., 4]
        f = ((1 - wt) * ((1 - wz) * g[k, j] + wz * g[k, j + 1])
             + wt * ((1 - wz) * g[k + 1, j] + wz * g[k + 1, j + 1]))
        prof.append(np.where(inside, f, np.nan))
    return [rest.reshape(-1, 8), np.array(prof), None]


def exact(case, seed):
    kind = case["kind"]
    if kind == "analysis":
        return _exact_analysis(case, seed)
    sites = case["nz"] * case["ny"] * case["nx"]
    # a step of one site takes about 30 ns (SU(3)), an improved one 12 times
    # as long, a gradient 6 times
    cost = sites * case["steps"] * (1.0 if case["nc"] == 3 else 0.3)
    cost *= 12 if case["scheme"] == "implicit" else 6 if kind == "gradient" else 1
    if kind == "run" or cost > 4.5e8:
        return None
    cfg = _cfg(case)
    if kind == "observables":
        x = _Exact(cfg, fields=_fields(case, seed))
        tab = x.table()
        return [x.gauss(), tab, tab[:, 0].sum().item() * case["a_z"] * case["ny"] * case["nx"]]
    if kind == "steps":
        x = _Exact(cfg, fields=_fields(case, seed))
        for _ in range(case["steps"]):
            x.step()
        return x.state()
    if kind == "gradient":
        return _exact_gradient(cfg, _rho(case, seed), case["steps"], _half_width(case))
    if kind == "ensemble":      # the first event of each size
        out = [None] * case["events"]
        sizes = _events(case)
        for k, (ny, nx) in enumerate(sizes):
            if sizes.index((ny, nx)) == k:
                out[k] = _exact_event(_cfg(case, ny=ny, nx=nx), _rho(case, [seed, k], nx, ny),
                                      case["steps"], case["steps"])[1][0]
        return out
    x, tabs = _exact_event(cfg, _rho(case, seed), case["steps"], case["every"])
    return [tabs] + (x.state() if case["precision"] == "fp64" else [])
