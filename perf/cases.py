"""Measured calls of the framework: what a user has it do, over the range of sizes it is used on.

A case names one public call and the problem it is made on:

  apply      y = A x or A^H x (``wri.apply_A``): residual and adjoint checks on given wavefields
  solve      the batched CGLS solve of every (source, frequency) system at a fixed number of
             iterations (``wri.solve``): the part of an inversion that takes the time
  gradient   source weights and model gradient on given wavefields (``wri.source_estimate`` and
             ``wri.gradient``), with complex64 wavefields or with their FP64 masters
  objective  f4(m) and its gradient through autograd (``objective.objective``): complex64 solves
             inside FP64 refinement, the certified configuration, for a float32 model
  tv         the total-variation term and its gradient (``wri.tv``) of the outer loop

Grids are given as physical nodes ("128x128x128", x first) with ``npml`` absorbing cells added on
every face; several frequency groups are separated by ";".  Systems are sources at the surface with a
borehole of receivers or an areal receiver grid.  Everything random comes from the seed.

The iteration counts are those up to which two correct roundings of the same CGLS stay together: the strong
layer entries are the first eigenvalues to converge, and from there (20 to 60 iterations on, earlier from a warm
start) an FP32 Krylov basis has lost its orthogonality and any two roundings part.
"""
import math

import numpy as np
import torch

LAYER_R = 1e-3      # target reflection of the absorbing layer
V_MAX = 3300.0      # velocity that sets the layer's damping: layers up to 3000 m/s, +10 % anomaly
V_REF = 2000.0      # medium of the synthetic traces and wavefields


def _solve(name, grid, npml, h, freq, nsys, iters, **kw):
    c = {"name": name, "call": "solve", "grid": grid, "npml": npml, "h": h, "freq": freq, "nsys": nsys, "nrec": 48,
         "iters": iters, "dtype": "c64", "mode": "free", "warm": False, "tuned": False}
    c.update(kw)
    return c


def listed():
    return [
        # the smallest call: one operator application on the 24^3 + 6 grid of the plain configuration,
        # where the launch is the cost
        {"name": "apply_c64_36", "call": "apply", "grid": "24x24x24", "npml": 6, "h": "10", "freq": "5", "nsys": 1,
         "dtype": "c64", "adjoint": False},
        # A^H in complex128 on the 61^3 + 10 timing case (odd extents), 9 sources: the FP64 residual check of a solve
        {"name": "apply_adjoint_c128_81", "call": "apply", "grid": "61x61x61", "npml": 10, "h": "50", "freq": "5",
         "nsys": 9, "dtype": "c128", "adjoint": True},
        # the plain method's configuration: complex128, one source, lambda = 10, 20 receivers on 24^3 + 6
        _solve("solve_c128_config1", "24x24x24", 6, "10", "5", 1, 40, nrec=20, dtype="c128", lam=10.0),
        # one source of the 8 Hz grid on its own: a batch too small to fill the chip
        _solve("solve_one_source_148", "128x128x128", 10, "20", "8", 1, 24, nrec=96),
        # the adaptive loop's solves: 16 sources x 3 frequencies on 64^3 + 10, starting from the last model's wavefields
        _solve("solve_config2_warm", "64x64x64;64x64x64;64x64x64", 10, "10;10;10", "3;5;7", 16, 40, warm=True),
        # the multi-frequency batch on grids of their own, kernel chosen by the autotuner as in the benchmark
        _solve("solve_multigrid_batch", "64x64x64;96x96x96;128x128x128", 10, "40;26.6666666667;20", "3;5;8", 64, 24,
               nrec=96, tuned=True),
        # the largest grid: 256 x 256 x 160 + 10 at 10 Hz, four sources
        _solve("solve_config5", "256x256x160", 10, "8", "10", 4, 24, nrec=96),
        # one misfit + gradient evaluation of the timing case: 9 sources, 45 x 45 receivers, odd extents
        {"name": "objective_81", "call": "objective", "grid": "61x61x61", "npml": 10, "h": "50", "freq": "5", "nsys": 9,
         "nrec": 2025, "iters": 16, "recompute": False},
        # differentiation: 32 sources on 96^3 + 10
        {"name": "objective_config3", "call": "objective", "grid": "96x96x96", "npml": 10, "h": "10", "freq": "6",
         "nsys": 32, "nrec": 48, "iters": 24, "recompute": False},
        # the gradient on complex64 wavefields (32 sources, 5 Hz grid) ...
        {"name": "gradient_c64_116", "call": "gradient", "grid": "96x96x96", "npml": 10, "h": "26.6666666667",
         "freq": "5", "nsys": 32, "nrec": 96, "dtype": "c64", "wide": False},
        # ... and on FP64 wavefields (16 sources, 8 Hz grid): the accurate variant
        {"name": "gradient_fp64_148", "call": "gradient", "grid": "128x128x128", "npml": 10, "h": "20", "freq": "8",
         "nsys": 16, "nrec": 96, "dtype": "c64", "wide": True},
        # the total-variation term on the largest model
        {"name": "tv_config5", "call": "tv", "grid": "256x256x160", "npml": 10, "h": "8", "freq": "10"},
    ]


def draw(rng):
    """Another case of the same calls: odd and ragged grids, every option that is used in earnest."""

    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    call = rng.choice(("apply", "solve", "solve", "solve", "solve", "gradient", "objective", "objective", "tv"))
    if call == "tv":
        n = [log_int(20, 256) for _ in range(3)]
        return {"call": "tv", "grid": "%dx%dx%d" % tuple(n), "npml": rng.choice((0, 6, 10)), "h": "10", "freq": "5"}
    npml = rng.choice((0, 4, 6, 10, 10))
    dtype = rng.choice(("c64", "c64", "c64", "c128")) if call != "objective" else "c64"
    cap = {"apply": 6e7, "solve": 1.2e9 if dtype == "c64" else 1.2e8, "gradient": 4e7, "objective": 6e8}[call]
    warm = call == "solve" and rng.random() < 0.25
    iters = rng.randint(4, 40 if npml == 0 else 8 if warm else 16) if call in ("solve", "objective") else 1
    groups = rng.choice((1, 1, 2, 3)) if call == "solve" else 1
    step = rng.choice((1, 1, 2, 4))  # extents: any, even, multiples of four
    grids, total = [], 0
    for _ in range(groups):
        n = [max(12, log_int(14, 150) // step * step) for _ in range(3)]
        grids.append(n)
        total += np.prod([v + 2 * npml for v in n])
    nsys = max(1, min(log_int(1, 48), int(cap / (total * iters))))
    h = [rng.choice((8.0, 10.0, 20.0, 40.0)) for _ in grids]
    freq = ["%.3f" % (V_REF / (hh * rng.uniform(8.0, 24.0))) for hh in h]   # 8 to 24 points per wavelength
    c = {"call": call, "grid": ";".join("%dx%dx%d" % tuple(n) for n in grids), "npml": npml,
         "h": ";".join(str(v) for v in h), "freq": ";".join(freq), "nsys": nsys}
    if call == "apply":
        c.update(dtype=dtype, adjoint=rng.random() < 0.5)
    elif call == "solve":
        c.update(nrec=rng.choice((1, 7, 48, 96, 400)), iters=iters, dtype=dtype,
                 mode=rng.choice(("free", "free", "free", "known", "rhs")), warm=warm,
                 tuned=dtype == "c64" and rng.random() < 0.2)
    elif call == "gradient":
        c.update(nrec=rng.choice((7, 48, 96)), dtype=dtype, wide=dtype == "c64" and rng.random() < 0.5)
    else:
        c.update(nrec=rng.choice((7, 48, 400)), iters=iters, recompute=rng.random() < 0.25)
    return c


# ------------------------------------------------------------------ the problem of a case
def _groups(case):
    """Per frequency group: physical extents, computational extents (nx, ny, nz), h, omega."""
    out = []
    for g, h, f in zip(case["grid"].split(";"), case["h"].split(";"), case["freq"].split(";")):
        ext = tuple(int(v) for v in g.split("x"))
        out.append((ext, tuple(v + 2 * case["npml"] for v in ext), float(h), 2 * math.pi * float(f)))
    return out


def _model(ext, npml, seed, dtype):
    """Squared slowness [nz, ny, nx] on the GPU: four flat layers (1500-3000 m/s) with seeded interface
    depths and a seeded +10 % Gaussian anomaly, copied outwards into the layer."""
    nx, ny, nz = ext
    r = np.random.Generator(np.random.PCG64(seed))
    ax = [torch.clamp(torch.arange(-npml, n + npml, device="cuda"), 0, n - 1).double() for n in (nz, ny, nx)]
    z, y, x = ax[0][:, None, None], ax[1][None, :, None], ax[2][None, None, :]
    v = torch.full((nz + 2 * npml, ny + 2 * npml, nx + 2 * npml), 1500.0, dtype=torch.float64, device="cuda")
    for layer in range(3):
        v += 500.0 * (z >= (layer + 1) * nz / 4 + r.uniform(-0.1, 0.1) * nz)
    c = r.uniform(0.3, 0.7, 3) * (nx, ny, nz)
    sig = max(2.0, min(ext) / 12.0)
    v *= 1 + 0.1 * torch.exp(-0.5 * ((x - c[0]) ** 2 + (y - c[1]) ** 2 + (z - c[2]) ** 2) / sig ** 2)
    return (1.0 / v ** 2).to(dtype).contiguous()


def _geometry(ext, npml, nsys, nrec):
    """Source nodes on a surface lattice and receiver nodes (a borehole, or an areal grid when there are more
    than fit in it), as physical (x, y, z) and as linear nodes of the computational grid."""
    nx, ny, nz = ext
    cols = math.ceil(math.sqrt(nsys * nx / ny))
    rows = math.ceil(nsys / max(cols, 1))
    src = [(int((i % cols + 0.5) * nx / cols), int((i // cols + 0.5) * ny / rows), min(2, nz - 1)) for i in range(nsys)]
    if nrec <= nz - 4:
        rec = [(nx // 2 + 1, ny // 2 + 1, int(z)) for z in np.unique(np.linspace(3, nz - 2, nrec).round())]
    else:
        k = max(1, min(int(round(math.sqrt(nrec))), nx - 2, ny - 2))
        rec = [(int(x), int(y), (3 * nz) // 4) for y in np.unique(np.linspace(1, ny - 2, k).round())
               for x in np.unique(np.linspace(1, nx - 2, k).round())]
    cx, cy = nx + 2 * npml, ny + 2 * npml
    lin = lambda p: [((z + npml) * cy + (y + npml)) * cx + x + npml for x, y, z in p]  # noqa: E731
    return np.array(src, float), np.array(rec, float), np.array(lin(src), np.int64), np.array(lin(rec), np.int32)


def _weights(nsys, seed):
    r = np.random.Generator(np.random.PCG64(seed))
    return r.uniform(5.0, 15.0, nsys) * np.exp(1j * r.uniform(-np.pi, np.pi, nsys))


def _traces(src, rec, h, omega, alpha, seed):
    """Receiver traces [nsys, nrec]: spreading and phase of a homogeneous medium, 2 % noise."""
    r = np.random.Generator(np.random.PCG64(seed))
    dist = h * np.linalg.norm(rec[None] - src[:, None], axis=2) + 0.5 * h
    tr = -alpha[:, None] * h ** 3 * np.exp(1j * omega / V_REF * dist) / (4 * np.pi * dist)
    return tr * (1 + 0.02 * (r.standard_normal(tr.shape) + 1j * r.standard_normal(tr.shape)))


def _wavefield(shape, src, npml, h, omega, alpha, seed, dtype):
    """Wavefield-like vectors [nsys, n] on the GPU: the homogeneous medium's outgoing waves, 1 % noise, dying
    out in the absorbing layer."""
    nz, ny, nx = shape
    gen = torch.Generator(device="cuda").manual_seed(seed)
    out = torch.empty(len(src), nz * ny * nx, dtype=dtype, device="cuda")
    ax = [torch.arange(n, device="cuda", dtype=torch.float64) for n in (nz, ny, nx)]
    fade = [1.0 / (1 + torch.clamp(torch.maximum(npml - a, a - (len(a) - 1 - npml)), min=0.0)) ** 4 for a in ax]
    fade = fade[0][:, None, None] * fade[1][None, :, None] * fade[2][None, None, :]
    for s in range(len(src)):
        d = torch.sqrt((ax[0][:, None, None] - src[s, 2] - npml) ** 2 + (ax[1][None, :, None] - src[s, 1] - npml) ** 2
                       + (ax[2][None, None, :] - src[s, 0] - npml) ** 2) * h + 0.5 * h
        amp = (abs(alpha[s]) * h ** 3 / (4 * math.pi)) * fade / d
        u = torch.polar(amp, d * (omega / V_REF) + math.pi + float(np.angle(alpha[s])))
        z = torch.randn(nz, ny, nx, dtype=torch.complex64, device="cuda", generator=gen)
        out[s] = (u * (1 + 0.01 * z)).reshape(-1)
    return out


def _specs(case, seed):
    """The GroupSpecs of a case, with what prepare() and exact() both need beside them."""
    from paper_2410_18429_gb300 import wri
    c128 = case.get("dtype") == "c128"
    rdt, cdt = (torch.float64, torch.complex128) if c128 else (torch.float32, torch.complex64)
    call, mode, nsys = case["call"], case.get("mode", "free"), case["nsys"]
    specs = []
    for j, (ext, dim, h, omega) in enumerate(_groups(case)):
        nx, ny, nz = dim
        n, s0 = nx * ny * nz, 1000 * seed + 10 * j
        src, rec, src_n, rec_n = _geometry(ext, case["npml"], nsys, case.get("nrec", 1))
        alpha = _weights(nsys, s0 + 1)
        d = _traces(src, rec, h, omega, alpha, s0 + 2)
        lam = 0.0 if mode == "rhs" else case.get("lam", 1.0 / h ** 2)
        al = q = u64 = None
        if mode == "known":
            al = torch.view_as_real(torch.from_numpy(alpha)).contiguous().cuda()
        waves = lambda k, t: _wavefield((nz, ny, nx), src, case["npml"], h, omega, alpha, s0 + k, t)  # noqa: E731
        if mode == "rhs":  # the adjoint solves of reduced FWI: data residuals at the receivers
            q = torch.zeros(nsys, n, dtype=cdt, device="cuda")
            q[:, torch.from_numpy(rec_n.astype(np.int64)).cuda()] = torch.from_numpy(d.conj()).to(cdt).cuda()
        if call == "objective":
            u = torch.empty(0, dtype=cdt, device="cuda")
        elif call in ("apply", "gradient"):
            u = waves(4, torch.complex128 if case.get("wide") else cdt)
            if case.get("wide"):
                u64, u = u, u.to(cdt)
        else:
            u = torch.zeros(nsys, n, dtype=cdt, device="cuda")
        specs.append(wri.GroupSpec(nx, ny, nz, case["npml"], h, omega, V_MAX, _model(ext, case["npml"], s0, rdt), src_n,
                                   np.arange(nsys + 1, dtype=np.int32) * len(rec_n), np.tile(rec_n, nsys),
                                   torch.from_numpy(d.reshape(-1)).to(cdt).cuda(), lam, u, al, LAYER_R, u64, q))
        if case.get("warm"):
            specs[-1].u.copy_(waves(5, cdt))
    return specs


def prepare(case, seed):
    from paper_2410_18429_gb300 import wri
    call = case["call"]
    if call == "tv":
        (ext, dim, h, omega), = _groups(case)
        m = _model(ext, case["npml"], 1000 * seed, torch.float64)
        spec = wri.GroupSpec(*dim, case["npml"], h, omega, V_MAX, m, np.zeros(1, np.int64), np.zeros(2, np.int32),
                             np.zeros(0, np.int32), None, 1.0, None)
        return {"call": call, "spec": spec, "m": m, "beta": 1e-9}
    specs = _specs(case, seed)
    code = wri.C128 if case.get("dtype") == "c128" else wri.C64
    st = {"call": call, "specs": specs, "code": code}
    if call == "apply":
        st["adjoint"] = case["adjoint"]
    elif call == "solve":
        opts = wri.make_opts(tol=0.0, max_iter=case["iters"], dtype=code, warm_start=case["warm"])
        st["work"] = torch.empty(wri.workspace_size(specs, opts), dtype=torch.uint8, device="cuda")
        st["u0"] = [s.u.clone() for s in specs] if case["warm"] else None
        if case["tuned"]:
            opts = wri.autotune(specs, opts, trial_iters=8, workspace=st["work"])
        st["opts"] = opts
    elif call == "gradient":
        st["work"] = torch.empty(wri.aux_workspace_size(specs), dtype=torch.uint8, device="cuda")
    else:
        st["m"] = specs[0].m.clone().requires_grad_(True)
        st["recompute"] = case["recompute"]
        st["opts"] = wri.make_opts(tol=0.0, max_iter=case["iters"], dtype=wri.C64, max_refine=1, refine_tol=0.0,
                                   inner_tol=1e-12)
    return st


def run(state):
    from paper_2410_18429_gb300 import objective, wri
    call = state["call"]
    if call == "tv":
        grad = torch.zeros_like(state["m"])
        tv, _ = wri.tv(state["spec"], state["m"], state["beta"], 0.02, grad=grad)
        return {"tv": tv, "grad": grad}
    specs = state["specs"]
    if call == "apply":
        return wri.apply_A(specs[0], specs[0].u, adjoint=state["adjoint"])
    if call == "solve":
        if state["u0"] is not None:
            for s, u in zip(specs, state["u0"]):  # the wavefields of the last model
                s.u.copy_(u)
        iters, _, status = wri.solve(specs, state["opts"], workspace=state["work"])
        return {"u": [s.u for s in specs], "iters": iters, "status": status}
    if call == "gradient":
        alpha = wri.source_estimate(specs, state["code"], workspace=state["work"])
        grads, f = wri.gradient(specs, state["code"], alpha, workspace=state["work"])
        return {"alpha": alpha, "grads": grads, "f": f}
    m = state["m"]
    m.grad = None
    stats = {}
    objective.objective(m, specs, state["opts"], recompute=state["recompute"], stats=stats).backward()
    return {"grad": m.grad, "iters": stats["iters"]}


def work(case):
    """Solves: each CGLS iteration reads and writes its four vectors once per product with A (s, p -> p, t and
    r, t -> r, s); everything else: each input read and each output written once."""
    if case["call"] == "tv":
        (_, dim, _, _), = _groups(case)
        n = np.prod(dim)
        return {"bytes": float(24 * n), "flops": float(45 * n)}
    n = float(sum(np.prod(g[1]) for g in _groups(case)))
    ns, cb = n * case["nsys"], 16 if case.get("dtype") == "c128" else 8
    if case["call"] == "apply":
        return {"bytes": 2 * cb * ns + cb / 2 * n, "flops": 18 * ns}
    if case["call"] == "gradient":
        return {"bytes": (16 if case["wide"] else cb) * ns + (cb / 2 + 8) * n, "flops": 28 * ns}
    it = case["iters"] * (2 if case.get("recompute") else 1)
    if case["call"] == "objective":   # and the FP64 residual: x and r read, r written, read for the gradient
        return {"bytes": it * 64 * ns + 64 * ns + 8 * n, "flops": it * 60 * ns + 70 * ns}
    return {"bytes": it * 8 * cb * ns + cb * ns + cb / 2 * n, "flops": it * 60 * ns}


# ------------------------------------------------------------------ the same in 64 bits
class _Operator:
    """A and A^H on [k, nz, ny, nx] complex128: omega^2 w m u + the 7-point Laplacian with the axes stretched
    by s = 1 + i sigma / omega in the layer, zero outside the grid."""

    def __init__(self, spec):
        self.m = (spec.m.double() * spec.omega ** 2)
        self.shape = (spec.nz, spec.ny, spec.nx)
        self.s, self.half = [], []
        for a, n in enumerate(self.shape):
            view = [1, 1, 1]
            view[a] = -1
            node = torch.arange(n, dtype=torch.float64, device="cuda")
            edge = torch.arange(n + 1, dtype=torch.float64, device="cuda") - 0.5
            self.s.append(self._stretch(spec, n, node).view(view))
            self.half.append((1.0 / (self._stretch(spec, n, edge) * spec.h ** 2)).view(view))
        self.w = self.s[0] * self.s[1] * self.s[2]

    @staticmethod
    def _stretch(spec, n, pos):
        if spec.npml == 0:
            return torch.ones_like(pos) + 0j
        length = spec.npml * spec.h
        top = 3.0 * spec.v_max * math.log(1.0 / spec.pml_R) / (2.0 * length)
        xi = torch.clamp(torch.maximum(spec.npml - pos, pos - (n - 1 - spec.npml)), min=0.0) * spec.h
        return torch.complex(torch.ones_like(pos), top * (xi / length) ** 2 / spec.omega)

    def __call__(self, u):
        out = self.w * self.m * u
        for a in range(3):
            size = list(u.shape)
            size[a + 1] += 2
            pad = torch.zeros(size, dtype=u.dtype, device=u.device)
            pad.narrow(a + 1, 1, self.shape[a]).copy_(u)
            flux = torch.diff(pad, dim=a + 1)
            del pad
            flux *= self.half[a]
            lap = torch.diff(flux, dim=a + 1)
            del flux
            b, c = (self.s[k] for k in range(3) if k != a)
            lap *= b * c
            out += lap
        return out

    def adjoint(self, u):
        return self(u.conj().resolve_conj()).conj().resolve_conj()


def _cgls(A, src, rec, lam, b1, b2, x, iters):
    """``iters`` CGLS iterations of min ||Z A x - b1||^2 + ||lam P x - b2||^2 for a chunk of systems; ``src``
    None: Z = I."""
    k = x.shape[0]
    row = torch.arange(k, device="cuda")
    flat = lambda v: v.view(k, -1)  # noqa: E731
    dot = lambda v: torch.linalg.vector_norm(flat(v), dim=1) ** 2  # noqa: E731

    def fwd(v):
        t = A(v)
        if src is not None:
            flat(t)[row, src] = 0
        return t, lam * flat(v)[:, rec]

    def adj(r1, r2):
        s = A.adjoint(r1)
        flat(s)[:, rec] += lam * r2
        return s

    t1, t2 = fwd(x)
    r1, r2 = b1 - t1, b2 - t2
    s = adj(r1, r2)
    p, gamma = s.clone(), dot(s)
    up = lambda c: c.view(k, 1, 1, 1)  # noqa: E731
    for _ in range(iters):
        t1, t2 = fwd(p)
        alpha = gamma / (dot(t1) + dot(t2))
        x = x + up(alpha) * p
        r1 -= up(alpha) * t1
        r2 = r2 - alpha[:, None] * t2
        s = adj(r1, r2)
        new = dot(s)
        p = s + up(new / gamma) * p
        gamma = new
    return x


def _solved(spec, A, iters, warm, lo, hi):
    """The wavefields of systems lo..hi-1 after the iterations."""
    shape = (hi - lo,) + A.shape
    rec = torch.from_numpy(np.asarray(spec.rec_idx[:spec.rec_off[1]], np.int64)).cuda()
    src = torch.from_numpy(np.asarray(spec.src[lo:hi])).cuda()
    b1 = torch.zeros(shape, dtype=torch.complex128, device="cuda")
    if spec.q is not None:
        b1 = spec.q[lo:hi].to(torch.complex128).view(shape)
    elif spec.alpha is not None:
        b1.view(hi - lo, -1)[torch.arange(hi - lo, device="cuda"), src] = torch.view_as_complex(spec.alpha)[lo:hi]
    free = spec.q is None and spec.alpha is None
    b2 = spec.lam * spec.d.to(torch.complex128).view(len(spec.src), -1)[lo:hi]
    x = spec.u[lo:hi].to(torch.complex128).view(shape) if warm else torch.zeros_like(b1)
    return _cgls(A, src if free else None, rec, spec.lam, b1, b2, x, iters)


def _gradient(spec, A, u, lo, hi, grad):
    """alpha = (A u)[src], f and grad += omega^2 Re(conj(w u)(A u - alpha e)) of systems lo..hi-1."""
    r = A(u)
    src = torch.from_numpy(np.asarray(spec.src[lo:hi])).cuda()
    row = torch.arange(hi - lo, device="cuda")
    alpha = r.view(hi - lo, -1)[row, src].clone()
    r.view(hi - lo, -1)[row, src] = 0
    rec = torch.from_numpy(np.asarray(spec.rec_idx[:spec.rec_off[1]], np.int64)).cuda()
    miss = u.view(hi - lo, -1)[:, rec] - spec.d.to(torch.complex128).view(len(spec.src), -1)[lo:hi]
    f = 0.5 * torch.linalg.vector_norm(r) ** 2 + 0.5 * spec.lam ** 2 * torch.linalg.vector_norm(miss) ** 2
    grad += spec.omega ** 2 * torch.real(torch.conj(A.w * u) * r).sum(dim=0)
    return alpha, f


def exact(case, seed):
    call = case["call"]
    if call == "tv":
        st = prepare(case, seed)
        m, beta = st["m"].clone().requires_grad_(True), st["beta"]
        d2 = torch.full_like(m, beta ** 2)
        for a in range(3):
            zero = torch.zeros_like(m.narrow(a, 0, 1))
            d2 = d2 + torch.cat([torch.diff(m, dim=a), zero], dim=a) ** 2
        tv = 0.02 * torch.sqrt(d2).sum()
        tv.backward()
        return {"tv": tv.detach().reshape(1), "grad": m.grad}
    if work(case)["bytes"] > 1.5e12:  # more than about 20 s
        return None
    specs = _specs(case, seed)
    found = []
    for spec in specs:
        A = _Operator(spec)
        nsys = len(spec.src)
        step = max(1, min(nsys, int(2.4e7 / (spec.nx * spec.ny * spec.nz))))
        parts = [(b, min(b + step, nsys)) for b in range(0, nsys, step)]
        if call == "apply":
            op = A.adjoint if case["adjoint"] else A
            return torch.cat([op(spec.u[b:e].to(torch.complex128).view((e - b,) + A.shape)).view(e - b, -1)
                              for b, e in parts])
        if call == "solve":
            found.append(torch.cat([_solved(spec, A, case["iters"], case["warm"], b, e).view(e - b, -1)
                                    for b, e in parts]))
            continue
        grad, f, alphas = torch.zeros(A.shape, dtype=torch.float64, device="cuda"), 0.0, []
        for b, e in parts:
            if call == "objective":
                u = _solved(spec, A, case["iters"], False, b, e)
            else:
                u = (spec.u if spec.u64 is None else spec.u64)[b:e].to(torch.complex128).view((e - b,) + A.shape)
            a, fb = _gradient(spec, A, u, b, e, grad)
            alphas.append(a)
            f = f + fb
        if call == "objective":
            return {"grad": grad, "iters": None}
        return {"alpha": torch.cat(alphas), "grads": [grad], "f": f.reshape(1)}
    return {"u": found, "iters": None, "status": None}

