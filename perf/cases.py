"""Workloads of the smoothing library, one pass each through its public calls.

A case names a lattice, a precision and storage, a smoother and its
parameters; `prepare` makes what a user's program holds before the call (the
seeded inputs on the GPU, a field), `run` is one pass of that program, `exact`
is the same pass in plain FP64 torch.  The vortex fields are iid Z(3) labels
with P(0) = 0.7 as in the 4^4 workload (6 of 10 plaquettes pierced, like the
projected hot starts of the other workloads); a pass starts from the labels,
so it can be repeated.  Passes have a few sweeps where a production run has
hundreds: the sweeps are alike, and the flow has not yet amplified rounding.
"""

import math

import numpy as np
import torch

from paper_2203_09764_gb300 import vs

OMEGA, CENTRIFUGE_SEED = 0.02, 1234
CHUNK = 1 << 19          # sites handled at once by the FP64 restatement


def _case(name, path, dims, **more):
    case = dict(name=name, path=path, lx=dims[0], ly=dims[1], lz=dims[2], lt=dims[3], precision="fp32", storage=18,
                epsilon=-0.25, step=0.06, sweeps=4, start="vortex", preserve=True, gauge=False, schedule="annealed",
                report=False)
    case.update(more)
    return case


def listed():
    return [
        # the smallest workload: 4^4 pure vortex field in FP64, 10 standard stout sweeps and the checks
        _case("stout_4_fp64", "stout", (4, 4, 4, 4), precision="fp64", epsilon=1.0, step=0.1, sweeps=10, report=True),
        # over-improved smoothing of the served shapes, one field alone
        _case("stout_8", "stout", (8, 8, 8, 8)),
        _case("stout_16_12real", "stout", (16, 16, 16, 32), storage=12),
        _case("stout_24", "stout", (24, 24, 24, 48)),
        # the benchmark's lattice: smoothing and the checks that follow it
        _case("stout_32", "stout", (32, 32, 32, 64), report=True),
        # the largest lattice
        _case("stout_48", "stout", (48, 48, 48, 96)),
        # the FP64 path of the 16^3x32 workload
        _case("stout_16_fp64", "stout", (16, 16, 16, 32), precision="fp64", sweeps=1),
        # a small ensemble of fields of four shapes through the serving loop
        _case("serve_mix", "serve", (24, 24, 24, 48), jobs=12, sweeps=10),
        # Wilson flow by Runge-Kutta of a rough gauge field
        _case("flow_32", "flow", (32, 32, 32, 64), epsilon=1.0, step=0.02, start="rough", preserve=False),
        # annealed MaxReTr smearing in a random gauge on the paper's own lattice
        _case("aus_20", "aus", (20, 20, 20, 40), step=0.02, gauge=True),
        # cooling of a hot start: the input generator, and the first phase of a served job
        _case("cool_24", "aus", (24, 24, 24, 48), epsilon=1.0, step=1.0, sweeps=3, start="hot", preserve=False),
        # the measurements made on a smoothed field
        _case("measure_32", "measure", (32, 32, 32, 64), gauge=True, sweeps=0),
    ]


def _sites(dims):
    return dims[0] * dims[1] * dims[2] * dims[3]


def draw(rng):
    """One more case: extents multiples of 4, volumes spread over their logarithm from 4^4 to 48^3x96."""
    path = rng.choice(["stout", "stout", "stout", "stout", "aus", "cool", "ape", "flow", "measure", "fp64", "serve"])
    most = {"fp64": 16 ** 3 * 32, "serve": 16 ** 3 * 32}.get(path, 48 ** 3 * 96)
    # rough links and gauge transforms come in as FP64 matrices: a smaller top keeps their preparation short
    if path in ("cool", "flow", "measure", "aus", "ape"):
        most = 32 ** 3 * 64
    while True:
        target = math.exp(rng.uniform(math.log(256), math.log(most)))
        side = target ** 0.25
        dims = tuple(4 * max(1, round(side * math.exp(rng.uniform(-0.4, 0.4)) / 4)) for _ in range(4))
        if _sites(dims) <= most and max(dims) <= 96:
            break
    storage = rng.choice([18, 18, 12])
    eps = rng.choice([-0.25, -0.25, 1.0])
    if path == "stout":
        return _case("", path, dims, storage=storage, epsilon=eps, step=round(rng.uniform(0.04, 0.06), 3),
                     sweeps=rng.randint(1, 4), preserve=rng.random() < 0.7,
                     schedule=rng.choice(["annealed", "annealed", "annealed", "simultaneous"]),
                     report=rng.random() < 0.3)
    if path == "aus":
        return _case("", "aus", dims, storage=storage, epsilon=eps, step=round(rng.uniform(0.01, 0.03), 3), gauge=True,
                     sweeps=rng.randint(1, 4))
    if path == "cool":
        return _case("", "aus", dims, storage=storage, epsilon=1.0, step=1.0, sweeps=rng.randint(1, 3), start="hot",
                     preserve=False)
    if path == "ape":
        return _case("", "ape", dims, storage=storage, epsilon=eps, step=round(rng.uniform(0.01, 0.03), 3), gauge=True,
                     sweeps=rng.randint(1, 3), schedule=rng.choice(["annealed", "simultaneous"]))
    if path == "flow":
        return _case("", "flow", dims, storage=storage, epsilon=eps, step=round(rng.uniform(0.01, 0.03), 3),
                     sweeps=rng.randint(1, 4), start="rough", preserve=False)
    if path == "measure":
        return _case("", "measure", dims, storage=storage, gauge=True, sweeps=0)
    if path == "serve":
        return _case("", "serve", dims, jobs=rng.randint(4, 12), sweeps=10, epsilon=eps, storage=storage)
    return _case("", "stout", dims, precision="fp64", epsilon=eps, sweeps=1, step=round(rng.uniform(0.04, 0.06), 3),
                 report=rng.random() < 0.3)


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------

def _dims(case):
    return case["lx"], case["ly"], case["lz"], case["lt"]


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _labels(dims, gen):
    u = torch.rand((4, _sites(dims)), generator=gen, device="cuda")
    return torch.where(u < 0.7, 0, torch.where(u < 0.85, 1, -1)).to(torch.int8)


def _haar(n, gen):
    """n Haar-distributed SU(3) matrices: Gram-Schmidt of Gaussian rows, the third row from the first two."""
    z = torch.randn((n, 2, 3, 2), generator=gen, device="cuda", dtype=torch.float64)
    z = torch.view_as_complex(z)
    a = z[:, 0] / z[:, 0].norm(dim=1, keepdim=True)
    b = z[:, 1] - (a.conj() * z[:, 1]).sum(1, keepdim=True) * a
    b = b / b.norm(dim=1, keepdim=True)
    return torch.stack([a, b, torch.linalg.cross(a, b, dim=1).conj()], 1)


def _rough(n, gen):
    """n SU(3) matrices spread around the identity like the links of a thermal field."""
    out = torch.empty((n, 3, 3), dtype=torch.complex128, device="cuda")
    for k in range(0, n, CHUNK):
        m = min(CHUNK, n - k)
        h = torch.view_as_complex(torch.randn((m, 3, 3, 2), generator=gen, device="cuda", dtype=torch.float64))
        h = 0.15 * (h + _dag(h))
        h = h - torch.eye(3, device="cuda") * (h.diagonal(dim1=1, dim2=2).sum(1) / 3)[:, None, None]
        out[k:k + m] = _exp(1j * h)
    return out


def _inputs(case, seed):
    """What the pass reads: labels (vortex), or FP64 links (hot, rough), and the random gauge if it has one."""
    gen = _generator(seed)
    dims = _dims(case)
    V = _sites(dims)
    labels = links = gauge = None
    if case["start"] == "vortex":
        labels = _labels(dims, gen)
    elif case["start"] == "hot":
        links = _haar(4 * V, gen).reshape(4, V, 3, 3)
    else:
        links = _rough(4 * V, gen).reshape(4, V, 3, 3)
    if case["gauge"]:
        gauge = _haar(V, gen)
    return labels, links, gauge


SHAPES = ((8, 8, 8, 8), (12, 12, 12, 24), (8, 8, 8, 8), (16, 16, 16, 32), (12, 12, 12, 24))


def _jobs(case, seed):
    """The jobs of a served ensemble: one field of the case's own lattice, then the smaller shapes of the mix in turn,
    each with its labels and a step size between 0.04 and 0.1."""
    gen = _generator(seed)
    jobs = []
    for k in range(case["jobs"]):
        dims = _dims(case) if k == 0 else SHAPES[(k - 1) % len(SHAPES)]
        jobs.append((dims, round(0.04 + 0.06 * ((k * 7) % 12) / 12, 4), _labels(dims, gen)))
    return jobs


class _State:
    """A field (or a serving context) with the buffers of a user's program; freed with the object."""

    def __init__(self, **k):
        self.field = None
        self.__dict__.update(k)

    def __del__(self):
        if self.field is not None:
            vs.vs_field_destroy(self.field)
        vs.vs_destroy(self.ctx)


def _precision(case):
    return vs.VS_FP64 if case["precision"] == "fp64" else vs.VS_FP32


def _storage(case):
    return vs.VS_LINK12 if case["storage"] == 12 else vs.VS_LINK18


def prepare(case, seed):
    if case["path"] == "serve":
        jobs = [(d, rho, lab.cpu().numpy()) for d, rho, lab in _jobs(case, seed)]
        return _State(case=case, ctx=vs.vs_create(0, hbm_budget_bytes=512 << 20, max_slots=8), jobs=jobs)
    labels, links, gauge = _inputs(case, seed)
    ctx = vs.vs_create(0)
    field = vs.vs_field_create(ctx, _dims(case), _precision(case), _storage(case), torch.cuda.current_stream())
    shape = (4, _sites(_dims(case)), 3, 3)
    state = _State(case=case, ctx=ctx, field=field, labels=labels, links=links, gauge=gauge)
    if case["path"] == "measure":
        state.current = torch.empty(shape[:2], dtype=torch.int8, device="cuda")
        _load(state)
        vs.vs_synchronize(field)
        state.labels = state.gauge = None
    else:
        state.out = torch.empty(shape, dtype=torch.complex128, device="cuda")
    return state


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------

def _load(s):
    if s.links is not None:
        vs.vs_load_field(s.field, links=s.links)
    else:
        vs.vs_load_field(s.field, labels=s.labels)
        vs.vs_centrifuge(s.field, OMEGA, CENTRIFUGE_SEED)
    if s.gauge is not None:
        vs.vs_gauge_transform(s.field, s.gauge)


def _number(case, v):
    """A result of an FP32 field carries FP32 precision."""
    return float(v) if case["precision"] == "fp64" else np.float32(v)


def _check(case, f):
    r = vs.vs_vortex_check(f)
    r["min_margin"] = _number(case, r["min_margin"])
    return r


def run(s):
    c = s.case
    if c["path"] == "serve":
        tickets = [vs.vs_submit(s.ctx, vs.make_job(d, rho, c["sweeps"], epsilon=c["epsilon"], labels=lab, omega=OMEGA,
                                                   centrifuge_seed=CENTRIFUGE_SEED, storage=_storage(c)))
                   for d, rho, lab in s.jobs]
        done = [vs.vs_poll(s.ctx, t) for t in tickets]
        return [dict(action=np.float32(r["action"]), n_label_diff=r["n_label_diff"], status=r["status"]) for r in done]
    f = s.field
    if c["path"] == "measure":
        o = vs.vs_observables(f)
        vs.vs_current_labels(f, s.current)
        return dict(observables={k: _number(c, v) for k, v in o.items()}, action=_number(c, vs.vs_action(f)),
                    check=_check(c, f), labels=s.current)
    _load(s)
    kind = vs.VS_SIMULTANEOUS if c["schedule"] == "simultaneous" else vs.VS_ANNEALED
    if c["path"] == "stout":
        vs.vs_smooth(f, c["sweeps"], c["step"], c["epsilon"], kind=kind, vortex_preserve=c["preserve"])
    elif c["path"] == "aus":
        vs.vs_smooth_aus(f, c["sweeps"], c["step"], c["epsilon"], vortex_preserve=c["preserve"])
    elif c["path"] == "ape":
        vs.vs_smooth_ape(f, c["sweeps"], c["step"], c["epsilon"], schedule=kind, vortex_preserve=c["preserve"])
    else:
        vs.vs_flow_rk3(f, c["sweeps"], c["step"], c["epsilon"])
    out = {}
    if c["report"]:
        out["action"] = _number(c, vs.vs_action(f))
        out["check"] = _check(c, f)
    vs.vs_read_field(f, s.out)
    out["links"] = s.out if c["precision"] == "fp64" else s.out.to(torch.complex64)
    return out


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------

ROWS2, FULL = 144, 216   # flops of two rows (the third of an SU(3) product follows from them) and of three


def _flops_per_update(epsilon):
    if epsilon == 1.0:
        return 6 * 2 * ROWS2 + 2 * FULL
    return 6 * (9 * ROWS2 + FULL) + 4 * FULL


def work(case):
    V = _sites(_dims(case))
    if case["path"] == "serve":
        shapes = [_dims(case)] + [SHAPES[k % len(SHAPES)] for k in range(case["jobs"] - 1)]
        V = sum(_sites(d) for d in shapes)
        return {"bytes": 4 * V, "flops": 4 * V * case["sweeps"] * _flops_per_update(case["epsilon"])}
    link = 144 if case["precision"] == "fp64" else 72
    if case["path"] == "measure":
        stored = link * case["storage"] // 18
        # six clovers of four leaves, the plaquettes of the action among them
        return {"bytes": V * (4 * stored + 4 + 4), "flops": V * 6 * 12 * FULL}
    read = 4 * V if case["start"] == "vortex" else 4 * V * 144
    if case["gauge"]:
        read += 144 * V
    stages = 3 if case["path"] == "flow" else 1
    return {"bytes": read + 4 * V * link, "flops": 4 * V * case["sweeps"] * stages * _flops_per_update(case["epsilon"])}


# ---------------------------------------------------------------------------
# The same pass in FP64 torch, path by path from the definitions
# ---------------------------------------------------------------------------

def _mm(a, b):
    return a[:, :, 0:1] * b[:, 0:1, :] + a[:, :, 1:2] * b[:, 1:2, :] + a[:, :, 2:3] * b[:, 2:3, :]


def _dag(a):
    return a.conj().transpose(-1, -2)


def _trace(a):
    return a[..., 0, 0] + a[..., 1, 1] + a[..., 2, 2]


def _eye(like):
    return torch.eye(3, dtype=like.dtype, device=like.device)


def _exp(x):
    """Taylor series of the matrix exponential; |x| is at most about 2."""
    term = _eye(x).expand_as(x).clone()
    total = term.clone()
    for n in range(1, 31):
        term = _mm(term, x) / n
        total += term
    return total


class _Lattice:
    def __init__(self, dims):
        self.dims = dims
        self.V = _sites(dims)
        self.stride = (1, dims[0], dims[0] * dims[1], dims[0] * dims[1] * dims[2])

    def coord(self, s, d):
        return (s // self.stride[d]) % self.dims[d]

    def shift(self, s, d, k):
        x = self.coord(s, d)
        return s + ((x + k) % self.dims[d] - x) * self.stride[d]

    def sites(self):
        return torch.arange(self.V, device="cuda")

    def path(self, U, s, steps):
        """Product of the links along steps (+-1 .. +-4: one site along direction |step| - 1) from sites s."""
        out = None
        for step in steps:
            d = abs(step) - 1
            if step > 0:
                link = U[d][s]
                s = self.shift(s, d, 1)
            else:
                s = self.shift(s, d, -1)
                link = _dag(U[d][s])
            out = link if out is None else _mm(out, link)
        return out

    def staples(self, U, s, mu, epsilon):
        """Over-improved staple sum: 6 plaquette staples and 18 rectangles (u0 = 1)."""
        c0, c1 = (5 - 2 * epsilon) / 3, (epsilon - 1) / 12
        m = mu + 1
        total = 0
        for nu in range(4):
            if nu == mu:
                continue
            for n in (nu + 1, -nu - 1):
                total = total + c0 * self.path(U, s, (n, m, -n))
                if c1:
                    for steps in ((n, n, m, -n, -n), (n, m, m, -n, -m), (-m, n, m, m, -n)):
                        total = total + c1 * self.path(U, s, steps)
        return total

    def classes(self, mu):
        """The sites of each colour class of direction mu."""
        s = self.sites()
        colour = (sum(self.coord(s, d) for d in range(4)) + self.coord(s, mu)) % 4
        return [s[colour == c] for c in range(4)]


def _centre_label(t):
    phi = torch.atan2(torch.where(t.imag == 0, 0.0, t.imag), t.real)
    return torch.where(phi.abs() < math.pi / 3, 0, torch.where(phi > 0, 1, -1)).to(torch.int8)


def _margin(t):
    phi = torch.atan2(t.imag, t.real).abs()
    return torch.minimum((phi - math.pi / 3).abs(), math.pi - phi)


def _splitmix(seed, i):
    def shr(z, k):
        return (z >> k) & ((1 << (64 - k)) - 1)

    def wrap(v):
        v &= (1 << 64) - 1
        return v - (1 << 64) if v >> 63 else v

    z = (i + 1) * wrap(0x9E3779B97F4A7C15) + seed
    z = (z ^ shr(z, 30)) * wrap(0xBF58476D1CE4E5B9)
    z = (z ^ shr(z, 27)) * wrap(0x94D049BB133111EB)
    return z ^ shr(z, 31)


def _centrifuge(lat, labels):
    lab = labels.to(torch.int64)
    s = lat.sites()
    U = torch.zeros((4, lat.V, 3, 3), dtype=torch.complex128, device="cuda")
    for mu in range(4):
        m = torch.zeros_like(s)
        up = lat.shift(s, mu, 1)
        for nu in range(4):
            if nu != mu:
                fwd, back = lat.shift(s, nu, 1), lat.shift(s, nu, -1)
                m += lab[nu][s] + lab[mu][fwd] - lab[nu][up] - lab[nu][back] + lab[mu][back]
                m += lab[nu][lat.shift(back, mu, 1)]
        n = lab[mu]
        delta = OMEGA * (m - 6 * n).double() / 9
        z = _splitmix(CENTRIFUGE_SEED, mu * lat.V + s)
        j = ((((z >> 1) & ((1 << 63) - 1)) % 3) * 2 + (z & 1)) % 3
        for c in range(3):
            phase = math.pi * (2 * n.double() / 3 + delta * ((j == c).double() - ((j + 1) % 3 == c).double()))
            U[mu, :, c, c] = torch.polar(torch.ones_like(phase), phase)
    return U


def _start(case, seed):
    labels, links, gauge = _inputs(case, seed)
    lat = _Lattice(_dims(case))
    if links is not None:
        return lat, None, links, None
    U = _centrifuge(lat, labels)
    if gauge is not None:
        for mu in range(4):
            for s in lat.sites().split(CHUNK):
                U[mu][s] = _mm(_mm(gauge[s], U[mu][s]), _dag(gauge[lat.shift(s, mu, 1)]))
    return lat, labels, U, gauge


def _vortex_trace(lat, link, s, mu, gauge):
    if gauge is None:
        return _trace(link)
    return _trace(_mm(_mm(_dag(gauge[s]), link), gauge[lat.shift(s, mu, 1)]))


def _generator_q(sigma, link):
    omega = _mm(sigma, _dag(link))
    q = (omega - _dag(omega)) / 2
    return q - _eye(q) * (_trace(q) / 3)[:, None, None]


def _maxretr(link, target, hits):
    u = link.clone()
    for _ in range(hits):
        for p, q in ((0, 1), (1, 2), (0, 2)):
            rows = torch.stack([u[:, p], u[:, q]], 1)
            block = rows @ torch.stack([target[:, p], target[:, q]], 1).conj().transpose(1, 2)
            a = (block[:, 0, 0] + block[:, 1, 1].conj()) / 2
            b = (block[:, 0, 1] - block[:, 1, 0].conj()) / 2
            k = (a.abs() ** 2 + b.abs() ** 2).sqrt()
            scale = block.abs().square().sum((1, 2)).sqrt()
            good = k > 1e-6 * scale
            k = torch.where(good, k, 1.0)
            a, b = a / k, b / k
            turn = torch.stack([torch.stack([a.conj(), -b], 1), torch.stack([b.conj(), a], 1)], 1)
            rows = torch.where(good[:, None, None], turn @ rows, rows)
            u[:, p], u[:, q] = rows[:, 0], rows[:, 1]
    return u


def _unit_circle(v):
    x = v
    for _ in range(30):
        x = (x + torch.linalg.inv(x).conj().transpose(1, 2)) / 2
    det = torch.linalg.det(x)
    return x * torch.polar(torch.ones_like(det.real), -torch.angle(det) / 3)[:, None, None]


def _candidate(case, lat, U, s, mu):
    sigma, link = lat.staples(U, s, mu, case["epsilon"]), U[mu][s]
    if case["path"] == "stout" or case["path"] == "serve":
        return _mm(_exp(case["step"] * _generator_q(sigma, link)), link)
    blocked = (1 - case["step"]) * link + (case["step"] / 6) * sigma
    return _maxretr(link, blocked, 3) if case["path"] == "aus" else _unit_circle(blocked)


def _smooth(case, lat, labels, U, gauge):
    for _ in range(case["sweeps"]):
        source = U.clone() if case["schedule"] == "simultaneous" else U
        for mu in range(4):
            for sites in lat.classes(mu):
                for s in sites.split(CHUNK):
                    new = _candidate(case, lat, source, s, mu)
                    if case["preserve"]:
                        keep = _centre_label(_vortex_trace(lat, new, s, mu, gauge)) == labels[mu][s]
                        new = torch.where(keep[:, None, None], new, source[mu][s])
                    U[mu][s] = new
    return U


def _flow(case, lat, U):
    Z = torch.zeros_like(U)
    for _ in range(case["sweeps"]):
        for a, b, c in ((1, 0, 1 / 4), (8 / 9, -17 / 36, 1), (3 / 4, -1, 1)):
            old = U.clone()
            for mu in range(4):
                for s in lat.sites().split(CHUNK):
                    q = _generator_q(lat.staples(old, s, mu, case["epsilon"]), old[mu][s])
                    Z[mu][s] = a * case["step"] * q + b * Z[mu][s]
                    U[mu][s] = _mm(_exp(c * Z[mu][s]), old[mu][s])
    return U


def _action(lat, U):
    total = 0.0
    for mu in range(3):
        for nu in range(mu + 1, 4):
            for s in lat.sites().split(CHUNK):
                total += float((3 - _trace(lat.path(U, s, (mu + 1, nu + 1, -mu - 1, -nu - 1))).real).sum())
    return total / 36 / lat.V


def _observables(lat, U):
    def clover(s, mu, nu):
        m, n = mu + 1, nu + 1
        c = sum(lat.path(U, s, p) for p in ((m, n, -m, -n), (n, -m, -n, m), (-m, -n, m, n), (-n, m, n, -m))) / 4
        f = (c - _dag(c)) / 2j
        return f - _eye(f) * (_trace(f) / 3)[:, None, None]

    sr = charge = 0.0
    for s in lat.sites().split(CHUNK // 4):
        for sign, a, b in ((1, (0, 1), (2, 3)), (-1, (0, 2), (1, 3)), (1, (0, 3), (1, 2))):
            fa, fb = clover(s, *a), clover(s, *b)
            sr += float(_trace(_mm(fa, fa)).real.sum() + _trace(_mm(fb, fb)).real.sum()) / 72
            charge += sign * float(_trace(_mm(fa, fb)).real.sum()) / (4 * math.pi ** 2)
    return dict(mean_S=_action(lat, U), mean_SR=sr / lat.V, Q=charge)


def _min_margin(lat, U, gauge):
    return min(float(_margin(_vortex_trace(lat, U[mu][s], s, mu, gauge)).min())
               for mu in range(4) for s in lat.sites().split(CHUNK))


def exact(case, seed):
    if case["path"] == "serve":
        out = []
        for dims, rho, labels in _jobs(case, seed):
            lat = _Lattice(dims)
            one = dict(case, step=rho, path="stout")
            U = _smooth(one, lat, labels, _centrifuge(lat, labels), None)
            out.append(dict(action=_action(lat, U), n_label_diff=None, status=None))
        return out
    lat, labels, U, gauge = _start(case, seed)
    if case["path"] == "measure":
        o = _observables(lat, U)
        return dict(observables=o, action=o["mean_S"], check=dict(min_margin=_min_margin(lat, U, gauge)), labels=None)
    U = _flow(case, lat, U) if case["path"] == "flow" else _smooth(case, lat, labels, U, gauge)
    out = dict(links=U)
    if case["report"]:
        out["action"] = _action(lat, U)
        out["check"] = dict(min_margin=_min_margin(lat, U, gauge))
    return out
