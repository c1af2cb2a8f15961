"""The work that a user of this framework has it do, as cases to be measured.

Every case but two is one run of a simulation through the public calls of
``paper_2405_02410_gb300.pss``: the initial fields are set from device
tensors, the system takes its steps, the final real fields are read back into
device tensors (and, where the workload reports it, the binned structure
factor).  The other two are the ensemble (many instances of uneven sides,
stepped together) and the adjoint (forward run and gradients through
``torch.autograd``).

``exact`` is an independent double-precision statement of the same method in
plain torch: the half spectrum, the Philox4x32-10 noise, the semi-implicit
update, de-aliasing, product terms, boundary frames, S(q) and the gradients.
"""
import math

import numpy as np
import torch

from paper_2405_02410_gb300 import autograd as pss_autograd
from paper_2405_02410_gb300 import pss

DEVICE = "cuda" if torch.cuda.is_available() else "cpu"
NBINS = 64

# half width of the uniform initial field, time step of each model
MODELS = {
    "b": dict(amp=0.1, dt=0.01, fields=1),        # Model B (Cahn-Hilliard with conserved noise)
    "a": dict(amp=0.1, dt=0.01, fields=1),        # Model A (Allen-Cahn)
    "pair": dict(amp=0.05, dt=0.005, fields=2),   # Model A + Model B side by side in one system
    "kpz": dict(amp=0.5, dt=0.01, fields=1),      # KPZ, one gradient-square term
    "coupled": dict(amp=0.1, dt=0.01, fields=2),  # conserved and non-conserved field, product terms
    "bath": dict(amp=0.5, dt=0.5, fields=1),      # heat bath: diffusion between two held ends
}
A, B, K, D = -1.0, 1.0, 1.0, 0.01
FRAME_WIDTH, FRAME_LO, FRAME_HI = 10, 10.0, 0.0


def listed():
    return [
        # 1D: the smallest calls, a line of 1024 sites (Model B), where launches are everything
        dict(name="line_1024_f32", kind="run", model="b", nx=1024, ny=1, nz=1, prec="f32", steps=200, order=2),
        # the heat-bath example of the boundary callbacks: 256 sites between two baths
        dict(name="heat_bath_256_f64", kind="run", model="bath", nx=256, ny=1, nz=1, prec="f64", steps=100, order=2),
        # the 64 x 64 parity workload of Model B, 100 steps
        dict(name="square_64_f32", kind="run", model="b", nx=64, ny=64, nz=1, prec="f32", steps=100, order=2),
        # double precision, as one takes it for reference runs
        dict(name="square_128_f64", kind="run", model="b", nx=128, ny=128, nz=1, prec="f64", steps=50, order=2),
        # the headline workload: 1024 x 1024 Model B with an output (field, S(q)) after a run of steps
        dict(name="square_1024_f32", kind="run", model="b", nx=1024, ny=1024, nz=1, prec="f32", steps=200, order=2,
             sq=True),
        # a channel, longer than wide: two fields
        dict(name="rect_512x128_pair_f32", kind="run", model="pair", nx=512, ny=128, nz=1, prec="f32", steps=50,
             order=2),
        # the 3D workload: Model A + Model B at 256^3
        dict(name="cube_256_pair_f32", kind="run", model="pair", nx=256, ny=256, nz=256, prec="f32", steps=6,
             order=2),
        # a small box with three different sides, double precision
        dict(name="box_64x32x128_f64", kind="run", model="b", nx=64, ny=32, nz=128, prec="f64", steps=20, order=2),
        # the interface-growth workload
        dict(name="kpz_512_f32", kind="run", model="kpz", nx=512, ny=512, nz=1, prec="f32", steps=100, order=2),
        # coupled fields (product terms), the paper's order-3 rule for cubic products
        dict(name="coupled_256_f32", kind="run", model="coupled", nx=256, ny=256, nz=1, prec="f32", steps=20,
             order=3),
        # the ensemble workload: instances of four sides, stepped together, fields and S(q) of each
        dict(name="ensemble_128_f32", kind="ensemble", count=128, lo=64, hi=512, prec="f32", steps=200),
        # the adjoint workload: gradients of an S(q) loss with respect to a, b, K, D and the initial field
        dict(name="adjoint_256_f32", kind="adjoint", nx=256, ny=256, nz=1, prec="f32", steps=400),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _side(rng, lo, hi):
    """A power of two (the lattice sides the library takes) in [lo, hi]."""
    return 1 << rng.randint(int(math.log2(lo)), int(math.log2(hi)))


def draw(rng):
    """One more case of the same ranges: 1D lines of 64..1024 sites, 2D lattices of 32..1024 by
    32..1024, 3D boxes of 16..256 a side, ensembles and adjoint runs."""
    kind = rng.choice(["line", "line", "plane", "plane", "plane", "box", "box", "ensemble", "adjoint", "coupled"])
    prec = rng.choice(["f32", "f32", "f64"])
    order = rng.choice([2, 2, 2, 3])
    if kind == "ensemble":
        hi = _side(rng, 64, 512)
        lo = _side(rng, 64, hi)
        return dict(kind="ensemble", count=_log_int(rng, 4, 100), lo=lo, hi=hi, prec="f32", steps=_log_int(rng, 20, 200))
    if kind == "adjoint":
        nx, ny = _side(rng, 64, 256), _side(rng, 64, 256)
        return dict(kind="adjoint", nx=nx, ny=ny, nz=1, prec="f32", steps=_log_int(rng, 20, 400))
    if kind == "line":
        return dict(kind="run", model=rng.choice(["b", "a", "kpz", "bath"]), nx=_side(rng, 64, 1024), ny=1, nz=1,
                    prec=prec, steps=_log_int(rng, 20, 200), order=order)
    if kind == "coupled":
        return dict(kind="run", model="coupled", nx=_side(rng, 32, 512), ny=_side(rng, 32, 512), nz=1, prec=prec,
                    steps=_log_int(rng, 10, 50), order=order)
    if kind == "plane":
        return dict(kind="run", model=rng.choice(["b", "b", "pair", "a", "kpz"]), nx=_side(rng, 32, 1024),
                    ny=_side(rng, 32, 1024), nz=1, prec=prec, steps=_log_int(rng, 20, 200), order=order)
    sides = [_side(rng, 16, 256) for _ in range(3)]
    while sides[0] * sides[1] * sides[2] > (1 << 22):   # at most a quarter of the largest listed lattice
        sides = [_side(rng, 16, 256) for _ in range(3)]
    return dict(kind="run", model=rng.choice(["b", "pair", "a"]), nx=sides[0], ny=sides[1], nz=sides[2], prec=prec,
                steps=_log_int(rng, 4, 30), order=order)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _shape(case):
    return tuple(n for n in (case["nz"], case["ny"], case["nx"]) if n > 1)


def _philox_seed(seed):
    return (int(seed) * 0x9E3779B1 + 12345) & 0xFFFFFFFFFFFF


def _initial(case, seed):
    """The initial real fields, one tensor per field: uniform around the model's mean."""
    m = MODELS[case["model"]]
    g = np.random.default_rng([int(seed), 1])
    mean = 5.0 if case["model"] == "bath" else 0.0
    out = []
    for _ in range(m["fields"]):
        u = g.random(_shape(case), dtype=np.float64 if case["prec"] == "f64" else np.float32)
        out.append(torch.from_numpy(mean + m["amp"] * (2 * u - 1)).to(DEVICE))
    return out


def _instances(case, seed):
    """Sides, noise seeds and coefficients a of an ensemble's instances, in increasing side."""
    g = np.random.default_rng([int(seed), 2])
    n = int(math.log2(case["hi"] // case["lo"])) + 1
    sides = [case["lo"] << i for i in range(n)]
    side = sorted(sides[i % n] for i in range(case["count"]))   # an equal share of every side
    a = g.uniform(-1.5, -0.5, size=case["count"])
    return [(int(side[i]), _philox_seed(seed) + i, float(a[i])) for i in range(case["count"])]


def _instance_fields(case, seed):
    """{side: initial fields of its instances, stacked}."""
    out = {}
    inst = _instances(case, seed)
    for side in sorted({s for s, _, _ in inst}):
        n = sum(1 for s, _, _ in inst if s == side)
        g = np.random.default_rng([int(seed), 3, side])
        u = g.random((n, side, side), dtype=np.float32)
        out[side] = torch.from_numpy(0.1 * (2 * u - 1)).to(DEVICE)
    return out


def _adjoint_inputs(case, seed):
    g = np.random.default_rng([int(seed), 4])
    phi = torch.from_numpy(0.1 * (2 * g.random(_shape(case)) - 1)).to(DEVICE)
    h0 = torch.fft.rfftn(phi).to(torch.complex64 if case["prec"] == "f32" else torch.complex128)
    target = torch.from_numpy(0.002 * (1 + g.random(NBINS))).to(DEVICE)
    rd = torch.float32 if case["prec"] == "f32" else torch.float64
    params = torch.tensor([-1.0 + 0.2 * g.random(), 1.0 + 0.2 * g.random(), 1.0 - 0.1 * g.random(), 0.01], dtype=rd,
                          device=DEVICE)
    return h0, params, target


def _build(case, seed):
    m = MODELS[case["model"]]
    s = pss.System(_shape(case), dt=m["dt"], seed=_philox_seed(seed), precision=case["prec"])
    model, order = case["model"], case["order"]
    if model == "b":
        pss.add_model_b_field(s, a=A, b=B, K=K, D=D, dealias_order=order)
    elif model == "a":
        pss.add_model_a_field(s, a=A, b=B, K=K, D=D, dealias_order=order)
    elif model == "pair":
        pss.add_model_a_field(s, a=A, b=B, K=K, D=0.05, dealias_order=order, name="psi")
        pss.add_model_b_field(s, a=A, b=B, K=K, D=0.05, dealias_order=order, name="phi")
    elif model == "kpz":
        pss.add_kpz_field(s, sigma=1.0, lam=0.5, D=D, dealias_order=order)
    elif model == "bath":
        f = s.add_field("T")
        s.add_term(f, True, [(-1, 1.0, 1)], [(f, 1)])
        s.set_frame(f, FRAME_WIDTH, FRAME_LO, FRAME_HI)
    else:   # coupled: dt phi + (a q^2 + K q^4) phi = -b q^2 F[phi^3] - g q^2 F[phi psi^2]; dt psi + (c + q^2) psi = -h F[phi^2 psi]
        f0, f1 = s.add_field("phi"), s.add_field("psi")
        p = {k: s.add_param(k, v) for k, v in (("a", A), ("K", K), ("b", B), ("g", 0.5), ("c", 0.3), ("L", 1.0),
                                              ("h", 0.7), ("D0", D), ("D1", D))}
        s.add_term(f0, True, [(p["a"], 1.0, 1), (p["K"], 1.0, 2)], [(f0, 1)])
        s.add_term(f0, False, [(p["b"], -1.0, 1)], [(f0, 3)])
        s.add_product_term(f0, [(p["g"], -1.0, 1)], [(f0, 1), (f1, 2)])
        s.add_term(f1, True, [(p["c"], 1.0, 0), (p["L"], 1.0, 1)], [(f1, 1)])
        s.add_product_term(f1, [(p["h"], -1.0, 0)], [(f0, 2), (f1, 1)])
        s.set_noise(f0, p["D0"], 1)
        s.set_noise(f1, p["D1"], 0)
        for f in (f0, f1):
            s.set_dealias(f, order)
    return s


def prepare(case, seed):
    if case["kind"] == "ensemble":
        fields = _instance_fields(case, seed)
        inst = _instances(case, seed)
        groups = []
        for side, phi0 in fields.items():
            mine = [(sd, a) for s, sd, a in inst if s == side]
            s = pss.System((side, side), dt=0.01, batch=len(mine), seeds=[sd for sd, _ in mine], precision=case["prec"])
            pss.add_model_b_field(s, a=A, b=B, K=K, D=D)
            s.set_param_batch(0, np.array([a for _, a in mine]))
            groups.append((s, phi0, torch.empty_like(phi0)))
        return dict(case=case, groups=groups)
    if case["kind"] == "adjoint":
        h0, params, target = _adjoint_inputs(case, seed)
        s = pss.model_b(_shape(case), dt=0.01, a=A, b=B, K=K, D=D, seed=_philox_seed(seed), precision=case["prec"])
        return dict(case=case, system=s, h0=h0, params=params, target=target)
    phi0 = _initial(case, seed)
    return dict(case=case, system=_build(case, seed), phi0=phi0, out=[torch.empty_like(x) for x in phi0])


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(state):
    case = state["case"]
    if case["kind"] == "ensemble":
        for s, phi0, _ in state["groups"]:
            s.set_step(0)
            for j in range(s.batch):
                s.select_instance(j)
                s.set_field(0, phi0[j])
        pss.step_many([s for s, _, _ in state["groups"]], case["steps"])
        fields, sq = [], []
        for s, _, out in state["groups"]:
            for j in range(s.batch):
                s.select_instance(j)
                s.get_field(0, out=out[j])
                sq.append(s.structure_factor(0, NBINS)[0])
            fields.append(out)
        return dict(fields=fields, sq=np.asarray(sq, dtype=np.float32))   # kept in the precision of the run
    if case["kind"] == "adjoint":
        h0 = state["h0"].detach().requires_grad_(True)
        params = state["params"].detach().requires_grad_(True)
        hT = pss_autograd.run(h0, params, state["system"], (0, 1, 2, 3), case["steps"])
        S, _ = pss_autograd.binned_structure_factor(hT, _shape(case), NBINS)
        ((S - state["target"]) ** 2).mean().backward()
        return dict(hT=hT.detach(), dh0=h0.grad, dparams=params.grad)
    s = state["system"]
    s.set_step(0)
    for f, x in enumerate(state["phi0"]):
        s.set_field(f, x)
    s.step(case["steps"])
    res = dict(fields=[s.get_field(f, out=x) for f, x in enumerate(state["out"])])
    if case.get("sq"):
        res["sq"] = s.structure_factor(0, NBINS)[0].astype(np.float32)   # kept in the precision of the run
    return res


def _flops(sites, steps, transforms, modes_noise):
    """Real transforms of `sites` points (5/2 n log2 n each), and per mode about 60 operations of noise and update."""
    return steps * (transforms * 2.5 * sites * math.log2(max(2, sites)) + 60.0 * modes_noise + 4.0 * sites)


def work(case):
    """Initial fields read and results written once.  A state larger than the chip's memory (the
    129 MB L2) also crosses to HBM and back every step; a smaller one need not."""
    size = 8 if case["prec"] == "f64" else 4
    if case["kind"] == "ensemble":
        inst = _instances(case, 0)
        sites = sum(s * s for s, _, _ in inst)
        flops = sum(_flops(s * s, case["steps"], 2, s * s / 2) for s, _, _ in inst)
        state = sites * size
        return dict(bytes=2 * state * (case["steps"] if state > 129e6 else 1), flops=flops)
    sites = case["nx"] * case["ny"] * case["nz"]
    if case["kind"] == "adjoint":
        # forward, recomputed forward, and per adjoint step four transforms more
        return dict(bytes=4 * sites * size, flops=2 * _flops(sites, case["steps"], 2, sites / 2) +
                    _flops(sites, case["steps"], 4, sites / 2))
    m = MODELS[case["model"]]
    dim = len(_shape(case))
    transforms = {"kpz": dim + 1, "coupled": 5, "bath": 2}.get(case["model"], 2 * m["fields"])
    noise = 0 if case["model"] == "bath" else m["fields"] * sites / 2
    state = sites * size * m["fields"]
    return dict(bytes=2 * state * (case["steps"] if state > 129e6 else 1), flops=_flops(sites, case["steps"], transforms, noise))


# ---------------------------------------------------------------------------
# the method in double precision, in plain torch
# ---------------------------------------------------------------------------
_MASK = 0xFFFFFFFF


def _philox(c0, c1, c2, c3, k0, k1):
    """Philox4x32-10 on int64 tensors holding 32-bit words (64-bit products wrap modulo 2^64)."""
    x, y, z, w = c0, torch.full_like(c0, c1), torch.full_like(c0, c2), torch.full_like(c0, c3)
    for _ in range(10):
        pa, pb = 0xD2511F53 * x, 0xCD9E8D57 * z
        x, y, z, w = ((pb >> 32) & _MASK) ^ y ^ k0, pb & _MASK, ((pa >> 32) & _MASK) ^ w ^ k1, pa & _MASK
        k0, k1 = (k0 + 0x9E3779B9) & _MASK, (k1 + 0xBB67AE85) & _MASK
    return x, y, z, w


class _Lattice:
    """Wave numbers, masks and noise of a batch of half spectra [batch, (nz,) (ny,) nx/2+1]."""

    def __init__(self, shape, seeds):
        self.shape, self.dim = tuple(shape), len(shape)
        self.n = int(np.prod(shape))
        nx = shape[-1]
        self.axes = tuple(range(1, self.dim + 1))
        ks = [torch.from_numpy(np.fft.fftfreq(m) * m) for m in shape[:-1]] + [torch.arange(nx // 2 + 1, dtype=torch.float64)]
        grids = torch.meshgrid(*[k.to(DEVICE).double() for k in ks], indexing="ij")
        self.k = grids                                            # slowest axis first
        self.q = [2 * math.pi * g / m for g, m in zip(grids, shape)]
        self.q2 = sum(q * q for q in self.q)
        # noise counters: each Hermitian pair is drawn by its member of the smaller half-spectrum index
        idx = torch.meshgrid(*[torch.arange(m, device=DEVICE) for m in shape[:-1]],
                             torch.arange(nx // 2 + 1, device=DEVICE), indexing="ij")
        kx = idx[-1]
        row = torch.zeros_like(kx)
        prow = torch.zeros_like(kx)
        for m, i in zip(shape[:-1], idx[:-1]):
            row = row * m + i
            prow = prow * m + (m - i) % m
        plane = (kx == 0) | (2 * kx == nx)
        self.conj = plane & (prow < row)
        self.selfc = plane & (prow == row)
        crow = torch.where(self.conj, prow, row)
        hxe = (nx // 2 + 1) + ((nx // 2 + 1) & 1)
        self.counter = ((crow * hxe + kx) >> 1).unsqueeze(0).expand(len(seeds), *kx.shape).contiguous()
        self.odd = (kx & 1) == 1
        one = [len(seeds)] + [1] * self.dim
        self.k0 = torch.tensor([s & _MASK for s in seeds], device=DEVICE).reshape(one)
        self.k1 = torch.tensor([(s >> 32) & _MASK for s in seeds], device=DEVICE).reshape(one)

    def noise(self, step, field, power):
        """xi_q / sqrt(D) of a step, per unit sqrt(dt): standard deviation sqrt(sites) |q|^power a component."""
        x, y, z, w = _philox(self.counter, step, field, 0, self.k0, self.k1)
        u0 = ((torch.where(self.odd, z, x) >> 8).double() + 0.5) / 2.0 ** 24
        u1 = ((torch.where(self.odd, w, y) >> 8).double() + 0.5) / 2.0 ** 24
        r = torch.sqrt(-2.0 * torch.log(u0)) * math.sqrt(self.n) * self.q2 ** (0.5 * power)
        re = torch.where(self.selfc, math.sqrt(2.0) * r * torch.cos(2 * math.pi * u1), r * torch.cos(2 * math.pi * u1))
        im = torch.where(self.selfc, torch.zeros_like(r), r * torch.sin(2 * math.pi * u1))
        return torch.complex(re, torch.where(self.conj, -im, im))

    def mask(self, order):
        keep = torch.ones_like(self.q2)
        for g, m in zip(self.k, self.shape):
            keep = keep * ((order + 1) * g.abs() < m if order > 0 else torch.ones_like(keep)).double()
        return keep

    def deriv(self, axis):
        """i q along axis (0 = x), zero at a Nyquist index."""
        g, m = self.k[self.dim - 1 - axis], self.shape[self.dim - 1 - axis]
        q = torch.where(2 * g.abs() == m, torch.zeros_like(g), self.q[self.dim - 1 - axis])
        return torch.complex(torch.zeros_like(q), q)

    def forward(self, r):
        return torch.fft.rfftn(r, dim=self.axes)

    def back(self, h):
        return torch.fft.irfftn(h, s=self.shape, dim=self.axes)

    def hermitian(self, h):
        """The part of a half spectrum that belongs to a real field."""
        out = h.clone()
        for col in (0, self.shape[-1] // 2):
            p = h[..., col]
            m = p
            for ax in range(1, self.dim):
                m = torch.roll(torch.flip(m, (ax,)), 1, ax)
            out[..., col] = 0.5 * (p + m.conj())
        return out


def _equations(model, lat, order):
    """Per field: (implicit operator, noise D or None, noise power), and the explicit part of all fields."""
    q2, m = lat.q2, lat.mask(order)
    if model in ("b", "a", "pair"):
        d = 0.05 if model == "pair" else D
        kinds = {"b": ["b"], "a": ["a"], "pair": ["a", "b"]}[model]
        lhs = [(A + K * q2, d, 0) if k == "a" else (A * q2 + K * q2 * q2, d, 1) for k in kinds]

        def rhs(h):
            return [(-B if k == "a" else -B * q2) * lat.forward(lat.back(m * x) ** 3) for k, x in zip(kinds, h)]
    elif model == "kpz":
        lhs = [(q2, D, 0)]

        def rhs(h):
            g2 = sum(lat.back(lat.deriv(j) * m * h[0]) ** 2 for j in range(lat.dim))
            return [0.5 * lat.forward(g2)]
    elif model == "bath":
        lhs = [(q2, None, 0)]

        def rhs(h):
            return [0.0]
    else:
        lhs = [(A * q2 + K * q2 * q2, D, 1), (0.3 + q2, D, 0)]

        def rhs(h):
            p, s = (lat.back(m * x) for x in h)
            return [-B * q2 * lat.forward(p ** 3) - 0.5 * q2 * lat.forward(p * s * s), -0.7 * lat.forward(p * p * s)]
    return lhs, rhs


def _structure_factor(lat, h):
    """Bin means of |phi_q|^2 / sites over 0 < |q| <= pi, one row per half spectrum of the batch."""
    s = torch.sqrt(sum((2.0 * NBINS * g / m) ** 2 for g, m in zip(lat.k, lat.shape)))
    valid = (s > 0) & (s <= NBINS)
    kx = lat.k[-1]
    w = (2.0 - ((kx == 0) | (2 * kx == lat.shape[-1])).double()) * valid.double()
    b = torch.where(valid, torch.ceil(s).long() - 1, torch.zeros_like(s, dtype=torch.long)).reshape(-1)
    cnt = torch.zeros(NBINS, dtype=torch.float64, device=h.device).index_add(0, b, w.reshape(-1))
    p = ((h.real ** 2 + h.imag ** 2) * w / lat.n).reshape(h.shape[0], -1)
    return torch.zeros(h.shape[0], NBINS, dtype=torch.float64, device=h.device).index_add(1, b, p) / cnt.clamp(min=1)


def exact(case, seed):
    if case["kind"] == "ensemble":
        inst = _instances(case, seed)
        fields, sq = [], []
        for side, phi0 in _instance_fields(case, seed).items():
            mine = [(sd, a) for s, sd, a in inst if s == side]
            lat = _Lattice((side, side), [sd for sd, _ in mine])
            a = torch.tensor([x for _, x in mine], dtype=torch.float64, device=DEVICE).reshape(-1, 1, 1)
            m, q2 = lat.mask(2), lat.q2
            h = lat.forward(phi0.double())
            for n in range(case["steps"]):
                P = -q2 * lat.forward(lat.back(m * h) ** 3)
                h = lat.hermitian((h + 0.01 * P + math.sqrt(0.01 * D) * lat.noise(n, 0, 1)) / (1 + 0.01 * (a * q2 + q2 * q2)))
            fields.append(lat.back(h))
            sq.append(_structure_factor(lat, h))
        return dict(fields=fields, sq=torch.cat(sq))
    lat = _Lattice(_shape(case), [_philox_seed(seed)])
    if case["kind"] == "adjoint":
        h0, params, target = _adjoint_inputs(case, seed)
        h0 = h0.to(torch.complex128).unsqueeze(0).requires_grad_(True)
        # the library takes the parameters as doubles made from these values
        p = params.double().detach().requires_grad_(True)
        m, q2 = lat.mask(2), lat.q2
        g = 1 / (1 + 0.01 * (p[0] * q2 + p[2] * q2 * q2))
        h = h0
        for n in range(case["steps"]):
            P = -p[1] * q2 * lat.forward(lat.back(m * h) ** 3)
            h = lat.hermitian(g * (h + 0.01 * P + torch.sqrt(0.01 * p[3]) * lat.noise(n, 0, 1)))
        S = _structure_factor(lat, h)[0]
        ((S - target) ** 2).mean().backward()
        return dict(hT=h.detach()[0], dh0=h0.grad[0], dparams=p.grad)
    model, dt = case["model"], MODELS[case["model"]]["dt"]
    lhs, rhs = _equations(model, lat, case["order"])
    h = [lat.forward(x.double().unsqueeze(0)) for x in _initial(case, seed)]
    for n in range(case["steps"]):
        N = rhs(h)
        new = []
        for f, (O, d, power) in enumerate(lhs):
            xi = math.sqrt(dt * d) * lat.noise(n, f, power) if d is not None else 0.0
            new.append(lat.hermitian((h[f] + dt * N[f] + xi) / (1 + dt * O)))
        if model == "bath":
            r = lat.back(new[0])
            r[..., :FRAME_WIDTH] = FRAME_LO
            r[..., -FRAME_WIDTH:] = FRAME_HI
            new = [lat.forward(r)]
        h = new
    res = dict(fields=[lat.back(x)[0] for x in h])
    if case.get("sq"):
        res["sq"] = _structure_factor(lat, h[0])[0]
    return res
