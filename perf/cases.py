"""The workloads that the library's speed is followed on: what a program calls, at the sizes it calls it.

Inputs are synthetic and made from a seed alone, on the GPU, without the library's kernels: smooth periodic
bands (a few cosines per band, sorted at each k-point) with positive orbital weights normalised over the
orbitals, or the hoppings of a random Hermitian tight-binding model. Energy grids cover the band range with
a margin, as a user lays them. ``exact`` gives the results in 64 bits from the method's formulas, one
tetrahedron at a time, in plain torch.
"""
import math

import numpy as np
import torch

from paper_1710_10789_gb300 import BatchPlan, Plan
from paper_1710_10789_gb300.autograd import model_dos

#: Independent lattice vectors of the tetragonal model: 1st to 3rd in-plane neighbours and +z.
R_VECTORS = ((1, 0, 0), (0, 1, 0), (1, 1, 0), (1, -1, 0), (2, 0, 0), (0, 2, 0), (0, 0, 1))
#: The six tetrahedra of a cube, corner labels at offsets (c & 1, c >> 1 & 1, c >> 2).
TETRAHEDRA = ((0, 1, 2, 5), (1, 2, 3, 5), (0, 2, 4, 5), (2, 3, 5, 7), (2, 4, 5, 6), (2, 5, 6, 7))
DTYPES = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # one-band simple-cubic grid: a small exploratory DOS, where latency and launches count
        dict(name="dos_16_1band", kind="dos", mode="point", n1=16, n2=16, n3=16, bands=1, orbitals=1, energies=401, weights="f32"),
        # the published benchmark's shape: few planes in z, five projected orbitals of eight bands
        dict(name="dos_60x60x10_5orb", kind="dos", mode="point", n1=60, n2=60, n3=10, bands=8, orbitals=5, energies=1024, weights="f32"),
        # the ordinary calculation: 64^3 k-points, orbital-resolved DOS at 2000 energies
        dict(name="dos_64", kind="dos", mode="point", n1=64, n2=64, n3=64, bands=8, orbitals=8, energies=2000, weights="f32"),
        # the largest calculation, whole: eigenvectors of a model at 256^3 k-points and its DOS at 4000 energies
        dict(name="model_256", kind="model", n1=256, n2=256, n3=256, bands=8, orbitals=8, energies=4000, weights="f32"),
        # bin averages with few bins and weights stored in 16 bits, at the largest grid
        dict(name="bins_256_bf16", kind="dos", mode="bin", n1=256, n2=256, n3=256, bands=8, orbitals=8, energies=200, weights="bf16"),
        # occupation as a function of energy
        dict(name="occupation_128", kind="dos", mode="integrated", n1=128, n2=128, n3=128, bands=8, orbitals=8, energies=1000, weights="f32"),
        # Fermi level for a given filling, grid with odd sides
        dict(name="fermi_95x97x96", kind="fermi", n1=95, n2=97, n3=96, bands=8, orbitals=8, weights="f32", filling=0.47),
        # many models of uneven grids and energy counts in one call
        dict(name="batch_64_models", kind="batch", models=64, n_lo=16, n_hi=96, e_lo=500, e_hi=3000, mode="point", bands=8, orbitals=8, weights="f32"),
        # one step of a fit of the hoppings to a target DOS: forward, loss and gradient
        dict(name="fit_64", kind="fit", n1=64, n2=64, n3=64, bands=8, energies=200),
        # bare susceptibility at finite temperature: transition bands and their spectral function
        dict(name="lindhard_64", kind="lindhard", n1=64, n2=64, n3=64, bands=8, energies=400, qx=16, qy=0, qz=0, kT=0.025),
        # bare susceptibility at T = 0, imaginary part
        dict(name="spectral_64", kind="spectral", mode="point", n1=64, n2=64, n3=64, bands=8, energies=400, qx=16, qy=0, qz=0),
        # bare susceptibility at T = 0, real part: every transition reaches every energy
        dict(name="chi0_real_48", kind="chi0", n1=48, n2=48, n3=48, bands=8, energies=400, qx=12, qy=0, qz=0),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["dos", "dos", "dos", "dos", "model", "fermi", "batch", "fit", "lindhard", "spectral", "chi0"])
    c = dict(kind=kind)
    if kind == "batch":
        n_lo = log_int(8, 32)
        e_lo = log_int(64, 800)
        c.update(models=log_int(2, 64), n_lo=n_lo, n_hi=n_lo + rng.randint(4, 48), e_lo=e_lo, e_hi=e_lo + rng.randint(16, 2000),
                 mode=rng.choice(["point", "point", "bin"]), bands=8, orbitals=rng.choice([1, 5, 8]), weights=rng.choice(["f32", "f32", "bf16"]))
        return c
    susceptibility = kind in ("lindhard", "spectral", "chi0")
    hi = {"dos": 160, "model": 160, "fermi": 128, "fit": 72, "lindhard": 72, "spectral": 72, "chi0": 56}[kind]
    n = log_int(12, hi)   # the three sides lie around it
    for a in ("n1", "n2", "n3"):
        c[a] = max(2, min(hi, int(round(n * math.exp(rng.uniform(-0.35, 0.25))))))
    c["bands"] = rng.choice([2, 4, 8, 8]) if susceptibility or kind in ("model", "fit") else rng.choice([1, 3, 4, 7, 8, 8, 8])
    if kind == "fit":
        c["energies"] = log_int(40, 600)
        return c
    if susceptibility:
        c["energies"] = log_int(50, 800 if kind != "chi0" else 400)
        c.update(qx=rng.randint(0, c["n1"] - 1), qy=rng.randint(0, c["n2"] - 1), qz=rng.randint(0, c["n3"] - 1))
        if kind == "lindhard":
            c["kT"] = rng.choice([0.01, 0.025, 0.1])
        if kind == "spectral":
            c["mode"] = rng.choice(["point", "bin"])
        return c
    c["orbitals"] = c["bands"] if kind == "model" or c["bands"] < 8 else rng.choice([1, 5, 8, 8, 8, 16])
    c["weights"] = rng.choice(["f32", "f32", "f16", "bf16"])
    if kind == "fermi":
        c["filling"] = round(rng.uniform(0.1, 0.9), 3)
        return c
    c["energies"] = log_int(64, 4000)
    if kind == "dos":
        c["mode"] = rng.choice(["point", "point", "bin", "integrated"])
        if c["mode"] != "point":
            c["energies"] = min(c["energies"], 1200)
    return c


# ------------------------------------------------------------------ inputs
def _rng(seed):
    return np.random.Generator(np.random.PCG64(int(seed)))


def _smooth(n1, n2, n3, terms):
    """sum of a cos(2 pi m.k + p) over the padded grid (the plane n repeats the plane 0)."""
    dev = torch.device("cuda")
    x = (torch.arange(n1 + 1, device=dev) % n1).float() / n1
    y = ((torch.arange(n2 + 1, device=dev) % n2).float() / n2)[:, None]
    z = ((torch.arange(n3 + 1, device=dev) % n3).float() / n3)[:, None, None]
    acc = torch.zeros((n3 + 1, n2 + 1, n1 + 1), device=dev)
    for a, m, p in terms:
        acc += a * torch.cos(2 * math.pi * (float(m[0]) * x + float(m[1]) * y + float(m[2]) * z) + p)
    return acc


def _bands(rng, n1, n2, n3, bands):
    """Band energies (n3+1, n2+1, n1+1, bands), ascending at each point."""
    e = torch.empty((n3 + 1, n2 + 1, n1 + 1, bands), device="cuda")
    for n in range(bands):
        terms = []
        for _ in range(3):
            m = rng.integers(-2, 3, size=3)
            if not m.any():
                m[0] = 1
            terms.append((float(rng.normal(0.0, 1.2)), m, float(rng.uniform(0, 2 * math.pi))))
        e[..., n] = _smooth(n1, n2, n3, terms) + (-8.0 + 16.0 * (n + 0.5) / bands)
    return e.sort(dim=-1).values


def _weights(rng, n1, n2, n3, bands, orbitals, out):
    """Positive orbital weights of each band, normalised over the orbitals, into out (..., bands * orbitals)."""
    for n in range(bands):
        b = torch.empty((n3 + 1, n2 + 1, n1 + 1, orbitals), device="cuda")
        for s in range(orbitals):
            term = (float(rng.uniform(0.2, 0.9)), rng.integers(-1, 2, size=3), float(rng.uniform(0, 2 * math.pi)))
            b[..., s] = 1.0 + _smooth(n1, n2, n3, [term])
        b /= b.sum(dim=-1, keepdim=True)
        out[..., n * orbitals:(n + 1) * orbitals] = b.to(out.dtype)


def _grid(lo, hi, n):
    return torch.linspace(lo, hi, n, dtype=torch.float64, device="cuda").float()


def _energies(e, case):
    lo, hi = float(e.min()) - 0.1, float(e.max()) + 0.1
    return _grid(lo, hi, case["energies"] + (case["mode"] == "bin"))


def _fields(case, seed, eps=None, w=None):
    """(eps, w, energies) of the padded grid, into the given arrays where there are some."""
    rng = _rng(seed)
    n = case["n1"], case["n2"], case["n3"]
    nb, no = case["bands"], case["orbitals"]
    e = _bands(rng, *n, nb)
    if eps is None:
        eps = torch.empty_like(e)
        w = torch.empty(e.shape[:3] + (nb * no,), dtype=DTYPES[case["weights"]], device="cuda")
    eps[..., :nb] = e
    _weights(rng, *n, nb, no, w)
    return eps, w, _energies(e, case) if "energies" in case else None


def _model(case, seed):
    """Packed parameters of a random tight-binding model and the range of its bands on a coarse grid."""
    rng = _rng(seed)
    n = case["bands"]
    on = rng.uniform(-2.0, 2.0, n)
    t = rng.normal(0.0, 0.3, (2, len(R_VECTORS), n, n))
    params = torch.from_numpy(np.concatenate([on, t.ravel()]).astype(np.float32)).cuda()
    R = torch.tensor(R_VECTORS, dtype=torch.int32, device="cuda")
    ev = np.linalg.eigvalsh(_hamiltonian(params.double(), n, 8, 8, 8).cpu().numpy())
    return params, R, float(ev.min()) - 0.3, float(ev.max()) + 0.3


def _hamiltonian(params, n, n1, n2, n3):
    """H(k) (points, n, n) in 128-bit complex numbers, point x + n1 (y + n2 z)."""
    dev = params.device
    nR = len(R_VECTORS)
    t = torch.complex(*params[n:].reshape(2, nR, n, n))
    z, y, x = torch.meshgrid(*(torch.arange(m, device=dev, dtype=torch.float64) / m for m in (n3, n2, n1)), indexing="ij")
    H = torch.diag(params[:n]).to(t.dtype).expand(n1 * n2 * n3, n, n).clone()
    for r, v in enumerate(R_VECTORS):
        f = torch.exp(2j * math.pi * (v[0] * x + v[1] * y + v[2] * z).reshape(-1, 1, 1))
        H = H + f * t[r] + f.conj() * t[r].conj().T
    return H


def _batch(case, seed):
    rng = _rng(seed * 7919 + 5)
    sizes = _rng(case["models"] * 1000003 + case["n_hi"] * 1009 + case["e_hi"])   # the plan's, the same for every seed
    out = []
    for _ in range(case["models"]):
        n = int(sizes.integers(case["n_lo"], case["n_hi"] + 1))
        out.append((dict(case, n1=n, n2=n, n3=n, energies=int(sizes.integers(case["e_lo"], case["e_hi"] + 1))), int(rng.integers(1 << 30))))
    return out


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case=case)
    if kind == "batch":
        models = _batch(case, seed)
        plan = BatchPlan([(c["n1"], c["n2"], c["n3"]) for c, _ in models], [c["energies"] for c, _ in models], case["bands"],
                         case["orbitals"], mode=case["mode"], weight_dtype=case["weights"])
        data = []
        for m, (c, sd) in enumerate(models):
            eps, w = plan.empty_inputs(m)
            data.append(_fields(c, sd, eps, w))
        s.update(plan=plan, eps=[d[0] for d in data], w=[d[1] for d in data], omega=[d[2] for d in data])
        return s
    n = case["n1"], case["n2"], case["n3"]
    nb = case["bands"]
    if kind in ("model", "fit"):
        params, R, lo, hi = _model(case, seed)
        mode = "point" if kind == "model" else "bin"
        s.update(params=params, R=R, plan=Plan(*n, nb, nb, case["energies"], mode=mode, weight_dtype=case.get("weights", "f32")),
                 omega=_grid(lo, hi, case["energies"] + (mode == "bin")))
        if kind == "fit":
            params.requires_grad_(True)
            s["target"] = _target(seed, nb, s["omega"])
        else:
            s["eps"], s["w"] = s["plan"].empty_inputs()   # a program keeps these between models
        return s
    if kind in ("lindhard", "spectral", "chi0"):
        e, mu, omega = _transitions(case, seed)
        plan = Plan(*n, nb, 1, 64)
        eps, _ = plan.empty_inputs()
        eps[..., :nb] = e
        s.update(plan=plan, eps=eps, mu=mu, omega=omega, q=(case["qx"], case["qy"], case["qz"]))
        if kind == "lindhard":
            s["pair_plan"] = Plan(*n, nb * nb, 1, case["energies"])
        return s
    if kind == "fermi":
        plan = Plan(*n, nb, case["orbitals"], 64, weight_dtype=case["weights"])
    else:
        plan = Plan(*n, nb, case["orbitals"], case["energies"], mode=case["mode"], weight_dtype=case["weights"])
    eps, w, omega = _fields(case, seed, *plan.empty_inputs())
    s.update(plan=plan, eps=eps, w=w, omega=omega)
    return s


def _target(seed, nb, edges):
    """A target DOS: a few Gaussian peaks per orbital, normalised."""
    rng = _rng(seed + 1)
    lo, hi = float(edges[0]), float(edges[-1])
    x = 0.5 * (edges[1:] + edges[:-1])
    out = torch.zeros((nb, x.numel()), device="cuda")
    for s in range(nb):
        for _ in range(4):
            c, d = rng.uniform(lo, hi), rng.uniform(0.05, 0.15) * (hi - lo)
            out[s] += 0.25 / (d * math.sqrt(2 * math.pi)) * torch.exp(-0.5 * ((x - c) / d) ** 2)
    return out


def _transitions(case, seed):
    """Bands, a chemical potential inside them and energies up to 4 eV."""
    e = _bands(_rng(seed), case["n1"], case["n2"], case["n3"], case["bands"])
    mu = float(e[::4, ::4, ::4].flatten().median()) + 0.01
    return e, mu, _grid(0.0, 4.0, case["energies"] + (case.get("mode") == "bin"))


# ------------------------------------------------------------------ one pass
def run(s):
    kind, plan = s["case"]["kind"], s["plan"]
    if kind in ("dos", "batch"):
        return plan.dos(s["eps"], s["w"], s["omega"])
    if kind == "model":
        eps, w = plan.eig(s["params"], s["R"], s["eps"], s["w"])
        return eps, w, plan.dos(eps, w, s["omega"])
    if kind == "fermi":
        return plan.fermi_level(s["eps"], s["w"], s["case"]["filling"] * s["case"]["bands"])
    if kind == "fit":
        dos = model_dos(s["params"], s["R"], s["omega"], plan)
        loss = ((dos - s["target"]) ** 2).sum()
        grad, = torch.autograd.grad(loss, s["params"])
        return dos.detach(), loss.detach(), grad
    if kind == "lindhard":
        eps, w = plan.pair_bands(s["eps"], s["q"], s["case"]["kT"], s["mu"], s["pair_plan"])
        return eps, w, s["pair_plan"].dos(eps, w, s["omega"])
    if kind == "spectral":
        return plan.spectral_t0(s["eps"], s["q"], s["mu"], s["omega"], mode=s["case"]["mode"])
    return plan.chi0_real_t0(s["eps"], s["q"], s["mu"], s["omega"])


def _window(case):
    """Energies inside a tetrahedron, on average: its spread is about 1/N of the band range."""
    return case["energies"] / (case["n1"] * case["n2"] * case["n3"]) ** (1 / 3) + 1


def work(case):
    """Inputs read once and outputs written once; per (tetrahedron, band) 40 operations to sort and set up and,
    per energy inside it, the corner derivatives and the projection (two operations per multiply-add)."""
    if case["kind"] == "batch":
        each = [work(dict(c, kind="dos")) for c, _ in _batch(case, 0)]
        return {k: sum(e[k] for e in each) for k in ("bytes", "flops")}
    kind, nb = case["kind"], case["bands"]
    no = case.get("orbitals", nb if kind == "fit" else 1)
    k = case["n1"] * case["n2"] * case["n3"]
    wb = 2 if case.get("weights") in ("f16", "bf16") else 4
    data = k * nb * (4 + wb * no)
    tet = 6 * k * nb
    eig = k * (2 * len(R_VECTORS) * nb * (nb + 1) * 2 + 2 * (8 / 3 + 3 + 4) * nb ** 3)
    if kind == "fermi":   # the bracket's end: one pass over the bands and weights, and one count
        return {"bytes": data, "flops": tet * (40 + 2 * 24)}
    n_e = case["energies"]
    if kind in ("dos", "model"):
        f = tet * (40 + _window(case) * 2 * (12 + 4 * no))
        return {"bytes": data + 4 * n_e * (no + 1), "flops": f + (eig if kind == "model" else 0)}
    if kind == "fit":   # forward, adjoint (weights and energies) and the adjoint of the eigenvectors
        return {"bytes": 4 * data + 4 * n_e * (2 * no + 1), "flops": 3 * eig + 3 * tet * (40 + _window(case) * 2 * (24 + 4 * no))}
    near = 6 * k * nb * nb * 0.25   # (tetrahedron, band pair) with a transition across the chemical potential in reach
    if kind == "lindhard":
        return {"bytes": k * nb * 4 + 2 * k * nb * nb * 8 + 8 * n_e, "flops": near * (40 + _window(case) * 32)}
    if kind == "spectral":
        return {"bytes": k * nb * 4 + 8 * n_e, "flops": near * (80 + _window(case) * 16)}
    return {"bytes": k * nb * 4 + 8 * n_e, "flops": near * (80 + _window(case) * 40)}


# ------------------------------------------------------------------ results in 64 bits
def _safe(x):
    return torch.where(x > 0, x, torch.ones_like(x))


def _corner_weights(e, E, f):
    """w_l(E) of tetrahedra with sorted corner energies e (m, 4): the integrated weights, full weight f each."""
    e1, e2, e3, e4 = e.unbind(-1)
    d21, d31, d41, d32, d42, d43 = (_safe(a) for a in (e2 - e1, e3 - e1, e4 - e1, e3 - e2, e4 - e2, e4 - e3))
    x, t, c, y = E - e1, E - e2, e3 - E, e4 - E
    C = f * x ** 3 / (d21 * d31 * d41)
    one = (C * (4 - x * (1 / d21 + 1 / d31 + 1 / d41)), C * x / d21, C * x / d31, C * x / d41)
    C1 = f * x * x / (d41 * d31)
    C2 = f * x * t * c / (d41 * d32 * d31)
    C3 = f * t * t * y / (d42 * d32 * d41)
    two = (C1 + (C1 + C2) * c / d31 + (C1 + C2 + C3) * y / d41, C1 + C2 + C3 + (C2 + C3) * c / d32 + C3 * y / d42,
           (C1 + C2) * x / d31 + (C2 + C3) * t / d32, (C1 + C2 + C3) * x / d41 + C3 * t / d42)
    D = f * y ** 3 / (d41 * d42 * d43)
    three = (f - D * y / d41, f - D * y / d42, f - D * y / d43, f - D * (4 - y * (1 / d41 + 1 / d42 + 1 / d43)))
    z = torch.zeros_like(x)
    pick = lambda a, b, g: torch.where(E <= e1, z, torch.where(E >= e4, z + f, torch.where(E <= e2, a, torch.where(E <= e3, b, g))))  # noqa: E731
    return torch.stack([pick(*v) for v in zip(one, two, three)], -1)


def _corner_densities(e, E, f):
    """dw_l/dE of the same: the section's area density times the mean barycentric coordinate over it."""
    e1, e2, e3, e4 = e.unbind(-1)
    d21, d31, d41, d32, d42, d43 = (_safe(a) for a in (e2 - e1, e3 - e1, e4 - e1, e3 - e2, e4 - e2, e4 - e3))
    x, t, y = E - e1, E - e2, e4 - E
    f21, f31, f41, f32, f42 = x / d21, x / d31, x / d41, t / d32, t / d42
    a = f21 * f31
    one = (a * (3 - f21 - f31 - f41), a * f21, a * f31, a * f41)
    f23, f24 = 1 - f32, 1 - f42
    a, b = f23 * f31, f32 * f24
    two = ((1 - f41) * (a + b) + (1 - f31) * a, f23 * (a + b) + f24 * b, f32 * (a + b) + f31 * a, f41 * (a + b) + f42 * b)
    g34, g24, g14 = y / d43, y / d42, y / d41
    b = g34 * g24
    three = (b * g14, b * g24, b * g34, b * (3 - g14 - g24 - g34))
    z = torch.zeros_like(x)
    pick = lambda p, q, r: torch.where((E <= e1) | (E >= e4), z, torch.where(E <= e2, p, torch.where(E <= e3, q, r)))  # noqa: E731
    return torch.stack([4 * f / d41 * pick(*v) for v in zip(one, two, three)], -1)


def _items(eps, w, case, zs):
    """Sorted corner energies (m, 4) and weights (m, 4, orbitals) in 64 bits of the tetrahedra in the planes zs, per tetrahedron."""
    n1, n2, nb = case["n1"], case["n2"], case["bands"]
    for tet in TETRAHEDRA:
        e, b = [], []
        for c in tet:
            at = (slice(zs.start + (c >> 2), zs.stop + (c >> 2)), slice(c >> 1 & 1, n2 + (c >> 1 & 1)), slice(c & 1, n1 + (c & 1)))
            e.append(eps[at][..., :nb].double().reshape(-1))
            b.append(w[at].double().reshape(e[-1].numel(), -1))
        e, at = torch.stack(e, -1).sort(-1)
        yield e, torch.stack(b, 1).gather(1, at[..., None].expand(-1, -1, b[0].shape[1]))


def _planes(case, per_plane):
    step = max(1, int(2.5e6 / per_plane))
    return [range(z, min(case["n3"], z + step)) for z in range(0, case["n3"], step)]


def _exact_dos(eps, w, omega, case):
    """DOS (orbitals, energies) in 64 bits."""
    mode = case["mode"]
    om = omega.double()
    n, no = case["energies"], case.get("orbitals", 1)
    f = 0.25 / (6.0 * case["n1"] * case["n2"] * case["n3"])
    out = torch.zeros((n + 1, no), dtype=torch.float64, device="cuda")
    for zs in _planes(case, case["n1"] * case["n2"] * case["bands"]):
        for e, b in _items(eps, w, case, zs):
            if mode == "bin":   # bins that reach into (e1, e4), and the one that holds a flat tetrahedron
                lo = (torch.searchsorted(om, e[:, 0].contiguous(), right=True) - 1).clamp(0, n)
                hi = torch.maximum(torch.searchsorted(om, e[:, 3].contiguous()), lo + (e[:, 0] >= om[0]).long()).clamp(max=n)
            else:
                lo = torch.searchsorted(om, e[:, 0].contiguous(), right=True)
                hi = torch.searchsorted(om, e[:, 3].contiguous())
            if mode == "integrated":   # full from the first energy at or above e4 (and above e1) on: summed up at the end
                full = (f * b).sum(1)
                at = torch.maximum(hi, lo)
                out.index_add_(0, at, full)
            K = hi - lo
            order = K.argsort(descending=True)
            K, lo, e, b = K[order], lo[order], e[order], b[order]
            counts = torch.bincount(K.clamp(min=0))
            left = (counts.sum() - counts.cumsum(0)).tolist()   # items with more than j energies
            last = None
            for j, m in enumerate(left):
                if m == 0:
                    break
                i = lo[:m] + j
                if mode == "point":
                    d = _corner_densities(e[:m], om[i], f)
                elif mode == "bin":
                    a = _corner_weights(e[:m], om[i], f) if last is None else last[:m]
                    last = _corner_weights(e[:m], om[i + 1], f)
                    d = (last - a) / (om[i + 1] - om[i])[:, None]
                else:   # what the next energy adds to the last one's occupation: differences, summed up at the end
                    d = _corner_weights(e[:m], om[i], f) - (0.0 if last is None else last[:m])
                    last = d + (0.0 if last is None else last[:m])
                v = (d[:, :, None] * b[:m]).sum(1)
                out.index_add_(0, i, v)
                if mode == "integrated":   # taken away again where the full weight comes in
                    ends = K[:m] == j + 1
                    out.index_add_(0, (i + 1)[ends], -(last[ends][:, :, None] * b[:m][ends]).sum(1))
    out = out.cumsum(0) if mode == "integrated" else out
    return out[:n].T.contiguous()


def _exact_fermi(case, seed):
    eps, w, _ = _fields(case, seed)
    target = case["filling"] * case["bands"]
    total = w.double().reshape(w.shape[:3] + (case["bands"], -1)).sum(-1).to(torch.float64)
    one = dict(case, mode="integrated", energies=64, orbitals=1)
    lo, hi = float(eps.min()), float(eps.max())
    while hi - lo > 1e-9 * max(1.0, abs(lo) + abs(hi)):
        om = torch.linspace(lo, hi, 64, dtype=torch.float64, device="cuda")
        n = _exact_dos(eps, total, om, one)[0]
        j = int(torch.searchsorted(n, target).clamp(1, 63))
        lo, hi = float(om[j - 1]), float(om[j])
    return 0.5 * (lo + hi)


def _strides(bands, orbitals, size):
    ws = -(-bands * orbitals * size // 16) * 16 // size
    return -(-bands // 4) * 4, ws + (16 // size if ws * size % 128 == 0 else 0)


def _padded(a, case, stride):
    """Values per grid point (points, m) in the padded layout, the stride's rest zero."""
    n1, n2, n3 = case["n1"], case["n2"], case["n3"]
    a = a.reshape(n3, n2, n1, -1)
    z, y, x = ((torch.arange(n + 1, device=a.device) % n) for n in (n3, n2, n1))
    out = torch.zeros((n3 + 1, n2 + 1, n1 + 1, stride), dtype=a.dtype, device=a.device)
    out[..., :a.shape[-1]] = a[z][:, y][:, :, x]
    return out


def _eigh(H):
    """Eigenvalues and eigenvectors of many small matrices (the library takes a limited batch)."""
    parts = [torch.linalg.eigh(h) for h in H.split(4096)]
    return torch.cat([p[0] for p in parts]), torch.cat([p[1] for p in parts])


def _exact_model(case, seed):
    params, _, lo, hi = _model(case, seed)
    nb = case["bands"]
    e, V = _eigh(_hamiltonian(params.double(), nb, case["n1"], case["n2"], case["n3"]))
    b = V.abs().square().transpose(1, 2).reshape(e.shape[0], -1)
    se, sw = _strides(nb, nb, 4 if case["weights"] == "f32" else 2)
    eps, w = _padded(e, case, se), _padded(b, case, sw)
    return eps, w, _exact_dos(eps, w[..., :nb * nb], _grid(lo, hi, case["energies"]), dict(case, mode="point"))


def _exact_fit(case, seed):
    nb, n1, n2, n3 = case["bands"], case["n1"], case["n2"], case["n3"]
    params, _, lo, hi = _model(case, seed)
    edges = _grid(lo, hi, case["energies"] + 1)
    target = _target(seed, nb, edges).double()
    p = params.double().requires_grad_(True)
    e, V = _eigh(_hamiltonian(p, nb, n1, n2, n3))
    b = V.abs().square().transpose(1, 2).reshape(e.shape[0], -1)
    full = dict(case, mode="bin", orbitals=nb)
    eps, w = _padded(e.detach(), case, nb), _padded(b.detach(), case, nb * nb)
    dos = _exact_dos(eps, w, edges, full)
    g = 2 * (dos - target)
    # dL/d eps and dL/d w: d w_l / d e_r by autograd on the formula, one tetrahedron's corners at a time
    om, f, n = edges.double(), 0.25 / (6.0 * n1 * n2 * n3), case["energies"]
    ge, gw = torch.zeros_like(eps), torch.zeros_like(w).reshape(-1, nb, nb)
    index = torch.arange(eps[..., 0].numel(), device="cuda").reshape(eps.shape[:3])
    for zs in _planes(case, n1 * n2 * nb):
        for tet in TETRAHEDRA:
            at = torch.stack([index[zs.start + (c >> 2):zs.stop + (c >> 2), (c >> 1 & 1):n2 + (c >> 1 & 1), (c & 1):n1 + (c & 1)].reshape(-1) for c in tet], -1)
            ev, order = eps.reshape(-1, nb)[at].transpose(1, 2).reshape(-1, 4).sort(-1)   # (points * bands, 4)
            at = at[:, None, :].expand(-1, nb, -1).reshape(-1, 4).gather(1, order)
            band = torch.arange(nb, device="cuda").repeat(ev.shape[0] // nb)
            bv = w.reshape(-1, nb, nb)[at, band[:, None]]
            i0 = (torch.searchsorted(om, ev[:, 0].contiguous(), right=True) - 1).clamp(0, n)
            i1 = torch.searchsorted(om, ev[:, 3].contiguous()).clamp(max=n)
            K = i1 - i0
            for j in range(int(K.max())):
                m = (K > j).nonzero()[:, 0]
                i = i0[m] + j
                x = ev[m].requires_grad_(True)
                d = (_corner_weights(x, om[i + 1], f) - _corner_weights(x, om[i], f)) / (om[i + 1] - om[i])[:, None]
                gi = g.T[i]
                gx, = torch.autograd.grad((d * (bv[m] * gi[:, None]).sum(-1)).sum(), x)
                ge.view(-1, nb).index_put_((at[m], band[m][:, None].expand(-1, 4)), gx, accumulate=True)
                gw.index_put_((at[m], band[m][:, None].expand(-1, 4)), d.detach()[..., None] * gi[:, None], accumulate=True)
    fold = lambda a: torch.zeros((n1 * n2 * n3, a.shape[-1]), dtype=a.dtype, device="cuda").index_add_(  # noqa: E731
        0, _padded(torch.arange(n1 * n2 * n3, device="cuda")[:, None], case, 1).reshape(-1), a.reshape(-1, a.shape[-1]))
    gp, = torch.autograd.grad([e, b], p, [fold(ge), fold(gw.reshape(-1, nb * nb))])
    return dos, (dos - target).square().sum(), gp


def _shifted(e, case):
    q = [case[k] % case[n] for k, n in (("qx", "n1"), ("qy", "n2"), ("qz", "n3"))]
    return _padded(e[:-1, :-1, :-1].roll((-q[2], -q[1], -q[0]), (0, 1, 2)), case, e.shape[-1])


def _exact_lindhard(case, seed):
    e, mu, omega = _transitions(case, seed)
    nb = case["bands"]
    e = e.double()
    s = _shifted(e, case)
    mu32, kT = float(np.float32(mu)), float(np.float32(case["kT"]))
    f = lambda v: 0.5 * (1 - torch.tanh(0.5 * (v - mu32) / kT))  # noqa: E731
    pe = (s[..., None, :] - e[..., :, None]).flatten(-2)
    pw = (f(e)[..., :, None] - f(s)[..., None, :]).flatten(-2)
    se, sw = _strides(nb * nb, 1, 4)
    eps, w = torch.zeros(e.shape[:3] + (se,), dtype=torch.float64, device="cuda"), torch.zeros(e.shape[:3] + (sw,), dtype=torch.float64, device="cuda")
    eps[..., :nb * nb], w[..., :nb * nb] = pe, pw
    return eps, w, _exact_dos(pe, pw, omega, dict(case, mode="point", bands=nb * nb))


def _cut(V, s):
    """The parts of tetrahedra V (m, 4, fields) where the linear field with corner values s (m, 4) is negative, as tetrahedra."""
    s, order = s.sort(-1)
    V = V.gather(1, order[..., None].expand_as(V))
    k = (s < 0).sum(-1)

    def at(m, i, j):   # where the field vanishes on the edge from corner i to corner j
        t = (s[m, i] / (s[m, i] - s[m, j]))[:, None]
        return V[m, i] + t * (V[m, j] - V[m, i])

    m1, m2, m3 = k == 1, k == 2, k == 3
    a, b, c, d = at(m2, 0, 2), at(m2, 0, 3), at(m2, 1, 2), at(m2, 1, 3)
    p, q, r = at(m3, 0, 3), at(m3, 1, 3), at(m3, 2, 3)
    v = lambda m, i: V[m, i]  # noqa: E731
    parts = [[v(m1, 0), at(m1, 0, 1), at(m1, 0, 2), at(m1, 0, 3)],
             [v(m2, 0), a, b, v(m2, 1)], [a, b, v(m2, 1), c], [b, v(m2, 1), c, d],
             [v(m3, 0), v(m3, 1), v(m3, 2), p], [v(m3, 1), v(m3, 2), p, q], [v(m3, 2), p, q, r]]
    return torch.cat([V[k == 4]] + [torch.stack(t, 1) for t in parts])


def _clipped(case, seed):
    """(sorted transition energies (m, 4), signed volume fractions) of the parts of tetrahedra across the chemical potential."""
    e, mu, _ = _transitions(case, seed)
    mu = float(np.float32(mu))
    nb, n1, n2 = case["bands"], case["n1"], case["n2"]
    A, C = e.double() - mu, _shifted(e.double(), case) - mu
    corner = torch.eye(4, dtype=torch.float64, device="cuda")[:, :3]
    held = []
    for zs in _planes(case, n1 * n2):
        for tet in TETRAHEDRA:
            at = [(slice(zs.start + (c >> 2), zs.stop + (c >> 2)), slice(c >> 1 & 1, n2 + (c >> 1 & 1)), slice(c & 1, n1 + (c & 1))) for c in tet]
            a, c = (torch.stack([F[i].reshape(-1, nb) for i in at], 1) for F in (A, C))
            for i in range(nb):
                for j in range(nb):
                    for sign in (1.0, -1.0):
                        m = ((sign * a[..., i]).amin(1) < 0) & ((sign * c[..., j]).amax(1) > 0)
                        if not bool(m.any()):
                            continue
                        x, y = a[m, :, i], c[m, :, j]
                        V = torch.cat([corner.expand(x.shape[0], 4, 3), x[..., None], y[..., None]], -1)
                        V = _cut(V, sign * V[..., 3])
                        V = _cut(V, -sign * V[..., 4])
                        if V.shape[0]:
                            u, v, x = (V[:, :3, :3] - V[:, 3:, :3]).unbind(1)
                            held.append(((V[..., 4] - V[..., 3]).sort(-1).values, sign * (torch.linalg.cross(u, v) * x).sum(-1).abs()))
                        if sum(h[1].numel() for h in held) > 4e6:
                            yield tuple(torch.cat(h) for h in zip(*held))
                            held.clear()
    if held:
        yield tuple(torch.cat(h) for h in zip(*held))


def _exact_spectral(case, seed):
    _, _, omega = _transitions(case, seed)
    om, n = omega.double(), case["energies"]
    out = torch.zeros(n + 1, dtype=torch.float64, device="cuda")
    vtvg = 1.0 / (6.0 * case["n1"] * case["n2"] * case["n3"])
    for d, amp in _clipped(case, seed):
        if case["mode"] == "point":
            lo, hi = torch.searchsorted(om, d[:, 0].contiguous(), right=True), torch.searchsorted(om, d[:, 3].contiguous())
        else:
            lo = (torch.searchsorted(om, d[:, 0].contiguous(), right=True) - 1).clamp(0, n)
            hi = torch.maximum(torch.searchsorted(om, d[:, 3].contiguous()), lo + (d[:, 0] >= om[0]).long()).clamp(max=n)
        K = hi - lo
        for j in range(max(0, int(K.max()))):
            m = (K > j).nonzero()[:, 0]
            i = lo[m] + j
            if case["mode"] == "point":
                v = _corner_densities(d[m], om[i], 0.25).sum(-1)
            else:
                v = (_corner_weights(d[m], om[i + 1], 0.25) - _corner_weights(d[m], om[i], 0.25)).sum(-1) / (om[i + 1] - om[i])
            out.index_add_(0, i, vtvg * amp[m] * v)
    return out[:n]


def _inverse_average(d, w):
    """Principal-value average of 1/(w - D) over tetrahedra on which D is linear, corner values d (m, 4), w (m,)."""
    d0, d1, d2, d3 = d.unbind(-1)
    d41 = _safe(d3 - d0)
    G1 = torch.where(d2 > d0, 3 * (d1 - d0) / (_safe(d2 - d0) * d41), 0.0)
    G2 = torch.where(d3 > d1, 3 * (d3 - d2) / (_safe(d3 - d1) * d41), 0.0)
    zero = torch.zeros_like(w)
    total = zero
    for b0, b1, b2, a, b in ((zero, zero, G1, d0, d1), (G1, 3 / d41, G2, d1, d2), (G2, zero, zero, d2, d3)):
        h = _safe(b - a)
        s = (w - a) / h
        u = s - 0.5
        la, lb = (torch.where(v == 0, 0.0, v.abs().clamp(min=1e-300).log()) for v in (w - a, w - b))
        p = b0 * (1 - s) ** 2 + 2 * b1 * s * (1 - s) + b2 * s * s
        closed = p * (la - lb) + b0 * (1.5 - s) + b1 * (2 * s - 1) - b2 * (s + 0.5)
        A, B, C = 0.25 * (b0 + 2 * b1 + b2), b2 - b0, b0 - 2 * b1 + b2
        v = 1 / torch.where(u.abs() < 1.5, 1.5, u)
        series = zero
        for j in range(30, -1, -1):
            m = (A * 0.5 ** j / (j + 1) + C * 0.5 ** (j + 2) / (j + 3)) if j % 2 == 0 else B * 0.5 ** (j + 1) / (j + 2)
            series = series * v + m
        total = total + torch.where(b > a, torch.where(u.abs() < 1.5, closed, series * v), 0.0)
    return torch.where(d3 > d0, total, 1 / torch.where(w == d0, math.inf, w - d0))


def _exact_chi0(case, seed):
    _, _, omega = _transitions(case, seed)
    om = omega.double()
    out = torch.zeros_like(om)
    vtvg = 1.0 / (6.0 * case["n1"] * case["n2"] * case["n3"])
    step = max(1, int(8e6 / om.numel()))
    for d, amp in _clipped(case, seed):
        for i in range(0, d.shape[0], step):
            x, a = d[i:i + step], amp[i:i + step]
            c = x.mean(-1)
            far = 4 * (x - c[:, None]).abs().amax(-1)
            u = om[None, :] - c[:, None]
            near = u.abs() <= far[:, None]
            # beyond: the series of the moments about the mean (complete homogeneous polynomials of the corner values)
            top = 24
            h = [torch.ones_like(c)] + [torch.zeros_like(c) for _ in range(top)]
            for k in range(4):
                for n in range(1, top + 1):
                    h[n] = h[n] + (x[:, k] - c) * h[n - 1]
            v = 1 / torch.where(near, math.inf, u)
            r = torch.zeros_like(u)
            for n in range(top, -1, -1):
                r = torch.addcmul((h[n] * (6.0 / ((n + 1) * (n + 2) * (n + 3))))[:, None], r, v)
            r = r * v
            j, k = near.nonzero(as_tuple=True)
            if j.numel():
                r[j, k] = _inverse_average(x[j], om[k])
            out.add_((a[:, None] * r).sum(0), alpha=vtvg)
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        if sum(6 * c["n1"] ** 3 * c["bands"] * (_window(c) + 4) for c, _ in _batch(case, 0)) > 3e9:
            return None
        return [exact(dict(c, kind="dos"), sd) for c, sd in _batch(case, seed)]
    k = case["n1"] * case["n2"] * case["n3"]
    if kind == "dos":
        # (the cost goes with the energies inside the tetrahedra)
        if 6 * k * case["bands"] * (_window(case) + 4) > 6e9:
            return None
        eps, w, omega = _fields(case, seed)
        return _exact_dos(eps, w, omega, case)
    if kind == "fermi":
        return _exact_fermi(case, seed) if k * case["bands"] <= 1e7 else None
    if kind == "model":
        return _exact_model(case, seed) if k <= 64 ** 3 else None
    if kind == "fit":
        return _exact_fit(case, seed) if k <= 72 ** 3 else None
    if kind == "lindhard":
        return _exact_lindhard(case, seed) if k * case["bands"] ** 2 <= 2e7 else None
    if kind == "spectral":
        return _exact_spectral(case, seed) if k * case["bands"] ** 2 <= 2e7 else None
    return _exact_chi0(case, seed) if k * case["bands"] ** 2 * case["energies"] <= 3e9 else None
