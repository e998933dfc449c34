"""The work that users of this library have it do, as measurable cases.

Families (``case["kind"]``):

  grad       the differentiable projector: forward projection, Poisson loss with a smoothness prior,
             and the gradient with respect to the image (float32, or float64 as in derivative checks)
  mlem       a reconstruction by ML-EM from a resident system matrix
  osem       ordered subsets with the dual matrix and an additive scatter estimate
  penalised  the penalised-likelihood solver
  serve      many acquisitions of mixed sizes reconstructed as one batch
  build      photon transport, detection and assembly of a system matrix, and its first use
  forced     the same by forced detection (weighted tallies)
  assemble   a system matrix from tally keys made elsewhere (one acquisition split into parts)

The matrices of the reconstruction families come from synthetic tally keys: history start voxels
uniform over the grid, views uniform, two thirds of the photons detected through the collimator's
blur and one third scattered widely, which gives the row and column structure of a built system at a
density that is chosen by the number of detections.
"""
import math

import numpy as np
import torch

from paper_2105_13324_gb300 import autograd as ag
from paper_2105_13324_gb300 import mcspect as mc
from paper_2105_13324_gb300 import phantoms as ph

FOV_MM = 256.0
ACCEPT = (1.5 / 35.0) ** 2 / 16.0  # collimator acceptance per view of an isotropic photon


def listed():
    return [
        # the smallest call: one gradient of the differentiable projector at the 32^3 workload's size
        dict(name="grad_water32", kind="grad", n=32, views=16, arc=180.0, events=25_000, histories=2_000_000,
             beta=1e-2, dtype="float32"),
        # a small reconstruction that watches its likelihood: 20 iterations, host read of 20 values
        dict(name="mlem_water32", kind="mlem", n=32, views=16, arc=180.0, events=25_000, histories=2_000_000,
             iters=20, values="f32", loglik=True),
        # ordered subsets at the 64^3 torso's size: 8 subsets, dual matrix, additive term, 3 sweeps
        dict(name="osem_torso64", kind="osem", n=64, views=60, arc=180.0, events=400_000, histories=100_000_000,
             iters=3, subsets=8, additive=True),
        # the benchmark's reconstruction: 128^3, 120 views, 10^9 histories' matrix, 50 iterations
        dict(name="mlem_torso128", kind="mlem", n=128, views=120, arc=360.0, events=7_300_000,
             histories=1_000_000_000, iters=50, values="f32", loglik=False),
        # ten times the histories, counts stored in half precision
        dict(name="mlem_torso128_f16", kind="mlem", n=128, views=120, arc=360.0, events=73_000_000,
             histories=10_000_000_000, iters=20, values="f16", loglik=False),
        # a low-noise matrix (rows of ~300 entries), the largest a user keeps
        dict(name="mlem_torso128_dense", kind="mlem", n=128, views=120, arc=360.0, events=600_000_000,
             histories=100_000_000_000, iters=6, values="f32", loglik=False),
        # the penalised solver on the benchmark's matrix
        dict(name="penalised_torso128", kind="penalised", n=128, views=120, arc=360.0, events=7_300_000,
             histories=1_000_000_000, iters=4, beta=1e-2),
        # a serving batch: 64 acquisitions of mixed sizes, 30 iterations each
        dict(name="serve_mixed64", kind="serve", systems=64, iters=30),
        # one-shot build from host inputs at the 32^3 workload's size, the matrix exported
        dict(name="build_water32", kind="build", phantom="water", n=32, views=16, arc=180.0, histories=2_000_000,
             primary=False, oneshot=True),
        # the headline build: 10^9 histories from a resident plan
        dict(name="build_torso128", kind="build", phantom="torso", n=128, views=120, arc=360.0,
             histories=1_000_000_000, primary=False, oneshot=False),
        # a forced-detection build, one history per voxel
        dict(name="forced_torso128", kind="forced", phantom="torso", n=128, views=120, arc=360.0,
             histories=2_097_152, primary=False),
        # a part's matrix from routed tally keys, columns too long for the short-column path
        dict(name="assemble_keys128", kind="assemble", n=128, views=60, arc=360.0, events=73_000_000,
             histories=20_000_000_000),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["grad", "mlem", "mlem", "mlem", "osem", "penalised", "serve", "build", "build", "forced",
                       "assemble"])
    n = rng.randint(24, 128)
    views = rng.randint(8, 120)
    arc = rng.choice([180.0, 360.0])
    c = dict(kind=kind, n=n, views=views, arc=arc)
    # detections in proportion to the grid's and the detector's size, over the densities of use
    scale = (n / 128.0) ** 3 * views / 120.0
    lo, hi = 4e6 * scale + 2e4, 4e8 * scale + 4e4
    if kind == "serve":
        return dict(kind=kind, systems=rng.randint(1, 64), iters=rng.randint(5, 40))
    if kind in ("build", "forced"):
        c["phantom"] = rng.choice(["water", "torso"])
        c["primary"] = rng.random() < 0.25
        if kind == "build":
            c["histories"] = _log(rng, 1e6, 8e8)
            c["oneshot"] = rng.random() < 0.3
        else:
            c["histories"] = _log(rng, 1e4, 2e6)
        return c
    c["events"] = _log(rng, lo, hi)
    c["histories"] = max(n ** 3, int(c["events"] / (views * ACCEPT * 0.53)))
    if kind == "grad":
        c["dtype"] = rng.choice(["float32", "float32", "float64"])
        c["beta"] = 10.0 ** rng.uniform(-4, -1)
    elif kind == "mlem":
        c["iters"] = rng.randint(3, 30)
        c["values"] = rng.choice(["f32", "f32", "f16", "bf16"])
        c["loglik"] = rng.random() < 0.3
    elif kind == "osem":
        c["subsets"] = rng.choice([2, 4, 5, 8])
        c["iters"] = rng.randint(1, 4)
        c["additive"] = rng.random() < 0.5
    elif kind == "penalised":
        c["iters"] = rng.randint(2, 5)
        c["beta"] = 10.0 ** rng.uniform(-4, -1)
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _rows(case):
    return case["views"] * case["n"] * case["n"]


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) % (2 ** 62))
    return g


def _keys(case, gen, count, primary=None):
    """`count` drawn detections (those that miss the detector are left out): keys v * M + j, int64; with
    `primary` a list, also appends which of them are unscattered."""
    n, views = case["n"], case["views"]
    m, h = _rows(case), FOV_MM / case["n"]
    out, step = [], 1 << 26
    for lo in range(0, count, step):
        k = min(step, count - lo)
        f = dict(generator=gen, device="cuda")
        v = torch.randint(0, n ** 3, (k,), dtype=torch.int64, **f)
        view = torch.randint(0, views, (k,), dtype=torch.int64, **f)
        th = view.float() * (math.radians(case["arc"]) / views)
        ct, st = torch.cos(th), torch.sin(th)
        x, y = (v % n).float() + 0.5 - 0.5 * n, (v // n % n).float() + 0.5 - 0.5 * n
        prim = torch.rand(k, **f) < 0.66
        # blur in voxels: intrinsic + collimator at the voxel's distance, or a wide scatter
        dist = 0.75 * n - (x * ct + y * st)
        sig = torch.where(prim, 1.5 / h + 0.011 * dist, 0.12 * n + 0.0 * dist)
        u = torch.floor(y * ct - x * st + sig * torch.randn(k, **f) + 0.5 * n)
        w = torch.floor((v // (n * n)).float() + 0.5 + sig * torch.randn(k, **f))
        ok = (u >= 0) & (u < n) & (w >= 0) & (w < n)
        j = (view * n + w.long()) * n + u.long()
        out.append((v * m + j)[ok])
        if primary is not None:
            primary.append(prim[ok])
        del v, view, th, ct, st, x, y, prim, dist, sig, u, w, ok, j
    return torch.cat(out) if len(out) > 1 else out[0]


def _activity(n, gen):
    """Integer uptake levels of a body, a liver and a heart shell at a drawn place."""
    p = torch.rand(3, generator=gen, device="cuda")
    c = (torch.arange(n, device="cuda", dtype=torch.float32) + 0.5) / n - 0.5
    z, y, x = torch.meshgrid(c, c, c, indexing="ij")
    a = ((x / 0.47) ** 2 + (y / 0.39) ** 2 <= 1).long()
    liver = ((x + 0.2) / 0.22) ** 2 + (y / 0.2) ** 2 + ((z + 0.25) / 0.17) ** 2 <= 1
    a = torch.where(liver & (a > 0), 2 * a, a)
    d = torch.sqrt((x - 0.1 + 0.04 * p[0]) ** 2 + (y - 0.08) ** 2 + (z - 0.05 * p[1]) ** 2)
    return torch.where((d < 0.08 + 0.03 * p[2]) & (d > 0.05) & (a > 0), 8 * a, a).reshape(-1)


def _data(case, gen, total):
    """Poisson counts of an independent realisation, float32 (integer sums, so the same from run to run)."""
    m = _rows(case)
    k = _keys(case, gen, min(case["events"], 20_000_000))
    q = torch.zeros(m, dtype=torch.int64, device="cuda")
    q.index_add_(0, k % m, _activity(case["n"], gen)[k // m])
    lam = q.double() * (total / max(int(q.sum().item()), 1))
    return torch.poisson(lam.float(), generator=gen)


def _total(case):
    return 2e7 * (case["n"] / 128.0) ** 2 * case["views"] / 120.0


def _serve_cases(case):
    rng = np.random.Generator(np.random.Philox(5 + case["systems"]))
    out = []
    for _ in range(case["systems"]):
        n = int((48, 64, 96, 128)[rng.integers(0, 4)])
        views = int(rng.integers(40, 121))
        out.append(dict(n=n, views=views, arc=360.0, histories=20_000_000,
                        events=int(20_000_000 * views * ACCEPT * 0.53), counts=float(10.0 ** rng.uniform(6.0, 7.0))))
    return out


def _phantom(case, seed):
    n, h = case["n"], FOV_MM / case["n"]
    if case["phantom"] == "water":
        r = np.random.Generator(np.random.Philox(int(seed) % (2 ** 62))).uniform(0.16, 0.24)
        p = ph.water_cylinder_phantom(n, h, FOV_MM * r)
    else:
        p = ph.torso_phantom(n, h, seed=int(seed) % (2 ** 31))
    return p, ph.spect_geometry(case["views"], case["arc"], n, h, n, h)


def prepare(case, seed):
    kind = case["kind"]
    gen = _gen(seed)
    st = dict(case=case, seed=int(seed) % (2 ** 32))
    if kind in ("build", "forced"):
        p, g = _phantom(case, seed)
        st.update(phantom=p, geometry=g, x=torch.as_tensor(p.activity.reshape(-1)).cuda(),
                  r=torch.rand(g.n_rows, generator=gen, device="cuda"))
        if not case.get("oneshot", False):
            st["plan"] = mc.mc_plan_create(p, g, primary_only=case["primary"], forced=kind == "forced")
        return st
    if kind == "serve":
        st.update(systems=[], ys=[], xs=[])
        for c in _serve_cases(case):
            st["systems"].append(mc.mc_system_from_keys(_rows(c), c["n"] ** 3, _keys(c, gen, c["events"]), 0,
                                                        c["histories"]))
            st["ys"].append(_data(c, gen, c["counts"]))
            st["xs"].append(torch.empty(c["n"] ** 3, dtype=torch.float32, device="cuda"))
        st["batch"] = mc.mc_batch_create(st["systems"], st["ys"], st["xs"])
        return st
    m, n3 = _rows(case), case["n"] ** 3
    prim = [] if kind == "osem" else None
    keys = _keys(case, gen, case["events"], prim)
    if kind == "assemble":
        st.update(keys=keys, x=torch.rand(n3, generator=gen, device="cuda"),
                  r=torch.rand(m, generator=gen, device="cuda"))
        return st
    st["system"] = mc.mc_system_from_keys(m, n3, keys, 0, case["histories"])
    st["y"] = _data(case, gen, _total(case))
    if kind == "grad":
        dt = getattr(torch, case["dtype"])
        st["x"] = (0.5 + torch.rand(n3, generator=gen, device="cuda")).to(dt)
        st["y"] = st["y"].to(dt)
        st["bg"] = torch.full((m,), 0.05, dtype=dt, device="cuda")
    elif kind == "mlem":
        st["system"].set_value_type(case["values"], allow_rounding=True)
        st["x"] = torch.empty(n3, dtype=torch.float32, device="cuda")
    elif kind == "osem":
        back = mc.mc_system_from_keys(m, n3, keys[torch.cat(prim)].contiguous(), 0, case["histories"])
        rpv, s = case["n"] ** 2, min(case["subsets"], case["views"])
        st["fwd"] = [mc.mc_system_subset(st["system"], rpv, s, k) for k in range(s)]
        st["back"] = [mc.mc_system_subset(back, rpv, s, k) for k in range(s)]
        st["add"] = 0.1 * torch.rand(m, generator=gen, device="cuda") if case["additive"] else None
        st["x"] = torch.empty(n3, dtype=torch.float32, device="cuda")
    return st


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def _matrix_outputs(system, st):
    """The first use of a new matrix: sensitivity, a projection and a back-projection, with its statistics."""
    i = system.info()
    dev = st["r"].device
    s = mc.mc_sensitivity(system, torch.empty(i["n_cols"], dtype=torch.float64, device=dev))
    q = mc.mc_project(system, st["x"], torch.empty(i["n_rows"], dtype=torch.float32, device=dev))
    b = mc.mc_backproject(system, st["r"], torch.empty(i["n_cols"], dtype=torch.float32, device=dev))
    return [s, q, b, np.array([i["nnz"], i["n_events"], i["max_count"]] + i["fates"], dtype=np.int64)]


def run(st):
    case, kind = st["case"], st["case"]["kind"]
    if kind in ("build", "forced"):
        if "plan" in st:
            system = mc.mc_plan_build(st["plan"], 0, case["histories"], st["seed"])
        else:
            system = mc.mc_build_system(st["phantom"], st["geometry"], case["histories"], st["seed"],
                                        primary_only=case["primary"])
        out = _matrix_outputs(system, st)
        if case["n"] <= 32 and kind == "build":  # a small matrix is saved
            col_ptr, _, _, n_v = system.export_csc()
            out += [col_ptr, n_v]
        system.free()
        return out
    if kind == "assemble":
        system = mc.mc_system_from_keys(_rows(case), case["n"] ** 3, st["keys"], 0, case["histories"])
        out = _matrix_outputs(system, st)
        system.free()
        return out
    if kind == "serve":
        mc.mc_batch_mlem(st["batch"], case["iters"])
        return list(st["xs"])
    if kind == "mlem":
        mc.mc_mlem_init(st["system"], st["y"], st["x"])
        ll = mc.mlem_iterate(st["system"], st["y"], st["x"], case["iters"], loglik=case["loglik"])
        return [st["x"], ll] if case["loglik"] else [st["x"]]
    if kind == "osem":
        mc.mc_mlem_init(st["system"], st["y"], st["x"])
        mc.osem_iterate(st["fwd"], st["back"], st["y"], st["x"], case["iters"], add=st["add"])
        return [st["x"]]
    shape = (case["n"],) * 3
    if kind == "penalised":
        hist = []
        x = ag.penalised_reconstruct(st["system"], st["y"], shape, case["beta"] * _mean_sens(case), case["iters"],
                                     history=hist)
        return [x, np.array(hist)]
    x = st["x"].detach().requires_grad_(True)
    q = ag.project(x, st["system"])
    ybar = q + st["bg"]
    loss = (ybar - st["y"] * torch.log(ybar)).sum() + ag.quadratic_prior(x, shape, case["beta"] * _mean_sens(case))
    loss.backward()
    return [q.detach(), x.grad]


def _mean_sens(case):
    return case["events"] / case["histories"]


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    kind = case["kind"]
    if kind == "serve":
        b = f = 0
        for c in _serve_cases(case):
            b += case["iters"] * (16 * c["events"]) + 4 * (_rows(c) + c["n"] ** 3)
            f += case["iters"] * 4 * c["events"]
        return dict(bytes=b, flops=f)
    m, n3 = _rows(case), case["n"] ** 3
    if kind in ("build", "forced"):
        hist = case["histories"]
        prim = 0.6 if case["primary"] else 1.0
        if kind == "build":
            nnz = hist * case["views"] * ACCEPT * 0.53 * prim
            return dict(bytes=int(n3 + 16 * nnz + 4 * (m + n3) + 2 * 8 * nnz), flops=int(482 * hist))
        loc = 1.0 if case["primary"] else 2.0
        nnz = hist * loc * case["views"] * 0.5
        return dict(bytes=int(n3 + 16 * nnz + 4 * (m + n3) + 2 * 8 * nnz), flops=int(650 * hist * loc * case["views"]))
    nnz = case["events"]
    if kind == "assemble":
        return dict(bytes=int(8 * nnz + 16 * nnz + 4 * (m + n3) + 2 * 8 * nnz), flops=int(4 * nnz))
    vecs = 4 * (m + 1) + 4 * (n3 + 1) + 4 * (n3 + 3 * m + 4 * n3)  # pointers, image, data, ratio, normalisers
    if kind == "grad":
        e = 8 if case["dtype"] == "float64" else 4
        return dict(bytes=2 * (4 + 4) * nnz + 4 * (m + n3) + e * (3 * m + 2 * n3), flops=4 * nnz + 10 * m + 14 * n3)
    if kind == "osem":
        s = min(case["subsets"], case["views"])
        return dict(bytes=case["iters"] * (16 * nnz + 4 * (4 * m + 5 * n3 * s)), flops=case["iters"] * 4 * nnz)
    if kind == "penalised":
        return dict(bytes=case["iters"] * (24 * nnz + vecs + 4 * (2 * m + 6 * n3)), flops=case["iters"] * (6 * nnz + 28 * n3))
    v = 4 if case["values"] == "f32" else 2
    return dict(bytes=case["iters"] * (2 * (4 + v) * nnz + vecs), flops=case["iters"] * 4 * nnz)


# ---------------------------------------------------------------------------
# the same results in 64 bits
# ---------------------------------------------------------------------------
class _Ref:
    """A = C diag(1/n_v) from tally keys, in float64."""

    def __init__(self, case, keys, rounded=None):
        self.m, self.n = _rows(case), case["n"] ** 3
        k, c = torch.unique(keys, return_counts=True)
        self.v, self.j = k // self.m, k % self.m
        self.c = c.double() if rounded is None else c.to(rounded).double()
        h = case["histories"]
        self.nv = (h // self.n + (torch.arange(self.n, device="cuda") < h % self.n).long()).double()
        self.has = torch.zeros(self.m, dtype=torch.bool, device="cuda")
        self.has[self.j] = True

    def fwd(self, x, sel=slice(None)):
        xs = torch.where(self.nv > 0, x / self.nv.clamp(min=1), torch.zeros_like(x))
        return torch.zeros(self.m, dtype=torch.float64, device="cuda").index_add_(
            0, self.j[sel], self.c[sel] * xs[self.v[sel]])

    def back(self, r, sel=slice(None)):
        b = torch.zeros(self.n, dtype=torch.float64, device="cuda").index_add_(
            0, self.v[sel], self.c[sel] * r[self.j[sel]])
        return torch.where(self.nv > 0, b / self.nv.clamp(min=1), torch.zeros_like(b))

    def sens(self, sel=slice(None)):
        return self.back(torch.ones(self.m, dtype=torch.float64, device="cuda"), sel)

    def start(self, y):
        s = self.sens()
        return torch.where(s > 0, y.sum() / s.sum(), torch.zeros_like(s))

    def loglik(self, q, y):
        t = torch.where((y > 0) & self.has, y * torch.log(torch.where(self.has, q, torch.ones_like(q))),
                        torch.zeros_like(q))
        return float((t - q).sum())


def _div(a, b):
    return torch.where(b > 0, a / torch.where(b > 0, b, torch.ones_like(b)), torch.zeros_like(a))


def _prior(x, shape, beta):
    g = torch.zeros_like(x).reshape(shape)
    xx, val = x.reshape(shape), 0.0
    for a in range(3):
        d = torch.diff(xx, dim=a)
        val += 0.5 * beta * float((d * d).sum())
        lo = [slice(None)] * 3
        hi = [slice(None)] * 3
        lo[a], hi[a] = slice(0, -1), slice(1, None)
        g[tuple(hi)] += beta * d
        g[tuple(lo)] -= beta * d
    return val, g.reshape(-1)


def _em(a, y, x, iters, lls=None):
    s = a.sens()
    for _ in range(iters):
        q = a.fwd(x)
        if lls is not None:
            lls.append(a.loglik(q, y))
        x = _div(x * a.back(_div(y, q)), s)
    return x


def exact(case, seed):
    kind = case["kind"]
    if kind in ("build", "forced"):
        return None  # sampled by the library's own transport: there is no such value
    gen = _gen(seed)
    if kind == "serve":
        out = []
        for c in _serve_cases(case):
            a = _Ref(c, _keys(c, gen, c["events"]))
            y = _data(c, gen, c["counts"]).double()
            out.append(_em(a, y, a.start(y), case["iters"]))
        return out
    prim = [] if kind == "osem" else None
    keys = _keys(case, gen, case["events"], prim)
    rounded = {"f16": torch.float16, "bf16": torch.bfloat16}.get(case.get("values"))
    a = _Ref(case, keys, rounded)
    m, n3, shape = a.m, a.n, (case["n"],) * 3
    if kind == "assemble":
        x = torch.rand(n3, generator=gen, device="cuda").double()
        r = torch.rand(m, generator=gen, device="cuda").double()
        return [a.sens(), a.fwd(x), a.back(r),
                np.array([a.c.numel(), keys.numel(), int(a.c.max()), 0, 0, 0, 0], dtype=np.int64)]
    y = _data(case, gen, _total(case)).double()
    beta = case.get("beta", 0.0) * _mean_sens(case)
    if kind == "grad":
        x = (0.5 + torch.rand(n3, generator=gen, device="cuda")).double()
        q = a.fwd(x)
        # the backgrounds and weights that the call has in hand are of its own type
        bg = torch.tensor(0.05, dtype=getattr(torch, case["dtype"]), device="cuda").double()
        return [q, a.back(1.0 - y / (q + bg)) + _prior(x, shape, beta)[1]]
    if kind == "mlem":
        lls = [] if case["loglik"] else None
        x = _em(a, y, a.start(y), case["iters"], lls)
        return [x, np.array(lls)] if case["loglik"] else [x]
    if kind == "osem":
        b = _Ref(case, keys[torch.cat(prim)])
        s = min(case["subsets"], case["views"])
        add = 0.1 * torch.rand(m, generator=gen, device="cuda") if case["additive"] else torch.zeros(m, device="cuda")
        add, x, rpv = add.double(), a.start(y), case["n"] ** 2
        fs = [torch.nonzero(a.j // rpv % s == k)[:, 0] for k in range(s)]
        bs = [torch.nonzero(b.j // rpv % s == k)[:, 0] for k in range(s)]
        for _ in range(case["iters"]):
            for k in range(s):
                r = _div(y, a.fwd(x, fs[k]) + add)
                t, w = b.back(r, bs[k]), b.sens(bs[k])
                x = torch.where(w > 0, _div(x * t, w), x)
        return [x]
    # penalised: EM-preconditioned gradient steps, halved until the objective does not increase
    sens, x, hist = a.sens(), a.start(y), []

    def phi(img):
        return -a.loglik(a.fwd(img), y) + _prior(img, shape, beta)[0]

    cur = phi(x)
    for _ in range(case["iters"]):
        grad = sens - a.back(_div(y, a.fwd(x))) + _prior(x, shape, beta)[1]
        t = 1.0
        for _ in range(21):
            xn = torch.where(sens > 0, (x - t * _div(x, sens) * grad).clamp(min=0), torch.zeros_like(x))
            new = phi(xn)
            if new <= cur or t < 2.0 ** -19:
                break
            t *= 0.5
        if new <= cur:
            x, cur = xn, new
        hist.append(cur)
    return [x, np.array(hist)]
