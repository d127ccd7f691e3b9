"""The work a user has this library do, as measurable cases.

Each case is one pass through the public entry points: a live lattice advanced
some steps and read back (`Simulation`), a window from given fields
(init, step, read), a batch of ragged columns through the C ABI, one call of
the learned surrogate, one training sample, one BF16 product.  Sizes are the
workloads' own (lbm_inputs.py, bench.py, the tests) and ragged ones of the
same range.

Outputs are kept in the type of the run's arithmetic: FP64 lattices return
their FP64 fields, float and half stores return the fields as float32 (what a
run of that precision is worth keeping), the BF16 surrogate its increment and
gradients as bfloat16.
"""
import ctypes
import math
import random

import numpy as np
import torch

import paper_2409_10399_gb300 as lbm

DEV = "cuda" if torch.cuda.is_available() else "cpu"
FIELDS = ("alpha_g", "u_g", "u_l", "p_k")
D_OF = {"D1Q3": 1, "D2Q9": 2, "D3Q19": 3}
Q_OF = {1: 3, 2: 9, 3: 19}
# bytes per direction and node of the six schemes together; of a held value
DIR_BYTES = {"fp64": 48, "fp32": 24, "fp16ab": 16, "fp16dev": 12}
HELD_BYTES = {"fp64": 8, "fp32": 4, "fp16ab": 4, "fp16dev": 4}
# arithmetic operations of one node update as the method's formulas count them
NODE_FLOPS = {1: 450, 2: 1200, 3: 2700}
L2_BYTES = 126e6
CIN = COUT = 16


# ----------------------------------------------------------------- the cases

def listed():
    return [
        # the 1D gas-liquid column (512 nodes, FP64, lag latch every 200
        # steps): the smallest lattice, 10,000 steps in use, nothing but the
        # latency of a step
        dict(name="column1d_fp64", kind="run", recipe="column1d", nx=512, ny=1, nz=1, precision="fp64", steps=200),
        # the paper's open tube (TEST #1, 200 nodes, inlet and outlet, ramped
        # inlet values, so every step's arguments differ): 6e6 steps in use
        dict(name="tube1d_fp64", kind="run", recipe="tube1d", nx=200, ny=1, nz=1, precision="fp64", steps=200),
        # the 2D bubble-column box, the benchmark: FP32, bottom inlet strip,
        # a snapshot every 64 steps
        dict(name="box2d_fp32", kind="run", recipe="box2d", nx=512, ny=2048, nz=1, precision="fp32", steps=64),
        # the same box in the mixed store (momenta in float, the rest in half)
        dict(name="box2d_fp16ab", kind="run", recipe="box2d", nx=512, ny=2048, nz=1, precision="fp16ab", steps=64),
        # the accuracy reference every form is judged against, on a box of
        # ragged sides
        dict(name="box2d_fp64", kind="run", recipe="box2d", nx=500, ny=1030, nz=1, precision="fp64", steps=20),
        # the 3D column at its full size in the half store: the largest lattice
        dict(name="column3d_fp16", kind="run", recipe="column3d", nx=256, ny=256, nz=512, precision="fp16dev", steps=16),
        # a 3D column of ragged sides in FP32
        dict(name="column3d_fp32", kind="run", recipe="column3d", nx=150, ny=122, nz=250, precision="fp32", steps=16),
        # the parameter sweep: ragged 2D columns (nx 64..512, ny = 4 nx), each
        # with its own density ratio and drag, advanced together
        dict(name="batch_fp32", kind="batch", columns=48, sweep=4, lo=64, hi=512, precision="fp32", steps=100),
        # the surrogate's training data: a 256 x 1024 box restarted from
        # device fields and advanced one 64-step window
        dict(name="window2d_fp32", kind="window", recipe="plume2d", nx=256, ny=1024, nz=1, precision="fp32", steps=64),
        # one call of the learned surrogate: 64 steps' worth
        dict(name="surrogate_advance", kind="advance", nx=256, ny=1024, channels=64, modes=32, layers=4),
        # one training sample of it: forward and backward, the gradients out
        dict(name="surrogate_train", kind="train", nx=256, ny=1024, channels=64, modes=32, layers=4),
        # the surrogate's channel mixing as a product of its own
        dict(name="product_pointwise", kind="product", m=64, n=262144, k=64, ta=False, tb=False, out="f32"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("1d", "2d", "2d", "3d", "3d", "batch", "window", "advance", "train", "product"))
    if kind == "1d":
        recipe = rng.choice(("column1d", "tube1d"))
        return dict(kind="run", recipe=recipe, nx=_log(rng, 64, 4096), ny=1, nz=1,
                    precision=rng.choice(("fp64", "fp32")), steps=rng.randrange(50, 201))
    if kind in ("2d", "window"):
        precision = "fp32" if kind == "window" else rng.choice(("fp32", "fp32", "fp16ab", "fp16dev", "fp64"))
        nx = _log(rng, 48, 512)
        ny = _log(rng, 96, 2048)
        if precision == "fp64":
            ny = min(ny, 500000 // nx)
        steps = rng.randrange(10, 21) if precision == "fp64" else rng.randrange(16, 65)
        return dict(kind="window" if kind == "window" else "run", recipe=rng.choice(("box2d", "plume2d")), nx=nx, ny=ny,
                    nz=1, precision=precision, steps=steps)
    if kind == "3d":
        return dict(kind="run", recipe="column3d", nx=_log(rng, 30, 256), ny=_log(rng, 30, 256), nz=_log(rng, 32, 256),
                    precision=rng.choice(("fp32", "fp16dev", "fp16ab")), steps=rng.randrange(8, 17))
    if kind == "batch":
        return dict(kind="batch", columns=_log(rng, 4, 48), sweep=rng.randrange(1000), lo=64,
                    hi=rng.randrange(100, 401), precision=rng.choice(("fp32", "fp32", "fp16dev")),
                    steps=rng.randrange(20, 61))
    if kind in ("advance", "train"):
        wide = rng.random() < 0.7
        return dict(kind=kind, nx=16 * rng.randrange(8, 17), ny=16 * _log(rng, 8, 64), channels=64 if wide else 32,
                    modes=32 if wide else rng.choice((8, 16, 24)), layers=rng.randrange(2, 5))
    return dict(kind="product", m=16 * rng.randrange(1, 9), n=16 * _log(rng, 64, 16384), k=16 * rng.randrange(1, 17),
                ta=rng.random() < 0.5, tb=rng.random() < 0.5, out=rng.choice(("f32", "bf16")))


# ------------------------------------------------------- lattice parameters

def _physics(R=1000.0, d_m=1e-3):
    """The workloads' physics in lattice units: dynamic viscosity ratio 50,
    Clift-Grace-Weber drag of bubbles of diameter d_m at lattice speed 69.2,
    buoyancy (R - 1) g_hat = 1e-6, stabilisers gamma = 1, n_gamma = 200."""
    g_hat = 1e-6 / (R - 1.0)
    kappa = 3.0 * 0.66 / (4.0 * d_m) * 69.2 ** 2 * g_hat / 9.81
    nu_l = (1.0 / 0.6 - 0.5) / 3.0 / 20.0
    return dict(R=R, omega_g=0.6, omega_l=1.0 / (0.5 + 3.0 * nu_l), omega_alpha=1.5, drag_model=1, kappa_I=kappa,
                kappa_W=0.0, g_hat=g_hat, gamma=1.0, n_gamma=200, spalding_mode=2)


def _lattice(case):
    """(lattice, dims, params) of a lattice case."""
    recipe, dims = case["recipe"], (case["nx"], case["ny"], case["nz"])
    p = _physics()
    if recipe == "column1d":
        p.update(g_axis=0, kappa_W=p["kappa_I"], bc_lo=(1, 0, 0), bc_hi=(1, 0, 0))
        lattice = "D1Q3"
    elif recipe == "tube1d":
        p = dict(R=2.0, omega_g=0.6, omega_l=0.6, omega_alpha=1.9997, drag_model=0, kappa_I=1e-2, kappa_W=1e-2, g_hat=1e-6,
                 g_axis=0, gamma=0.0, n_gamma=1, spalding_mode=2, bc_lo=(2, 0, 0), bc_hi=(3, 0, 0), in_alpha=(0.01, 0.8),
                 in_ug=(math.sqrt(0.01 * 0.99 * 1e-6 / 1e-2), 1e-2), in_ul=(0.0, 1e-3), ramp_nt=500000)
        lattice = "D1Q3"
    elif recipe == "box2d":
        p.update(g_axis=1, bc_lo=(0, 2, 0), bc_hi=(0, 1, 0), inlet_lo=3 * dims[0] // 8, inlet_hi=5 * dims[0] // 8,
                 in_alpha=(0.01, 0.3), in_ug=(4.3e-4, 4.3e-3), inlet_ul_mode=1, ramp_nt=1667)
        lattice = "D2Q9"
    elif recipe == "plume2d":
        p.update(g_axis=1, bc_lo=(0, 1, 0), bc_hi=(0, 1, 0))
        lattice = "D2Q9"
    else:
        p.update(g_axis=2, bc_lo=(1, 1, 0), bc_hi=(1, 1, 0))
        lattice = "D3Q19"
    return lattice, dims, dict(p, precision=case["precision"])


def _sweep(case):
    """[(dims, params)] of a batch case."""
    r = random.Random(case["sweep"])
    out = []
    for _ in range(case["columns"]):
        nx = r.randint(case["lo"], case["hi"])
        p = _physics(math.exp(r.uniform(math.log(10.0), math.log(1000.0))), r.uniform(0.5e-3, 5e-3))
        p.update(g_axis=1, bc_lo=(0, 1, 0), bc_hi=(0, 1, 0), precision=case["precision"])
        out.append(((nx, 4 * nx, 1), p))
    return out


# --------------------------------------------------------------- the inputs

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _waves(g, dims, n=8, shortest=16.0):
    """A smooth periodic random field of unit variance: plane waves no shorter
    than `shortest` nodes."""
    nx, ny, nz = dims
    out = torch.zeros((nz, ny, nx), dtype=torch.float64, device=DEV)
    ax = [torch.arange(m, dtype=torch.float64, device=DEV) / m for m in (nz, ny, nx)]
    r = torch.rand((n, 4), generator=g, dtype=torch.float64, device=DEV).cpu().numpy()
    for k in range(n):
        most = [max(1, int(m / shortest)) if m > 1 else 0 for m in (nz, ny, nx)]
        kz, ky, kx = [round((2.0 * r[k, i] - 1.0) * most[i]) for i in range(3)]
        ph = (kz * ax[0])[:, None, None] + (ky * ax[1])[None, :, None] + (kx * ax[2])[None, None, :]
        out += torch.cos(2.0 * math.pi * (ph + r[k, 3]))
    return out.reshape(-1) * math.sqrt(2.0 / n)


def _fields(recipe, dims, seed):
    """Initial fields of a recipe: what such a run starts from."""
    g = _gen(seed)
    nx, ny, nz = dims
    N = nx * ny * nz
    D = 1 if ny == 1 and nz == 1 else (2 if nz == 1 else 3)

    def uni(*shape):
        return torch.rand(shape, generator=g, dtype=torch.float64, device=DEV) * 2.0 - 1.0

    pk = torch.full((N,), 1.0 / 3.0, dtype=torch.float64, device=DEV)
    if recipe == "tube1d":
        a = torch.full((N,), 0.01, dtype=torch.float64, device=DEV) + 1e-3 * uni(N).abs()
        u = math.sqrt(0.01 * 0.99 * 1e-6 / 1e-2)
        return dict(alpha_g=a, u_g=u * (1.0 + 0.01 * uni(1, N)), u_l=1e-5 * uni(1, N), p_k=pk)
    if recipe in ("column1d", "column2d"):
        n = ny if D == 2 else nx  # gas below, liquid above
        at = torch.arange(N, device=DEV) // (nx if D == 2 else 1)
        a = torch.where(at < n // 2, 0.9, 0.1).double() + 1e-3 * uni(N)
        return dict(alpha_g=a, u_g=1e-6 * uni(D, N), u_l=1e-6 * uni(D, N), p_k=pk)
    if recipe == "box2d":
        a = 0.01 + 5e-4 * _waves(g, dims)
        return dict(alpha_g=a.clamp(0.005, 0.1), u_g=4.3e-5 * uni(2, N), u_l=4.3e-5 * uni(2, N), p_k=pk)
    if recipe == "plume2d":
        a = 0.1 + 0.03 * _waves(g, dims)
        return dict(alpha_g=a.clamp(0.01, 0.6), u_g=1e-5 * uni(2, N), u_l=1e-5 * uni(2, N), p_k=pk)
    # 3D column in motion: smooth gas fraction about 0.05, smooth velocities
    ug = torch.stack([1e-3 * _waves(g, dims, 4) for _ in range(3)])
    ul = torch.stack([5e-4 * _waves(g, dims, 4) for _ in range(3)])
    a = (0.05 + 0.01 * _waves(g, dims)).clamp(0.01, 0.99)
    return dict(alpha_g=a, u_g=ug, u_l=ul, p_k=pk)


def _weights(case, seed):
    """Seeded weights of the surrogate in the library's parameter order, and
    its normalisation: unit-variance layers, a trained-size output."""
    C, K, L = case["channels"], case["modes"], case["layers"]
    r = np.random.Generator(np.random.PCG64(int(seed)))

    def normal(std, *shape):
        return (r.standard_normal(int(np.prod(shape)), dtype=np.float32) * np.float32(std))

    parts = [normal(1 / math.sqrt(6.0), C, CIN), normal(0.1, C)]
    for _ in range(L):
        parts += [normal(1 / math.sqrt(C), C, C), normal(0.1, C)]
        parts += [normal(1 / math.sqrt(2.0 * C * K), K, C, C) for _ in range(4)]
    parts += [normal(0.5 / math.sqrt(C), COUT, C), normal(0.01, COUT)]
    mean = np.array([0.1, 0.0, 0.0, 0.0, 0.0, 1.0 / 3.0], np.float32)
    std_in = np.array([0.03, 1e-3, 1e-3, 5e-4, 5e-4, 1e-5], np.float32)
    std_out = np.array([2e-3, 2e-4, 2e-4, 5e-5, 5e-5, 5e-6], np.float32)
    return np.concatenate(parts), (mean, std_in, std_out)


def _states(case, seed):
    """A state (6, N) of a 2D box in motion and the one 64 steps later, as a
    training set has them."""
    g = _gen(seed + 77)
    dims = (case["nx"], case["ny"], 1)
    _, (mean, std_in, std_out) = _weights(dict(case, layers=0), seed)
    col = lambda v: torch.tensor(v, dtype=torch.float64, device=DEV)[:, None]  # noqa: E731
    now = col(mean) + col(std_in) * torch.stack([_waves(g, dims, 6) for _ in range(6)])
    now[0].clamp_(0.01, 0.6)
    nxt = now + col(std_out) * torch.stack([_waves(g, dims, 6, 32.0) for _ in range(6)])
    return now.contiguous(), nxt.contiguous()


def _operands(case, seed):
    g = _gen(seed)
    m, n, k = case["m"], case["n"], case["k"]
    a = torch.randn((k, m) if case["ta"] else (m, k), generator=g, device=DEV).to(torch.bfloat16)
    b = torch.randn((n, k) if case["tb"] else (k, n), generator=g, device=DEV).to(torch.bfloat16)
    return a, b


# ------------------------------------------------------------ prepare / run

class _Batch:
    """A batch handle of the C ABI, as a C program keeps it."""

    def __init__(self, items):
        self.lib = lbm.load_library()
        n = len(items)
        dims = (ctypes.c_int * (3 * n))(*[v for d, _ in items for v in d])
        params = (lbm.Params * n)(*[lbm.make_params(p) for _, p in items])
        self.h = ctypes.c_void_p()
        self.check(self.lib.lbm_batch_create(2, n, dims, params, ctypes.byref(self.h)))

    def check(self, rc):
        if rc:
            raise RuntimeError("batch call failed: %d %s" % (rc, (self.lib.lbm_batch_last_error(self.h) or b"").decode()))

    def __del__(self):
        if self.h:
            self.lib.lbm_batch_destroy(self.h)
            self.h = None


def _empty_fields(D, N):
    return dict(alpha_g=torch.empty(N, dtype=torch.float64, device=DEV), u_g=torch.empty((D, N), dtype=torch.float64, device=DEV),
                u_l=torch.empty((D, N), dtype=torch.float64, device=DEV), p_k=torch.empty(N, dtype=torch.float64, device=DEV))


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("run", "window"):
        lattice, dims, params = _lattice(case)
        f = _fields(case["recipe"], dims, seed)
        sim = lbm.Simulation(lattice, dims, params)
        sim.init(**f)
        return dict(case=case, sim=sim, fields=f if kind == "window" else None, out=_empty_fields(sim.D, sim.N))
    if kind == "batch":
        items = _sweep(case)
        b = _Batch(items)
        sizes = [d[0] * d[1] for d, _ in items]
        for i, (d, _) in enumerate(items):
            f = _fields("column2d", d, seed + i)
            b.check(b.lib.lbm_batch_init(b.h, i, *[f[k].data_ptr() for k in FIELDS], 1))
        torch.cuda.synchronize()
        total = sum(sizes)
        out = {k: torch.empty(v * total, dtype=torch.float64, device=DEV) for k, v in zip(FIELDS, (1, 2, 2, 1))}
        return dict(case=case, batch=b, sizes=sizes, out=out)
    if kind in ("advance", "train"):
        w, norm = _weights(case, seed)
        m = lbm.Surrogate(case["nx"], case["ny"], case["channels"], case["modes"], case["layers"])
        m.set_params(w)
        m.set_norm(*norm)
        now, nxt = _states(case, seed)
        if kind == "train":
            m.set_loss(1.0)
        return dict(case=case, model=m, now=now, nxt=nxt, out=torch.empty_like(now),
                    step=torch.empty_like(now, dtype=torch.bfloat16))
    a, b = _operands(case, seed)
    c = torch.empty((case["m"], case["n"]), dtype=torch.float32 if case["out"] == "f32" else torch.bfloat16, device=DEV)
    return dict(case=case, a=a, b=b, c=c)


def _kept(out, precision):
    return out if precision == "fp64" else {k: v.float() for k, v in out.items()}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind in ("run", "window"):
        sim = state["sim"]
        if kind == "window":
            sim.init(**state["fields"])
        sim.step(case["steps"])
        return _kept(sim.moments(out=state["out"]), case["precision"])
    if kind == "batch":
        b, out = state["batch"], state["out"]
        b.check(b.lib.lbm_batch_step(b.h, case["steps"]))
        at = 0
        for i, n in enumerate(state["sizes"]):
            ptr = [out[k].data_ptr() + 8 * w * at for k, w in zip(FIELDS, (1, 2, 2, 1))]
            b.check(b.lib.lbm_batch_get_moments(b.h, i, *ptr, None, None, 1))
            at += n
        return _kept(out, case["precision"])
    if kind == "advance":
        _, ok = state["model"].advance(state["now"], state["out"], max_drift=1.0)
        # the predicted change over the window, in the model's type
        inc = torch.sub(state["out"], state["now"], out=state["step"])
        return dict(zip(FIELDS, (inc[0], inc[1:3], inc[3:5], inc[5])), ok=ok)
    if kind == "train":
        m = state["model"]
        m.zero_grads()
        loss = m.accumulate(state["now"], state["nxt"])
        return dict(grads=torch.from_numpy(m.grads()).bfloat16(), loss=torch.tensor(loss).bfloat16())
    lbm.fno_gemm(state["a"], state["b"], state["c"], ta=case["ta"], tb=case["tb"])
    return state["c"]


# ------------------------------------------------------------------- work

def work(case):
    kind = case["kind"]
    if kind in ("run", "window", "batch"):
        if kind == "batch":
            D, N = 2, sum(d[0] * d[1] for d, _ in _sweep(case))
        else:
            lattice, dims, _ = _lattice(case)
            D, N = D_OF[lattice], dims[0] * dims[1] * dims[2]
        store = Q_OF[D] * DIR_BYTES[case["precision"]] * N
        held = 3 * HELD_BYTES[case["precision"]] * N
        fields = 8 * (2 + 2 * D) * N
        # a store beyond L2 crosses memory every step, a smaller one once
        crossings = case["steps"] if store > L2_BYTES else 1
        b = crossings * (2 * store + held) + fields * (2 if kind == "window" else 1)
        return dict(bytes=b, flops=NODE_FLOPS[D] * N * case["steps"])
    if kind in ("advance", "train"):
        C, K, L, P = case["channels"], case["modes"], case["layers"], case["nx"] * case["ny"]
        np_ = C * CIN + C + L * (C * C + C + 4 * K * C * C) + COUT * C + COUT
        axes = case["nx"] + case["ny"]
        # per layer: channel mixing, the two axes' projections and
        # reconstructions as truncated sums, the modes' mixings
        per = 2 * C * C * P + 2 * 2 * (2 * 2 * K * C * P) + 2 * K * 4 * C * C * axes
        f = 2 * P * C * 12 + L * per
        if kind == "advance":
            return dict(bytes=2 * 48 * P + 2 * np_, flops=f)
        return dict(bytes=2 * 48 * P + 4 * np_ + 4 * np_, flops=3 * f)
    m, n, k = case["m"], case["n"], case["k"]
    return dict(bytes=2 * (m * k + k * n) + (4 if case["out"] == "f32" else 2) * m * n, flops=2 * m * n * k)


# ------------------------------------------- the same outputs in 64 bits

class _Plain:
    """The six coupled schemes in plain float64 torch: two arrays, the
    formulas as the paper writes them (arXiv 2409.10399, Secs. 2-3), psi = 0."""

    def __init__(self, D, dims, p, f):
        self.D, self.p, self.t = D, p, 0
        self.n = dims[:D]
        self.N = int(np.prod(dims))
        vs = [v for v in np.ndindex(*([3] * D))]
        vs = sorted((np.array(v) - 1 for v in vs), key=lambda v: int(np.abs(v).sum()))
        vs = [v for v in vs if np.abs(v).sum() <= 2]
        wt = {1: (2 / 3, 1 / 6), 2: (4 / 9, 1 / 9, 1 / 36), 3: (1 / 3, 1 / 18, 1 / 36)}[D]
        self.v = [tuple(int(c) for c in v) for v in vs]
        self.Q = len(vs)
        self.opp = [self.v.index(tuple(-c for c in v)) for v in self.v]
        self.V = torch.tensor(np.array(self.v, np.float64), device=DEV)
        self.w = torch.tensor([wt[int(np.abs(v).sum())] for v in vs], dtype=torch.float64, device=DEV)[:, None]
        self.k0 = (1 - wt[0]) / wt[0]
        self._faces()
        a, ug, ul = f["alpha_g"], f["u_g"], f["u_l"]
        eps = f["p_k"] * 3.0
        phi = 1.0 + (eps - 1.0) / p["R"]
        one = torch.ones_like(a)
        self.f = [self.feq_I(one, eps, ug), self.feq_I(phi, one, ul), self.feq_S(a, ug), self.feq_S(1 - a, ul),
                  self.feq_S(one, (1 - a) * (ug - ul)), self.feq_S(one, a * (ul - ug))]

    def _faces(self):
        p, D, n = self.p, self.D, self.n
        idx = torch.arange(self.N, device=DEV)
        co, s = [], 1
        for d in range(D):
            co.append((idx // s) % n[d])
            s *= n[d]
        self.stride = int(np.prod(n[:p["g_axis"]]))
        ga = p["g_axis"]
        tr = next((d for d in range(D) if d != ga), None)
        self.cross = []
        for q in range(self.Q):
            wall = torch.zeros(self.N, dtype=torch.bool, device=DEV)
            inl, outl = wall.clone(), wall.clone()
            for d in range(D):
                vd = self.v[q][d]
                if vd == 0:
                    continue
                bc = (p["bc_hi"] if vd > 0 else p["bc_lo"])[d]
                at = co[d] == (n[d] - 1 if vd > 0 else 0)
                if bc == 1:
                    wall |= at
                elif bc == 2:
                    strip = at if tr is None else at & (co[tr] >= p["inlet_lo"]) & (co[tr] < p["inlet_hi"])
                    inl |= strip
                    wall |= at & ~strip
                elif bc == 3:
                    outl |= at
            self.cross.append([m.nonzero()[:, 0] for m in (wall, inl & ~wall, outl & ~wall)])

    def even(self, u):
        vu = self.V @ u
        return vu, 4.5 * vu * vu - 1.5 * (u * u).sum(0)

    def eta(self, phi):
        e = phi.expand(self.Q, -1).clone()
        e[0] = 1.0 + self.k0 * (1.0 - e[0])
        return e

    def feq_I(self, phi, eps, u):
        vu, e = self.even(u)
        return self.w * (eps * self.eta(phi) + 3.0 * vu + e)

    def feq_S(self, alpha, u):
        vu, e = self.even(u)
        return self.w * alpha * (1.0 + 3.0 * vu + e)

    def feq_L(self, S, G):
        e = S.expand(self.Q, -1).clone() * 0.0
        e[0] = S * (1.0 + self.k0)
        return self.w * (e + 3.0 * (self.V @ G))

    def moments(self):
        f, V = self.f, self.V
        m = dict(eg=f[0].sum(0), el=f[1].sum(0), ag=f[2].sum(0), al=f[3].sum(0), Sg=1 - f[4].sum(0), Sl=1 - f[5].sum(0))
        for k, s in (("ug", 0), ("ul", 1), ("Jg", 2), ("Jl", 3)):
            m[k] = V.t() @ f[s]
        if self.p["spalding_mode"]:
            bg, bl = m["ag"].clamp(0, 1), m["al"].clamp(0, 1)
            m["Ag"] = bg / (bg + bl)
            m["Al"] = 1 - m["Ag"]
        else:
            m["Ag"], m["Al"] = m["ag"], m["al"]
        return m

    def ramp(self, mm):
        nt = self.p.get("ramp_nt", 0)
        return mm[1] if nt <= 0 else (mm[1] - mm[0]) * math.tanh(self.t / nt) + mm[0]

    def step(self):
        p, D, R = self.p, self.D, self.p["R"]
        m = self.moments()
        eg, el, ug, ul, Ag, Al = m["eg"], m["el"], m["ug"], m["ul"], m["Ag"], m["Al"]
        cg, cl = Al * (ug - ul), Ag * (ul - ug)
        phi = (1 + (eg - 1) / R) / el
        if self.t % p["n_gamma"] == 0:
            self.Sg = m["Sg"] - p["gamma"] * (ug * ug).sum(0) * (eg - 1)
            self.Sl = m["Sl"] - p["gamma"] * (ul * ul).sum(0) * (phi * el - 1)
            self.Lam = Ag * Al * (Ag + Al * R)
        Sg, Sl = self.Sg, self.Sl
        grg = 3 * p["omega_alpha"] * (m["ag"] * ug - m["Jg"])
        grl = 3 * p["omega_alpha"] * (m["al"] * ul - m["Jl"])
        gG = 0.5 * (grg - grl)
        sG, sL = torch.zeros_like(ug), torch.zeros_like(ul)
        if D == 1:
            Ag_, Al_ = [(1 / p[k] - 0.5) * p[k] for k in ("omega_g", "omega_l")]
        else:
            Ag_, Al_ = [1 - 0.5 * p[k] for k in ("omega_g", "omega_l")]
        for d in range(D):
            for e in range(D):
                vv = (self.V[:, d] * self.V[:, e])[None]
                Pg, Pl = (vv @ self.f[0])[0], (vv @ self.f[1])[0]
                qg = ug[d] * ug[e] + (eg / 3 if d == e else 0)
                ql = ul[d] * ul[e] + (phi * el / 3 if d == e else 0)
                sG[d] += Ag_ * (qg - Pg) * gG[e]
                sL[d] -= Al_ * (ql - Pl) * gG[e]
        KI = p["kappa_I"] * (self.Lam if p["drag_model"] else 1.0)
        KW = p["kappa_W"] * (self.Lam if p["drag_model"] else 1.0)
        du = ul - ug
        ndu, nul = (du * du).sum(0).sqrt(), (ul * ul).sum(0).sqrt()
        Gg = Sg * ug + (sG + KI * ndu * du) / Ag.clamp_min(1e-8)
        Gg[p["g_axis"]] += (R - 1) * p["g_hat"]
        Gl = Sl * ul + (sL - (KI * ndu * du + KW * nul * ul) / R) / Al.clamp_min(1e-8)
        f, one = self.f, torch.ones_like(eg)
        mode2 = p["spalding_mode"] == 2
        out = [f[0] + p["omega_g"] * (self.feq_I(one, eg, ug) - f[0]) + self.feq_L(Sg, Gg),
               f[1] + p["omega_l"] * (self.feq_I(phi, el, ul) - f[1]) + self.feq_L(Sl, Gl),
               f[2] + p["omega_alpha"] * (self.feq_S(Ag if mode2 else m["ag"], ug) - f[2]),
               f[3] + p["omega_alpha"] * (self.feq_S(Al if mode2 else m["al"], ul) - f[3]),
               self.feq_S(one, cg), self.feq_S(one, cl)]
        self.f = f = None
        back = self._rules(out, m, cg, cl)
        shape = tuple(reversed(self.n))
        new = []
        for s in range(6):
            o = out[s].reshape((self.Q,) + shape)
            fs = torch.empty_like(o)
            for q in range(self.Q):
                fs[q] = torch.roll(o[q], tuple(reversed(self.v[q])), tuple(range(D)))
            fs = fs.reshape(self.Q, self.N)
            for q in range(self.Q):
                for (ii, val) in back[s][q]:
                    fs[self.opp[q], ii] = val
            new.append(fs)
            out[s] = None
        self.f = new
        self.t += 1

    def _rules(self, out, m, cg, cl):
        """(nodes, value streamed back along opp(q)) of every scheme and q."""
        p, D, ga = self.p, self.D, self.p["g_axis"]
        back = [[[] for _ in range(self.Q)] for _ in range(6)]
        for q in range(self.Q):
            wall, inl, outl = self.cross[q]
            if len(wall):
                for s in range(6):
                    back[s][q].append((wall, out[s][q][wall]))
            for ii, side in ((inl, 1), (outl, -1)):
                if not len(ii):
                    continue
                jj, qo = ii + side * self.stride, self.opp[q]
                ext = lambda x: 2 * x[..., ii] - x[..., jj]  # noqa: E731
                hw = lambda x: 1.5 * x[..., ii] - 0.5 * x[..., jj]  # noqa: E731
                one = torch.ones(len(ii), dtype=torch.float64, device=DEV)
                if side == 1:
                    a, u = self.ramp(p["in_alpha"]), self.ramp(p["in_ug"])
                    v = -a * u / (1 - a) if p.get("inlet_ul_mode", 0) else self.ramp(p["in_ul"])
                    uu, vv = torch.zeros((D, len(ii)), dtype=torch.float64, device=DEV), torch.zeros((D, len(ii)), dtype=torch.float64, device=DEV)
                    uu[ga], vv[ga] = u, v
                    w = float(self.w[q, 0])
                    val = [out[0][q][ii] - 6 * w * self.v[q][ga] * u, out[1][q][ii] - 6 * w * self.v[q][ga] * v,
                           self.feq_S(a * one, uu)[qo], self.feq_S((1 - a) * one, vv)[qo]]
                else:
                    ub, lb = hw(m["ug"]), hw(m["ul"])
                    both = lambda e, u: self.feq_S(e, u)[q] + self.feq_S(e, -u)[q]  # noqa: E731
                    val = [both(one, ub) - out[0][q][ii], both(one, lb) - out[1][q][ii],
                           both(hw(m["Ag"]), ub) - out[2][q][ii], both(hw(m["Al"]), lb) - out[3][q][ii]]
                val += [self.feq_S(one, ext(cg))[qo], self.feq_S(one, ext(cl))[qo]]
                for s in range(6):
                    back[s][q].append((ii, val[s]))
        return back

    def fields(self):
        m = self.moments()
        return dict(alpha_g=m["Ag"], u_g=m["ug"], u_l=m["ul"], p_k=m["eg"] / 3)


def _plain_run(D, dims, p, f, steps):
    s = _Plain(D, dims, p, f)
    for _ in range(steps):
        s.step()
    return s.fields()


def _gelu(z):
    return 0.5 * z * (1 + torch.tanh(math.sqrt(2 / math.pi) * (z + 0.044715 * z ** 3)))


def _plain_model(case, w, x):
    """The surrogate's output (16, ny, nx) in plain float64 torch."""
    C, K, L = case["channels"], case["modes"], case["layers"]
    at = 0

    def take(*shape):
        nonlocal at
        n = int(np.prod(shape))
        at += n
        return w[at - n:at].reshape(shape)

    def spectral(h, A, B, dim):
        F = torch.fft.rfft(h, dim=dim).narrow(dim, 0, K)
        W = torch.complex(A, -B)
        G = torch.einsum("koi,iyk->oyk", W, F) if dim == 2 else torch.einsum("koi,ikx->okx", W, F)
        return torch.fft.irfft(G, n=h.shape[dim], dim=dim)  # the higher modes are zero

    W_in, b_in = take(C, CIN), take(C)
    h = torch.einsum("oi,iyx->oyx", W_in, x) + b_in[:, None, None]
    for _ in range(L):
        W, b, Ax, Bx, Ay, By = take(C, C), take(C), take(K, C, C), take(K, C, C), take(K, C, C), take(K, C, C)
        z = torch.einsum("oi,iyx->oyx", W, h) + b[:, None, None]
        h = _gelu(z + spectral(h, Ax, Bx, 2) + spectral(h, Ay, By, 1))
    W_out, b_out = take(COUT, C), take(COUT)
    return torch.einsum("oi,iyx->oyx", W_out, h) + b_out[:, None, None]


def exact(case, seed):
    kind = case["kind"]
    if kind in ("run", "window"):
        lattice, dims, p = _lattice(case)
        return _plain_run(D_OF[lattice], dims, p, _fields(case["recipe"], dims, seed), case["steps"])
    if kind == "batch":
        got = [_plain_run(2, d, p, _fields("column2d", d, seed + i), case["steps"]) for i, (d, p) in enumerate(_sweep(case))]
        return {k: torch.cat([g[k].reshape(-1) for g in got]) for k in FIELDS}
    if kind in ("advance", "train"):
        wf, norm = _weights(case, seed)
        mean, std_in, std_out = [torch.tensor(v.astype(np.float64), device=DEV)[:, None] for v in norm]
        w = torch.tensor(wf.astype(np.float64), device=DEV)
        now, nxt = _states(case, seed)
        shape = (CIN, case["ny"], case["nx"])
        x = torch.zeros((CIN, now.shape[1]), dtype=torch.float64, device=DEV)
        x[:6] = (now - mean) / std_in
        if kind == "advance":
            with torch.no_grad():
                inc = std_out * _plain_model(case, w, x.reshape(shape))[:6].reshape(6, -1)
            return dict(zip(FIELDS, (inc[0], inc[1:3], inc[3:5], inc[5])), ok=None)
        w.requires_grad_(True)
        y = _plain_model(case, w, x.reshape(shape))[:6].reshape(6, -1)
        e = y - (nxt - now) / std_out
        loss = (e * e).mean() + 1.0 * e[0].mean() ** 2
        loss.backward()
        return dict(grads=w.grad.cpu(), loss=loss.detach().cpu())
    a, b = _operands(case, seed)
    a, b = a.double(), b.double()
    return (a.t() if case["ta"] else a) @ (b.t() if case["tb"] else b)
