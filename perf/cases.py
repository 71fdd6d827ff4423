"""Performance cases: what a user of the library has it do, through its public
entry points, with the inputs, plans and handles such a program holds.

Five kinds of case:

* ``grid``   a 2D run: initial fields in, ``steps`` time steps of the fused
             MRT-FD step, the state out (checkpoint populations; FP64-class
             runs also the fields). Flows: the Sod tube, the regular shock
             reflection, the Mach reflection (sides that switch kind at a
             moving position), the shock-bubble interaction and the doubly
             periodic quadrant problem of the corrector's training data.
* ``tubes``  a batch of independent quasi-1D shock tubes of uneven length.
* ``train``  one training step of the coarse-grid corrector network.
* ``infer``  the corrector applied to a coarse field.
* ``vn``     spectral radii of the Sec. IV amplification matrix over a table of
             states, rates and wave vectors (a stability map).

The parameters are those of the paper's problems as ``workloads.py`` states
them; every seed perturbs the initial fields, so that inputs differ.
"""
import math

import numpy as np
import torch

from paper_0908_3749_gb300 import lbm

SQ2 = math.sqrt(2.0)
FLOPS_PER_NODE = 389       # 2D step, factorised moments, FMA = 2
FLOPS_PER_TUBE_NODE = 325  # the same without the y terms


# ----------------------------------------------------------------------------
# The cases
# ----------------------------------------------------------------------------
def listed():
    return [
        # The smallest run: the Sod tube on 200 x 4 nodes, 100 of its 10 000
        # steps (one output interval). A step is a few microseconds: latency.
        {"name": "sod_fp64_200x4", "kind": "grid", "flow": "sod", "precision": "fp64",
         "nx": 200, "ny": 4, "steps": 100, "audit": 0},
        # The regular shock reflection at its configured 600 x 200 in FP32 with
        # audits: a grid that fits in the L2, between two outputs.
        {"name": "reflection_fp32_600x200", "kind": "grid", "flow": "reflection",
         "precision": "fp32", "nx": 600, "ny": 200, "steps": 200, "audit": 50},
        # The Mach reflection in FP64 on an odd, ragged grid near the paper's
        # 600 x 300, whose top side switches kind at a moving position.
        {"name": "mach_fp64_601x299", "kind": "grid", "flow": "mach", "precision": "fp64",
         "nx": 601, "ny": 299, "steps": 20, "audit": 10},
        # The largest 2D workload (the benchmark's grid) in each precision that
        # is used on it: the paper's FP64, FP32, double-word and tensor cores.
        {"name": "bubble_fp64_2048x1024", "kind": "grid", "flow": "bubble", "precision": "fp64",
         "nx": 2048, "ny": 1024, "steps": 10, "audit": 10},
        {"name": "bubble_fp32_2048x1024", "kind": "grid", "flow": "bubble", "precision": "fp32",
         "nx": 2048, "ny": 1024, "steps": 70, "audit": 10},
        {"name": "bubble_df64_2048x1024", "kind": "grid", "flow": "bubble", "precision": "df64",
         "nx": 2048, "ny": 1024, "steps": 20, "audit": 10},
        {"name": "bubble_tc_2048x1024", "kind": "grid", "flow": "bubble",
         "precision": "tc_tf32x3", "nx": 2048, "ny": 1024, "steps": 70, "audit": 10},
        # The batched Riemann problems: the configured 4096 tubes, and a small
        # parameter study of 61.
        {"name": "tubes_4096", "kind": "tubes", "ntubes": 4096, "nx_min": 128, "nx_max": 2048,
         "steps": 100},
        {"name": "tubes_61", "kind": "tubes", "ntubes": 61, "nx_min": 128, "nx_max": 2048,
         "steps": 200},
        # The corrector on the configured 512 x 512 coarse grid: one training
        # step (forward, loss, backward, Adam), and inference.
        {"name": "train_512x512", "kind": "train", "h": 512, "w": 512, "loss": "mse"},
        {"name": "infer_512x512", "kind": "infer", "h": 512, "w": 512},
        # A stability map: 32 states x 1024 wave numbers.
        {"name": "vn_32x1024", "kind": "vn", "ncases": 32, "nk": 1024},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["grid", "grid", "grid", "tubes", "train", "infer", "vn"])
    if kind == "grid":
        precision = rng.choice(["fp64", "fp32", "fp32", "df64", "tc_tf32x3", "fp32_dwmom"])
        flow = rng.choice(["sod", "reflection", "mach", "bubble", "quadrant"])
        if flow == "sod":
            nx, ny = _log_int(rng, 100, 4000), rng.randint(1, 8)
        else:
            nodes = math.exp(rng.uniform(math.log(6e3), math.log(2.0e6)))
            aspect = rng.uniform(1.0, 3.0)
            nx = max(64, int(math.sqrt(nodes * aspect)))
            ny = max(48, min(int(nodes / nx), 2097152 // nx))
        most = {"fp64": 10, "df64": 20}.get(precision, 60)  # steps at 2048 x 1024
        steps = min(_log_int(rng, 5, 200), max(5, int(most * 2097152.0 / (nx * ny))))
        return {"kind": "grid", "flow": flow, "precision": precision, "nx": nx, "ny": ny,
                "steps": steps, "audit": rng.choice([0, 1, 10, 50])}
    if kind == "tubes":
        lo = _log_int(rng, 32, 1024)
        return {"kind": "tubes", "ntubes": _log_int(rng, 8, 4096), "nx_min": lo,
                "nx_max": min(2048, lo + _log_int(rng, 8, 1920)), "steps": _log_int(rng, 4, 100)}
    if kind in ("train", "infer"):
        c = {"kind": kind, "h": _log_int(rng, 13, 512), "w": _log_int(rng, 11, 512)}
        if kind == "train":
            c["loss"] = rng.choice(["mse", "l1"])
        return c
    return {"kind": "vn", "ncases": _log_int(rng, 1, 32), "nk": _log_int(rng, 11, 1024)}


# ----------------------------------------------------------------------------
# Inputs
# ----------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device="cpu")
    g.manual_seed(int(seed))
    return g


def _smooth(gen, ny, nx, modes=4):
    """A smooth field of unit size: a few random Fourier modes."""
    x = torch.arange(nx, device="cuda", dtype=torch.float64)[None, :] / nx
    y = torch.arange(ny, device="cuda", dtype=torch.float64)[:, None] / ny
    out = torch.zeros((ny, nx), device="cuda", dtype=torch.float64)
    for _ in range(modes):
        kx, ky = (int(v) for v in torch.randint(0, 5, (2,), generator=gen))
        a, ph = (float(v) for v in torch.rand(2, generator=gen))
        out += (2 * a - 1) * torch.cos(2 * math.pi * (kx * x + ky * y) + 2 * math.pi * ph)
    return out / modes


def _rates(default=1e5, **given):
    s = [float(default)] * 16
    for key, val in given.items():
        s[int(key[1:]) - 1] = float(val)
    return s


SOD = ((1.0, 0.0, 0.0, 1.0), (0.125, 0.0, 0.0, 0.8))
REFLECT_IN = (1.0, 2.9 * SQ2, 0.0, 1.0)
REFLECT_TOP = (1.5374771480804381, 3.742789341797761, -0.6208189520502188, 1.6065279429250885)
MACH_PRE = (2.0, 0.0, 0.0, 0.5)
MACH_POST = (3.17647, 0.555556 * math.cos(math.pi / 6), -0.555556 * math.sin(math.pi / 6), 0.839506)
BUBBLE_POST = (1.28, -0.3774, 0.0, 1.6512 / 1.28)


def _flow(case, seed):
    """(dx, dt, rates, boundary sides, fields [4][ny][nx] on the GPU)."""
    nx, ny, flow = case["nx"], case["ny"], case["flow"]
    gen = _gen(seed)
    one = torch.ones((ny, nx), device="cuda", dtype=torch.float64)
    x = torch.arange(nx, device="cuda", dtype=torch.float64)[None, :] + 0.5
    y = torch.arange(ny, device="cuda", dtype=torch.float64)[:, None] + 0.5

    def two(mask, a, b):
        mask = mask.expand(ny, nx)
        return [torch.where(mask, p * one, q * one) for p, q in zip(a, b)]

    if flow == "sod":
        dx, dt = 0.005, 1e-5
        s = _rates(s5=200, s6=200, s7=400, s8=400, s11=1000)
        bc = (("eq", SOD[0]), ("eq", SOD[1]), ("periodic", None), ("periodic", None))
        f = two(x <= 0.5 * nx, *SOD)
    elif flow == "reflection":
        dx, dt = 1e-3, 2e-6
        s = _rates(s5=1e4, s6=2e3, s7=1e4, s8=1e4)
        bc = (("eq", REFLECT_IN), ("extrap", None), ("reflect", None), ("eq", REFLECT_TOP))
        f = [q * one for q in REFLECT_IN]
    elif flow == "mach":
        dx, dt = 0.003, 1e-5
        foot = 0.25 * nx
        s = _rates(s5=1e3, s6=5e2, s7=1e3, s8=1e3)
        t30 = math.tan(math.pi / 6)
        bc = (("eq", MACH_POST), ("extrap", None), ("eq", MACH_POST, ("reflect", foot * dx, 0.0)),
              ("eq", MACH_POST, ("extrap", foot * dx + t30 * ny * dx,
                                 t30 * 1.5 / math.sin(math.pi / 6))))
        f = two(y >= math.tan(math.pi / 3) * (x - foot), MACH_POST, MACH_PRE)
    elif flow == "bubble":
        dx, dt = 1e-3, 1e-5
        s = _rates(s5=1e4, s6=1e4, s7=1e4, s8=1e4)
        bc = (("extrap", None), ("eq", BUBBLE_POST), ("reflect", None), ("reflect", None))
        r = 0.125 * min(nx, ny)
        inside = (x - 0.5 * nx) ** 2 + (y - 0.5 * ny) ** 2 <= r * r
        pre = two(inside, (0.1358, 0.0, 0.0, 1.0 / 0.1358), (1.0, 0.0, 0.0, 1.0))
        post = (x > 0.5 * nx + 1.25 * r).expand(ny, nx)
        f = [torch.where(post, p * one, q) for p, q in zip(BUBBLE_POST, pre)]
    else:  # quadrant: doubly periodic checkerboard of four states
        dx, dt = 1.0 / 512, 1e-5
        k = 0.005 / dx
        s = _rates(s5=200 * k, s6=200 * k, s7=400 * k, s8=400 * k, s11=1000 * k)
        bc = (("periodic", None),) * 4
        st = torch.rand((4, 4), generator=gen, dtype=torch.float64)
        lo, hi = math.log(0.5), math.log(2.0)

        def h(c, n):
            c = c / n
            return 0.5 * (torch.tanh((c - 0.25) / 0.004) - torch.tanh((c - 0.75) / 0.004))
        hx, hy = h(x, nx), h(y, ny)
        wts = ((1 - hx) * (1 - hy), hx * (1 - hy), (1 - hx) * hy, hx * hy)
        f = []
        for q in range(4):
            val = [float(v) for v in (torch.exp(lo + (hi - lo) * st[:, q]) if q in (0, 3)
                                      else 0.6 * st[:, q] - 0.3)]
            f.append(sum(w * v for w, v in zip(wts, val)))
    f[0] = f[0] * (1.0 + 0.02 * _smooth(gen, ny, nx))
    f[1] = f[1] + 0.02 * _smooth(gen, ny, nx)
    f[2] = f[2] + 0.02 * _smooth(gen, ny, nx)
    f[3] = f[3] * (1.0 + 0.02 * _smooth(gen, ny, nx))
    return dx, dt, s, bc, [q.contiguous() for q in f]


def _tubes(case, seed):
    """Tube lengths, spacings, rates and end states (numpy), as the batch of
    seeded Riemann problems draws them, with densities and temperatures within
    [0.4, 2.5] so that every tube stays physical over the run."""
    n = case["ntubes"]
    lengths = np.random.default_rng([n, case["nx_min"], case["nx_max"]])
    nx = lengths.integers(case["nx_min"], case["nx_max"] + 1, n)
    rng = np.random.default_rng(seed)
    dx = 1.0 / np.maximum(nx, 128)
    lo, hi = math.log(0.4), math.log(2.5)
    ends = [np.stack([np.exp(rng.uniform(lo, hi, n)), rng.uniform(-0.3, 0.3, n),
                      rng.uniform(-0.3, 0.3, n), np.exp(rng.uniform(lo, hi, n))], 1)
            for _ in range(2)]
    s = np.full((n, 16), 1e5)
    for k, base in ((5, 200.0), (6, 200.0), (7, 400.0), (8, 400.0), (11, 1000.0)):
        s[:, k - 1] = np.minimum(base * 0.005 / dx, 1e5)
    return nx, dx, 1e-5, s, ends[0], ends[1]


def _tube_fields(nx, left, right):
    """Initial fields of all tubes, concatenated, [4][sum nx] on the GPU."""
    n = torch.as_tensor(nx, device="cuda")
    tube = torch.repeat_interleave(torch.arange(len(nx), device="cuda"), n)
    start = torch.cumsum(n, 0) - n
    at = torch.arange(len(tube), device="cuda") - start[tube]
    first = (2 * at + 1 <= n[tube])
    ends = [torch.as_tensor(e, device="cuda")[tube] for e in (left, right)]
    f = torch.where(first[:, None], ends[0], ends[1])
    return f.t().contiguous(), tube, at


def _params(seed):
    """He-normal weights, a small last layer and small biases (a network some
    way into its training)."""
    rng = np.random.default_rng(seed)
    parts = []
    ch = lbm.CNN_CHANNELS
    for l in range(len(ch) - 1):
        size = math.sqrt(2.0 / (9 * ch[l])) * (0.3 if l == len(ch) - 2 else 1.0)
        parts += [(rng.standard_normal((3, 3, ch[l], ch[l + 1])) * size).reshape(-1),
                  rng.standard_normal(ch[l + 1]) * 0.02]
    return np.concatenate(parts).astype(np.float32)


def _pair(case, seed):
    """(coarse, target) fields [4][h][w]: a corrector quadrant state, and the
    same with a correction of a few per cent."""
    c = _flow({"nx": case["w"], "ny": case["h"], "flow": "quadrant"}, seed)[4]
    gen = _gen(seed + 7919)
    d = [_smooth(gen, case["h"], case["w"], 8) for _ in range(4)]
    t = [c[0] * (1 + 0.05 * d[0]), c[1] + 0.03 * d[1], c[2] + 0.03 * d[2], c[3] * (1 + 0.05 * d[3])]
    return torch.stack(c), torch.stack(t)


def _vn(case, seed):
    rng = np.random.default_rng(seed)
    n = case["ncases"]
    states = np.stack([np.exp(rng.uniform(math.log(0.5), math.log(2.0), n)),
                       rng.uniform(-2.0, 2.0, n), rng.uniform(-2.0, 2.0, n),
                       np.exp(rng.uniform(math.log(0.5), math.log(2.0), n))], 1)
    rates = 10.0 ** rng.uniform(3.0, 5.0, (n, 16))
    dx = 2e-3
    th = rng.uniform(0.0, math.pi) * 0.05 + np.linspace(0.0, math.pi, case["nk"])
    ang = rng.uniform(0.0, 0.5 * math.pi)
    k = np.stack([th * math.cos(ang) / dx, th * math.sin(ang) / dx], 1)
    return lbm.vn_cases(states, rates), k, states, rates, dx, 1e-5


class _State:
    """The handles and buffers of one case; frees the handle with itself."""
    handle, destroy = None, None

    def __init__(self, case):
        self.case = case

    def __del__(self):
        if self.handle:
            self.destroy(self.handle)
            self.handle = None


def prepare(case, seed):
    st = _State(case)
    kind = case["kind"]
    if kind == "grid":
        dx, dt, s, bc, fields = _flow(case, seed)
        nx, ny = case["nx"], case["ny"]
        st.fields = fields
        st.handle = lbm.lbm_create(lbm.make_config(nx, ny, dx, dx, dt, s, bc, case["precision"],
                                                   case["audit"]))
        st.destroy = lbm.lbm_destroy
        fp64 = case["precision"] == "fp64"
        shape = (16, ny, nx, 2) if case["precision"] == "df64" else (16, ny, nx)
        st.f = torch.empty(shape, device="cuda", dtype=torch.float64 if fp64 else torch.float32)
        st.out = torch.empty((4, ny, nx), device="cuda", dtype=torch.float64)
    elif kind == "tubes":
        nx, dx, dt, s, left, right = _tubes(case, seed)
        st.handle = lbm.lbm_batch_create(nx, dx, dt, s, left, right)
        st.destroy = lbm.lbm_batch_destroy
        st.fields = _tube_fields(nx, left, right)[0]
        st.out = torch.empty_like(st.fields)
    elif kind in ("train", "infer"):
        st.coarse, st.target = _pair(case, seed)
        st.handle = lbm.lbm_cnn_create(case["h"], case["w"])
        st.destroy = lbm.lbm_cnn_destroy
        lbm.lbm_cnn_set_params(st.handle, _params(seed))
        lbm.lbm_cnn_set_output_scale(st.handle, lbm.lbm_cnn_residual_rms(st.handle, st.coarse, st.target))
        if kind == "train":
            lbm.lbm_cnn_set_loss(st.handle, case["loss"])
        st.params = torch.empty(lbm.CNN_NPARAMS, device="cuda", dtype=torch.float32)
        st.out = torch.empty_like(st.coarse)
    else:
        cases, k, _, _, st.dx, st.dt = _vn(case, seed)
        st.cases = torch.as_tensor(cases, device="cuda")
        st.k = torch.as_tensor(k, device="cuda")
        st.radius = torch.empty((case["ncases"], case["nk"]), device="cuda", dtype=torch.float64)
    return st


def run(st):
    kind = st.case["kind"]
    if kind == "grid":
        # A run between two outputs, from the initial fields.
        lbm.lbm_set_init(st.handle, *st.fields)
        lbm.lbm_step(st.handle, st.case["steps"])
        lbm.lbm_get_populations(st.handle, st.f)
        precision = st.case["precision"]
        if precision == "fp64":
            lbm.lbm_moments(st.handle, *st.out)
            return {"f": st.f, "fields": st.out}
        if precision == "df64":  # a population's value is the sum of its two words
            lbm.lbm_moments(st.handle, *st.out)
            return {"f": st.f[..., 0].double() + st.f[..., 1], "fields": st.out}
        return {"f": st.f}
    if kind == "tubes":
        lbm.lbm_batch_set_init(st.handle, *st.fields)
        lbm.lbm_batch_step(st.handle, st.case["steps"])
        lbm.lbm_batch_moments(st.handle, *st.out)
        return {"fields": st.out}
    if kind == "train":
        # One step of the training loop, which records the loss; the weights
        # after it. The loss is one of an FP32 / BF16 network: single precision.
        loss = lbm.lbm_cnn_train_step(st.handle, st.coarse, st.target)
        lbm.lbm_cnn_get_params(st.handle, st.params)
        return {"loss": np.float32(loss), "params": st.params}
    if kind == "infer":
        fallback = lbm.lbm_cnn_correct(st.handle, st.coarse, st.out)
        return {"fields": st.out, "fallback": fallback}
    _, _, failed = lbm.lbm_vn_spectrum(st.cases, st.k, st.dx, st.dx, st.dt, radius=st.radius)
    return {"radius": st.radius, "failed": failed}


def _layers():
    ch = lbm.CNN_CHANNELS
    return [(ch[l], ch[l + 1]) for l in range(len(ch) - 1)]


def work(case):
    kind = case["kind"]
    if kind == "grid":
        n = case["nx"] * case["ny"]
        fp64 = case["precision"] in ("fp64", "df64")
        out = 16 * (8 if fp64 else 4) + (32 if fp64 else 0)
        return {"bytes": n * (32 + out), "flops": FLOPS_PER_NODE * n * case["steps"]}
    if kind == "tubes":
        n = case["ntubes"] * (case["nx_min"] + case["nx_max"]) // 2
        return {"bytes": n * 64, "flops": FLOPS_PER_TUBE_NODE * n * case["steps"]}
    if kind in ("train", "infer"):
        p = case["h"] * case["w"]
        fwd = sum(2 * 9 * a * b for a, b in _layers()) * p
        first = 2 * 9 * 4 * 32 * p  # no gradient is taken with respect to the input
        if kind == "train":
            return {"bytes": 64 * p + 8 * lbm.CNN_NPARAMS, "flops": 3 * fwd - first}
        return {"bytes": 64 * p, "flops": fwd}
    # Hessenberg reduction 10/3 n^3 complex multiply-adds (8 flops), then about
    # 2.5 sweeps per eigenvalue on the shrinking active block (m^2 rotated
    # pairs, 20 flops each).
    n = case["ncases"] * case["nk"]
    per = 8 * 10 * 16 ** 3 / 3 + 2.5 * 20 * sum(m * m for m in range(2, 17))
    return {"bytes": 160 * case["ncases"] + 16 * case["nk"] + 8 * n, "flops": per * n}


# ----------------------------------------------------------------------------
# The same in 64 bits, in plain torch and numpy
# ----------------------------------------------------------------------------
def _velocities():
    v = []
    for c in (1.0, 6.0):
        v += [(c, 0.0), (0.0, c), (-c, 0.0), (0.0, -c)]
    for h in (SQ2, 3.0 / SQ2):
        v += [(h, h), (-h, h), (-h, -h), (h, -h)]
    return np.array(v)


def _moment_matrix():
    x, y = _velocities().T
    q = x * x + y * y
    c3, s3 = x * (x * x - 3 * y * y), y * (3 * x * x - y * y)
    M = np.stack([x * 0 + 1, x, y, q / 2, x * x - y * y, x * y, x * q / 2, y * q / 2, c3, s3,
                  q * q / 4, x ** 4 - 6 * x * x * y * y + y ** 4, q * (x * x - y * y), q * x * y,
                  c3 * q, s3 * q])
    inv = np.linalg.inv(M).astype(np.longdouble)
    for _ in range(3):  # Newton's iteration for the inverse, in extended precision
        inv = inv @ (2 * np.eye(16, dtype=np.longdouble) - M.astype(np.longdouble) @ inv)
    return M, inv.astype(np.float64)


def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), device="cuda", dtype=torch.float64)


def _equilibria(rho, jx, jy, e):
    """Eq. 14, stacked along the first axis."""
    P = e - (jx * jx + jy * jy) / (2 * rho)
    z = torch.zeros_like(rho)
    jj = jx * jx + jy * jy
    a = (6 * rho * e - 2 * jj) / rho ** 2
    m5, m6 = (jx * jx - jy * jy) / rho, jx * jy / rho
    return torch.stack([rho, jx, jy, e, m5, m6, (e + P) * jx / rho, (e + P) * jy / rho,
                        (jx * jx - 3 * jy * jy) * jx / rho ** 2,
                        (3 * jx * jx - jy * jy) * jy / rho ** 2,
                        2 * e * e / rho - jj * jj / (4 * rho ** 3), z, a * m5, a * m6, z, z])


def _feq(Minv, rho, u, v, T):
    m = _equilibria(rho, rho * u, rho * v, rho * T + 0.5 * rho * (u * u + v * v))
    return (Minv @ m.reshape(16, -1)).reshape(m.shape)


def _fields_of(M, f):
    m = (M[:4] @ f.reshape(16, -1)).reshape((4,) + f.shape[1:])
    u, v = m[1] / m[0], m[2] / m[0]
    return torch.stack([m[0], u, v, m[3] / m[0] - 0.5 * (u * u + v * v)])


def _collision(M, Minv, f, w):
    """M^-1 w (M f - m^eq), w = -dt s ([16] or [16][nodes])."""
    m = M @ f.reshape(16, -1)
    m = m - _equilibria(m[0], m[1], m[2], m[3])
    return (Minv @ (w.reshape(16, -1) * m)).reshape(f.shape)


def _ghost(M, Minv, kind, state, first, second, opposite, normal):
    if kind == "periodic":
        return opposite
    q1 = _fields_of(M, first)
    if kind == "eq":
        return _feq(Minv, *[torch.full_like(q1[0], s) for s in state])
    if kind == "reflect":
        q1[1 + normal] = -q1[1 + normal]
        return _feq(Minv, *q1)
    q = 2 * q1 - _fields_of(M, second)  # "extrap"
    return _feq(Minv, *torch.where((q[0] > 0) & (q[3] > 0), q, q1))


def _exact_grid(case, seed):
    dx, dt, s, bc, fields = _flow(case, seed)
    Mn, In = _moment_matrix()
    M, Minv, vel = _dev(Mn), _dev(In), _velocities()
    w = _dev([0.0] * 4 + [-dt * k for k in s[4:]])
    f = _feq(Minv, *fields)
    ax, ay = (_dev(vel[:, k] * dt / dx)[:, None, None] for k in (0, 1))
    for n in range(case["steps"]):
        lines = []
        for side in range(4):
            axis = 2 if side < 2 else 1
            size = f.shape[axis]
            at = [0, min(1, size - 1), size - 1] if side % 2 == 0 else [size - 1, max(size - 2, 0), 0]
            a, b, c = (f.select(axis, k) for k in at)
            kind, state = bc[side][0], bc[side][1]
            g = _ghost(M, Minv, kind, state, a, b, c, side // 2)
            if len(bc[side]) > 2:
                far, s0, s1 = bc[side][2]
                pos = (torch.arange(g.shape[1], device="cuda", dtype=torch.float64) + 0.5) * dx
                g = torch.where(pos <= s0 + s1 * n * dt, g,
                                _ghost(M, Minv, far, state, a, b, c, side // 2))
            lines.append(g.unsqueeze(axis))
        new = f + _collision(M, Minv, f, w)
        E, W_ = torch.cat([f[:, :, 1:], lines[1]], 2), torch.cat([lines[0], f[:, :, :-1]], 2)
        new += 0.5 * ax * ax * (E - 2 * f + W_) - 0.5 * ax * (E - W_)
        N, S_ = torch.cat([f[:, 1:], lines[3]], 1), torch.cat([lines[2], f[:, :-1]], 1)
        new += 0.5 * ay * ay * (N - 2 * f + S_) - 0.5 * ay * (N - S_)
        f = new
    out = {"f": f}
    if case["precision"] in ("fp64", "df64"):
        out["fields"] = _fields_of(M, f)
    return out


def _exact_tubes(case, seed):
    nx, dx, dt, s, left, right = _tubes(case, seed)
    fields, tube, at = _tube_fields(nx, left, right)
    Mn, In = _moment_matrix()
    M, Minv = _dev(Mn), _dev(In)
    gl, gr = (_feq(Minv, *_dev(e.T))[:, tube] for e in (left, right))
    w = -dt * _dev(s.T)[:, tube]
    w[:4] = 0
    a = _dev(_velocities()[:, 0])[:, None] * (dt / _dev(dx))[tube]
    first, last = at == 0, at == torch.as_tensor(nx, device="cuda")[tube] - 1
    f = _feq(Minv, *fields)
    for _ in range(case["steps"]):
        E = torch.where(last, gr, torch.roll(f, -1, 1))
        W_ = torch.where(first, gl, torch.roll(f, 1, 1))
        f = f + _collision(M, Minv, f, w) + 0.5 * a * a * (E - 2 * f + W_) - 0.5 * a * (E - W_)
    return {"fields": _fields_of(M, f)}


def _features(q):
    return torch.stack([torch.log(q[0]), q[1], q[2], torch.log(q[3])])


def _network(params, x):
    h, o = x[None], 0
    for l, (cin, cout) in enumerate(_layers()):
        w = params[o:o + 9 * cin * cout].reshape(3, 3, cin, cout).permute(3, 2, 0, 1)
        o += 9 * cin * cout
        cols = torch.nn.functional.unfold(h, 3, padding=1)[0]  # [cin * 9][pixels]
        h = w.reshape(cout, -1) @ cols + params[o:o + cout, None]
        o += cout
        h = h.reshape(1, cout, *x.shape[1:])
        h = torch.relu(h) if l < len(_layers()) - 1 else h
    return h[0]


def _exact_cnn(case, seed):
    coarse, target = _pair(case, seed)
    x, t = _features(coarse), _features(target)
    scale = (t - x).square().mean(dim=(1, 2)).sqrt()[:, None, None]
    p = _dev(_params(seed)).requires_grad_(case["kind"] == "train")
    out = x + scale * _network(p, x)
    if case["kind"] == "infer":
        return {"fields": torch.stack([torch.exp(out[0]), out[1], out[2], torch.exp(out[3])]),
                "fallback": None}
    d = out - t
    loss = (d.square() if case["loss"] == "mse" else d.abs()).mean()
    loss.backward()
    # Adam's first step: both moments are the gradient's own after correction.
    new = p.detach() - 1e-3 * p.grad / (p.grad.abs() + 1e-8)
    return {"loss": np.float64(loss.item()), "params": new}


def _exact_vn(case, seed):
    _, k, states, rates, dx, dt = _vn(case, seed)
    Mn, In = _moment_matrix()
    M, Minv, vel = _dev(Mn), _dev(In), _velocities()
    ax, ay = vel[:, 0] * dt / dx, vel[:, 1] * dt / dx
    ex, ey = np.exp(1j * k[:, :1] * dx), np.exp(1j * k[:, 1:] * dx)
    diag = (1.0 + 0.5 * ax ** 2 * (ex - 2 + 1 / ex) - 0.5 * ax * (ex - 1 / ex)
            + 0.5 * ay ** 2 * (ey - 2 + 1 / ey) - 0.5 * ay * (ey - 1 / ey))
    out = np.empty((len(states), len(k)))
    for c, (rho, u, v, T) in enumerate(states):
        cons = _dev([rho, rho * u, rho * v, rho * T + 0.5 * rho * (u * u + v * v)])
        J = torch.autograd.functional.jacobian(lambda q: _equilibria(q[0], q[1], q[2], q[3]), cons)
        w = -dt * _dev(rates[c])
        w[:4] = 0
        C = (Minv @ (w[:, None] * (M - J @ M[:4]))).cpu().numpy()
        G = C[None] + diag[:, :, None] * np.eye(16)[None]
        out[c] = np.abs(np.linalg.eigvals(G)).max(axis=1)
    return {"radius": out, "failed": None}


def exact(case, seed):
    kind = case["kind"]
    if kind == "grid":
        return _exact_grid(case, seed)
    if kind == "tubes":
        return _exact_tubes(case, seed)
    if kind in ("train", "infer"):
        return _exact_cnn(case, seed)
    return _exact_vn(case, seed)
