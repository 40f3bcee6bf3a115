"""Workloads of the library through its public entry points, for timing and for comparing results.

listed() and draw() name cases, prepare() makes what a user's program holds before the call (inputs on the GPU, a
plan or a network context), run() makes one pass, work() counts what the pass cannot do without, and exact() gives
the results in 64 bits from plain torch.  Everything random comes from the seed given to prepare().
"""
import math

import numpy as np
import torch

import paper_1805_07801_gb300 as fk

DEV = "cuda:0"
SCHEMES = {"rk2": fk.TARANG_RK2, "rk4": fk.TARANG_RK4}
RBC_BASES = {"fff": fk.TARANG_RBC_FFF, "sff": fk.TARANG_RBC_SFF}
MLP_DIMS = (5, 64, 64, 64, 6)
ADAM = (0.9, 0.999, 1e-8)
ADAM_STEP, LEARNING_RATE = 1000, 1e-3
PAIRS = ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))  # order of the six stress components


def listed():
    return [
        # the smallest transform a program makes in a loop (64^3 is the plain method's test size): launches count
        {"name": "fft_64", "kind": "fft", "nx": 64, "ny": 64, "nz": 64, "batch": 1, "basis": "FFF"},
        # the headline forward and inverse pair on a large cube
        {"name": "fft_1024", "kind": "fft", "nx": 1024, "ny": 1024, "nz": 1024, "batch": 1, "basis": "FFF"},
        # several fields on a box with different axes, two of them with the factor 3
        {"name": "fft_box", "kind": "fft", "nx": 384, "ny": 64, "nz": 192, "batch": 5, "basis": "FFF"},
        # two free-slip directions, one periodic
        {"name": "fft_ssf_512", "kind": "fft", "nx": 512, "ny": 512, "nz": 512, "batch": 1, "basis": "SCF"},
        # a coarse turbulence run: steps so short that launches count
        {"name": "ns_64", "kind": "ns", "n": 64, "scheme": "rk2", "force": False, "model": False},
        # the same with forcing and the learned subgrid stress in the right-hand side
        {"name": "ns_64_model", "kind": "ns", "n": 64, "scheme": "rk2", "force": True, "model": True},
        # the headline decaying-turbulence step
        {"name": "ns_512", "kind": "ns", "n": 512, "scheme": "rk2", "force": False, "model": False},
        # the grid of the published cluster runs (3 * 2^m)
        {"name": "ns_768", "kind": "ns", "n": 768, "scheme": "rk2", "force": False, "model": False},
        # convection in the periodic cube with the published scheme (52 transforms per step)
        {"name": "rbc_fff_512", "kind": "rbc", "n": 512, "scheme": "rk4", "basis": "fff"},
        # convection between free-slip plates
        {"name": "rbc_sff_256", "kind": "rbc", "n": 256, "scheme": "rk4", "basis": "sff"},
        # one training step of the closure network at the batch of its published schedule
        {"name": "train_65536", "kind": "train", "batch": 65536},
        # shell-to-shell transfer of a stored snapshot over octave shells
        {"name": "shells_256", "kind": "shells", "n": 256},
    ]


def _dim(rng, lo, hi):
    """An axis length 2^a or 3 * 2^a in [lo, hi], spread over the logarithm."""
    all_ = sorted({f << a for f in (1, 3) for a in range(12) if lo <= (f << a) <= hi and (f == 1 or (f << a) >= 12)})
    return rng.choice(all_)


def draw(rng):
    kind = rng.choices(("fft", "ns", "rbc", "train", "shells", "transfer"), (8, 6, 3, 3, 1, 2))[0]
    k0 = round(rng.uniform(2.0, 6.0), 1)  # where the spectrum of a state peaks
    if kind == "fft":
        while True:
            basis = rng.choices(("FFF", "SFF", "CSF", "SCF", "CCS", "SSC"), (10, 2, 1, 1, 1, 1))[0]
            nx, ny, nz = (_dim(rng, 16, 1024) for _ in range(3))
            if basis != "FFF":
                nx, ny, nz = (1 << (v.bit_length() - 1) for v in (nx, ny, nz))
            most = 2 ** rng.uniform(15, 30)
            batch = int(most / (nx * ny * nz))
            if batch >= 1:
                return {"kind": kind, "nx": nx, "ny": ny, "nz": nz, "batch": min(batch, rng.choice((1, 2, 3, 5, 7, 12, 31))),
                        "basis": basis}
    if kind == "ns":
        model = rng.random() < 0.25
        n = rng.choice((32, 64, 128)) if model else rng.choice((32, 48, 64, 96, 128, 192, 256, 384, 512, 768))
        scheme = "rk2" if n > 512 else rng.choice(("rk2", "rk4"))
        return {"kind": kind, "n": n, "scheme": scheme, "force": rng.random() < 0.5, "model": model, "k0": k0}
    if kind == "rbc":
        basis = rng.choice(("fff", "sff"))
        n = rng.choice((32, 64, 128, 256, 512) if basis == "sff" else (32, 48, 64, 96, 128, 192, 256, 384, 512))
        return {"kind": kind, "n": n, "scheme": rng.choice(("rk2", "rk4")), "basis": basis, "k0": k0}
    if kind == "train":
        return {"kind": kind, "batch": int(2 ** rng.uniform(8, 18))}
    return {"kind": kind, "n": rng.choice((32, 64, 128, 256) if kind == "shells" else (48, 64, 96, 128, 192, 256, 384, 512)),
            "k0": k0}


# ---------------------------------------------------------------- inputs --


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _axes(n, dtype):
    k = torch.fft.fftfreq(n, 1.0 / n, device=DEV, dtype=dtype)
    return k[:, None, None], k[None, :, None], torch.arange(n // 2 + 1, device=DEV, dtype=dtype)[None, None, :]


def _amplitude(k2, k0, n):
    """Per-mode amplitude of a broad turbulence spectrum with its peak near k0 and a tail to the last kept modes."""
    E = k2 ** 2 / (1.0 + k2 / k0 ** 2) ** (17.0 / 6.0) * torch.exp(-6.0 * torch.sqrt(k2) / n)
    return torch.sqrt(E / torch.clamp(k2, min=1.0))


def _kept(n):
    kx, ky, kz = _axes(n, torch.float32)
    return (3 * kx.abs() < n) & (3 * ky.abs() < n) & (3 * kz < n)


def _scaled(u, total):
    """Fields with 1/2 sum w |u|^2 = total (w = 1 on k_z = 0, else 2)."""
    e = sum(0.5 * (2.0 * f.abs().double().square().sum() - f[..., 0].abs().double().square().sum()) for f in u)
    return u * float(math.sqrt(total / float(e)))


def _turbulence(n, fields, seed, k0, energy=0.5):
    """Random-phase spectra [fields][n][n][n/2+1], 2/3-truncated; the first three are solenoidal."""
    g = _gen(seed)
    kx, ky, kz = _axes(n, torch.float32)
    k2 = kx * kx + ky * ky + kz * kz
    a = _amplitude(k2, k0, n) * _kept(n)
    u = torch.empty((fields, n, n, n // 2 + 1), dtype=torch.complex64, device=DEV)
    for f in range(fields):
        u[f] = torch.fft.rfftn(torch.randn((n, n, n), generator=g, device=DEV), norm="forward") * a
    k2[0, 0, 0] = 1.0
    d = (kx * u[0] + ky * u[1] + kz * u[2]) / k2
    for f, k in enumerate((kx, ky, kz)):
        u[f] -= k * d
    del d, a, k2
    u[..., 0] = 0.5 * (u[..., 0] + torch.roll(torch.flip(u[..., 0], (1, 2)), (1, 1), (1, 2)).conj())  # Hermitian plane
    u[:, 0, 0, 0] = 0
    return _scaled(u, energy)


def _plates(n, seed, k0):
    """Convection state between plates: u_x and theta in sine series along x, u_y and u_z in cosine series."""
    g = _gen(seed)
    ky, kz = _axes(n, torch.float32)[1:]
    kx = torch.arange(n, device=DEV, dtype=torch.float32)[:, None, None]  # cosine rows; a sine row a is k_x = a + 1
    keep_yz = (3 * ky.abs() < n) & (3 * kz < n)
    s = torch.empty((4, n, n, n // 2 + 1), dtype=torch.complex64, device=DEV)
    for f in range(4):
        k = kx + 1 if f in (0, 3) else kx
        k2 = k * k + ky * ky + kz * kz
        white = torch.fft.rfftn(torch.randn((n, n, n), generator=g, device=DEV), dim=(1, 2), norm="forward")
        s[f] = white * (_amplitude(k2, k0, n) * ((3 * k < 2 * n) & keep_yz))
    s[..., 0] = 0.5 * (s[..., 0] + torch.roll(torch.flip(s[..., 0], (2,)), 1, 2).conj())
    ux = torch.zeros_like(s[0])  # the sine rows at their cosine place
    ux[1:] = s[0, :-1]
    k2 = kx * kx + ky * ky + kz * kz
    k2[0, 0, 0] = 1.0
    p = -(kx * ux + 1j * (ky * s[1] + kz * s[2])) / k2
    s[1] -= 1j * ky * p
    s[2] -= 1j * kz * p
    s[0, :-1] += (kx * p)[1:]
    return _scaled(s, 0.5)


def _network(seed):
    """Parameters of a trained-scale network: uniform in +-1/sqrt(fan in), in the library's order."""
    g = _gen(seed)
    parts = []
    for din, dout in zip(MLP_DIMS, MLP_DIMS[1:]):
        for shape in (dout * din, dout):
            parts.append((2 * torch.rand(shape, generator=g, device=DEV) - 1) / math.sqrt(din))
    return torch.cat(parts)


def _physics(case):
    n = case["n"]
    return {"nu": 0.64 / n, "dt": 0.064 / n, "eps": 0.1, "k2": (1, 4), "Ra": 1e6 * (n / 64.0) ** 2, "Pr": 1.0}


MODEL_SHIFT, MODEL_SCALE, MODEL_OUT = (2.0, -2.0, 0.0, 0.0, -2.0), (0.2, 0.2, 0.1, 0.1, 0.05), (4e-3, 4e-3, 4e-3, 2e-3, 2e-3, 2e-3)


def _bounds(n):
    """Octave shells from 0 to the largest shell of the kept set."""
    b = [0, 1, 2]
    while b[-1] * 2 < n // 3:
        b.append(b[-1] * 2)
    return b + [int(math.sqrt(3.0) * ((n - 1) // 3) + 0.5) + 1]


class _Handle:
    """A plan or network context, given back with the state that holds it."""

    def __init__(self, handle, destroy):
        self.h, self.destroy = handle, destroy

    def __del__(self):
        self.destroy(self.h)


def _plan(nx, ny, nz):
    return _Handle(fk.fftk_plan_create(nx, ny, nz), fk.fftk_plan_destroy)


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case, "stream": torch.cuda.current_stream().cuda_stream}
    if kind == "fft":
        nx, ny, nz, b = case["nx"], case["ny"], case["nz"], case["batch"]
        s["plan"] = _plan(nx, ny, nz)
        s["x"] = torch.randn((b, nx, ny, nz), generator=_gen(seed), device=DEV)
        if case["basis"][2] == "F":
            s["F"] = torch.empty((b, nx, ny, nz // 2 + 1), dtype=torch.complex64, device=DEV)
        else:
            s["F"] = torch.empty((b, nx, ny, nz), device=DEV)
        s["back"] = torch.empty_like(s["x"])
    elif kind == "train":
        b, g = case["batch"], _gen(seed)
        s["mlp"] = _Handle(fk.tarang_mlp_create(b), fk.tarang_mlp_destroy)
        s["params"] = _network(seed + 1000003)
        s["x"] = torch.randn((b, 5), generator=g, device=DEV)
        s["x"] *= s["x"].abs() ** 0.5  # heavier tails, as the invariants have
        s["t"] = torch.tanh(s["x"][:, (0, 1, 2, 3, 4, 0)]) + 0.5 * torch.randn((b, 6), generator=g, device=DEV)
        s["m"] = 1e-3 * torch.randn(s["params"].shape, generator=g, device=DEV)
        s["v"] = 1e-6 * (0.5 + torch.rand(s["params"].shape, generator=g, device=DEV))
        s["loss"] = torch.zeros(1, dtype=torch.float64, device=DEV)
    else:
        n, p, k0 = case["n"], _physics(case), case.get("k0", 4.0)
        s["plan"] = _plan(n, n, n)
        if kind == "rbc":
            s["u"] = _plates(n, seed, k0) if case["basis"] == "sff" else _turbulence(n, 4, seed, k0)
            s["physics"] = p
        else:
            s["u"] = _turbulence(n, 3, seed, k0)
        if kind == "ns":
            model = None
            if case["model"]:
                s["net"] = _network(seed + 1000003)
                model = fk.make_sgs_model(s["net"].data_ptr(), MODEL_SHIFT, MODEL_SCALE, MODEL_OUT)
            s["params"] = fk.make_params(p["nu"], p["dt"], p["eps"] if case["force"] else 0.0, p["k2"], model,
                                         SCHEMES[case["scheme"]])
    return s


def run(s):
    case, st = s["case"], s["stream"]
    kind = case["kind"]
    if kind == "fft":
        x, F, back, b, plan = s["x"], s["F"], s["back"], case["batch"], s["plan"].h
        if case["basis"] == "FFF":
            fk.fftk_r2c(plan, x.data_ptr(), F.data_ptr(), b, st)
            fk.fftk_c2r(plan, F.data_ptr(), back.data_ptr(), b, st)
        else:
            fk.fftk_forward(plan, case["basis"], x.data_ptr(), F.data_ptr(), b, st)
            fk.fftk_inverse(plan, case["basis"], F.data_ptr(), back.data_ptr(), b, st)
        return {"spectrum": F, "back": back}
    if kind == "ns":
        fk.tarang_ns_step(s["plan"].h, s["u"].data_ptr(), s["params"], 1, False, st)
        return {"u": s["u"]}
    if kind == "rbc":
        p = s["physics"]
        fk.tarang_rbc_step(s["plan"].h, s["u"].data_ptr(), p["Ra"], p["Pr"], p["dt"], 1, SCHEMES[case["scheme"]], st,
                           RBC_BASES[case["basis"]])
        return {"state": s["u"]}
    if kind == "train":
        fk.tarang_mlp_train_step(s["mlp"].h, s["params"].data_ptr(), s["m"].data_ptr(), s["v"].data_ptr(), ADAM_STEP,
                                 s["x"].data_ptr(), s["t"].data_ptr(), case["batch"], LEARNING_RATE,
                                 s["loss"].data_ptr(), st)
        # the loss is a 64-bit sum of 32-bit errors: it is logged in 32 bits
        return {"params": s["params"], "m": s["m"], "v": s["v"], "loss": s["loss"].float()}
    if kind == "shells":
        T = fk.tarang_shell_transfer(s["plan"].h, s["u"].data_ptr(), _bounds(case["n"]), st)
        return {"T": np.asarray(T, dtype=np.float32)}  # 64-bit sums of a 32-bit nonlinear term
    _, T, _ = fk.tarang_transfer(s["plan"].h, s["u"].data_ptr(), None, st)
    return {"T": np.asarray(T, dtype=np.float32)}  # (the flux is the host's running sum of it)


def work(case):
    """Bytes with each input read once and each output written once, and the operations of the transforms (2.5 N log2 N
    for a real one of N points), products and layers."""
    kind = case["kind"]
    if kind == "train":
        macs = sum(a * b for a, b in zip(MLP_DIMS, MLP_DIMS[1:]))
        params = sum((a + 1) * b for a, b in zip(MLP_DIMS, MLP_DIMS[1:]))
        return {"bytes": 4.0 * (11 * case["batch"] + 6 * params), "flops": 2.0 * case["batch"] * (3 * macs - 5 * 64)}
    if kind == "fft":
        r = case["batch"] * case["nx"] * case["ny"] * case["nz"]
        f = case["batch"] * case["nx"] * case["ny"] * (case["nz"] // 2 + 1) * 8 if case["basis"][2] == "F" else 4 * r
        return {"bytes": 8.0 * r + 2.0 * f, "flops": 2 * 2.5 * r * math.log2(case["nx"] * case["ny"] * case["nz"])}
    n = case["n"]
    kd = (n - 1) // 3
    fields = 4 if kind == "rbc" else 3
    rows = (2 * n - 1) // 3 + 1 if case.get("basis") == "sff" else 2 * kd + 1
    state = 8.0 * fields * rows * (2 * kd + 1) * (kd + 1)
    stages = {"rk2": 2, "rk4": 4}.get(case.get("scheme"), 1)
    one = 2.5 * n ** 3 * 3 * math.log2(n)
    if kind == "ns":
        b = 2 * state
        f = stages * 9 * one + (stages * (15 * one + 4.0 * 8896 * n ** 3) if case["model"] else 0)
    elif kind == "rbc":
        b, f = 2 * state, stages * 13 * one
    elif kind == "transfer":
        b, f = state, 9 * one
    else:
        b, f = state, (3 + 12 * (len(_bounds(n)) - 1)) * one
    return {"bytes": b, "flops": f}


# --------------------------------------------------- results in 64 bits ---


def _to_real(u, n):
    return torch.fft.irfftn(u, s=(n, n, n), dim=(-3, -2, -1), norm="forward")


def _to_spec(r):
    return torch.fft.rfftn(r, dim=(-3, -2, -1), norm="forward")


def _cross(a, b, c):
    i, j = (c + 1) % 3, (c + 2) % 3
    return a[i] * b[j] - a[j] * b[i]


def _curl(u, k):
    return [1j * (k[(c + 1) % 3] * u[(c + 2) % 3] - k[(c + 2) % 3] * u[(c + 1) % 3]) for c in range(3)]


def _project(v, k, k2):
    d = sum(k[c] * v[c] for c in range(3)) / k2
    for c in range(3):
        v[c] -= k[c] * d
        v[c][0, 0, 0] = 0
    return v


def _modes(n):
    k = _axes(n, torch.float64)
    k2 = k[0] ** 2 + k[1] ** 2 + k[2] ** 2
    safe = k2.clone()
    safe[0, 0, 0] = 1.0
    return k, k2, safe, _kept(n)


def _bf16(x):
    return x.to(torch.bfloat16).double()


def _layers(params):
    at, out = 0, []
    for din, dout in zip(MLP_DIMS, MLP_DIMS[1:]):
        w = params[at:at + dout * din].double().view(dout, din)
        b = params[at + dout * din:at + dout * (din + 1)].double()
        out.append((w, b))
        at += dout * (din + 1)
    return out


def _stress_force(u, net, n, k, safe, keep):
    """P[-i k_j tau_ij] of the network's stress (five invariants in, the stress in the strain eigenframe out)."""
    A = torch.stack([torch.stack([_to_real(1j * k[j] * (torch.abs(2 * k[j]) != n) * u[i], n) for j in range(3)], -1) for i in range(3)], -2).reshape(-1, 3, 3)
    S, R = 0.5 * (A + A.mT), 0.5 * (A - A.mT)
    tr = lambda m: m.diagonal(dim1=-2, dim2=-1).sum(-1)  # noqa: E731
    S2, R2 = S @ S, R @ R
    inv = torch.stack([tr(S2), tr(R2), tr(S2 @ S), tr(R2 @ S), tr(R2 @ S2)], -1)
    Q = torch.linalg.eigh(S.cpu())[1].to(DEV).flip(-1)  # (the batch is too large for the GPU's solver)
    big = Q.gather(-2, Q.abs().argmax(-2, keepdim=True))
    Q = Q * torch.where(big < 0, -1.0, 1.0)
    h = (inv - torch.tensor(MODEL_SHIFT, device=DEV, dtype=torch.float64)) * torch.tensor(MODEL_SCALE, device=DEV, dtype=torch.float64)
    for i, (w, b) in enumerate(_layers(net)):
        h = _bf16(h) @ w.T + b
        h = torch.tanh(h) if i < 3 else h
    h = h * torch.tensor(MODEL_OUT, device=DEV, dtype=torch.float64)
    T = torch.empty_like(A)
    for c, (i, j) in enumerate(PAIRS):
        T[:, i, j] = T[:, j, i] = h[:, c]
    tau = (Q @ T @ Q.mT).reshape(n, n, n, 3, 3)
    f = [-1j * sum(k[j] * _to_spec(tau[..., i, j].contiguous()) for j in range(3)) * keep for i in range(3)]
    return _project(f, k, safe)


def _ns_term(u, case, n, modes, net=None):
    k, k2, safe, keep = modes
    ur = [_to_real(c, n) for c in u]
    wr = [_to_real(c, n) for c in _curl(u, k)]
    v = [_to_spec(_cross(ur, wr, c)) * keep for c in range(3)]
    del ur, wr
    v = _project(v, k, safe)
    if net is not None:
        v = [a + b for a, b in zip(v, _stress_force(u, net, n, k, safe, keep))]
    if case.get("force"):
        p = _physics(case)
        band = (k2 >= p["k2"][0]) & (k2 <= p["k2"][1])
        w = torch.where(k[2] == 0, 1.0, 2.0)
        e = 0.5 * sum((w * c.abs() ** 2)[band].sum() for c in u)
        v = [a + p["eps"] / (2 * e) * torch.where(band, c, 0) for a, c in zip(v, u)]
    return v


def _advance(u, term, E, H, dt, scheme):
    """One step with the integrating factors E (whole step) and H (half step), one per field."""
    def lin(*pairs):
        return [sum(a * x[c] if not isinstance(a, list) else a[c] * x[c] for a, x in pairs) for c in range(len(u))]

    if scheme == "rk2":
        u1 = lin((E, lin((1.0, u), (dt, term(u)))))
        n1 = term(u1)
        return lin((0.5, lin((E, u))), (0.5, u1), (0.5 * dt, n1))
    n1 = term(u)
    n2 = term(lin((H, lin((1.0, u), (0.5 * dt, n1)))))
    acc = lin((E, u), (dt / 6, lin((E, n1))), (dt / 3, lin((H, n2))))
    del n1
    n3 = term(lin((H, u), (0.5 * dt, n2)))
    del n2
    hn3 = lin((H, n3))
    del n3
    n4 = term(lin((E, u), (dt, hn3)))
    return lin((1.0, acc), (dt / 3, hn3), (dt / 6, n4))


def _exact_ns(case, s):
    n, p = case["n"], _physics(case)
    modes = _modes(n)
    u = [c.to(torch.complex128) for c in s["u"]]
    E = torch.exp(-p["nu"] * p["dt"] * modes[1])
    H = torch.exp(-0.5 * p["nu"] * p["dt"] * modes[1])
    u = _advance(u, lambda v: _ns_term(v, case, n, modes, s.get("net")), [E] * 3, [H] * 3, p["dt"], case["scheme"])
    return torch.stack(u)


def _rbc_factors(k2, p):
    nu, kappa = math.sqrt(p["Pr"] / p["Ra"]), 1.0 / math.sqrt(p["Ra"] * p["Pr"])
    f = [[torch.exp(-c * h * p["dt"] * k2) for c in (nu, kappa)] for h in (1.0, 0.5)]
    return [[a] * 3 + [b] for a, b in f]


def _exact_rbc_cube(case, s):
    n, p = case["n"], _physics(case)
    k, k2, safe, keep = _modes(n)

    def term(x):
        ur, tr = [_to_real(c, n) for c in x[:3]], _to_real(x[3], n)
        wr = [_to_real(c, n) for c in _curl(x, k)]
        v = [_to_spec(_cross(ur, wr, c)) * keep for c in range(3)]
        v[2] = v[2] + x[3]
        t = -1j * sum(k[c] * _to_spec(ur[c] * tr) for c in range(3)) * keep + x[2]
        t[0, 0, 0] = 0
        return _project(v, k, safe) + [t]

    E, H = _rbc_factors(k2, p)
    return torch.stack(_advance([c.to(torch.complex128) for c in s["u"]], term, E, H, p["dt"], case["scheme"]))


def _sc_matrix(n, sine, inverse):
    """The dense sine or cosine transform of n points s_j = (j + 1/2) pi / n."""
    j = (torch.arange(n, device=DEV, dtype=torch.float64) + 0.5) * math.pi / n
    k = torch.arange(n, device=DEV, dtype=torch.float64) + (1 if sine else 0)
    m = torch.sin(j[:, None] * k) if sine else torch.cos(j[:, None] * k)
    if inverse:
        return 2.0 * m
    f = m.T / n
    f[-1 if sine else 0] *= 0.5
    return f.contiguous()


def _along(m, x, axis):
    if x.is_complex():
        return torch.complex(_along(m, x.real, axis), _along(m, x.imag, axis))
    y = x.movedim(axis, 0)
    return (m @ y.reshape(y.shape[0], -1)).reshape(y.shape).movedim(0, axis)


def _exact_rbc_plates(case, s):
    n, p = case["n"], _physics(case)
    ky, kz = _axes(n, torch.float64)[1:]
    a = torch.arange(n, device=DEV, dtype=torch.float64)[:, None, None]
    keep_yz = (3 * ky.abs() < n) & (3 * kz < n)
    yz2 = ky ** 2 + kz ** 2
    kc, ks = a, a + 1  # wavenumber of a cosine row, of a sine row
    keep_c, keep_s = keep_yz & (3 * kc < 2 * n), keep_yz & (3 * ks < 2 * n)
    mat = {(q, i): _sc_matrix(n, q, i) for q in (False, True) for i in (False, True)}
    real = lambda x, q: torch.fft.irfft2(_along(mat[q, True], x, 0), s=(n, n), dim=(1, 2), norm="forward")  # noqa: E731
    spec = lambda r, q: _along(mat[q, False], torch.fft.rfft2(r, dim=(1, 2), norm="forward"), 0)  # noqa: E731

    def up(x):  # sine rows at their cosine place
        return torch.cat([torch.zeros_like(x[:1]), x[:-1]])

    def down(x):  # cosine rows at their sine place
        return torch.cat([x[1:], torch.zeros_like(x[:1])])

    def term(x):
        ux, uy, uz, th = x
        wx = 1j * (ky * uz - kz * uy)
        wy = 1j * kz * ux - down(-kc * uz)
        wz = down(-kc * uy) - 1j * ky * ux
        ur = [real(ux, True), real(uy, False), real(uz, False)]
        wr = [real(wx, False), real(wy, True), real(wz, True)]
        tr = real(th, True)
        vx = spec(_cross(ur, wr, 0), True) * keep_s + th
        vy, vz = (spec(_cross(ur, wr, c), False) * keep_c for c in (1, 2))
        k2 = kc ** 2 + yz2
        k2[0, 0, 0] = 1.0
        pr = -(kc * up(vx) + 1j * (ky * vy + kz * vz)) / k2
        pr[0, 0, 0] = 0
        d = down(-kc * 0 + kc * spec(ur[0] * tr, False))  # d_x (cosine) = -k (sine)
        t = d - 1j * ky * spec(ur[1] * tr, True) - 1j * kz * spec(ur[2] * tr, True)
        return [vx + down(kc * pr), vy - 1j * ky * pr, vz - 1j * kz * pr, t * keep_s + ux]

    Es, Hs = _rbc_factors(ks ** 2 + yz2, p)
    Ec, Hc = _rbc_factors(kc ** 2 + yz2, p)
    E, H = [Es[0], Ec[1], Ec[2], Es[3]], [Hs[0], Hc[1], Hc[2], Hs[3]]
    return torch.stack(_advance([c.to(torch.complex128) for c in s["u"]], term, E, H, p["dt"], case["scheme"]))


def _exact_fft(case, s):
    b = case["basis"]
    x = s["x"].double()
    if b == "FFF":
        F = torch.fft.rfftn(x, dim=(1, 2, 3), norm="forward")
    else:
        F = torch.fft.rfft(x, dim=3, norm="forward") if b[2] == "F" else _along(_sc_matrix(case["nz"], b[2] == "S", False), x, 3)
        for axis, n in ((2, case["ny"]), (1, case["nx"])):
            if b[axis - 1] == "F":
                F = torch.fft.fft(F, dim=axis, norm="forward")
            else:
                F = _along(_sc_matrix(n, b[axis - 1] == "S", False), F, axis)
    return {"spectrum": F, "back": x}


def _exact_train(case, s):
    layers = _layers(s["params"])
    acts, h = [], s["x"].double()
    for i, (w, b) in enumerate(layers):
        acts.append(_bf16(h))
        h = acts[-1] @ w.T + b
        h = torch.tanh(h) if i < 3 else h
    e = h - s["t"].double()
    d = e * (2.0 / e.numel())
    grads = []
    for i in (3, 2, 1, 0):
        grads = [(d.T @ acts[i]).reshape(-1), d.sum(0)] + grads
        if i:
            d = (d @ layers[i][0]) * (1.0 - acts[i] ** 2)
    g = torch.cat(grads)
    b1, b2, eps = ADAM
    m = b1 * s["m"].double() + (1 - b1) * g
    v = b2 * s["v"].double() + (1 - b2) * g * g
    mh, vh = m / (1 - b1 ** ADAM_STEP), v / (1 - b2 ** ADAM_STEP)
    return {"params": s["params"].double() - LEARNING_RATE * mh / (torch.sqrt(vh) + eps), "m": m, "v": v,
            "loss": (e * e).mean().reshape(1)}


def _shell(k2):
    return torch.floor(torch.sqrt(k2) + 0.5).long()


def _exact_transfer(case, s):
    n = case["n"]
    modes = _modes(n)
    u = [c.to(torch.complex128) for c in s["u"]]
    v = _ns_term(u, {}, n, modes)
    w = torch.where(modes[0][2] == 0, 1.0, 2.0)
    size = int(math.floor(math.sqrt(3.0) * (n // 2) + 0.5)) + 2
    t = sum(w * (a.conj() * b).real for a, b in zip(u, v)) * modes[3]
    T = torch.zeros(size, dtype=torch.float64, device=DEV).scatter_add_(0, _shell(modes[1]).reshape(-1).clamp(max=size - 1), t.reshape(-1))
    return {"T": T.cpu().numpy()}


def _exact_shells(case, s):
    n = case["n"]
    k, k2, _, keep = _modes(n)
    u = [c.to(torch.complex128) for c in s["u"]]
    ur = [_to_real(c, n) for c in u]
    bounds, K = _bounds(n), _shell(k2)
    w = torch.where(k[2] == 0, 1.0, 2.0) * keep
    out = np.zeros((len(bounds) - 1, len(bounds) - 1))
    inside = [(K >= a) & (K < b) for a, b in zip(bounds, bounds[1:])]
    for g, giver in enumerate(inside):
        t = 0.0
        for i in range(3):
            adv = sum(ur[j] * _to_real(1j * k[j] * u[i] * giver, n) for j in range(3))
            t = t - w * (u[i].conj() * _to_spec(adv)).real
        for r, receiver in enumerate(inside):
            out[r, g] = float(t[receiver].sum())
    return {"T": out}


def exact(case, seed):
    if case.get("model") and case["n"] > 64:
        return None  # the eigenvectors of millions of matrices in 64 bits take too long
    s = prepare(case, seed)
    kind = case["kind"]
    if kind == "fft":
        return _exact_fft(case, s)
    if kind == "ns":
        return {"u": _exact_ns(case, s)}
    if kind == "rbc":
        return {"state": (_exact_rbc_plates if case["basis"] == "sff" else _exact_rbc_cube)(case, s)}
    if kind == "train":
        return _exact_train(case, s)
    return _exact_shells(case, s) if kind == "shells" else _exact_transfer(case, s)
