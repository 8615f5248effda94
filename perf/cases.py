"""Workloads of the library, each run through its public entry points.

listed() are the sizes that the configurations and benchmarks of this repository use;
draw() gives others of the same ranges (grid sides, batches, steps, precisions, layouts).
exact() is the same quantity in complex128 by plain torch: the pseudo-spectral step on the
n-point grid, IMEX RK443 from its tableaux, Parareal from its definition.
"""
import math

import numpy as np
import torch

import paper_1902_00387_gb300 as kd

RB, GP = kd.KD_FLOW_ROBERTS, kd.KD_FLOW_GALLOWAY_PROCTOR


def listed():
    return [
        # the 32^2 Roberts problem in complex128: one slice's 125 fine steps, all 8 slices
        {"name": "fine_roberts32_c128", "kind": "fine", "flow": RB, "n": 32, "kz": 1.0, "Rm": 8.0, "dt": 1e-2,
         "double": True, "conv": False, "kept": False, "batch": 8, "steps": 125},
        # Parareal's parallel step at 128^2: 64 slices, the 158 steps of a slice
        {"name": "fine_gp128", "kind": "fine", "flow": GP, "n": 128, "kz": 0.57, "Rm": 100.0, "dt": 4.97e-3,
         "double": False, "conv": False, "kept": False, "batch": 64, "steps": 158},
        # the coarse-resolution study's grid (N_F = 160, 10 slices), not a power of two
        {"name": "fine_roberts160", "kind": "fine", "flow": RB, "n": 160, "kz": 2.87, "Rm": 512.0, "dt": 1e-2,
         "double": False, "conv": False, "kept": False, "batch": 10, "steps": 100},
        # 256^2, 128 slices
        {"name": "fine_gp256", "kind": "fine", "flow": GP, "n": 256, "kz": 0.57, "Rm": 1000.0, "dt": 2.5e-3,
         "double": False, "conv": False, "kept": False, "batch": 128, "steps": 8},
        # Table 1's Roberts row at 512^2 in the kept-mode layout, an odd number of fields
        {"name": "fine_roberts512_kept", "kind": "fine", "flow": RB, "n": 512, "kz": 7.5, "Rm": 4096.0, "dt": 2.5e-3,
         "double": False, "conv": False, "kept": True, "batch": 45, "steps": 4},
        # the large run: one step of all 256 slices of 1024^2
        {"name": "fine_gp1024", "kind": "fine", "flow": GP, "n": 1024, "kz": 0.57, "Rm": 1e4, "dt": 1e-3,
         "double": False, "conv": False, "kept": False, "batch": 256, "steps": 1},
        # complex128 reference steps of the 128^2 problem
        {"name": "fine_gp128_c128", "kind": "fine", "flow": GP, "n": 128, "kz": 0.57, "Rm": 100.0, "dt": 4.97e-3,
         "double": True, "conv": False, "kept": False, "batch": 64, "steps": 10},
        # the convolution form of the fine operator on the same 128^2 slices
        {"name": "conv_gp128", "kind": "fine", "flow": GP, "n": 128, "kz": 0.57, "Rm": 100.0, "dt": 4.97e-3,
         "double": False, "conv": True, "kept": False, "batch": 64, "steps": 158},
        # one slice of Parareal's serial sweep: 51 coarse steps of one field
        {"name": "coarse_gp128", "kind": "coarse", "flow": GP, "n": 128, "nc": 128, "kz": 0.57, "Rm": 100.0,
         "dt": 2.0 / 128, "double": False, "batch": 1, "steps": 51},
        # a whole Parareal solve: 128^2, 64 slices over [0, 16 pi], stopped at 1e-6
        {"name": "parareal_gp128", "kind": "parareal", "flow": GP, "n": 128, "nc": 128, "kz": 0.57, "Rm": 100.0,
         "dt": 5e-3, "dtc": 2.0 / 128, "T": 16 * math.pi, "slices": 64, "k_max": 64, "tol": 1e-6},
        # a batched sweep of uneven instances (their grid sides grow with Rm), two iterations
        {"name": "sweep_uneven", "kind": "sweep", "n_lo": 64, "n_hi": 256, "instances": 7, "T": 1.0, "slices": 32,
         "k_max": 2},
        # loss and gradient of the learned coarse operator on |k| <= 24, one phase's 256 pairs
        {"name": "learned_grad49", "kind": "learned", "n": 256, "m": 49, "pairs": 256},
    ]


def _even(rng, lo, hi):
    """An even integer, uniform in the logarithm."""
    return max(lo, min(hi, 2 * round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / 2)))


def _log_int(rng, lo, hi):
    return max(lo, min(hi, round(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def _side(rng, lo, hi):
    """A grid side the FFT operator takes: any even one to 286, else 512 or 1024."""
    n = _even(rng, lo, hi)
    if n > 286:
        return 512 if n < 724 else 1024
    if rng.random() < 0.5:
        return n
    return min((32, 64, 96, 128, 160, 192, 256), key=lambda s: abs(math.log(s / n)))


def draw(rng):
    kind = rng.choice(["fine"] * 6 + ["double"] * 2 + ["conv", "coarse", "coarse", "parareal", "sweep", "learned"])
    flow = rng.choice([RB, GP])
    kz = round(rng.uniform(0.2, 1.5), 3)
    if kind in ("fine", "double", "conv"):
        n = _side(rng, 32, {"fine": 1024, "double": 256, "conv": 190}[kind]) if kind != "conv" else _even(rng, 32, 190)
        budget = {"fine": 1.6e8, "double": 5e6, "conv": 1.2e8}[kind]
        batch = _log_int(rng, 1, max(1, min(256, int(budget / n ** 2))))
        steps = _log_int(rng, 1, max(1, min(200, int(budget / n ** 2 / batch))))
        return {"kind": "fine", "flow": flow, "n": n, "kz": kz, "Rm": round(8.0 * (n / 32.0) ** 2, 2),
                "dt": 0.64 / n, "double": kind == "double", "conv": kind == "conv",
                "kept": kind == "fine" and rng.random() < 0.4, "batch": batch, "steps": steps}
    if kind == "coarse":
        n = _side(rng, 64, 512)
        nc = _even(rng, 16, min(n, 190))
        batch = _log_int(rng, 1, 64)
        return {"kind": "coarse", "flow": flow, "n": n, "nc": nc, "kz": kz, "Rm": round(8.0 * (n / 32.0) ** 2, 2),
                "dt": 2.0 / nc, "double": rng.random() < 0.3, "batch": batch, "steps": _log_int(rng, 4, 64)}
    if kind == "parareal":
        n = _side(rng, 32, 192)
        slices = _log_int(rng, 8, 64)
        return {"kind": "parareal", "flow": flow, "n": n, "nc": _even(rng, max(16, n // 2), n), "kz": kz,
                "Rm": round(8.0 * (n / 32.0) ** 2, 2), "dt": 0.64 / n, "dtc": 2.0 / n, "T": slices * 32 * 0.64 / n,
                "slices": slices, "k_max": 2, "tol": 0.0}
    if kind == "sweep":
        return {"kind": "sweep", "n_lo": 64, "n_hi": 128, "instances": rng.randint(2, 6), "T": 1.0,
                "slices": rng.randint(8, 32), "k_max": 2}
    return {"kind": "learned", "n": 256, "m": rng.randint(16, 49), "pairs": _log_int(rng, 64, 512)}


# ---------------------------------------------------------------------------- inputs
def _waves(n):
    i = torch.arange(n, device="cuda")
    return torch.where(i < n // 2, i, i - n).to(torch.float64)


def _mask(n, K):
    k = _waves(n).abs() <= K
    return k[:, None] & k[None, :]


def _fields(n, kz, batch, seed, dtype):
    """Seeded solenoidal fields [batch][3][n][n] with a |k3|^-2 spectrum and unit norm."""
    g = torch.Generator(device="cuda").manual_seed(1000003 * (seed + 1) + n)
    out = torch.empty((batch, 3, n, n), dtype=dtype, device="cuda")
    work = torch.complex64 if n >= 512 and dtype == torch.complex64 else torch.complex128
    k = _waves(n)
    kk = torch.stack(torch.broadcast_tensors(k[None, :], k[:, None], torch.full((1, 1), float(kz), device="cuda",
                                                                              dtype=torch.float64)))
    k2 = (kk * kk).sum(0)
    keep = _mask(n, n // 3).to(work)
    kk, k2 = kk.to(work), k2.to(work)
    for lo in range(0, batch, 16):
        m = min(16, batch - lo)
        b = torch.randn((m, 3, n, n), dtype=work, device="cuda", generator=g) * (keep / k2)
        b -= kk * ((kk * b).sum(1, keepdim=True) / k2)
        b /= torch.linalg.vector_norm(b, dim=(1, 2, 3), keepdim=True)
        out[lo:lo + m] = b
    return out


def _to_kept(b):
    n = b.shape[-1]
    i = torch.arange(-(n // 3), n // 3 + 1, device="cuda") % n
    return b[..., i, :][..., i].contiguous()


def _times(batch, seed):
    """Start times of the fields: slices of length pi / 4 from a seeded origin."""
    return math.pi / 4 * torch.arange(batch, dtype=torch.float64, device="cuda") + 0.1 * (seed % 61)


def _instances(case, seed):
    """Flow, side, kz and Rm of the sweep's instances: Rm log-uniform, the side with its root."""
    rng = np.random.default_rng(seed + 17)
    lo, hi = case["n_lo"], case["n_hi"]
    out = []
    for i in range(case["instances"]):
        # the sides cover the range evenly, so that every seed has the same work
        n = 2 ** round(math.log2(lo) + (math.log2(hi) - math.log2(lo)) * i / max(1, case["instances"] - 1))
        Rm = 50.0 * (n / 64.0) ** 2 * math.exp(rng.uniform(-0.3, 0.3))
        nc = n // 2
        dtc = 2.0 / nc
        out.append({"flow": i % 2, "n": n, "kz": float(rng.uniform(0.2, 1.5)), "Rm": Rm, "dt": 0.32 / n, "nc": nc,
                    "dtc": dtc})
    return out


class State:
    """What a user's program keeps: inputs, output buffers and the context."""

    def __init__(self, case):
        self.case = case
        self.ctx = None
        self.sweep = None

    def __del__(self):
        try:
            torch.cuda.synchronize()
            if self.ctx is not None:
                kd.kd_destroy(self.ctx)
            if self.sweep is not None:
                self.sweep.close()
        except Exception:
            pass


def prepare(case, seed):
    s = State(case)
    kind = case["kind"]
    if kind == "fine":
        prec = kd.KD_C128 if case["double"] else kd.KD_C64
        dtype = torch.complex128 if case["double"] else torch.complex64
        b = _fields(case["n"], case["kz"], case["batch"], seed, dtype)
        s.x = _to_kept(b) if case["kept"] else b
        s.y = torch.empty_like(s.x)
        s.t0 = _times(case["batch"], seed)
        s.prec = prec
        s.ctx = kd.kd_create(kd.make_params(case["flow"], case["n"], case["kz"], case["Rm"], case["dt"], prec,
                                            fine_operator=kd.KD_FINE_CONV if case["conv"] else kd.KD_FINE_FFT))
    elif kind == "coarse":
        s.x = _fields(case["n"], case["kz"], case["batch"], seed, torch.complex128)
        s.y = torch.empty_like(s.x)
        s.t0 = _times(case["batch"], seed)
        prec = kd.KD_C128 if case["double"] else kd.KD_C64
        s.ctx = kd.kd_create(kd.make_params(case["flow"], case["n"], case["kz"], case["Rm"], case["dt"], kd.KD_C64,
                                            n_coarse=case["nc"], dt_coarse=case["dt"], prec_coarse=prec))
    elif kind == "parareal":
        n = case["n"]
        s.x = _fields(n, case["kz"], 1, seed, torch.complex128)[0]
        s.u = torch.empty((case["slices"] + 1, 3, n, n), dtype=torch.complex128, device="cuda")
        s.ctx = kd.kd_create(kd.make_params(case["flow"], n, case["kz"], case["Rm"], case["dt"], kd.KD_C64,
                                            n_coarse=case["nc"], dt_coarse=case["dtc"], prec_coarse=kd.KD_C64,
                                            fine_form=kd.KD_FINE_INCREMENT))
    elif kind == "sweep":
        q = _instances(case, seed)
        s.x = [_fields(i["n"], i["kz"], 1, seed + 7 * j, torch.complex128)[0] for j, i in enumerate(q)]
        s.u = [torch.empty_like(b) for b in s.x]
        s.sweep = kd.kd_sweep_create([kd.make_instance(i["flow"], i["n"], i["kz"], i["Rm"], i["dt"], i["nc"], i["dtc"])
                                      for i in q], case["T"], case["slices"])
    else:
        m, nb = case["m"], case["pairs"]
        nc = 3 * m * m
        g = torch.Generator(device="cuda").manual_seed(seed + 5)
        s.w0 = torch.randn((2 * nc, nc), device="cuda", generator=g) * (0.02 / math.sqrt(nc))
        s.w0[:nc].diagonal().add_(0.9)
        s.w = s.w0 + torch.randn((2 * nc, nc), device="cuda", generator=g) * (0.01 / math.sqrt(nc))
        s.x = torch.randn((nb, 3, m, m), dtype=torch.complex64, device="cuda", generator=g)
        s.y = 0.9 * s.x + 0.1 * torch.randn((nb, 3, m, m), dtype=torch.complex64, device="cuda", generator=g)
        s.grad = torch.empty((2 * nc, nc), device="cuda")
        s.ctx = kd.kd_create(kd.make_params(GP, case["n"], 0.57, 1000.0, 2.5e-3, kd.KD_C64, n_coarse=64,
                                            dt_coarse=2.0 / 64, fine_form=kd.KD_FINE_INCREMENT, learned_modes=m))
    return s


def run(s):
    case, kind = s.case, s.case["kind"]
    if kind == "fine":
        call = kd.kd_fine_batched_kept if case["kept"] else kd.kd_fine_batched
        call(s.ctx, s.x, s.y, s.t0, case["steps"], case["batch"], s.prec)
        return s.y
    if kind == "coarse":
        kd.kd_coarse(s.ctx, s.x, s.y, s.t0, case["steps"], case["batch"])
        return s.y if case["double"] else s.y.to(torch.complex64)   # kept in the propagator's precision
    if kind == "parareal":
        _, st = kd.kd_parareal_run(s.ctx, s.x, case["T"], case["slices"], case["k_max"], case["tol"], s.u)
        return {"u": s.u.to(torch.complex64), "k": int(st.k_con)}
    if kind == "sweep":
        kd.kd_sweep_exec(s.sweep, s.x, case["k_max"], 0.0, u_final=s.u)
        return [u.to(torch.complex64) for u in s.u]
    loss = kd.kd_learned_loss_grad(s.ctx, s.w, s.w0, 1e-4, s.x, s.y, case["pairs"], s.grad)
    return {"loss": loss, "grad": s.grad}


# ------------------------------------------------------------------------------ work
def _fine_flops(n, steps, batch):
    """A step of one field: at each of 4 stages six pruned 2D transforms on the smallest grid
    without aliasing of the kept set, 15 flops a grid point for u x b, ~60 a kept mode."""
    P = 2 * (n // 3) + 1
    m = P + 1
    return steps * batch * 4.0 * (6 * (P + m) * 5.0 * m * math.log2(m) + 30.0 * m * m + 3 * 40.0 * P * P)


def _conv_flops(n, steps, batch):
    P = 2 * (n // 3) + 1
    return 540.0 * P * P * steps * batch


def work(case):
    kind = case["kind"]
    if kind == "fine":
        n, es = case["n"], 16 if case["double"] else 8
        P = 2 * (n // 3) + 1
        out = P * P if case["kept"] else n * n
        f = (_conv_flops if case["conv"] else _fine_flops)(n, case["steps"], case["batch"])
        return {"bytes": 3.0 * (P * P + out) * es * case["batch"], "flops": f}
    if kind == "coarse":
        n = case["n"]
        Pc = 2 * (case["nc"] // 3) + 1
        return {"bytes": 3.0 * (Pc * Pc + n * n) * 16 * case["batch"],
                "flops": _conv_flops(case["nc"], case["steps"], case["batch"])}
    if kind == "parareal":
        n, N = case["n"], case["slices"]
        S, Sc = _steps(case["T"] / N, case["dt"]), _steps(case["T"] / N, case["dtc"])
        it = min(2, case["k_max"])
        return {"bytes": 48.0 * n * n * (N + 2),
                "flops": it * _fine_flops(n, S, N) + (it + 1) * _conv_flops(case["nc"], Sc, N)}
    if kind == "sweep":
        b = f = 0.0
        for q in _instances(case, 0):
            dT = case["T"] / case["slices"]
            b += 96.0 * q["n"] ** 2
            f += case["k_max"] * _fine_flops(q["n"], _steps(dT, q["dt"]), case["slices"])
            f += (case["k_max"] + 1) * _conv_flops(q["nc"], _steps(dT, q["dtc"]), case["slices"])
        return {"bytes": b, "flops": f}
    nc, nb = 3 * case["m"] ** 2, case["pairs"]
    return {"bytes": 3 * 8.0 * nc * nc + 16.0 * nc * nb, "flops": 2 * 8.0 * nc * nc * nb}


# ----------------------------------------------------------------------------- exact
_C = (0.0, 0.5, 2.0 / 3.0, 0.5)
_H = ((1 / 2,), (11 / 18, 1 / 18), (5 / 6, -5 / 6, 1 / 2), (1 / 4, 7 / 4, 3 / 4, -7 / 4))
_A = ((1 / 2,), (1 / 6, 1 / 2), (-1 / 2, 1 / 2, 1 / 2), (3 / 2, -3 / 2, 1 / 2, 1 / 2))


class _Exact:
    """The pseudo-spectral IMEX RK443 step in complex128 on the n-point grid."""

    def __init__(self, flow, n, kz, Rm):
        self.flow, self.n = flow, n
        k = _waves(n)
        kk = torch.stack(torch.broadcast_tensors(k[None, :], k[:, None],
                                                 torch.full((1, 1), float(kz), device="cuda", dtype=torch.float64)))
        self.lam = (kk * kk).sum(0) / Rm
        self.mask = _mask(n, n // 3).to(torch.float64)
        self.ik = (1j * kk.to(torch.complex128) * self.mask)
        self.x = 2 * math.pi / n * torch.arange(n, device="cuda", dtype=torch.float64)

    def _u(self, t):
        """u(x, y, t) for start times t: [len(t)][3][n][n]."""
        if self.flow == GP:
            A, px, py = math.sqrt(1.5), torch.cos(t), torch.sin(t)
        else:
            A, px, py = 1.0, torch.zeros_like(t), torch.zeros_like(t)
        ax = (self.x[None, None, :] + px[:, None, None])
        ay = (self.x[None, :, None] + py[:, None, None])
        shape = (len(t), self.n, self.n)
        return A * torch.stack([torch.cos(ay).expand(shape), torch.sin(ax).expand(shape),
                                torch.cos(ax) + torch.sin(ay)], 1).to(torch.complex128)

    def rhs(self, b, t):
        w = torch.linalg.cross(self._u(t), torch.fft.ifft2(b, norm="forward"), dim=-3)
        return torch.linalg.cross(self.ik.expand_as(b), torch.fft.fft2(w, norm="forward"), dim=-3)

    def steps(self, b, t0, dt, nsteps):
        b = b * self.mask
        for s in range(nsteps):
            F, L = [], []
            for i in range(4):
                F.append(self.rhs(b if i == 0 else X, t0 + (s + _C[i]) * dt))
                r = b + sum((dt * h) * f for h, f in zip(_H[i], F))
                if L:
                    r = r - sum((dt * a) * l for a, l in zip(_A[i], L))
                X = r / (1 + 0.5 * dt * self.lam)
                L.append(self.lam * X)
            b = X
        return b

    def batch(self, b, t0, dt, nsteps):
        """steps() in parts that fit the memory."""
        part = max(1, (1 << 23) // self.n ** 2)
        return torch.cat([self.steps(b[i:i + part].to(torch.complex128), t0[i:i + part], dt, nsteps)
                          for i in range(0, b.shape[0], part)])


def _resample(b, n):
    """Fourier truncation / zero padding to the kept set of the smaller of the two grids."""
    m = b.shape[-1]
    K = min(n, m) // 3
    i = torch.arange(-K, K + 1, device="cuda")
    out = torch.zeros((*b.shape[:-2], n, n), dtype=b.dtype, device="cuda")
    out[..., (i % n)[:, None], (i % n)[None, :]] = b[..., (i % m)[:, None], (i % m)[None, :]]
    return out


def _steps(dT, dt):
    q = dT / dt
    return max(1, math.ceil(q - 1e-9 * max(1.0, q)))


def _exact_parareal(q, b0, T, N, k_max, tol):
    """(states at the slice boundaries, iterations) of Parareal in complex128."""
    n, nc, dT = q["n"], q["nc"], T / N
    S, Sc = _steps(dT, q["dt"]), _steps(dT, q["dtc"])
    f, g = _Exact(q["flow"], n, q["kz"], q["Rm"]), _Exact(q["flow"], nc, q["kz"], q["Rm"])
    times = dT * torch.arange(N, device="cuda", dtype=torch.float64)

    def G(u, i):
        return _resample(g.steps(_resample(u[None], nc), times[i:i + 1], dT / Sc, Sc), n)[0]

    U, Go, k = [b0 * f.mask], [], 0
    for i in range(N):
        Go.append(G(U[i], i))
        U.append(Go[i])
    for k in range(1, k_max + 1):
        F = f.batch(torch.stack(U[:N]), times, dT / S, S)
        new = [U[0]]
        for i in range(N):
            Gn = G(new[i], i)
            new.append(F[i] + (Gn - Go[i]))
            Go[i] = Gn
        sigma = float(torch.linalg.vector_norm(new[N] - U[N]) / torch.linalg.vector_norm(new[N]))
        U = new
        if sigma <= tol:
            break
    return torch.stack(U), k


def exact(case, seed):
    kind = case["kind"]
    if kind == "fine":
        # the input rounded to the precision the call takes
        b = _fields(case["n"], case["kz"], case["batch"], seed,
                    torch.complex128 if case["double"] else torch.complex64)
        e = _Exact(case["flow"], case["n"], case["kz"], case["Rm"])
        r = e.batch(b, _times(case["batch"], seed), case["dt"], case["steps"])
        return _to_kept(r) if case["kept"] else r
    if kind == "coarse":
        b = _fields(case["n"], case["kz"], case["batch"], seed, torch.complex128)
        e = _Exact(case["flow"], case["nc"], case["kz"], case["Rm"])
        return _resample(e.batch(_resample(b, case["nc"]), _times(case["batch"], seed), case["dt"], case["steps"]),
                         case["n"])
    if kind == "parareal":
        b0 = _fields(case["n"], case["kz"], 1, seed, torch.complex128)[0]
        u, k = _exact_parareal(case, b0, case["T"], case["slices"], case["k_max"], case["tol"])
        return {"u": u, "k": k}
    if kind == "sweep":
        out = []
        for j, q in enumerate(_instances(case, seed)):
            b0 = _fields(q["n"], q["kz"], 1, seed + 7 * j, torch.complex128)[0]
            out.append(_exact_parareal(q, b0, case["T"], case["slices"], case["k_max"], 0.0)[0][-1])
        return out
    s = prepare(case, seed)
    nc, nb = 3 * case["m"] ** 2, case["pairs"]
    W = torch.complex(s.w[:nc].double(), s.w[nc:].double())
    X = s.x.reshape(nb, nc).to(torch.complex128)
    R = X @ W.T - s.y.reshape(nb, nc).to(torch.complex128)
    loss = float(R.abs().square().sum()) / nb
    G = (2.0 / nb) * (R.T @ X.conj())
    grad = torch.cat([G.real, G.imag]) + 2e-4 * (s.w.double() - s.w0.double())
    return {"loss": loss, "grad": grad}
