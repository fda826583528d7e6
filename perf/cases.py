"""The work whose speed this repository looks after, as plain cases.

Each case is one thing a program that uses the library has it do, through the
calls of `paper_2202_10647_gb300.ionize` and `multistep`:

  pulse      a whole run of the 2D nitrogen pulse (N_0 = 1 everywhere), its
             time steps captured in one graph (`StepGraph`).
  step       one `ionize.step` of a PIC code's nitrogen or ladder cells.
  field      one `ionize.step_field` from field components, with a gas density.
  batch      one `ionize.step_batched` over several species.
  beams      a run of captured steps of a ladder gas in crossed laser beams,
             with the step's own conservation measure.
  surrogate  one `Surrogate.step` (rates from the network where it is trusted).
  train      one optimizer step of the surrogate's training (`mlp_loss_grad`,
             `mlp_adam`).
  targets    the surrogate's training data (`log2_rates`, `mlp_inputs`,
             `mlp_standardize`).
  rates      a table of rates of every state (`ionize.rates`).

A step moves its populations and windows on in place, as in a PIC code.  So
that a pass is the same work however often it is repeated, `run` hands the
call the windows it had at first (one copy of two bytes per cell; a PIC code
places them when cells move), or keeps them (ION_NO_WINDOW_UPDATE), and the
multi-step runs begin from fresh gas; what a call costs depends on the fields
and the windows.
"""
import math

import numpy as np
import torch

from paper_2202_10647_gb300 import ionize, multistep, workloads

DT = 0.05  # fs
HIDDEN = 64
FLOOR = -40.0  # log2 W below which the surrogate's targets are cut
LOG10E = (1.0, 5.0)  # its trained range, GV/m


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # the nitrogen pulse of the paper's kind on a small 2D grid, 200 steps
        # in FP64: many tiny steps one after another, nothing but latency
        {"name": "pulse_2d_f64_200_steps", "kind": "pulse", "nx": 128, "ny": 128, "steps": 200,
         "f64": True},
        # one call on a small patch of a PIC code's grid, windows kept by the
        # caller: argument checks, launches and the shortest kernels
        {"name": "step_n_patch_16k", "kind": "step", "gas": "N", "n": 16384, "f64": False,
         "keep": True, "odd_ld": False, "adaptive": False},
        # the main path: nitrogen on a 3D grid of 33.5M cells, FP32
        {"name": "step_n_33m", "kind": "step", "gas": "N", "n": 33554432, "f64": False,
         "keep": False, "odd_ld": False, "adaptive": False},
        # the same cells in the plain FP64 form
        {"name": "step_n_33m_f64", "kind": "step", "gas": "N", "n": 33554432, "f64": True,
         "keep": False, "odd_ld": False, "adaptive": False},
        # a heavy gas with windows that grow and shrink, on a ragged cell count
        {"name": "step_kr_4m_adaptive", "kind": "step", "gas": "Kr", "n": 4000037, "f64": False,
         "keep": False, "odd_ld": False, "adaptive": True},
        # a PIC code's three field components and gas density, on an odd cell
        # count with unpadded planes
        {"name": "field_ar_1m_odd", "kind": "field", "gas": "Ar", "n": 1000003, "f64": False,
         "components": 3},
        # three gases of uneven size and charge in one launch
        {"name": "batch_mixed_30m", "kind": "batch", "n": 30000000},
        # a heavy gas in sixteen crossed beams, 20 captured steps from fresh gas
        {"name": "beams_kr_16m_20_steps", "kind": "beams", "nz": 256, "ny": 256, "nx": 256,
         "steps": 20},
        # the step with the learned rates, on the Ar-like cells of the plain one
        {"name": "surrogate_ar_33m", "kind": "surrogate", "gas": "Ar", "n": 33554432},
        # one of the 40,000 optimizer steps that train the network
        {"name": "train_ar_8192", "kind": "train", "k": 18, "batch": 8192, "pairs": False},
        # the training set of a million fields
        {"name": "targets_ar_1m", "kind": "targets", "gas": "Ar", "n": 1048576},
        # every rate of a heavy gas on an odd number of fields
        {"name": "rates_kr_4m", "kind": "rates", "gas": "Kr", "n": 4000001, "f64": False},
    ]


def _log_size(rng, lo, hi, odd=0.5):
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return n if rng.random() < odd else max(64, n // 64 * 64)


def draw(rng):
    kind = rng.choice(["pulse", "step", "step", "step", "field", "batch", "beams", "surrogate",
                       "train", "targets", "rates"])
    gas = rng.choice(["N", "Ar", "Kr"])
    if kind == "pulse":
        return {"kind": kind, "nx": rng.randint(48, 256), "ny": rng.randint(48, 256),
                "steps": rng.randint(40, 200), "f64": rng.random() < 0.5}
    if kind == "step":
        f64 = rng.random() < 0.3
        return {"kind": kind, "gas": gas, "n": _log_size(rng, 1000, 8e6 if f64 else 2.4e7),
                "f64": f64, "keep": rng.random() < 0.3, "odd_ld": rng.random() < 0.3,
                "adaptive": rng.random() < 0.25}
    if kind == "field":
        return {"kind": kind, "gas": gas, "n": _log_size(rng, 3000, 1.2e7),
                "f64": rng.random() < 0.3, "components": rng.randint(1, 3)}
    if kind == "batch":
        return {"kind": kind, "n": _log_size(rng, 30000, 3e7)}
    if kind == "beams":
        return {"kind": kind, "nz": rng.randint(24, 160), "ny": rng.randint(48, 256),
                "nx": 4 * rng.randint(12, 64), "steps": rng.randint(5, 20)}
    if kind == "surrogate":
        return {"kind": kind, "gas": gas, "n": _log_size(rng, 20000, 1.6e7)}
    if kind == "train":
        return {"kind": kind, "k": rng.choice([7, 18, 36, rng.randint(1, 63)]),
                "batch": _log_size(rng, 500, 32768), "pairs": rng.random() < 0.3}
    if kind == "targets":
        return {"kind": kind, "gas": gas, "n": _log_size(rng, 20000, 2e6)}
    return {"kind": kind, "gas": gas, "n": _log_size(rng, 10000, 8e6), "f64": rng.random() < 0.4}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _gas(name):
    return {"N": workloads.nitrogen, "Ar": workloads.argon_like,
            "Kr": workloads.krypton_like}[name]()


def _grid(n):
    """nz, ny, nx of a nitrogen grid holding at least n cells."""
    nx = 512 if n >= 1 << 20 else 128
    side = max(8, int(math.ceil(math.sqrt(n / nx))))
    ny = (side + 7) // 8 * 8
    return -(-n // (ny * nx)), ny, nx


def _cells(gas, n, seed, device):
    """|E|, N (planes, n), k_lo, k_hi of n cells: nitrogen in a pulse on a 3D
    grid, the heavier gases in a lognormal field."""
    if gas == "N":
        nz, ny, nx = _grid(n)
        total = nz * ny * nx
        # the n cells around the middle of the grid (the pulse's centre)
        at = (total - n) // 2 + torch.arange(n, dtype=torch.int64, device=device)
        return workloads.nitrogen_3d(nz, ny, nx, seed=seed, device=device, cells=at)
    return workloads.ladder_cells(_gas(gas), n, seed, device)


def _windows(lo, hi):
    """k_lo and k_hi in one buffer, each 16-byte aligned (one copy hands a
    call both)."""
    n = lo.numel()
    w = torch.zeros((2, (n + 63) // 64 * 64), dtype=torch.uint8, device=lo.device)
    w[0, :n] = lo
    w[1, :n] = hi
    return w


def _planes(N, n, ld, dtype):
    out = torch.zeros((N.shape[0], ld), dtype=dtype, device=N.device)
    out[:, :n] = N[:, :n]
    return out


class _State:
    pass


_WINDOW = {"w_min": 2, "w_max": 6, "eps_grow": 1e-6}


def _pulse_fields(case, seed, device):
    """The pulse's |E| at each step; its peak, waist and phase are the seed's."""
    u = np.random.RandomState(seed % (1 << 31)).rand(3)
    return [workloads.nitrogen_pulse_2d((s + 0.5) * DT + 4.0 * u[2], case["nx"], case["ny"],
                                        E0=1500.0 + 1000.0 * u[0], waist=7.0 + 2.0 * u[1],
                                        device=device) for s in range(case["steps"])]


def _beam_fields(case, seed, device):
    A, B = workloads.krypton_beam_terms(case["nz"], case["ny"], case["nx"], seed=seed,
                                        device=device)
    scale = workloads.krypton_scale(A)
    return [workloads.krypton_field(A, B, (s + 0.5) * DT, scale) for s in range(case["steps"])]


def _components(E, count, seed, dtype):
    """Field components of magnitude E in directions of the seed."""
    if count == 1:
        sign = workloads.uniform(seed, 70, torch.arange(E.numel(), device=E.device)) < 0.5
        return [torch.where(sign, E, -E).to(dtype)]
    i = torch.arange(E.numel(), device=E.device)
    phi = 2 * math.pi * workloads.uniform(seed, 71, i)
    if count == 2:
        return [(E * torch.cos(phi)).to(dtype), (E * torch.sin(phi)).to(dtype)]
    ct = 2 * workloads.uniform(seed, 72, i) - 1
    st = torch.sqrt(1 - ct * ct)
    return [(E * st * torch.cos(phi)).to(dtype), (E * st * torch.sin(phi)).to(dtype),
            (E * ct).to(dtype)]


def _train_inputs(case, seed):
    """Parameters, a batch with targets of a smooth function of the input,
    and Adam's moments some way into a training run."""
    K, B, H = case["k"], case["batch"], HIDDEN
    g = torch.Generator().manual_seed(seed % (1 << 31))
    W1 = torch.randn(H, generator=g) * 4.0
    b1 = (torch.rand(H, generator=g) * 2 - 1) * 4.0
    W2 = torch.randn(H, H, generator=g) * math.sqrt(2.0 / H)
    b2 = torch.randn(H, generator=g) * 0.1
    W3 = torch.randn(K, H, generator=g) * math.sqrt(1.0 / H)
    b3 = torch.randn(K, generator=g) * 0.1
    P = torch.cat([W1, b1, W2.reshape(-1), b2, W3.reshape(-1), b3]).float()
    x = torch.rand(B, generator=g) * 2 - 1
    k = torch.arange(K)
    t = torch.tanh(3.0 * (x[:, None] - (k[None, :] - K / 2) / max(K, 2))) + 0.5 * x[:, None]
    m = torch.randn(P.numel(), generator=g) * 1e-3
    v = torch.rand(P.numel(), generator=g) * 1e-5 + 1e-6
    return P, x.float(), t.float().contiguous(), m.float(), v.float()


def _network(gas, seed):
    """Parameters and scaling of a network for one gas, without training:
    layers 1 and 2 make 64 smooth ramps over the input, layer 3 is the
    least-squares fit of the standardized log-rates on them."""
    r = np.random.RandomState(seed % (1 << 31))
    H = HIDDEN
    knots = -1.06 + 2.1 * (np.arange(H) + 0.3 * (r.rand(H) - 0.5)) / (H - 1)
    W1 = 14.0 + r.rand(H)
    b1 = -W1 * knots
    W2 = 0.25 * np.eye(H) + 0.002 * r.randn(H, H)
    b2 = 0.05 * r.randn(H)
    W1, b1, W2, b2 = (a.astype(np.float32).astype(np.float64) for a in (W1, b1, W2, b2))
    l2 = [v * math.log2(10.0) for v in LOG10E]
    x = np.linspace(-1, 1, 6001)
    E = torch.from_numpy(2.0 ** (l2[0] + (x + 1) / 2 * (l2[1] - l2[0])))
    Y = np.maximum(_log2_rates(_gas(gas), E).numpy().T, FLOOR)
    mean, scale = Y.mean(0), np.maximum(Y.std(0, ddof=1), 1e-3)

    def gelu(z):
        return 0.5 * z * (1 + np.tanh(math.sqrt(2 / math.pi) * (z + 0.044715 * z ** 3)))

    h = gelu(gelu(x[:, None] * W1 + b1) @ W2.T + b2)
    F = np.concatenate([h, np.ones((len(x), 1))], 1)
    T = (Y - mean) / scale
    c = np.linalg.solve(F.T @ F + 1e-3 * np.eye(H + 1), F.T @ T)
    P = np.concatenate([W1, b1, W2.reshape(-1), b2, c[:H].T.reshape(-1), c[H]])
    norm = {"log2E_min": l2[0], "log2E_max": l2[1], "y_floor": FLOOR,
            "y_mean": mean.tolist(), "y_scale": scale.tolist()}
    return torch.from_numpy(P.astype(np.float32)), norm


def _species(gas):
    return ionize.Species(gas.U, gas.l, gas.m)


def prepare(case, seed):
    dev = torch.device("cuda")
    s = _State()
    s.case, s.kind = case, case["kind"]
    seed = int(seed) % (1 << 31)
    f64 = bool(case.get("f64"))
    s.dtype = torch.float64 if f64 else torch.float32
    s.flags = ionize.ION_F64_PLAIN if f64 else ionize.ION_F32
    if s.kind in ("pulse", "beams"):
        beams = s.kind == "beams"
        gas = _gas("Kr" if beams else "N")
        fields = (_beam_fields if beams else _pulse_fields)(case, seed, dev)
        fields = [E.to(s.dtype) for E in fields]
        n = fields[0].numel()
        s.sp = _species(gas)
        s.N = torch.zeros((gas.Z + 1, (n + 3) // 4 * 4), dtype=s.dtype, device=dev)
        s.win = _windows(*(torch.zeros(n, dtype=torch.uint8, device=dev) for _ in range(2)))
        s.lo, s.hi = s.win[0, :n], s.win[1, :n]
        s.dne = torch.empty(n, dtype=s.dtype, device=dev)
        s.graph = multistep.StepGraph(s.sp, fields, s.N, s.lo, s.hi, s.dne, DT, flags=s.flags,
                                      conservation="fused" if beams else False)
        return s
    if s.kind in ("step", "field", "surrogate"):
        n = case["n"]
        wl = _cells(case["gas"], n, seed, dev)
        s.sp = _species(wl.species)
        odd = case.get("odd_ld") or s.kind == "field"
        s.N = _planes(wl.N, n, n if odd else (n + 3) // 4 * 4, s.dtype)
        s.win0 = _windows(wl.lo, wl.hi)
        s.win = s.win0.clone()
        s.lo, s.hi = s.win[0, :n], s.win[1, :n]
        s.dne = torch.empty(n, dtype=s.dtype, device=dev)
        if s.kind == "field":
            s.comps = _components(wl.E.double(), case["components"], seed, s.dtype)
            s.n_gas = _density(n, seed, dev).to(s.dtype)
            nb = int(ionize.lib().ion_step_field_workspace_bytes(n, s.flags))
            s.ws = torch.empty(nb, dtype=torch.uint8, device=dev)
            return s
        s.E = wl.E.to(s.dtype)
        s.ws = ionize.workspace(n, s.flags, dev)
        if s.kind == "surrogate":
            P, norm = _network(case["gas"], seed)
            s.net = ionize.Surrogate(s.sp, P.to(dev), norm)
            s.net.validate()
            return s
        s.window = _WINDOW if case["adaptive"] else None
        if case["keep"]:
            s.flags |= ionize.ION_NO_WINDOW_UPDATE
        return s
    if s.kind == "batch":
        s.jobs, s.wins = [], []
        for wl in workloads.mixed_batch(case["n"] / 3e7, seed=seed, device=dev):
            n = wl.ncells
            win0 = _windows(wl.lo, wl.hi)
            win = win0.clone()
            s.wins.append((win, win0))
            s.jobs.append((_species(wl.species), wl.E, wl.N, win[0, :n], win[1, :n],
                           torch.empty(n, dtype=torch.float32, device=dev)))
        s.ws = ionize.batched_workspace(s.jobs)
        return s
    if s.kind == "train":
        s.P, s.x, s.t, s.m, s.v = (a.to(dev) for a in _train_inputs(case, seed))
        s.grad = torch.empty_like(s.P)
        s.loss = torch.empty(1, dtype=torch.float32, device=dev)
        s.ws = ionize.mlp_workspace(case["k"], case["batch"], dev)
        s.step = 1000
        return s
    s.sp = _species(_gas(case["gas"]))
    lo, hi = LOG10E if s.kind == "targets" else (1.0, 3.9)
    s.E = workloads.log_uniform_fields(seed, 60, case["n"], lo, hi, device=dev).to(s.dtype)
    return s


def _density(n, seed, device):
    """Gas density in units of a reference density, a smooth ramp with noise."""
    i = torch.arange(n, dtype=torch.int64, device=device)
    return 0.5 + i.double() / n + 0.1 * workloads.uniform(seed, 73, i)


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(s):
    kind = s.kind
    if kind in ("pulse", "beams"):
        # fresh gas, then the run
        s.N.zero_()
        s.N[0].fill_(1.0)
        s.win[0].zero_()
        s.win[1].fill_(3)
        s.graph.replay()
        out = {"N": s.N, "k_lo": s.lo, "k_hi": s.hi, "dne": s.dne}
        if kind == "beams":
            out["change"] = s.graph.cons
            out["total"] = s.graph.cons_full
        return out
    if kind == "step":
        if not s.case["keep"]:
            s.win.copy_(s.win0)
        ionize.step(s.sp, s.E, s.N, s.lo, s.hi, DT, s.dne, ws=s.ws, flags=s.flags,
                    window=s.window)
        return {"N": s.N, "k_lo": s.lo, "k_hi": s.hi, "dne": s.dne}
    if kind == "field":
        s.win.copy_(s.win0)
        ionize.step_field(s.sp, s.comps, s.N, s.lo, s.hi, DT, s.dne, n_gas=s.n_gas, ws=s.ws,
                          flags=s.flags)
        return {"N": s.N, "k_lo": s.lo, "k_hi": s.hi, "dne": s.dne}
    if kind == "surrogate":
        s.win.copy_(s.win0)
        s.net.step(s.E, s.N, s.lo, s.hi, DT, s.dne, ws=s.ws)
        return {"N": s.N, "k_lo": s.lo, "k_hi": s.hi, "dne": s.dne}
    if kind == "batch":
        for win, win0 in s.wins:
            win.copy_(win0)
        ionize.step_batched(s.jobs, DT, ws=s.ws)
        return [{"N": j[2], "k_lo": j[3], "k_hi": j[4], "dne": j[5]} for j in s.jobs]
    if kind == "train":
        flags = ionize.ION_MLP_BF16 if s.case["pairs"] else 0
        ionize.mlp_loss_grad(s.P, s.case["k"], s.x, s.t, flags, grad=s.grad, loss=s.loss, ws=s.ws)
        ionize.mlp_adam(s.P, s.grad, s.m, s.v, 1e-4, s.step)
        return {"loss": s.loss, "grad": s.grad, "P": s.P, "m": s.m, "v": s.v}
    if kind == "targets":
        l2 = [v * math.log2(10.0) for v in LOG10E]
        Y = ionize.log2_rates(s.sp, s.E, 0, s.sp.Z, FLOOR)
        x = ionize.mlp_inputs(s.E, l2[0], l2[1])
        mean, scale, T = ionize.mlp_standardize(Y, 1e-3)
        return {"x": x, "Y": Y, "mean": mean, "scale": scale, "T": T}
    return ionize.rates(s.sp, s.E, 0, s.sp.Z)


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
_Z = {"N": 7, "Ar": 18, "Kr": 36}


def _step_work(n, width, elem):
    """Bytes and operations of one step: |E|, the windows and the window
    planes read; the planes, the windows and dne written.  Per rate an
    exponent and its power of two, then a few products per state."""
    return (n * (2 * elem + 4 + 2 * elem * width), n * (4 + 12 * (width - 1)))


def work(case):
    kind = case["kind"]
    elem = 8 if case.get("f64") else 4
    width = 3.5 if case.get("gas") == "N" else 4.0
    if kind in ("pulse", "beams"):
        n = case["nx"] * case["ny"] * case.get("nz", 1)
        b, f = _step_work(n, 4.0, elem)
        return {"bytes": float(b * case["steps"]), "flops": float(f * case["steps"])}
    if kind == "step":
        b, f = _step_work(case["n"], width, elem)
        return {"bytes": float(b), "flops": float(f)}
    if kind == "field":
        b, f = _step_work(case["n"], width, elem)
        return {"bytes": float(b + case["n"] * elem * case["components"]),
                "flops": float(f + 6 * case["n"])}
    if kind == "batch":
        b, f = _step_work(case["n"], 4.0, 4)
        return {"bytes": float(b), "flops": float(f)}
    if kind == "surrogate":
        b, f = _step_work(case["n"], width, 4)
        net = 2 * HIDDEN * (1 + HIDDEN + _Z[case["gas"]])
        return {"bytes": float(b), "flops": float(f + case["n"] * net)}
    if kind == "train":
        K, B = case["k"], case["batch"]
        p = HIDDEN * (HIDDEN + K + 3) + K
        return {"bytes": 4.0 * (7 * p + B * (1 + K)), "flops": 6.0 * B * HIDDEN * (1 + HIDDEN + K)}
    Z, n = _Z[case["gas"]], case["n"]
    if kind == "targets":
        # E read; x, Y (FP64) and T written
        return {"bytes": float(n * (4 + 4 + 12 * Z)), "flops": float(n * 10 * Z)}
    return {"bytes": float(n * elem * (1 + Z)), "flops": float(n * 8 * Z)}


# ---------------------------------------------------------------------------
# the same in 64 bits, in plain torch
# ---------------------------------------------------------------------------
def _log2_table(gas):
    """a, b, C with log2 W_k [1/fs] = a_k - b_k log2|E| - C_k/|E| (the ADK
    rate, cycle averaged, E_a = 510 GV/m, omega_a = 41.3/fs, U_H = 13.6 eV)."""
    f = math.factorial
    rows = []
    for k, (U, l, m) in enumerate(zip(gas.U, gas.l, gas.m)):
        Q, am = k + 1.0, abs(m)
        ns = Q * math.sqrt(13.6 / U)
        flm = (2 * l + 1) * f(l + am) / (2.0 ** am * f(am) * f(l - am))
        x = 2 * ns - am - 1
        lg = (math.log(41.3) + 0.5 * math.log(3 * ns ** 3 / (math.pi * Q ** 3))
              + math.log(Q * Q / (2 * ns * ns)) + 2 * ns * math.log(2 * math.e / ns)
              + math.log(flm / (2 * math.pi * ns)) + x * math.log(2 * Q ** 3 / ns ** 3))
        b = x - 0.5
        rows.append((lg / math.log(2) + b * math.log2(510.0), b,
                     (2.0 / 3.0) * (Q / ns) ** 3 * 510.0 / math.log(2)))
    return torch.tensor(rows, dtype=torch.float64)


def _log2_rates(gas, E):
    """log2 W_k(|E|) for every state, (Z, n) in FP64; -inf where W is 0."""
    t = _log2_table(gas).to(E.device)
    E = E.double().abs()
    q = t[:, 2, None] / E
    y = t[:, 0, None] - t[:, 1, None] * torch.log2(E) - q
    return torch.where((q > 700 / math.log(2)) | (E <= 1e-6), -math.inf, y)


def _expm_cells(lam, v, w):
    """exp(dt A) v for cells of one width w: lam (w-1, n) the rates times dt,
    v (w, n).  Scaling and squaring of the triangular matrix, by entries."""
    out = v.clone()
    if w < 2 or v.shape[1] == 0:
        return out
    lmax = lam.max(0).values
    squarings = torch.ceil(torch.log2(lmax.clamp(min=1e-30) / 0.25)).clamp(min=0).long()
    for sq in torch.unique(squarings).tolist():
        at = torch.nonzero(squarings == sq).squeeze(1)
        for part in torch.split(at, 1 << 22):
            L = lam[:, part] / 2.0 ** sq
            x = v[:, part]
            if sq == 0:
                out[:, part] = _taylor(L, [x[i] for i in range(w)])
                continue
            one, zero = torch.ones_like(x[0]), torch.zeros_like(x[0])
            M = [_taylor(L, [one if i == j else zero for i in range(w)]) for j in range(w)]
            for _ in range(sq):
                M = [[sum((M[k][i] * M[j][k] for k in range(j + 1, i + 1)), M[j][i] * M[j][j])
                      if i >= j else zero for i in range(w)] for j in range(w)]
            out[:, part] = torch.stack([sum((M[j][i] * x[j] for j in range(1, i + 1)),
                                            M[0][i] * x[0]) for i in range(w)])
    return out


def _taylor(L, x):
    """sum_k A^k x / k! for rates of at most 1/4."""
    w = len(x)
    acc, t = list(x), list(x)
    for k in range(1, 17):
        flow = [L[i] * t[i] / k for i in range(w - 1)]
        t = [(flow[i - 1] if i > 0 else 0) - (flow[i] if i < w - 1 else 0) for i in range(w)]
        acc = [a + b for a, b in zip(acc, t)]
    return torch.stack(acc)


def _step64(gas, E, N, lo, hi, slide=True, adaptive=False):
    """One step in FP64: N (Z+1, n), lo and hi (int64) are updated in place;
    returns the freed electrons per atom."""
    n, Z = E.numel(), gas.Z
    t = _log2_table(gas).to(E.device)
    dne = torch.zeros(n, dtype=torch.float64, device=E.device)
    width = hi - lo + 1
    for w in torch.unique(width).tolist():
        for part in torch.split(torch.nonzero(width == w).squeeze(1), 1 << 23):
            a = lo[part]
            e = E[part].double().abs()
            rows = [a + r for r in range(w)]
            v = torch.stack([N[k, part] for k in rows])
            lam = []
            for k in rows[:-1]:
                q = t[k, 2] / e
                y = t[k, 0] + math.log2(DT) - t[k, 1] * torch.log2(e) - q
                lam.append(torch.where((q > 700 / math.log(2)) | (e <= 1e-6), 0.0,
                                       torch.exp2(y)))
            if w < 2:
                continue
            u = _expm_cells(torch.stack(lam), v, w)
            for r, k in enumerate(rows):
                N[k, part] = u[r]
            d = u - v
            dne[part] = sum(r * d[r] for r in range(1, w))
            if not slide:
                continue
            b = hi[part].clone()
            a = a.clone()
            go = torch.ones_like(a, dtype=torch.bool)
            for r in range(w - 1):
                go = go & (u[r] < 1e-6)
                if adaptive:
                    drop = go & (b - a + 1 > _WINDOW["w_min"])
                    move = go & ~drop & (b < Z)
                    go = drop | move
                    a = a + go.long()
                    b = b + move.long()
                else:
                    go = go & (b < Z)
                    a = a + go.long()
                    b = b + go.long()
            if adaptive:
                grow = (u[w - 1] > _WINDOW["eps_grow"]) & (b < Z) & (b - a + 1 < _WINDOW["w_max"])
                b = b + grow.long()
            lo[part] = a
            hi[part] = b
    return dne


def _exact_cells(E, wl, n, ld, dtype, slide=True, adaptive=False, n_gas=None):
    N = _planes(wl.N, n, ld, dtype).double()
    lo, hi = wl.lo.long(), wl.hi.long()
    dne = _step64(wl.species, E, N, lo, hi, slide, adaptive)
    if n_gas is not None:
        dne = dne * n_gas.double()
    return {"N": N, "k_lo": None, "k_hi": None, "dne": dne}


def exact(case, seed):
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    seed = int(seed) % (1 << 31)
    kind = case["kind"]
    dtype = torch.float64 if case.get("f64") else torch.float32
    if kind in ("pulse", "beams"):
        beams = kind == "beams"
        gas = _gas("Kr" if beams else "N")
        fields = (_beam_fields if beams else _pulse_fields)(case, seed, dev)
        n = fields[0].numel()
        N = torch.zeros((gas.Z + 1, (n + 3) // 4 * 4), dtype=torch.float64, device=dev)
        N[0] = 1.0
        lo = torch.zeros(n, dtype=torch.int64, device=dev)
        hi = torch.full((n,), 3, dtype=torch.int64, device=dev)
        for E in fields:
            dne = _step64(gas, E, N, lo, hi)
        out = {"N": N, "k_lo": None, "k_hi": None, "dne": dne}
        if beams:  # the arithmetic's own rounding: nothing to compare
            out["change"] = out["total"] = None
        return out
    if kind in ("step", "field", "surrogate"):
        n = case["n"]
        wl = _cells(case["gas"], n, seed, dev)
        odd = case.get("odd_ld") or kind == "field"
        ld = n if odd else (n + 3) // 4 * 4
        if kind == "field":
            comps = _components(wl.E.double(), case["components"], seed, dtype)
            E = torch.sqrt(sum(c.double() ** 2 for c in comps))
            return _exact_cells(E, wl, n, ld, dtype,
                                n_gas=_density(n, seed, dev).to(dtype))
        return _exact_cells(wl.E, wl, n, ld, dtype, not case.get("keep"),
                            bool(case.get("adaptive")))
    if kind == "batch":
        return [_exact_cells(wl.E, wl, wl.ncells, wl.N.shape[1], torch.float32)
                for wl in workloads.mixed_batch(case["n"] / 3e7, seed=seed, device=dev)]
    if kind == "train":
        return _exact_train(case, seed, dev)
    gas = _gas(case["gas"])
    lo, hi = LOG10E if kind == "targets" else (1.0, 3.9)
    E = workloads.log_uniform_fields(seed, 60, case["n"], lo, hi, device=dev).to(dtype)
    y = _log2_rates(gas, E)
    if kind == "rates":
        return torch.exp2(y)
    Y = y.clamp(min=FLOOR).T.contiguous()
    l2 = [v * math.log2(10.0) for v in LOG10E]
    x = (2 * (torch.log2(E.double()) - l2[0]) / (l2[1] - l2[0]) - 1).clamp(-1, 1)
    mean, scale = Y.mean(0), Y.std(0).clamp(min=1e-3)
    return {"x": x, "Y": Y, "mean": mean, "scale": scale, "T": (Y - mean) / scale}


def _exact_train(case, seed, dev):
    K, B, H = case["k"], case["batch"], HIDDEN
    P, x, t, m, v = (a.to(dev).double() for a in _train_inputs(case, seed))
    W1, b1 = P[:H], P[H:2 * H]
    W2, b2 = P[2 * H:2 * H + H * H].view(H, H), P[2 * H + H * H:3 * H + H * H]
    W3, b3 = P[3 * H + H * H:3 * H + H * H + K * H].view(K, H), P[3 * H + H * H + K * H:]
    c = math.sqrt(2 / math.pi)

    def gelu(z):
        th = torch.tanh(c * (z + 0.044715 * z ** 3))
        return 0.5 * z * (1 + th), 0.5 * (1 + th) + 0.5 * z * (1 - th * th) * c * (
            1 + 3 * 0.044715 * z * z)

    z1 = x[:, None] * W1 + b1
    h1, g1 = gelu(z1)
    h2, g2 = gelu(h1 @ W2.T + b2)
    d = h2 @ W3.T + b3 - t
    dy = 2.0 / (B * K) * d
    dz2 = (dy @ W3) * g2
    dz1 = (dz2 @ W2) * g1
    grad = torch.cat([(dz1 * x[:, None]).sum(0), dz1.sum(0), (dz2.T @ h1).reshape(-1),
                      dz2.sum(0), (dy.T @ h2).reshape(-1), dy.sum(0)])
    m = 0.9 * m + 0.1 * grad
    v = 0.999 * v + 0.001 * grad * grad
    P = P - 1e-4 * (m / (1 - 0.9 ** 1000)) / (torch.sqrt(v / (1 - 0.999 ** 1000)) + 1e-8)
    return {"loss": (d * d).mean().reshape(1), "grad": grad, "P": P, "m": m, "v": v}
