"""Timed cases: the work a flow solver, or a user training a surrogate, has this library do.

Each case is one pass through the public entry points of ``paper_2312_13513_gb300`` on seeded
inputs made on the GPU: the FP64 chemistry advance of the two mechanisms (small requests, stiff
mixtures, whole fields), the surrogate step, the whole chemistry + thermo step, the per-species
networks, one training step, transport properties and the species-equation assembly.

``exact`` restates each path in plain FP64 torch (the Rodas4 step with its step control, the
networks without BF16 rounding, the closed forms of the properties and of the matrix).
"""
from __future__ import annotations

import functools
import math
import os
import struct

import numpy as np
import torch

import paper_2312_13513_gb300 as cg
from paper_2312_13513_gb300.train import PAD, Trainer
from synth.mechanism import ch4_mechanism, h2_mechanism
from synth.mesh import box_mesh
from synth.states import AIR_N2, AIR_O2, PATM, beta_params, load_table
from synth.transport import generate_transport

DEV = "cuda" if torch.cuda.is_available() else "cpu"
F64 = torch.float64
RU = 8.314462618e7
MODEL = os.path.join(os.path.dirname(os.path.abspath(cg.__file__)), "models", "h2_quasi_dns.chemsur")
PS_HIDDEN = (1600, 800, 400)


# ------------------------------------------------------------------------------------------
# the cases
# ------------------------------------------------------------------------------------------
def listed():
    return [
        # a small solver's (or one block's) mixing layer before ignition: few cells, many stiff sub-steps
        {"name": "h2_mixing_4096", "kind": "advance", "mech": "h2", "field": "mixing", "n": 4096, "dt": 1e-6},
        # the smallest request the serving loop sees: one block of a flame, ragged
        {"name": "h2_block_10007", "kind": "advance", "mech": "h2", "field": "front", "n": 10007, "dt": 5e-7},
        # the quasi-DNS field, half of a 128^3 box
        {"name": "h2_field_1048576", "kind": "advance", "mech": "h2", "field": "front", "n": 1 << 20, "dt": 5e-7},
        # a block of the LES on the 53-species mechanism
        {"name": "ch4_block_1021", "kind": "advance", "mech": "ch4", "field": "les", "n": 1021, "dt": 1e-6},
        # an LES field on the 53-species mechanism
        {"name": "ch4_field_131101", "kind": "advance", "mech": "ch4", "field": "les", "n": 131101, "dt": 1e-6},
        # the surrogate step on a small request and on two 128^3 boxes
        {"name": "surrogate_block_10007", "kind": "surrogate", "n": 10007},
        {"name": "surrogate_field_4194304", "kind": "surrogate", "n": 1 << 22},
        # the chemistry + thermo step of a solver's time loop: surrogate, T from h, transport, replayed
        {"name": "step_100003", "kind": "step", "n": 100003},
        # the per-species networks over one field block, two whole passes and a short last one
        {"name": "per_species_131089", "kind": "per_species", "n": 131089},
        # one training step of the 4 x 512 network at the training batch
        {"name": "train_step_4096", "kind": "train", "batch": 4096},
        # transport properties of the 53-species mechanism
        {"name": "transport_ch4_100003", "kind": "transport", "mech": "ch4", "n": 100003},
        # the species equation on a 128^3 box: PaSR factor, assembly, CSR values for the solver
        {"name": "species_eq_128", "kind": "fvm", "nx": 128, "ny": 128, "nz": 128, "permute": False},
    ]


def _log_size(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["advance"] * 5 + ["surrogate"] * 2 + ["step", "per_species", "train", "transport", "fvm"])
    if kind == "advance":
        if rng.random() < 0.4:
            return {"kind": kind, "mech": "ch4", "field": "les", "n": _log_size(rng, 300, 131101),
                    "dt": rng.choice([5e-7, 1e-6])}
        field, dt = rng.choice(["front", "front", "mixing"]), rng.choice([5e-7, 1e-6])
        most = 32768 if field == "mixing" else (1 << 20) if dt == 5e-7 else (1 << 19)
        return {"kind": kind, "mech": "h2", "field": field, "n": _log_size(rng, 1000, most), "dt": dt}
    if kind == "surrogate":
        return {"kind": kind, "n": _log_size(rng, 1000, 1 << 22)}
    if kind == "step":
        return {"kind": kind, "n": _log_size(rng, 1000, 1 << 19)}
    if kind == "per_species":
        return {"kind": kind, "n": _log_size(rng, 1000, 131089)}
    if kind == "train":
        return {"kind": kind, "batch": 128 * _log_size(rng, 2, 64)}
    if kind == "transport":
        return {"kind": kind, "mech": rng.choice(["h2", "ch4"]), "n": _log_size(rng, 1000, 100003)}
    nx, ny, nz = (_log_size(rng, 12, 128) for _ in range(3))
    return {"kind": "fvm", "nx": nx, "ny": ny, "nz": nz, "permute": rng.random() < 0.5}


# ------------------------------------------------------------------------------------------
# what a program keeps: mechanisms, models, meshes
# ------------------------------------------------------------------------------------------
@functools.lru_cache(maxsize=None)
def _mech_data(name):
    return h2_mechanism() if name == "h2" else ch4_mechanism()


@functools.lru_cache(maxsize=None)
def _mech(name):
    return cg.Mechanism(_mech_data(name))


@functools.lru_cache(maxsize=None)
def _surrogate():
    return cg.Surrogate(_mech("h2"), path=MODEL)


@functools.lru_cache(maxsize=None)
def _transport_data(name):
    return generate_transport(_mech_data(name))


@functools.lru_cache(maxsize=None)
def _transport(name):
    return cg.Transport(_mech(name), _transport_data(name))


@functools.lru_cache(maxsize=None)
def _model_params():
    """The shipped network's arrays (CHEMSUR1: magic, ns, width, dt, five layers, statistics)."""
    with open(MODEL, "rb") as f:
        raw = f.read()
    ns, hid = struct.unpack_from("<ii", raw, 8)
    dt, = struct.unpack_from("<d", raw, 16)
    a = np.frombuffer(raw, "<f4", offset=24)
    dims = [ns + 2, hid, hid, hid, hid, ns]
    W, b, o = [], [], 0

    def take(*shape):
        nonlocal o
        k = int(np.prod(shape))
        o += k
        return a[o - k:o].reshape(shape).copy()

    for l in range(5):
        W.append(take(dims[l + 1], dims[l]))
        b.append(take(dims[l + 1]))
    out = {"W": W, "b": b, "dt": dt}
    for key, k in (("x_mean", ns + 2), ("x_std", ns + 2), ("y_mean", ns), ("y_std", ns), ("box_lo", ns + 2),
                   ("box_hi", ns + 2)):
        out[key] = take(k)
    return out


@functools.lru_cache(maxsize=None)
def _ps_params():
    """Per-species networks of the published widths with seeded weights, on the shipped statistics."""
    p = dict(_model_params())
    rng = np.random.default_rng(31)
    dims = (p["x_mean"].size,) + PS_HIDDEN + (1,)
    nets = {}
    for k in range(p["y_std"].size):
        if p["y_std"][k] > 0.0:
            nets[k] = {"W": [(rng.standard_normal((dims[l + 1], dims[l])) * math.sqrt(2.0 / dims[l])).astype(np.float32)
                             for l in range(4)],
                       "b": [(0.1 * rng.standard_normal(dims[l + 1])).astype(np.float32) for l in range(4)]}
    p.pop("W"), p.pop("b")
    p.update(hidden=list(PS_HIDDEN), nets=nets)
    return p


@functools.lru_cache(maxsize=None)
def _per_species():
    return cg.Surrogate(_mech("h2"), params=_ps_params())


@functools.lru_cache(maxsize=2)
def _mesh_data(nx, ny, nz, permute):
    return box_mesh(nx, ny, nz, seed=21, stretch=1.5, permute=permute)


@functools.lru_cache(maxsize=2)
def _mesh(nx, ny, nz, permute):
    return cg.FvMesh(_mesh_data(nx, ny, nz, permute))


# ------------------------------------------------------------------------------------------
# seeded states, made on the GPU
# ------------------------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device=DEV, dtype=F64)


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device=DEV, dtype=F64)


def _dev(a):
    return torch.tensor(np.ascontiguousarray(a), device=DEV)


def _table_lookup(grid, vals, x):
    """vals [m, len(grid)] linearly interpolated at x [n] -> [m, n]."""
    i = torch.clamp(torch.searchsorted(grid, x.contiguous(), right=True) - 1, 0, grid.numel() - 2)
    w = torch.clamp((x - grid[i]) / (grid[i + 1] - grid[i]), 0.0, 1.0)
    return vals[:, i] * (1.0 - w) + vals[:, i + 1] * w


def _random_field(g, nz, side, corr):
    """Unit-variance periodic Gaussian random field [nz, side, side]."""
    noise = _randn(g, nz, side, side)
    k = [torch.fft.fftfreq(m, device=DEV, dtype=F64) * 2.0 * math.pi for m in (nz, side, side)]
    k2 = k[0][:, None, None] ** 2 + k[1][None, :, None] ** 2 + k[2][None, None, :] ** 2
    f = torch.fft.ifftn(torch.fft.fftn(noise) * torch.exp(-0.5 * k2 * corr ** 2)).real
    f = f - f.mean()
    return f / f.std()


def _front_states(n, seed):
    """The quasi-DNS-shaped flame: planar fronts along x, Gaussian random fields on T and Y."""
    g = _gen(seed)
    t = {k: _dev(v) for k, v in load_table("h2_flamelet.npz").items()}
    side = 128 if n > 65536 else 32
    nz = max(side, -(-n // (side * side)))
    x = torch.arange(side, device=DEV, dtype=F64)
    s = 8.0 - torch.abs(x % 32 - 16.0)
    c = (0.5 * (1.0 + torch.tanh(s / 2.0))).repeat(-(-n // side))[:n]
    T = _table_lookup(t["c"], t["T"][None], c)[0]
    Y = _table_lookup(t["c"], t["Y"], c)
    T = T * (1.0 + 0.05 * _random_field(g, nz, side, 8.0).reshape(-1)[:n])
    for k in range(Y.shape[0]):
        Y[k] = torch.clamp(Y[k] * (1.0 + 0.10 * _random_field(g, nz, side, 8.0).reshape(-1)[:n]), min=0.0)
    Y = Y / Y.sum(0, keepdim=True)
    return T.contiguous(), torch.full_like(T, PATM), Y.contiguous()


def _mixing_states(n, seed):
    """H2/air mixing layer: Z ~ U[0, 1], T ~ U[900, 2200] K; half of the cells carry burning gas
    (a flamelet state at random progress) instead of a fresh mixture."""
    m = _mech_data("h2")
    g = _gen(seed)
    t = {k: _dev(v) for k, v in load_table("h2_flamelet.npz").items()}
    Z = _rand(g, n)
    T = 900.0 + 1300.0 * _rand(g, n)
    Y = torch.zeros((m.ns, n), device=DEV, dtype=F64)
    Y[m.index("H2")] = Z
    Y[m.index("O2")] = AIR_O2 * (1.0 - Z)
    Y[m.index("N2")] = AIR_N2 * (1.0 - Z)
    Yb = _table_lookup(t["c"], t["Y"], _rand(g, n)) * (1.0 + 0.10 * _randn(g, m.ns, n)).clamp(min=0.0)
    share = torch.where(_rand(g, n) < 0.5, _rand(g, n), torch.zeros_like(Z))
    Y = (1.0 - share) * Y + share * Yb
    Y = Y / Y.sum(0, keepdim=True)
    return T.contiguous(), torch.full_like(T, PATM), Y.contiguous()


def _les_states(n, seed):
    """The LES-shaped CH4 field: Z ~ Beta(mean 0.3, var 0.05), c ~ U[0, 1], 5 % noise on T."""
    g = _gen(seed)
    t = {k: _dev(v) for k, v in load_table("ch4_flamelet.npz").items()}
    a, b = beta_params(0.3, 0.05)
    ga = torch._standard_gamma(torch.full((n,), a, device=DEV, dtype=F64), generator=g)
    gb = torch._standard_gamma(torch.full((n,), b, device=DEV, dtype=F64), generator=g)
    Z = ga / (ga + gb)
    c = _rand(g, n)
    zg, cgr = t["Z"], t["c"]
    iz = torch.clamp(torch.searchsorted(zg, Z) - 1, 0, zg.numel() - 2)
    ic = torch.clamp(torch.searchsorted(cgr, c) - 1, 0, cgr.numel() - 2)
    wz = torch.clamp((Z - zg[iz]) / (zg[iz + 1] - zg[iz]), 0.0, 1.0)
    wc = torch.clamp((c - cgr[ic]) / (cgr[ic + 1] - cgr[ic]), 0.0, 1.0)

    def bil(F):
        w0, w1 = (wz, wc) if F.dim() == 2 else (wz[:, None], wc[:, None])
        return ((1 - w0) * ((1 - w1) * F[iz, ic] + w1 * F[iz, ic + 1])
                + w0 * ((1 - w1) * F[iz + 1, ic] + w1 * F[iz + 1, ic + 1]))

    T = torch.clamp(bil(t["T"]) * (1.0 + 0.05 * _randn(g, n)), 300.0, 2200.0)
    Y = torch.clamp(bil(t["Y"]), min=0.0).T
    Y = Y / Y.sum(0, keepdim=True)
    return T.contiguous(), torch.full_like(T, PATM), Y.contiguous()


def _states(case, seed):
    return {"mixing": _mixing_states, "front": _front_states, "les": _les_states}[case.get("field", "front")](
        case["n"], seed)


def _train_inputs(case, seed):
    """One batch of normalised features and targets, and the network's starting weights."""
    g = _gen(seed)
    B, n_in, n_out = case["batch"], 11, 9
    x = _randn(g, B, n_in).float()
    hi = x.bfloat16()
    lo = (x - hi.float()).bfloat16()
    X = torch.zeros((B, PAD), dtype=torch.bfloat16, device=DEV)
    X[:, :n_in], X[:, n_in:2 * n_in], X[:, 2 * n_in:3 * n_in] = hi, lo, hi
    t = _randn(g, B, n_out).float()
    rng = np.random.default_rng(seed)
    dims = [n_in, 512, 512, 512, 512, n_out]
    W = [(rng.standard_normal((dims[l + 1], dims[l])) / math.sqrt(dims[l])).astype(np.float32) for l in range(5)]
    b = [(0.1 * rng.standard_normal(dims[l + 1])).astype(np.float32) for l in range(5)]
    return x, X, t, W, b


def _fvm_inputs(case, seed):
    m = _mesh_data(case["nx"], case["ny"], case["nz"], case["permute"])
    g = _gen(seed)
    n, nf, nb = m.n_cells, m.owner.size, m.b_cell.size
    u = lambda lo, hi, k: lo + (hi - lo) * _rand(g, k)
    kw = dict(dt=1e-6, rho=u(2e-4, 1.2e-3, n), rho_old=u(2e-4, 1.2e-3, n), Y_old=u(0.0, 0.3, n),
              phi=1e-6 * _randn(g, nf), phi_b=1e-6 * _randn(g, nb), gamma=u(1e-4, 1e-3, n),
              gamma_b=u(1e-4, 1e-3, nb), Y_b=u(0.0, 0.3, nb), S=_randn(g, n))
    pasr = dict(tau_c=10.0 ** u(-7.0, -2.0, n), rho=kw["rho"], mu=u(1e-4, 6e-4, n), strain=10.0 ** u(1.0, 5.0, n),
                delta=torch.full((n,), 1.0 / 128, device=DEV, dtype=F64))
    return kw, pasr


# ------------------------------------------------------------------------------------------
# prepare and run
# ------------------------------------------------------------------------------------------
def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind}
    if kind == "train":
        _, s["X"], s["t"], W, b = _train_inputs(case, seed)
        s["tr"] = Trainer(11, 9, case["batch"], W=W, b=b)
        s["loss"] = torch.zeros(1, dtype=F64, device=DEV)
        s["out"] = torch.empty((case["batch"], 9), dtype=torch.float32, device=DEV)
        s["flat"] = torch.empty(s["tr"].grad_count(), dtype=torch.float32, device=DEV)
        return s
    if kind == "fvm":
        s["mesh"] = _mesh(case["nx"], case["ny"], case["nz"], case["permute"])
        s["kw"], s["pasr"] = _fvm_inputs(case, seed)
        return s
    if kind == "transport":
        s["mech"], s["tr"] = _mech(case["mech"]), _transport(case["mech"])
        field = {"field": "les" if case["mech"] == "ch4" else "front", "n": case["n"]}
        s["T"], s["p"], s["Y"] = _states(field, seed)
        s["mu"], s["lam"] = torch.empty_like(s["T"]), torch.empty_like(s["T"])
        s["D"] = torch.empty_like(s["Y"])
        return s
    # a solver's resident state, restored from the flow's field before each chemistry step
    s["T0"], s["p"], s["Y0"] = _states(case, seed)
    s["T"], s["Y"] = torch.empty_like(s["T0"]), torch.empty_like(s["Y0"])
    n = case["n"]
    if kind == "advance":
        s["mech"], s["dt"] = _mech(case["mech"]), case["dt"]
        s["status"] = torch.empty(n, dtype=torch.int8, device=DEV)
    elif kind == "surrogate":
        s["model"], s["dt"] = _surrogate(), _model_params()["dt"]
        s["route"] = torch.empty(n, dtype=torch.int8, device=DEV)
    elif kind == "per_species":
        s["model"] = _per_species()
    else:
        e = lambda: torch.empty_like(s["T0"])
        s.update(h0=e(), cp0=e(), q=e(), mu=e(), lam=e(), D=torch.empty_like(s["Y0"]),
                 route=torch.empty(n, dtype=torch.int8, device=DEV),
                 thermo_status=torch.empty(n, dtype=torch.int8, device=DEV))
        s["step"] = cg.Step(_mech("h2"), s["T"], s["p"], s["Y"], _model_params()["dt"], model=_surrogate(),
                            transport=_transport("h2"), **{k: s[k] for k in (
                                "h0", "cp0", "q", "route", "thermo_status", "mu", "lam", "D")})
    return s


def run(s):
    kind = s["kind"]
    if kind == "train":
        tr = s["tr"]
        tr.forward(s["X"], s["out"])
        tr.backward(s["t"], s["loss"])
        tr.pack_grads(s["flat"])
        tr.adam(3e-4)
        return {"loss": s["loss"], "out": s["out"], "grad": s["flat"]}
    if kind == "fvm":
        kappa = cg.pasr_kappa(**s["pasr"])
        lower, upper, diag, source = s["mesh"].assemble(kappa=kappa, **s["kw"])
        vals = s["mesh"].to_csr(lower, upper, diag)
        return {"kappa": kappa, "lower": lower, "upper": upper, "diag": diag, "source": source, "csr": vals}
    if kind == "transport":
        s["tr"](s["T"], s["p"], s["Y"], mu=s["mu"], lam=s["lam"], D=s["D"])
        return {"mu": s["mu"], "lam": s["lam"], "D": s["D"]}
    if kind == "per_species":
        ynet, z, box = cg.surrogate_forward(s["model"], s["T0"], s["p"], s["Y0"], with_z=True)
        return {"ynet": ynet, "z": z, "box": box}
    s["T"].copy_(s["T0"])
    s["Y"].copy_(s["Y0"])
    if kind == "advance":
        cg.advance(s["mech"], s["T"], s["p"], s["Y"], s["dt"], status=s["status"])
        return {"T": s["T"], "Y": s["Y"], "status": s["status"]}
    if kind == "surrogate":
        cg.surrogate_advance(s["model"], s["T"], s["p"], s["Y"], s["dt"], route=s["route"])
        return {"T": s["T"], "Y": s["Y"], "route": s["route"]}
    s["step"].run(graph=True)
    return {k: s[k] for k in ("T", "Y", "h0", "cp0", "q", "route", "thermo_status", "mu", "lam", "D")}


def work(case):
    kind = case["kind"]
    if kind == "train":
        p = 11 * 512 + 3 * 512 * 512 + 512 * 9
        # X, targets and predictions; weights, gradients and both moments (read and written)
        return {"bytes": case["batch"] * (PAD * 2 + 9 * 8) + p * 4 * 7.0, "flops": 6.0 * p * case["batch"]}
    if kind == "fvm":
        nx, ny, nz = case["nx"], case["ny"], case["nz"]
        n = nx * ny * nz
        nf = 3 * n - nx * ny - ny * nz - nx * nz
        nb = 2 * (nx * ny + ny * nz + nx * nz)
        nnz = n + 2 * nf
        # PaSR: 5 reads, 1 write; assembly: V, rho, rho_old, Y_old, gamma, S and kappa, addressing and
        # geometry in, ldu and source out; CSR: pattern and ldu in, values out
        byts = 48 * n + n * (72 + 4) + nf * 56 + nb * 41 + (2 * nf + nb) * 4 + nnz * 12 + 8 * (n + 2 * nf)
        return {"bytes": float(byts), "flops": float(30 * n + 18 * nf)}
    n = case["n"]
    ns = 53 if case.get("mech") == "ch4" else 9
    if kind == "transport":
        return {"bytes": 8.0 * n * (2 * ns + 4), "flops": n * (ns * (ns - 1) / 2 * 26.0 + ns * ns * 8.0 + ns * 110.0)}
    state = 8.0 * n * (2 * (ns + 1) + 1) + n
    if kind == "advance":
        # mean attempts and accepted sub-steps of each field, times the plain operations of one
        att, acc = {"front": (6.37, 4.32), "mixing": (70.0, 56.0), "les": (3.74, 2.96)}[case["field"]]
        per = (acc * 4929.0 + att * 13361.0) if ns == 9 else (acc * 97300.0 + att * 289000.0)
        return {"bytes": state, "flops": n * per}
    if kind == "surrogate":
        return {"bytes": state, "flops": n * 1.593e6}
    if kind == "step":
        return {"bytes": state + 8.0 * n * (ns + 5) + n, "flops": n * 1.6e6}
    per = 8 * 2.0 * (11 * 1600 + 1600 * 800 + 800 * 400 + 400)
    return {"bytes": 8.0 * n * (ns + 2) + 8.0 * n * ns + n, "flops": n * per}


# ------------------------------------------------------------------------------------------
# the same results in plain FP64
# ------------------------------------------------------------------------------------------
class _Kinetics:
    """NASA-7 thermo, Arrhenius / third-body / Troe rates and the constant-pressure reactor."""

    def __init__(self, m):
        d = lambda a: torch.as_tensor(np.asarray(a), device=DEV).to(F64)
        self.ns, self.nr = m.ns, m.nr
        self.W, self.lo, self.hi = d(m.W), d(m.nasa_lo), d(m.nasa_hi)
        nu = np.zeros((m.nr, m.ns))
        for j in range(m.nr):
            for k in m.reac[j]:
                if k >= 0:
                    nu[j, k] -= 1
            for k in m.prod[j]:
                if k >= 0:
                    nu[j, k] += 1
        self.nu = d(nu)
        self.dnu = self.nu.sum(1)
        pad = lambda a: torch.as_tensor(np.where(np.asarray(a) < 0, m.ns, a).astype(np.int64), device=DEV)
        self.reac, self.prod = pad(m.reac), pad(m.prod)
        self.lnA = torch.log(d(m.A))
        self.b, self.Ta = d(m.b), d(m.Ea) / (RU / 4.184e7)
        self.tb = torch.as_tensor(np.nonzero(np.asarray(m.rtype) == 1)[0], device=DEV)
        self.fo = torch.as_tensor(np.nonzero(np.asarray(m.rtype) == 2)[0], device=DEV)
        eff = d(m.eff)
        self.eff_tb, self.eff_fo = eff[self.tb], eff[self.fo]
        t = d(m.troe)[self.fo]
        self.k0 = (torch.log(t[:, 0]), t[:, 1], t[:, 2] / (RU / 4.184e7))
        self.a, self.T3, self.T1, self.T2 = t[:, 3], t[:, 4], t[:, 5], t[:, 6]
        self.h2 = d(m.has_t2)[self.fo]

    def thermo(self, T):
        """cp/R, h/RT and s/R of every species, [n, ns]."""
        T = T[:, None]
        a = torch.where((T < 1000.0)[..., None], self.lo, self.hi)
        c = a.unbind(-1)
        cp = c[0] + T * (c[1] + T * (c[2] + T * (c[3] + T * c[4])))
        h = c[0] + T * (c[1] / 2 + T * (c[2] / 3 + T * (c[3] / 4 + T * c[4] / 5))) + c[5] / T
        s = c[0] * torch.log(T) + T * (c[1] + T * (c[2] / 2 + T * (c[3] / 3 + T * c[4] / 4))) + c[6]
        return cp, h, s

    def h_mass(self, T, Y):
        return RU * T * ((Y / self.W) * self.thermo(T)[1]).sum(1)

    def cp_mass(self, T, Y):
        return RU * ((Y / self.W) * self.thermo(T)[0]).sum(1)

    def rhs(self, y, p):
        """d(T, Y)/dt of [n, ns + 1] states."""
        T, Y = y[:, 0], y[:, 1:]
        cp, h, s = self.thermo(T)
        yw = Y / self.W
        S = yw.sum(1)
        rho = p / (RU * T * S)
        C = rho[:, None] * yw
        C1 = torch.cat([C, torch.ones_like(T)[:, None]], 1)
        lnT, iT = torch.log(T)[:, None], (1.0 / T)[:, None]
        kf = torch.exp(self.lnA + self.b * lnT - self.Ta * iT)
        mult = torch.ones_like(kf)
        if self.tb.numel():
            mult = mult.index_copy(1, self.tb, C @ self.eff_tb.T)
        if self.fo.numel():
            M = C @ self.eff_fo.T
            kinf = kf[:, self.fo]
            k0 = torch.exp(self.k0[0] + self.k0[1] * lnT - self.k0[2] * iT)
            Fc = ((1 - self.a) * torch.exp(-T[:, None] / self.T3) + self.a * torch.exp(-T[:, None] / self.T1)
                  + self.h2 * torch.exp(-self.T2 * iT))
            Pr = k0 * M / kinf
            L = torch.log10(Fc)
            u = torch.log10(Pr) - 0.4 - 0.67 * L
            f1 = u / (0.75 - 1.27 * L - 0.14 * u)
            F = 10.0 ** (L / (1.0 + f1 * f1))
            kf = kf.index_copy(1, self.fo, kinf * (Pr / (1.0 + Pr)) * F)
        dG = (h - s) @ self.nu.T
        kr = kf * torch.exp(dG - self.dnu * (math.log(1.01325e6 / RU) - lnT))
        cr, cpd = C1[:, self.reac], C1[:, self.prod]
        q = mult * (kf * (cr[..., 0] * cr[..., 1] * cr[..., 2]) - kr * (cpd[..., 0] * cpd[..., 1] * cpd[..., 2]))
        w = q @ self.nu
        dT = -(RU * T[:, None] * h * w).sum(1) / (rho * RU * (yw * cp).sum(1))
        return torch.cat([dT[:, None], self.W * w / rho[:, None]], 1)

    def jacobian(self, y, p):
        """df_i/dy_j by forward differentiation, one unknown at a time."""
        f = lambda v: self.rhs(v, p)
        cols = []
        for j in range(self.ns + 1):
            t = torch.zeros_like(y)
            t[:, j] = 1.0
            cols.append(torch.func.jvp(f, (y,), (t,))[1])
        return torch.stack(cols, 2)


# Rodas4 (Hairer & Wanner, Solving ODEs II, IV.7), transformed form
_RA = [[], [1.544], [0.9466785280815826, 0.2557011698983284],
       [3.314825187068521, 2.896124015972201, 0.9986419139977817],
       [1.221224509226641, 6.019134481288629, 12.53708332932087, -0.6878860361058950],
       [1.221224509226641, 6.019134481288629, 12.53708332932087, -0.6878860361058950, 1.0]]
_RC = [[], [-5.6688], [-2.430093356833875, -0.2063599157091915],
       [-0.1073529058151375, -9.594562251023355, -20.47028614809616],
       [7.496443313967647, -10.24680431464352, -33.99990352819905, 11.70890893206160],
       [8.083246795921522, -7.981132988064893, -31.52159432874371, 16.31930543123136, -6.058818238834054]]
_RM = [1.221224509226641, 6.019134481288629, 12.53708332932087, -0.6878860361058950, 1.0, 1.0]


def _rodas4(kin, T, p, Y, dt, rtol=1e-6, atol=1e-10):
    """Adaptive Rodas4 over [0, dt] from h = dt, all cells at once (finished cells drop out)."""
    y_all = torch.cat([T[:, None], Y.T], 1)
    live = torch.arange(T.numel(), device=DEV)
    t = torch.zeros_like(T)
    h = torch.full_like(T, dt)
    fmax = torch.full_like(T, 6.0)
    N = kin.ns + 1
    eye = torch.eye(N, device=DEV, dtype=F64)
    while live.numel():
        y, pl = y_all[live], p[live]
        last = h >= dt - t
        h = torch.where(last, dt - t, h)
        f0 = kin.rhs(y, pl)
        LU, piv = torch.linalg.lu_factor(eye / (0.25 * h)[:, None, None] - kin.jacobian(y, pl))
        u = []
        for s in range(6):
            f = f0 if s == 0 else kin.rhs(y + sum(a * v for a, v in zip(_RA[s], u)), pl)
            g = f + sum((c / h)[:, None] * v for c, v in zip(_RC[s], u)) if s else f
            u.append(torch.linalg.lu_solve(LU, piv, g[..., None])[..., 0])
        yn = y + sum(m * v for m, v in zip(_RM, u))
        sc = atol + rtol * torch.maximum(y.abs(), yn.abs())
        en = torch.sqrt(((u[5] / sc) ** 2).sum(1) / N)
        fac = torch.where(torch.isfinite(en), torch.clamp(0.9 * en ** -0.25, min=0.2), torch.full_like(en, 0.2))
        ok = en <= 1.0
        y_all[live] = torch.where(ok[:, None], yn, y)
        t = torch.where(ok, t + h, t)
        done = ok & last
        h = h * torch.where(ok, torch.minimum(fac, fmax), fac)
        fmax = torch.where(ok, torch.full_like(h, 6.0), torch.ones_like(h))
        keep = ~done
        live, t, h, fmax = live[keep], t[keep], h[keep], fmax[keep]
    return y_all


def _advanced(kin, T, p, Y, dt, chunk):
    got = [_rodas4(kin, T[i:i + chunk], p[i:i + chunk], Y[:, i:i + chunk], dt) for i in range(0, T.numel(), chunk)]
    y = torch.cat(got)
    return y[:, 0].contiguous(), y[:, 1:].T.contiguous()


def _gelu(v):
    return 0.5 * v * (1.0 + torch.erf(v / math.sqrt(2.0)))


def _boxcox(Y):
    return (torch.clamp(Y, min=0.0) ** 0.1 - 1.0) / 0.1


def _features(p_, T, p, Y):
    x = torch.cat([T[:, None], torch.log(p)[:, None], _boxcox(Y).T], 1)
    return (x - _dev(p_["x_mean"]).to(F64)) / _dev(np.where(p_["x_std"] > 0, p_["x_std"], 1.0)).to(F64)


def _dense(x, Ws, bs):
    for l, (W, b) in enumerate(zip(Ws, bs)):
        x = x @ _dev(W).to(F64).T + _dev(b).to(F64)
        if l + 1 < len(Ws):
            x = _gelu(x)
    return x


def _inverse(p_, Y, z):
    d = z * _dev(p_["y_std"]).to(F64) + _dev(p_["y_mean"]).to(F64)
    return (torch.clamp(1.0 + 0.1 * (_boxcox(Y).T + d), min=0.0) ** 10.0).T


def _surrogate_step(kin, T, p, Y):
    """Network, element-conservation projection, clipping and T from enthalpy."""
    q, m = _model_params(), _mech_data("h2")
    Yn = _inverse(q, Y, _dense(_features(q, T, p, Y), q["W"], q["b"])).T
    A = _dev(np.asarray(m.comp, np.float64).T * np.asarray(m.elem_mass)[:, None] / np.asarray(m.W)[None])
    D = Yn + 1e-12
    G = torch.einsum("ek,nk,fk->nef", A, D, A)
    lam = torch.linalg.solve(G, ((Yn - Y.T) @ A.T)[..., None])[..., 0]
    Yn = torch.clamp(Yn - D * (lam @ A), min=0.0)
    h0 = kin.h_mass(T, Y.T)
    Tn = T.clone()
    for _ in range(12):
        Tn = torch.clamp(Tn - (kin.h_mass(Tn, Yn) - h0) / kin.cp_mass(Tn, Yn), 200.0, 6000.0)
    return Tn, Yn.T.contiguous(), h0


def _transport_exact(name, T, p, Y):
    m, t = _mech_data(name), _transport_data(name)
    W = _dev(np.asarray(m.W, np.float64))
    d = lambda a: torch.as_tensor(a, device=DEV)
    wq = (W[None, :] / W[:, None]) ** 0.25                      # [k, j]: (W_j / W_k)^(1/4)
    cw = 1.0 / torch.sqrt(8.0 * (1.0 + W[:, None] / W[None, :]))  # [k, j]
    eye = torch.eye(m.ns, dtype=torch.bool, device=DEV)
    mu_all, lam_all, D_all = [], [], []
    for i in range(0, T.numel(), 4096):
        L = torch.log(T[i:i + 4096])
        V = torch.stack([torch.ones_like(L), L, L ** 2, L ** 3], 1)
        mu, lam = torch.exp(V @ d(t.mu_poly).T), torch.exp(V @ d(t.lambda_poly).T)
        y = Y[:, i:i + 4096].T
        X = y / W
        X = X / X.sum(1, keepdim=True)
        r = torch.sqrt(mu[:, :, None] / mu[:, None, :])
        den = (X[:, None, :] * (1.0 + r * wq) ** 2 * cw).sum(2)
        mu_all.append((X * mu / den).sum(1))
        lam_all.append(0.5 * ((X * lam).sum(1) + 1.0 / (X / lam).sum(1)))
        iD = torch.exp(-torch.einsum("nc,jkc->njk", V, d(t.diff_poly))) * (p[i:i + 4096] / 1.01325e6)[:, None, None]
        D_all.append(((1.0 - y) / (X[:, :, None] * iD.masked_fill(eye, 0.0)).sum(1)).T)
    return torch.cat(mu_all), torch.cat(lam_all), torch.cat(D_all, 1).contiguous()


def _train_exact(case, seed):
    x, X, t, W, b = _train_inputs(case, seed)
    n_in = x.shape[1]
    x = (X[:, :n_in].to(F64) + X[:, n_in:2 * n_in].to(F64))
    P = [(_dev(w).to(F64).requires_grad_(), _dev(v).to(F64).requires_grad_()) for w, v in zip(W, b)]
    v = x
    for l, (w, c) in enumerate(P):
        v = v @ w.T + c
        if l + 1 < len(P):
            v = _gelu(v)
    loss = ((v - t.to(F64)) ** 2).mean()
    loss.backward()
    grad = torch.cat([g.grad.reshape(-1) for pair in P for g in pair])
    return {"loss": loss.detach().reshape(1), "out": v.detach(), "grad": grad}


def _fvm_exact(case, seed):
    m = _mesh_data(case["nx"], case["ny"], case["nz"], case["permute"])
    kw, q = _fvm_inputs(case, seed)
    nu = (0.17 * q["delta"]) ** 2 * q["strain"]
    eps = nu * q["strain"] ** 2
    kappa = q["tau_c"] / (q["tau_c"] + torch.sqrt((q["mu"] + q["rho"] * nu) / (q["rho"] * eps)))
    i64 = lambda a: torch.as_tensor(np.asarray(a), device=DEV).long()
    o, nb, bc = i64(m.owner), i64(m.neighbour), i64(m.b_cell)
    V, w = _dev(m.volume), _dev(m.weight)
    c = (w * kw["gamma"][o] + (1.0 - w) * kw["gamma"][nb]) * _dev(m.mag_sf) * _dev(m.delta)
    F = kw["phi"]
    upper, lower = torch.clamp(F, max=0.0) - c, torch.clamp(-F, max=0.0) - c
    diag = kw["rho"] * V / kw["dt"]
    source = kw["rho_old"] * kw["Y_old"] * V / kw["dt"] + V * kappa * kw["S"]
    diag = diag.index_add(0, o, torch.clamp(F, min=0.0) + c).index_add(0, nb, torch.clamp(-F, min=0.0) + c)
    cb = torch.where(i64(m.b_type) == 1, kw["gamma_b"] * _dev(m.b_mag_sf) * _dev(m.b_delta), torch.zeros_like(kw["phi_b"]))
    diag = diag.index_add(0, bc, torch.clamp(kw["phi_b"], min=0.0) + cb)
    source = source.index_add(0, bc, (cb - torch.clamp(kw["phi_b"], max=0.0)) * kw["Y_b"])
    row = torch.cat([torch.arange(m.n_cells, device=DEV), o, nb])
    col = torch.cat([torch.arange(m.n_cells, device=DEV), nb, o])
    csr = torch.cat([diag, upper, lower])[torch.argsort(row * m.n_cells + col)]
    return {"kappa": kappa, "lower": lower, "upper": upper, "diag": diag, "source": source, "csr": csr}


def exact(case, seed):
    kind = case["kind"]
    if kind == "train":
        return _train_exact(case, seed)
    if kind == "fvm":
        return _fvm_exact(case, seed)
    if kind == "transport":
        T, p, Y = _states({"field": "les" if case["mech"] == "ch4" else "front", "n": case["n"]}, seed)
        return dict(zip(("mu", "lam", "D"), _transport_exact(case["mech"], T, p, Y)))
    if kind == "advance" and case["mech"] == "ch4" and case["n"] > 4096:
        return None                       # 54 unknowns a cell: minutes in plain torch
    T, p, Y = _states(case, seed)
    if kind == "per_species":
        q = _ps_params()
        z = torch.zeros((T.numel(), Y.shape[0]), device=DEV, dtype=F64)
        x = _features(q, T, p, Y)
        for k, net in q["nets"].items():
            for i in range(0, T.numel(), 32768):
                z[i:i + 32768, k] = _dense(x[i:i + 32768], net["W"], net["b"])[:, 0]
        return {"ynet": _inverse(q, Y, z).contiguous(), "z": z.T.contiguous(), "box": None}
    kin = _Kinetics(_mech_data(case.get("mech", "h2")))
    if kind == "advance":
        T1, Y1 = _advanced(kin, T, p, Y, case["dt"], 131072 if case["mech"] == "h2" else 512)
        return {"T": T1, "Y": Y1, "status": None}
    parts = [_surrogate_step(kin, T[i:i + 131072], p[i:i + 131072], Y[:, i:i + 131072])
             for i in range(0, T.numel(), 131072)]
    T1, Y1, h0 = torch.cat([a[0] for a in parts]), torch.cat([a[1] for a in parts], 1), torch.cat([a[2] for a in parts])
    if kind == "surrogate":
        return {"T": T1, "Y": Y1.contiguous(), "route": None}
    h = kin.thermo(T)[1] * RU * T[:, None]
    rho = p / (RU * T * (Y.T / kin.W).sum(1))
    q = -rho * (h * (Y1 - Y).T / kin.W).sum(1) / _model_params()["dt"]
    mu, lam, D = _transport_exact("h2", T1, p, Y1)
    return {"T": T1, "Y": Y1.contiguous(), "h0": h0, "cp0": kin.cp_mass(T, Y.T), "q": q, "route": None,
            "thermo_status": None, "mu": mu, "lam": lam, "D": D}
