"""The work that a user has this library do, as cases to be timed: one pass through the public entry points each.

A case is a dict of plain values. `kind` names the call chain, the other values its sizes and options:

  forward      neighbours, then coefficients and power spectrum: the feature calculator
  neighbours   the periodic pair list alone
  selected     neighbours, then coefficients and a listed part of the power spectrum
  forces       neighbours, coefficients, power spectrum, linear energy, forces and virial: a step of dynamics
  gpr          the same with the sparse GPR energy model: dE/dp from the model, forces from dE/dp
  spectrum     power spectrum of stored coefficients
  equivariants rank-lambda equivariants of stored coefficients
  surrogate    neighbours, then coefficients with the radial integrals of the learned network
  training     loss and parameter gradient of one minibatch of that network

Structures are thermally displaced lattices with vacancies: n of the m^3 >= n sites of a cubic lattice, each moved
inside a cube that keeps any two atoms d_min apart, which gives the pair counts and pair distances of a liquid.
`exact` is the same result from plain torch in 64 bits: brute-force pairs, the series of the 1F1 radial integrals on a
fine grid (Hermite interpolation, error below 1e-12), harmonics by recurrence, gradients by automatic differentiation.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2101_08814_gb300 import DeviceSystem, GprModel, SoapCalculator
from paper_2101_08814_gb300.autograd import LinearSoapEnergy

LABELS = [1, 6, 7, 8, 9, 15, 16, 17]
HIDDEN = 64  # hidden width of the learned radial network (the one the library supports)


def _hypers(r_cut, sigma, n_max, l_max, species):
    return dict(r_cut=r_cut, sigma=sigma, n_max=n_max, l_max=l_max, species=species)


def _cells(cells, lo, hi, density, d_min, periodic=True):
    return dict(cells=cells, atoms_lo=lo, atoms_hi=hi, density=density, d_min=d_min, periodic=periodic)


def listed():
    batch = _hypers(5.0, 0.5, 12, 9, 4)
    large = _hypers(6.0, 0.5, 10, 8, 3)
    return [
        # a single small crystal cell: what a script computes one structure at a time; latency and launches count
        dict(name="one_small_cell", kind="forward", **_cells(1, 64, 64, 0.064, 2.0), **_hypers(5.0, 0.5, 8, 6, 1),
             precision="fp32", layout="packed", include_center=False),
        # a data set of 512 molecular cells turned into features: the library's headline workload
        dict(name="dataset_features", kind="forward", **_cells(512, 64, 216, 0.05, 1.8), **batch, precision="fp32",
             layout="packed", include_center=False),
        # isolated molecules of 9 to 29 atoms, five species, the square layout and the centre's own density: a small
        # odd-sized basis, short neighbour lists, no periodicity
        dict(name="molecules_full", kind="forward", **_cells(1500, 9, 29, 0.09, 1.0, False), **_hypers(4.5, 0.4, 7, 5, 5),
             precision="fp32", layout="full", include_center=True),
        # neighbour list of a dense 32768-atom liquid, the first call of every step
        dict(name="liquid_neighbours", kind="neighbours", **_cells(1, 32768, 32768, 0.1, 1.0), **large),
        # a tenth of the features, as a fitted model with feature selection asks for
        dict(name="selected_features", kind="selected", **_cells(256, 64, 216, 0.05, 1.8), **batch, fraction=0.1),
        # a step of dynamics with the linear model: 4096 atoms, two species
        dict(name="dynamics_4096", kind="forces", **_cells(1, 4096, 4096, 0.05, 1.8), **_hypers(5.5, 0.4, 8, 6, 2)),
        # the same for the 32768-atom liquid, 90 neighbours per atom
        dict(name="dynamics_32768", kind="forces", **_cells(1, 32768, 32768, 0.1, 1.0), **large),
        # a step with the sparse GPR model, 256 sparse points per species, molecular cells
        dict(name="gpr_dynamics", kind="gpr", **_cells(64, 64, 216, 0.05, 1.8), **batch, sparse=256, zeta=2),
        # power spectrum of stored coefficients with 16-bit inputs on the tensor cores
        dict(name="spectrum_bf16", kind="spectrum", centres=20000, **batch, precision="bf16", layout="packed"),
        # rank-1 equivariants (dipoles) of stored coefficients
        dict(name="equivariants_1", kind="equivariants", centres=9001, **batch, rank=1),
        # coefficients with the learned radial integrals: 8192 atoms, eight species, the widest basis
        dict(name="surrogate_8192", kind="surrogate", **_cells(1, 8192, 8192, 0.06, 1.6), **_hypers(6.0, 0.5, 16, 12, 8)),
        # one minibatch of the network's training
        dict(name="training_4096", kind="training", batch=4096, **_hypers(6.0, 0.5, 16, 12, 8)),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["forward", "forward", "neighbours", "selected", "forces", "forces", "gpr", "spectrum",
                       "equivariants", "surrogate", "training"])
    S = rng.randint(1, 5)
    n_max = rng.randint(4, min(14, 60 // S))
    l_max = rng.randint(3, 9)
    h = _hypers(round(rng.uniform(4.0, 6.0), 2), round(rng.uniform(0.35, 0.55), 2), n_max, l_max, S)
    if kind == "training":
        return dict(kind=kind, batch=log_int(300, 4096), **h)
    Q = S * n_max
    if kind in ("spectrum", "equivariants"):
        rank = rng.randint(0, 3)
        per = 4.0 * Q * Q * (l_max + 1) * (2 * rank + 1 if kind == "equivariants" else 1)
        case = dict(kind=kind, centres=min(log_int(65, 20000), int(1.0e9 / per)), **h)
        if kind == "equivariants":
            return dict(case, rank=rank)
        return dict(case, precision=rng.choice(["fp32", "bf16", "tf32x3"]), layout=rng.choice(["packed", "full"]))
    density = round(rng.uniform(0.04, 0.1), 4)
    d_min = round(0.55 * density ** (-1.0 / 3.0), 2)
    most = min(30000, int(1.5e9 / (4.0 * Q * Q * (l_max + 1))))
    atoms = log_int(60, most)
    if rng.random() < 0.5:  # one cell, or many of 20 to 200 atoms
        cells = _cells(1, atoms, atoms, density, d_min)
    else:
        lo = rng.randint(20, 100)
        hi = lo + rng.randint(0, 100)
        cells = _cells(max(2, 2 * atoms // (lo + hi)), lo, hi, density, d_min, rng.random() < 0.7)
    case = dict(kind=kind, **cells, **h)
    if kind == "forward":
        return dict(case, precision=rng.choice(["fp32", "fp32", "tf32x3"]), layout=rng.choice(["packed", "packed", "full"]),
                    include_center=rng.random() < 0.3)
    if kind == "selected":
        return dict(case, fraction=round(rng.uniform(0.03, 0.3), 3))
    if kind == "gpr":
        return dict(case, sparse=rng.randint(17, 256), zeta=rng.randint(1, 4))
    return case


# ------------------------------------------------------------------------------------------------------- inputs
def _structures(case, seed):
    """positions [N, 3], species [N], cells [n_s, 3, 3], pbc [n_s, 3], offsets [n_s + 1] (numpy).

    The atom counts belong to the case, the rest to the seed. A pair list's length has to belong to the case too: there
    the seed moves the origin of one and the same arrangement, permutes its axes and renumbers its atoms."""
    rng = np.random.default_rng([int(seed), 1])
    counts = np.random.default_rng([case["cells"], case["atoms_lo"], case["atoms_hi"]]).integers(
        case["atoms_lo"], case["atoms_hi"] + 1, case["cells"])
    fixed = case["kind"] == "neighbours"
    base = np.random.default_rng(8) if fixed else rng
    pos, cells, offs = [], [], [0]
    for n in counts.tolist():
        L = (n / case["density"]) ** (1.0 / 3.0)
        m = math.ceil(round(n ** (1.0 / 3.0), 9))
        site = np.sort(base.permutation(m ** 3)[:n])
        grid = np.stack([site // (m * m), (site // m) % m, site % m], axis=1) + 0.5
        slack = max(0.0, 0.5 * (L / m - case["d_min"]))
        x = grid * (L / m) + base.uniform(-slack, slack, (n, 3))
        if fixed:
            x = x[rng.permutation(n)][:, rng.permutation(3)] + rng.uniform(0.0, L, 3) * case["periodic"]
        pos.append(np.mod(x, L) if case["periodic"] else x)
        cells.append(np.eye(3) * (L if case["periodic"] else 3.0 * L))
        offs.append(offs[-1] + n)
    n = offs[-1]
    species = np.asarray(LABELS[:case["species"]], dtype=np.int32)[rng.integers(0, case["species"], n)]
    pbc = np.full((case["cells"], 3), 1 if case["periodic"] else 0, dtype=np.int32)
    return np.concatenate(pos), species, np.stack(cells), pbc, np.asarray(offs, dtype=np.int32)


def _device_system(arrays):
    pos, species, cells, pbc, offs = arrays
    put = lambda a, t: torch.as_tensor(a, dtype=t).cuda().contiguous()  # noqa: E731
    return DeviceSystem(put(pos, torch.float64), put(species, torch.int32), put(cells, torch.float64), put(pbc, torch.int32),
                        put(offs, torch.int32))


def _calculator(case):
    return SoapCalculator(case["r_cut"], case["sigma"], case["n_max"], case["l_max"], LABELS[:case["species"]],
                          smooth_width=0.5, include_center=case.get("include_center", False))


def _n_features(case):
    Q = case["species"] * case["n_max"]
    return (case["l_max"] + 1) * Q * (Q + 1) // 2


def _generator(seed, k):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1000003 + k) % (1 << 62))
    return g


def _stored_coefficients(case, seed):
    """Coefficients as an expansion leaves them: magnitudes falling with n and l, blocks of absent species zero."""
    g = _generator(seed, 2)
    n, S, n_max, l_max = case["centres"], case["species"], case["n_max"], case["l_max"]
    c = torch.randn((n, S, n_max, (l_max + 1) ** 2), generator=g, device="cuda")
    c *= torch.exp(-0.25 * torch.arange(n_max, device="cuda"))[:, None]
    c *= torch.repeat_interleave(torch.exp(-0.2 * torch.arange(l_max + 1.0, device="cuda")),
                                 2 * torch.arange(l_max + 1, device="cuda") + 1)
    c *= (torch.rand((n, S, 1, 1), generator=g, device="cuda") < 0.95)
    return c.contiguous()


def _selection(case, seed):
    F = _n_features(case)
    rng = np.random.default_rng([int(seed), 3])
    return np.sort(rng.permutation(F)[:max(1, int(F * case["fraction"]))]).astype(np.int32)


def _linear_weights(case, seed):
    rng = np.random.default_rng([int(seed), 4])
    return rng.standard_normal((case["species"], _n_features(case))).astype(np.float32)


def _sparse_model(case, seed):
    """Sparse points (64-bit power spectra of environments of other structures), their species and weights."""
    per = case["sparse"]
    train = dict(case, cells=max(1, -(-2 * per * case["species"] // 100)), atoms_lo=100, atoms_hi=100)
    arrays = _structures(train, seed + 77)
    species = np.searchsorted(LABELS[:case["species"]], arrays[1])
    rng = np.random.default_rng([int(seed), 5])
    pick = np.concatenate([rng.permutation(np.flatnonzero(species == a))[:per] for a in range(case["species"])])
    pick = torch.as_tensor(np.sort(pick)).cuda()
    p = _spectrum64(train, _expansion64(train, arrays)[pick], "packed")
    return p.reshape(len(pick), -1), species[pick.cpu().numpy()], rng.standard_normal(len(pick))


def _network(case, seed):
    """Parameters [W1 | b1 | W2 | b2 | W3 | b3] and output scales of the 1 -> 64 -> 64 -> F network, float32."""
    rng = np.random.default_rng([int(seed), 6])
    F = case["n_max"] * (case["l_max"] + 1)
    parts = [2.0 * rng.standard_normal(HIDDEN), rng.uniform(-2.0, 2.0, HIDDEN),
             rng.standard_normal(HIDDEN * HIDDEN) / math.sqrt(HIDDEN), 0.1 * rng.standard_normal(HIDDEN),
             rng.standard_normal(F * HIDDEN) / math.sqrt(HIDDEN), 0.1 * rng.standard_normal(F)]
    table = _radial_table64(case)[0].abs().amax(dim=0)                       # [n, l]
    return np.concatenate(parts).astype(np.float32), table.t().reshape(-1).cpu().numpy().astype(np.float32)


def _minibatch(case, seed):
    """Inputs t = r / r_cut [B] and scaled targets [B, F] (f = l n_max + n), float32 on the device."""
    g = _generator(seed, 7)
    t = torch.rand(case["batch"], generator=g, device="cuda")
    values = _radial64(case, t.double() * case["r_cut"])                     # [B, n, l]
    scale = _radial_table64(case)[0].abs().amax(dim=0)
    y = (values / scale).transpose(1, 2).reshape(case["batch"], -1)
    return t, y.float().contiguous()


def prepare(case, seed):
    kind = case["kind"]
    state = dict(case=case, calc=_calculator(case))
    if kind in ("spectrum", "equivariants"):
        return dict(state, coeffs=_stored_coefficients(case, seed))
    if kind == "training":
        state["calc"].mlp_set_params(*_network(case, seed))
        t, y = _minibatch(case, seed)
        return dict(state, t=t, y=y)
    state["system"] = _device_system(_structures(case, seed))
    if kind == "selected":
        state["sel"] = torch.as_tensor(_selection(case, seed)).cuda()
    elif kind == "forces":
        state["model"] = LinearSoapEnergy(state["calc"], torch.as_tensor(_linear_weights(case, seed)))
    elif kind == "gpr":
        M, a, x = _sparse_model(case, seed)
        state["model"] = GprModel(state["calc"], M.cpu().numpy(), np.asarray(LABELS, dtype=np.int32)[a], x, zeta=case["zeta"])
    elif kind == "surrogate":
        state["calc"].mlp_set_params(*_network(case, seed))
        state["calc"].set_radial("mlp")
    return state


def run(state):
    case, calc = state["case"], state["calc"]
    kind = case["kind"]
    if kind == "spectrum":
        return {"p": calc.power_spectrum(state["coeffs"], precision=case["precision"], layout=case["layout"])}
    if kind == "equivariants":
        return {"t": calc.lambda_soap(state["coeffs"], case["rank"])}
    if kind == "training":
        g, loss = calc.mlp_gradients(state["t"], state["y"])
        return {"grad": g, "loss": loss}
    system = state["system"]
    if kind == "forces":
        energy, forces, virial = state["model"](system)
        # sums of 32-bit terms; a program that learns or moves atoms with them goes on in 32 bits
        return {"energy": energy.float(), "forces": forces.float(), "virial": virial.float()}
    pairs = calc.neighbours(system)
    if kind == "neighbours":
        return {"offsets": pairs.offsets, "j": pairs.nbr_j, "shifts": pairs.shifts, "rij": pairs.rij}
    if kind == "forward":
        c, p = calc.soap(system, pairs, layout=case["layout"], precision=case["precision"])
        return {"c": c, "p": p}
    if kind == "selected":
        c, p = calc.soap_selected(system, pairs, state["sel"])
        return {"c": c, "p": p}
    if kind == "surrogate":
        return {"c": calc.spherical_expansion(system, pairs)}
    c, p = calc.soap(system, pairs)
    energy, atomic, grad = state["model"].predict(system, p, grad=True)
    forces, virial = calc.gradients(system, pairs, c, grad_ps=grad)
    return {"energy": energy.float(), "atomic": atomic, "grad": grad, "forces": forces.float(), "virial": virial.float()}


def work(case):
    kind, S, n_max, L1 = case["kind"], case["species"], case["n_max"], case["l_max"] + 1
    Q, n_lm, F = S * n_max, L1 * L1, _n_features(case)
    if kind == "training":
        B, out = case["batch"], n_max * L1
        weights = HIDDEN * (HIDDEN + out)
        return {"bytes": 4.0 * B * (out + 1) + 8.0 * (weights + 3 * HIDDEN + out), "flops": 6.0 * B * weights}
    gram = 2.0 * n_lm * Q * (Q + 1) / 2  # flops of one centre's packed power spectrum
    if kind == "spectrum":
        f_out = F if case["layout"] == "packed" else L1 * Q * Q
        return {"bytes": 4.0 * case["centres"] * (Q * n_lm + f_out), "flops": case["centres"] * gram}
    if kind == "equivariants":
        lam, flops, out = case["rank"], 0.0, 0
        for l1 in range(L1):
            for l2 in range(l1, L1):
                if l2 - l1 <= lam <= l1 + l2 and (l1 + l2 + lam) % 2 == 0:
                    flops += 2.0 * (2 * lam + 1) * Q * Q * (2 * l2 + 1)
                    out += (2 * lam + 1) * Q * Q
        return {"bytes": 4.0 * case["centres"] * (Q * n_lm + out), "flops": case["centres"] * flops}
    mean = 0.5 * (case["atoms_lo"] + case["atoms_hi"])
    atoms = case["cells"] * mean
    pairs = atoms * min(4.18879 * case["r_cut"] ** 3 * case["density"], mean if not case["periodic"] else 1e9)
    given = 28.0 * atoms + 88.0 * case["cells"]
    if kind == "neighbours":
        return {"bytes": given + 8.0 * atoms + 32.0 * pairs, "flops": 8.0 * pairs}
    expansion = 2.0 * n_max * n_lm * pairs
    coeffs = 4.0 * atoms * Q * n_lm
    if kind == "surrogate":
        out = n_max * L1
        return {"bytes": given + coeffs, "flops": expansion + 2.0 * pairs * HIDDEN * (HIDDEN + out)}
    if kind == "forward":
        f_out = F if case["layout"] == "packed" else L1 * Q * Q
        return {"bytes": given + coeffs + 4.0 * atoms * f_out, "flops": expansion + atoms * gram}
    if kind == "selected":
        return {"bytes": given + coeffs + 4.0 * atoms * int(F * case["fraction"]),
                "flops": expansion + atoms * gram * case["fraction"]}
    back = 2.0 * 2.0 * Q * Q * n_lm / 2 * atoms + 10.0 * n_max * n_lm * pairs
    if kind == "forces":
        return {"bytes": given + 4.0 * S * F + 24.0 * atoms + 80.0 * case["cells"], "flops": expansion + atoms * gram + back}
    gemm = 2.0 * 2.0 * atoms * case["sparse"] * F  # kernel and its gradient
    return {"bytes": given + 4.0 * S * case["sparse"] * F + 4.0 * atoms * F + 28.0 * atoms,
            "flops": expansion + atoms * gram + gemm + back}


# ------------------------------------------------------------------------------------- the same in 64 bits, plain torch
def _pairs64(case, arrays):
    """Brute-force pairs (i, j, r_ji) in the order (i, j, n1, n2, n3)."""
    pos, _, cells, pbc, offs = arrays
    rc = case["r_cut"]
    out_i, out_j, out_r, out_k = [], [], [], []
    x_all = torch.as_tensor(pos).cuda()
    for s in range(len(offs) - 1):
        a, b = int(offs[s]), int(offs[s + 1])
        L = float(cells[s, 0, 0])
        R = math.ceil(rc / L) if pbc[s, 0] else 0
        x = x_all[a:b]
        n = torch.cartesian_prod(*[torch.arange(-R, R + 1, device="cuda")] * 3).reshape(-1, 3)
        step = max(1, int(4e6 // (b - a)))
        for lo in range(0, b - a, step):
            hi = min(b - a, lo + step)
            rel = x[None, :, :] - x[lo:hi, None, :]                          # [i, j, 3]
            each = max(1, int(2e7 // ((hi - lo) * (b - a))))                 # images at a time
            for k0 in range(0, len(n), each):
                nk = n[k0:k0 + each]
                d2 = 0.0
                for ax in range(3):
                    d2 = d2 + (rel[None, :, :, ax] + nk[:, ax, None, None] * L) ** 2
                keep = d2 < rc * rc
                own = (nk == 0).all(dim=1).nonzero().flatten()
                if len(own):
                    keep[own[0], torch.arange(hi - lo), torch.arange(lo, hi)] = False
                k, i, j = keep.nonzero(as_tuple=True)
                sh = nk[k]
                out_i.append(i + (lo + a))
                out_j.append(j + a)
                out_r.append(rel[i, j] + sh * L)
                out_k.append(((sh[:, 0] + 512) << 20) + ((sh[:, 1] + 512) << 10) + sh[:, 2] + 512)
    i, j, r, key = (torch.cat(v) for v in (out_i, out_j, out_r, out_k))
    at = torch.argsort(key)
    for by in (j, i):  # stable sorts, the least significant key first
        at = at[torch.argsort(by[at], stable=True)]
    return i[at], j[at], r[at]


_TABLES = {}


def _radial_table64(case, intervals=8192):
    """o-GTO radial integrals I_nl and dI_nl/dr on a uniform grid of [0, r_cut]: two [intervals + 1, n, l] tensors."""
    key = (case["r_cut"], case["sigma"], case["n_max"], case["l_max"])
    if key in _TABLES:
        return _TABLES[key]
    r_cut, sigma, n_max, l_max = key
    c = 1.0 / (2.0 * sigma * sigma)
    n = torch.arange(n_max, dtype=torch.float64)
    s = r_cut * torch.clamp(torch.sqrt(n), min=1.0) / n_max
    d = 1.0 / (2.0 * s * s)
    log_norm = 0.5 * (math.log(2.0) - (2 * n + 3) * torch.log(s) - torch.lgamma(n + 1.5))
    e = 0.5 * (n[:, None] + n[None, :] + 3)
    overlap = torch.exp(log_norm[:, None] + log_norm[None, :] + torch.lgamma(e) - e * torch.log(d[:, None] + d[None, :])) / 2
    w, V = torch.linalg.eigh(overlap)
    T = ((V / torch.sqrt(w)) @ V.t()).cuda()
    r = torch.linspace(0.0, r_cut, intervals + 1, dtype=torch.float64, device="cuda")[:, None, None]
    n, d, log_norm = (v.cuda()[None, :, None] for v in (n, d, log_norm))
    l = torch.arange(l_max + 1, dtype=torch.float64, device="cuda")[None, None, :]
    a, b = 0.5 * (n + l + 3), l + 1.5
    kappa = c * c / (c + d)
    z = kappa * r * r
    t, dt = torch.ones_like(z * l), torch.ones_like(z * l) * (a / b)
    M, dM = t.clone(), dt.clone()
    for k in range(int(float(z.max()) + 14.0 * math.sqrt(float(z.max())) + 60)):  # all terms positive
        t = t * ((a + k) / (b + k) / (k + 1)) * z
        dt = dt * ((a + k + 1) / (b + k + 1) / (k + 1)) * z
        M += t
        dM += dt
    pref = torch.exp(1.5 * math.log(math.pi) + log_norm + l * math.log(c) - a * torch.log(c + d) + torch.lgamma(a) - torch.lgamma(b))
    pref = pref * torch.exp(-c * r * r)
    rl = r ** l
    drl = torch.where(l > 0, l * r ** torch.clamp(l - 1, min=0.0), torch.zeros_like(l * r))
    value = pref * rl * M
    slope = pref * (drl * M + rl * (2.0 * kappa * r * dM - 2.0 * c * r * M))
    _TABLES.clear()
    _TABLES[key] = tuple(torch.einsum("nk,rkl->rnl", T, v) for v in (value, slope))
    return _TABLES[key]


def _radial64(case, r):
    """I_nl at r [P] by cubic Hermite interpolation of the fine table: [P, n, l]; differentiable in r."""
    v, dv = _radial_table64(case)
    h = case["r_cut"] / (v.shape[0] - 1)
    k = torch.clamp((r.detach() / h).long(), 0, v.shape[0] - 2)
    u = (r / h - k)[:, None, None]
    return ((1 + 2 * u) * (1 - u) ** 2 * v[k] + u * u * (3 - 2 * u) * v[k + 1]
            + h * u * (1 - u) ** 2 * dv[k] - h * u * u * (1 - u) * dv[k + 1])


def _harmonics64(u, l_max):
    """Real orthonormal harmonics at unit vectors u [P, 3], index l^2 + l + m, no Condon-Shortley phase: [P, lm]."""
    x, y, z = u.unbind(dim=1)
    out = [None] * (l_max + 1) ** 2
    cm, sm, k = torch.ones_like(x), torch.zeros_like(x), math.sqrt(1.0 / (4.0 * math.pi))
    for m in range(l_max + 1):
        if m:
            cm, sm = cm * x - sm * y, cm * y + sm * x
            k *= math.sqrt((2 * m + 1.0) / (2 * m)) * (math.sqrt(2.0) if m == 1 else 1.0)
        q1, q2 = torch.full_like(x, k), torch.zeros_like(x)
        for l in range(m, l_max + 1):
            if l > m:
                A = math.sqrt((4.0 * l * l - 1) / (l * l - m * m))
                B = math.sqrt(((l - 1.0) ** 2 - m * m) / (4.0 * (l - 1) ** 2 - 1)) if l - 1 > m else 0.0
                q1, q2 = A * (z * q1 - B * q2), q1
            out[l * l + l + m] = q1 * cm
            if m:
                out[l * l + l - m] = q1 * sm
    return torch.stack(out, dim=1)


def _pair_terms64(case, r, values):
    """f_cut(r) I_nl(r) Y_lm of pair vectors r [P, 3]: [P, n, lm]; `values` gives I_nl at the distances."""
    d = torch.sqrt((r * r).sum(dim=1))
    t = torch.clamp((d - case["r_cut"] + 0.5) / 0.5, min=0.0)
    f = 0.5 * (1.0 + torch.cos(math.pi * t))
    l_max = case["l_max"]
    lidx = torch.repeat_interleave(torch.arange(l_max + 1), 2 * torch.arange(l_max + 1) + 1).cuda()
    return f[:, None, None] * values(d)[:, :, lidx] * _harmonics64(r / d[:, None], l_max)[:, None, :]


def _species64(case, arrays):
    return torch.as_tensor(np.searchsorted(LABELS[:case["species"]], arrays[1])).cuda()


def _expansion64(case, arrays, pairs=None, values=None):
    """Coefficients [N, S, n, lm]."""
    i, j, r = pairs if pairs is not None else _pairs64(case, arrays)
    values = values or (lambda d: _radial64(case, d))
    a = _species64(case, arrays)
    S, n_max, n_lm = case["species"], case["n_max"], (case["l_max"] + 1) ** 2
    c = torch.zeros((len(a) * S, n_max, n_lm), dtype=torch.float64, device="cuda")
    step = max(1, int(1.5e8 // (n_max * n_lm)))
    for lo in range(0, len(i), step):
        sl = slice(lo, lo + step)
        c.index_add_(0, i[sl] * S + a[j[sl]], _pair_terms64(case, r[sl], values))
    if case.get("include_center", False):
        own = torch.arange(len(a), device="cuda") * S + a
        c[own, :, 0] += values(torch.zeros(1, dtype=torch.float64, device="cuda"))[0, :, 0] / math.sqrt(4.0 * math.pi)
    return c.reshape(len(a), S, n_max, n_lm)


def _spectrum64(case, c, layout):
    """Power spectrum [N, l, Q (Q + 1) / 2] or [N, l, Q, Q] of coefficients."""
    N, Q, L1 = c.shape[0], case["species"] * case["n_max"], case["l_max"] + 1
    C = c.reshape(N, Q, -1).double()
    iu = torch.triu_indices(Q, Q, device="cuda")
    out = torch.empty((N, L1, iu.shape[1]) if layout == "packed" else (N, L1, Q, Q), dtype=torch.float64, device="cuda")
    for l in range(L1):
        Cl = C[:, :, l * l:(l + 1) ** 2]
        p = Cl @ Cl.transpose(1, 2) / math.sqrt(2 * l + 1)
        out[:, l] = p[:, iu[0], iu[1]] if layout == "packed" else p
    return out


def _adjoint64(case, c, weights):
    """dE/dc of E = sum_i G_i . p_i; `weights(l)` gives the packed G_i of one l: [N, Q (Q + 1) / 2]."""
    N, Q = c.shape[0], case["species"] * case["n_max"]
    C = c.reshape(N, Q, -1)
    iu = torch.triu_indices(Q, Q, device="cuda")
    out = torch.empty_like(C)
    for l in range(case["l_max"] + 1):
        for lo in range(0, N, 8192):
            W = torch.zeros((min(N, lo + 8192) - lo, Q, Q), dtype=torch.float64, device="cuda")
            W[:, iu[0], iu[1]] = weights(l)[lo:lo + 8192]
            out[lo:lo + 8192, :, l * l:(l + 1) ** 2] = (W + W.transpose(1, 2)) @ C[lo:lo + 8192, :, l * l:(l + 1) ** 2] \
                / math.sqrt(2 * l + 1)
    return out.reshape(c.shape)


def _forces64(case, arrays, pairs, adjoint):
    """Forces [N, 3] and virial [n_s, 3, 3] from dE/dc, by differentiating each pair's share of the energy."""
    i, j, r = pairs
    a = _species64(case, arrays)
    offs = torch.as_tensor(arrays[4].astype(np.int64)).cuda()
    forces = torch.zeros((len(a), 3), dtype=torch.float64, device="cuda")
    virial = torch.zeros((len(offs) - 1, 3, 3), dtype=torch.float64, device="cuda")
    step = max(1, int(5e7 // (adjoint.shape[2] * adjoint.shape[3])))
    for lo in range(0, len(i), step):
        si, sj, x = i[lo:lo + step], j[lo:lo + step], r[lo:lo + step].clone().requires_grad_(True)
        e = (_pair_terms64(case, x, lambda d: _radial64(case, d)) * adjoint[si, a[sj]]).sum()
        g = torch.autograd.grad(e, x)[0]
        forces.index_add_(0, sj, -g)
        forces.index_add_(0, si, g)
        s = torch.searchsorted(offs, si, right=True) - 1
        virial.index_add_(0, s, g[:, :, None] * x.detach()[:, None, :])
    return forces, virial


def _per_structure64(arrays, atomic):
    offs = torch.as_tensor(arrays[4].astype(np.int64)).cuda()
    total = torch.cat([torch.zeros(1, dtype=torch.float64, device="cuda"), torch.cumsum(atomic, 0)])
    return total[offs[1:]] - total[offs[:-1]]


def _coupling64(l1, l2, lam):
    """Clebsch-Gordan coefficients in the real basis [mu, m1, m2] from the integral of three harmonics (l1+l2+lam even)."""
    deg = l1 + l2 + lam
    z, w = np.polynomial.legendre.leggauss(deg // 2 + 2)
    phi = 2.0 * math.pi * np.arange(deg + 2) / (deg + 2)
    Z, P = np.repeat(z, len(phi)), np.tile(phi, len(z))
    u = torch.as_tensor(np.stack([np.sqrt(1 - Z * Z) * np.cos(P), np.sqrt(1 - Z * Z) * np.sin(P), Z], axis=1)).cuda()
    wt = torch.as_tensor(np.repeat(w, len(phi)) * 2.0 * math.pi / len(phi)).cuda()
    Y = _harmonics64(u, max(l1, l2, lam))
    block = lambda l: Y[:, l * l:(l + 1) ** 2]  # noqa: E731
    gaunt = torch.einsum("p,pu,pm,pn->umn", wt, block(lam), block(l1), block(l2))
    g, f = deg // 2, math.factorial
    zero = (-1) ** (g - lam) * math.sqrt(2 * lam + 1) * f(g) / (f(g - l1) * f(g - l2) * f(g - lam)) * math.sqrt(
        f(2 * g - 2 * l1) * f(2 * g - 2 * l2) * f(2 * g - 2 * lam) / f(2 * g + 1))
    return gaunt / (math.sqrt((2 * l1 + 1) * (2 * l2 + 1) / (4 * math.pi * (2 * lam + 1))) * zero)


def _network64(case, params, t):
    """The network's outputs [B, F] from inputs t [B]."""
    F = case["n_max"] * (case["l_max"] + 1)
    W1, b1, W2, b2, W3, b3 = torch.split(params, [HIDDEN, HIDDEN, HIDDEN * HIDDEN, HIDDEN, F * HIDDEN, F])
    silu = torch.nn.functional.silu
    h = silu(t[:, None] * W1 + b1)
    h = silu(h @ W2.reshape(HIDDEN, HIDDEN).t() + b2)
    return h @ W3.reshape(F, HIDDEN).t() + b3


def exact(case, seed):
    kind = case["kind"]
    if kind == "spectrum":
        return {"p": _spectrum64(case, _stored_coefficients(case, seed), case["layout"]).flatten(1)}
    if kind == "equivariants":
        c, lam = _stored_coefficients(case, seed).double(), case["rank"]
        Q = case["species"] * case["n_max"]
        C, out = c.reshape(len(c), Q, -1), []
        for l1 in range(case["l_max"] + 1):
            for l2 in range(l1, case["l_max"] + 1):
                if l2 - l1 <= lam <= l1 + l2 and (l1 + l2 + lam) % 2 == 0:
                    X = torch.einsum("umn,iqm->iuqn", _coupling64(l1, l2, lam), C[:, :, l1 * l1:(l1 + 1) ** 2])
                    out.append(X @ C[:, None, :, l2 * l2:(l2 + 1) ** 2].transpose(2, 3))
        return {"t": torch.stack(out, dim=1)}
    if kind == "training":
        params = torch.as_tensor(_network(case, seed)[0]).cuda().double().requires_grad_(True)
        t, y = _minibatch(case, seed)
        loss = ((_network64(case, params, t.double()) - y.double()) ** 2).mean()
        return {"grad": torch.autograd.grad(loss, params)[0], "loss": loss.detach().reshape(1)}
    arrays = _structures(case, seed)
    pairs = _pairs64(case, arrays)
    if kind == "neighbours":
        return {"offsets": None, "j": None, "shifts": None,
                "rij": torch.cat([pairs[2], torch.sqrt((pairs[2] ** 2).sum(dim=1, keepdim=True))], dim=1)}
    if kind == "surrogate":
        params, scale = (torch.as_tensor(v).cuda().double() for v in _network(case, seed))

        def values(d):
            y = scale * _network64(case, params, d / case["r_cut"])
            return y.reshape(len(d), case["l_max"] + 1, case["n_max"]).transpose(1, 2)

        return {"c": _expansion64(case, arrays, pairs, values)}
    c = _expansion64(case, arrays, pairs)
    if kind == "forward":
        return {"c": c, "p": _spectrum64(case, c, case["layout"]).flatten(1)}
    if kind == "selected":
        sel = torch.as_tensor(_selection(case, seed)).cuda().long()
        return {"c": c, "p": _spectrum64(case, c, "packed").flatten(1)[:, sel]}
    a = _species64(case, arrays)
    L1 = case["l_max"] + 1
    if kind == "forces":
        w = torch.as_tensor(_linear_weights(case, seed)).cuda().double().reshape(case["species"], L1, -1)
        adjoint = _adjoint64(case, c, lambda l: w[a, l])
        atomic = 0.5 * (adjoint * c).flatten(1).sum(dim=1)                   # the energy is quadratic in c
        forces, virial = _forces64(case, arrays, pairs, adjoint)
        return {"energy": _per_structure64(arrays, atomic), "forces": forces, "virial": virial}
    M, sa, x = _sparse_model(case, seed)
    sa, x = torch.as_tensor(sa).cuda(), torch.as_tensor(x).cuda()
    p = _spectrum64(case, c, "packed").flatten(1)
    size = p.norm(dim=1, keepdim=True)
    p, size = torch.where(size > 0, p / size, p), torch.where(size > 0, size, torch.ones_like(size))
    M = M / M.norm(dim=1, keepdim=True)
    atomic, grad, zeta = torch.zeros(len(a), dtype=torch.float64, device="cuda"), torch.zeros_like(p), case["zeta"]
    for s in range(case["species"]):
        rows, pts = (a == s).nonzero().flatten(), (sa == s).nonzero().flatten()
        k = p[rows] @ M[pts].t()
        atomic[rows] = (k ** zeta) @ x[pts]
        g = (zeta * x[pts] * k ** (zeta - 1)) @ M[pts]
        grad[rows] = (g - zeta * atomic[rows, None] * p[rows]) / size[rows]
    packed = grad.reshape(len(a), L1, -1)
    forces, virial = _forces64(case, arrays, pairs, _adjoint64(case, c, lambda l: packed[:, l]))
    return {"energy": _per_structure64(arrays, atomic), "atomic": atomic, "grad": grad, "forces": forces, "virial": virial}
