"""Kernels at the sizes where their tiles can go wrong: remainders, single elements, the widest shapes they accept."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from oracle import lambda_soap as ols  # noqa: E402
from oracle import mlp as omlp  # noqa: E402
from oracle import soap as osoap  # noqa: E402
from oracle.neighbours import neighbour_list  # noqa: E402
from synth import System, config_batch, mlp_initial_params, random_cell_atoms  # noqa: E402
from tests.gpu_common import block_rel_err  # noqa: E402
from tests.test_gpu_gpr import _emulated_energies, _grad_checks, _predict, _unit_tf32, tf32_trunc  # noqa: E402

H = 64


@pytest.fixture(scope="module")
def rg():
    import paper_2101_08814_gb300 as rg

    return rg


def _network(p, F):
    p, out, o = np.asarray(p, dtype=np.float64), {}, 0
    for name, shape in (("W1", (H, 1)), ("b1", (H,)), ("W2", (H, H)), ("b2", (H,)), ("W3", (F, H)), ("b3", (F,))):
        out[name] = p[o:o + int(np.prod(shape))].reshape(shape)
        o += int(np.prod(shape))
    return out


# outputs not a multiple of the 4-wide tiles, batches of one sample, one past a tile of 8, 16 or 32, and the widest
# basis (512 outputs: 8 samples fit beside its weights, so a CTA takes several tiles). The bound is that of the other
# gradient test: 1e-4 of a parameter block's largest entry (fast exponentials and FP32 sums over 3 layers).
@pytest.mark.parametrize("n_max,l_max,batch", [(3, 2, 1), (3, 2, 9), (5, 0, 1217), (7, 6, 2433), (16, 12, 4865), (32, 15, 1300)])
def test_training_step_tiles(rg, n_max, l_max, batch):
    import torch

    calc = rg.SoapCalculator(5.0, 0.5, n_max, l_max, [1], spline_intervals=64)
    F = n_max * (l_max + 1)
    rng = np.random.default_rng(17)
    p0 = (mlp_initial_params(H, F, seed=9) + 0.05 * rng.standard_normal(3 * H + H * H + F * H + F)).astype(np.float32)
    calc.mlp_set_params(p0, np.ones(F, np.float32))
    t = rng.random(batch).astype(np.float32)
    y = rng.standard_normal((batch, F)).astype(np.float32)
    g, loss = calc.mlp_gradients(torch.tensor(t, device="cuda"), torch.tensor(y, device="cuda"))
    loss_ref, ref = omlp.loss_and_grads(_network(p0, F), t.astype(np.float64), y.astype(np.float64))
    assert abs(loss.item() - loss_ref) <= 1e-5 * loss_ref
    got = _network(g.cpu().numpy(), F)
    for k in ref:
        assert np.max(np.abs(got[k] - ref[k])) <= 1e-4 * np.max(np.abs(ref[k])), k
    # the minibatch order: the same step on a reversed order gives the same loss
    order = torch.arange(batch - 1, -1, -1, dtype=torch.int64, device="cuda")
    first = calc.mlp_train(torch.tensor(t, device="cuda"), torch.tensor(y, device="cuda"), order, batch=batch, steps=1)
    assert abs(first.item() - loss_ref) <= 1e-5 * loss_ref


# Q = 1, 5, 7, 18 (scalar stores), 36, 256 (16-byte stores); one row group per thread and several, a pair split into
# chunks of rows with a remainder, the widest basis the kernel takes (its smallest chunk), the top rank. FP32 products
# of FP32 inputs summed over at most 31 terms, twice: 2e-6 of a block's largest entry, as for the tiny cell.
@pytest.mark.parametrize("n_max,S,l_max,lam", [(1, 1, 0, 0), (1, 1, 15, 3), (5, 1, 3, 1), (7, 1, 4, 8), (9, 2, 6, 3),
                                               (12, 3, 5, 2), (16, 16, 12, 1)])
def test_equivariant_tiles(rg, n_max, S, l_max, lam):
    import torch

    species = list(range(1, S + 1))
    calc = rg.SoapCalculator(5.0, 0.5, n_max, l_max, species, spline_intervals=64)
    h = osoap.Hypers(5.0, 0.5, n_max, l_max, species)
    n = 2 if S == 16 else 5
    c = np.random.default_rng(23).standard_normal((n, S, n_max, (l_max + 1) ** 2)).astype(np.float32)
    T = calc.lambda_soap(torch.tensor(c, device="cuda"), lam)
    ref = ols.equivariants(c, h, lam)
    assert block_rel_err(T.cpu().numpy(), ref, 2) <= 2e-6


def _lists(rg, s):
    pl = rg.SoapCalculator(**s.hypers).neighbours(rg.DeviceSystem.from_numpy(s))
    return [getattr(pl, k).cpu().numpy() for k in ("offsets", "nbr_j", "shifts", "rij")]


def _cell(n, cell, r_cut, pbc=(1, 1, 1), d_min=0.7, seed=61):
    rng = np.random.Generator(np.random.PCG64(seed))
    cell = np.asarray(cell, np.float64)
    return System(random_cell_atoms(n, cell, d_min, rng), np.full(n, 6, np.int32), cell[None], np.asarray([pbc], np.int32),
                  np.array([0, n], np.int32), dict(r_cut=r_cut, sigma=0.5, n_max=2, l_max=1, smooth_width=0.5, species=[6]))


# stencils of one batch and of several (a flat cell: 9 x 9 x 3 bins), candidates of one chunk and of several (27 x 70 of
# one bin), bins that split into several work items, one with fewer centres than warps, one open axis: equal to the
# brute-force list, vectors to FP32 rounding
@pytest.mark.parametrize("n,cell,r_cut,pbc", [
    (1, np.eye(3) * 3.0, 5.0, (1, 1, 1)), (3, np.diag([1.4, 1.6, 9.0]), 5.0, (1, 1, 1)),
    (70, np.eye(3) * 5.5, 5.0, (1, 1, 1)), (70, np.diag([5.5, 5.5, 7.0]), 4.0, (1, 0, 1)), (200, np.eye(3) * 11.0, 5.0, (1, 1, 1))])
def test_neighbour_stencils(rg, n, cell, r_cut, pbc):
    s = _cell(n, cell, r_cut, pbc)
    off, j, sh, rij = _lists(rg, s)
    ref = neighbour_list(s, r_cut)
    assert np.array_equal(off, ref["offsets"]) and np.array_equal(j, ref["nbr_j"]) and np.array_equal(sh, ref["shifts"])
    assert np.allclose(rij[:, :3], ref["rij"], rtol=0, atol=2e-6)


def test_neighbours_far_from_their_cell(rg):
    s = _cell(40, np.diag([7.0, 8.0, 9.0]), 4.0)
    far = System(s.positions + np.array([600.0 * 7.0, -700.0 * 8.0, 0.0]), s.species, s.cells, s.pbc, s.struct_offsets, s.hypers)
    off, j, sh, rij = _lists(rg, far)
    ref = neighbour_list(far, 4.0)
    assert np.array_equal(off, ref["offsets"]) and np.array_equal(j, ref["nbr_j"]) and np.array_equal(sh, ref["shifts"])
    moved = far.positions.copy()
    moved[0] += np.array([7.0 * 1200.0, 0.0, 0.0])  # neighbours 1200 cells apart: beyond the shift range
    with pytest.raises(rg.RascalError) as e:
        _lists(rg, System(moved, s.species, s.cells, s.pbc, s.struct_offsets, s.hypers))
    assert e.value.code == rg._lib.RASCAL_E_UNSUPPORTED


def test_neighbours_of_many_atoms_and_loose_offsets(rg):
    # more atoms than the one-launch offsets take: copies of the same cells have the same lists
    s = config_batch(n_structures=24)
    off, j, sh, rij = _lists(rg, s)
    k = 131072 // s.n_atoms + 2
    big = System(np.tile(s.positions, (k, 1)), np.tile(s.species, k), np.tile(s.cells, (k, 1, 1)), np.tile(s.pbc, (k, 1)),
                 np.concatenate([[0]] + [s.struct_offsets[1:] + q * s.n_atoms for q in range(k)]).astype(np.int32), s.hypers)
    boff, bj, bsh, brij = _lists(rg, big)
    P = len(j)
    assert np.array_equal(boff, np.concatenate([[0]] + [off[1:] + q * P for q in range(k)]))
    assert np.array_equal(bj, np.concatenate([j + q * s.n_atoms for q in range(k)]))
    assert np.array_equal(bsh, np.tile(sh, (k, 1))) and np.array_equal(brij, np.tile(rij, (k, 1)))
    # atoms before the first offset count as the first structure's, atoms past the last as the last one's
    loose = System(s.positions, s.species, s.cells, s.pbc, s.struct_offsets.copy(), s.hypers)
    loose.struct_offsets[0], loose.struct_offsets[-1] = 5, s.n_atoms - 7
    for a, b in zip(_lists(rg, loose), (off, j, sh, rij)):
        assert np.array_equal(a, b)


# Q = 1 and 7 (one block of rows, partly empty), 16, 17, 24, 35, 48, 60 and 128 (32-row blocks with and without a lone
# 16-row block after them, several items left of the diagonal), and Q = 256, whose FULL l blocks do not fit the staging
# area. The bars are those of the other power-spectrum tests: 1e-5 per (centre, l) block in FP32 and TF32x3; BF16 inputs
# 2^-7 of a block's largest entry and 5e-3 of its norm.
@pytest.mark.parametrize("n_max,S,l_max", [(1, 1, 0), (7, 1, 3), (8, 2, 6), (17, 1, 2), (12, 2, 9), (7, 5, 5), (12, 4, 9),
                                           (15, 4, 4), (16, 8, 12), (16, 16, 1)])
def test_power_spectrum_items(rg, n_max, S, l_max):
    import torch

    species = list(range(1, S + 1))
    calc = rg.SoapCalculator(5.0, 0.5, n_max, l_max, species, spline_intervals=64)
    h = osoap.Hypers(5.0, 0.5, n_max, l_max, species)
    rng = np.random.default_rng(29)
    c = rng.standard_normal((4, S, n_max, (l_max + 1) ** 2)).astype(np.float32)
    c[-1] = 0.0
    c_dev = torch.tensor(c, device="cuda")
    for layout in ("packed", "full"):
        ref = osoap.power_spectrum(c.astype(np.float64), h, layout).reshape(4, l_max + 1, -1)
        for precision in ("fp32", "tf32x3", "bf16"):
            if precision != "fp32" and (h.q > 128 or (precision == "tf32x3" and h.q > 96)):
                continue  # refused by the library
            p = calc.power_spectrum(c_dev, precision=precision, layout=layout).cpu().numpy().reshape(ref.shape)
            assert np.all(p[-1] == 0.0)
            if precision == "bf16":
                assert block_rel_err(p, ref, 2) <= 2.0 ** -7
                fro = np.sqrt(np.sum((p - ref) ** 2, axis=-1) / np.maximum(np.sum(ref ** 2, axis=-1), 1e-300))
                assert np.max(fro) <= 5e-3
            else:
                assert block_rel_err(p, ref, 2) <= 1e-5, (layout, precision)


# Centres with 0, 1, 32, 33 and 65 neighbours (no chunk of 32 pairs, a single pair, full chunks, chunks with one left), odd
# and even n_max, l_max 0 and 15, one warp's rows of four and of six, packed blocks that do not all fit at once, compiled
# shapes, and the widest basis, whose tables do not fit and which takes the other kernel. Against sums in 64 bits over the
# pairs' explicit feature gradients; the bound is the longest chain of roundings that a product passes (rows, columns,
# l, and the pairs of an atom) times the sum of the products' magnitudes.
@pytest.mark.parametrize("n_max,l_max,S", [(1, 0, 1), (3, 1, 2), (5, 15, 1), (8, 6, 2), (10, 8, 3), (12, 9, 4), (11, 7, 5),
                                           (16, 12, 8), (12, 15, 8)])
def test_gradient_chunks(rg, n_max, l_max, S):
    import torch

    species = list(range(1, S + 1))
    calc = rg.SoapCalculator(6.0, 0.5, n_max, l_max, species, spline_intervals=64)
    rng = np.random.default_rng(43)
    sizes = (1, 2, 33, 34, 66)
    pos = np.concatenate([random_cell_atoms(n, np.eye(3) * (1.0 + 0.9 * n ** (1 / 3)), 0.4, rng) * 0.6 for n in sizes])
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int32)
    N, Q, L1, M = int(off[-1]), S * n_max, l_max + 1, (l_max + 1) ** 2
    s = System(pos, rng.integers(1, S + 1, N).astype(np.int32), np.tile(np.eye(3) * 40.0, (5, 1, 1)), np.zeros((5, 3), np.int32),
               off, {})
    ds = rg.DeviceSystem.from_numpy(s)
    pairs = calc.neighbours(ds)
    po = pairs.offsets.cpu().numpy()
    assert sorted(set(np.diff(po))) == [0, 1, 32, 33, 65]
    i, j = np.repeat(np.arange(N), np.diff(po)), pairs.nbr_j.cpu().numpy()
    c = rng.standard_normal((N, Q, M)).astype(np.float32)
    w = rng.standard_normal((S, L1 * Q * (Q + 1) // 2)).astype(np.float32)
    g = rng.standard_normal((N, w.shape[1])).astype(np.float32) if N * w.shape[1] < 2e7 else w[s.species - 1]
    d = torch.cat([calc.debug_pair_gradients(r).double() for r in pairs.rij.split(256)]).cuda()  # [P, 3, n_max, M]
    ti, tj = torch.tensor(i, device="cuda"), torch.tensor(j, device="cuda").long()
    lo, hi = np.triu_indices(Q)
    sid = torch.tensor(np.searchsorted(off, i, side="right") - 1, device="cuda")
    rij = pairs.rij[:, :3].double()
    eps = 2.0 ** -24 * (Q + 2 * n_max + 8 * L1 + 32 + 130)
    cd = torch.tensor(c, device="cuda").double()
    for weights in (True, False):
        wi = torch.tensor(w[s.species - 1] if weights else g, device="cuda").double().view(N, L1, -1)
        pair = torch.zeros(len(i), 3, device="cuda", dtype=torch.float64)
        size = torch.zeros(len(i), device="cuda", dtype=torch.float64)
        own = torch.tensor((s.species - 1)[j], device="cuda")
        for l in range(L1):
            W = torch.zeros(N, Q, Q, device="cuda", dtype=torch.float64)
            W[:, lo, hi] = wi[:, l]
            W = W + W.transpose(1, 2)
            sl = slice(l * l, (l + 1) ** 2)
            rows = lambda A, C: ((A @ C) / np.sqrt(2 * l + 1)).view(N, S, n_max, -1)[ti, own]  # noqa: E731
            chat, mag = rows(W, cd[:, :, sl]), rows(W.abs(), cd[:, :, sl].abs())
            pair += torch.einsum("pnm,pxnm->px", chat, d[..., sl])
            size += (mag.norm(dim=2) * d[..., sl].norm(dim=(1, 3))).sum(dim=1)
        f = torch.zeros(N, 3, device="cuda", dtype=torch.float64).index_add(0, ti, pair).index_add(0, tj, -pair)
        f_size = torch.zeros(N, device="cuda", dtype=torch.float64).index_add(0, ti, size).index_add(0, tj, size)
        v = torch.zeros(5, 3, 3, device="cuda", dtype=torch.float64).index_add(0, sid, pair[:, :, None] * rij[:, None, :])
        v_size = torch.zeros(5, device="cuda", dtype=torch.float64).index_add(0, sid, size * rij.norm(dim=1))
        kw = dict(weights=torch.tensor(w, device="cuda")) if weights else dict(grad_ps=torch.tensor(g, device="cuda"))
        fg, vg = calc.gradients(ds, pairs, torch.tensor(c, device="cuda"), **kw)
        assert bool(((fg - f).abs().amax(dim=1) <= eps * f_size).all()), (weights, float(((fg - f).abs().amax(1) / (eps * f_size)).nan_to_num().max()))
        assert bool(((vg - v).abs().amax(dim=(1, 2)) <= eps * v_size).all())
        if not weights:
            continue
        # the energies from the coefficients: half of chat . c, at most rows, columns and 130 atoms of roundings
        e, fe, ve = calc.linear_gradients(ds, pairs, torch.tensor(c, device="cuda"), kw["weights"])
        p = calc.power_spectrum(torch.tensor(c, device="cuda")).double()
        pa = calc.power_spectrum(torch.tensor(np.abs(c), device="cuda")).double()
        at = torch.tensor(np.repeat(np.arange(5), sizes), device="cuda")
        wa = torch.tensor(w[s.species - 1], device="cuda").double()
        ref = torch.zeros(5, device="cuda", dtype=torch.float64).index_add(0, at, (p * wa).sum(1))
        e_size = torch.zeros(5, device="cuda", dtype=torch.float64).index_add(0, at, (pa * wa.abs()).sum(1))
        assert bool(((e - ref).abs() <= eps * e_size).all())
        assert bool(((fe - f).abs().amax(dim=1) <= eps * f_size).all()) and bool(((ve - v).abs().amax(dim=(1, 2)) <= eps * v_size).all())


# Tiles of 128, 256 and 512 sparse points (one and several to a species, the wider ones where there are centres for every
# SM), a species whose points are not a multiple of 32, features of less than a stage, of an odd number (4-byte copies) and of
# half a stage past a whole one; gradient tiles of 256 features and what is left of them. Against the arithmetic on the inputs
# as the tensor core sees them; the bounds are those of the model's other tests (1e-5 zeta sum |x|, 1e-4 of the terms).
@pytest.mark.parametrize("N,F,points", [(140, 12, (3, 17)), (300, 301, (130, 40)), (260, 1040, (256, 48)), (19500, 36, (200, 16)),
                                        (13000, 20, (600, 32)), (130, 272, (560, 0))])
def test_gpr_tiles(rg, N, F, points):
    rng = np.random.default_rng(47)
    spe = rng.choice([1, 6], size=N).astype(np.int32)
    s = System(rng.uniform(0, 20, size=(N, 3)), spe, np.eye(3)[None] * 20, np.ones((1, 3), np.int32), np.array([0, N], np.int32),
               dict(r_cut=4.0, sigma=0.5, n_max=2, l_max=1, smooth_width=0.5, species=[1, 6]), "gpr-tiles")
    p32 = np.abs(rng.normal(size=(N, F))).astype(np.float32)
    M = np.abs(rng.normal(size=(sum(points), F)))
    labels = np.repeat([1, 6], points).astype(np.int32)
    x = rng.standard_normal(len(M)) / 30
    Mt, zeta = _unit_tf32(M), 2
    calc = rg.SoapCalculator(**s.hypers)
    _, ea, g = _predict(rg, s, calc, p32, Mt, labels, x, zeta)
    cs, ms = np.searchsorted([1, 6], spe), np.searchsorted([1, 6], labels)
    E = _emulated_energies(p32, cs, Mt, ms, x, zeta, tf32_trunc)
    assert np.max(np.abs(ea - E)) <= 1e-5 * zeta * np.sum(np.abs(x))
    part = rng.choice(N, size=min(N, 600), replace=False)
    r_emul, r_exact = _grad_checks(g[part], p32[part], cs[part], Mt, ms, x, zeta, Mt)
    assert r_emul <= 1.0 and r_exact <= 1.0
    assert np.all(g[~np.isin(cs, ms)] == 0.0)


# Coefficients alone equal those of the fused call bit for bit: one and several species rounds, coefficients of a round that fit
# the pair rows and that do not (16 species), targets at every alignment, four warps and eight (at most two centres per SM), no
# neighbours, one chunk and several.
@pytest.mark.parametrize("n_max,l_max,S,n,copies", [(1, 0, 1, 40, 1), (8, 6, 1, 64, 1), (8, 6, 2, 50, 8), (5, 3, 3, 50, 8),
                                                    (4, 6, 16, 60, 1), (16, 12, 8, 30, 1), (10, 8, 3, 90, 1)])
def test_coefficients_alone(rg, n_max, l_max, S, n, copies):
    import torch

    calc = rg.SoapCalculator(5.0, 0.5, n_max, l_max, list(range(1, S + 1)), include_center=True, spline_intervals=64)
    rng = np.random.default_rng(53)
    L = (n / 0.08) ** (1 / 3)
    pos = np.concatenate([np.concatenate([random_cell_atoms(n, np.eye(3) * L, 1.0, rng), [[0.0, 0.0, 60.0]]])] * copies)
    s = System(pos, rng.integers(1, S + 1, len(pos)).astype(np.int32), np.tile(np.diag([L, L, 200.0])[None], (copies, 1, 1)),
               np.tile([[1, 1, 0]], (copies, 1)).astype(np.int32), np.arange(0, len(pos) + 1, n + 1).astype(np.int32), {})
    ds = rg.DeviceSystem.from_numpy(s)
    pairs = calc.neighbours(ds)
    ref, _ = calc.soap(ds, pairs)
    for shift in range(4):
        out = torch.full((ref.numel() + 8,), 7.0, device="cuda")
        calc.spherical_expansion(ds, pairs, out=out[shift:])
        assert torch.equal(out[shift:shift + ref.numel()].view_as(ref), ref)
        assert bool((out[:shift] == 7.0).all()) and bool((out[shift + ref.numel():] == 7.0).all())


# The fill pass is queued before the host knows the counts: where they do not fit it writes nothing (too small a capacity, a
# flagged geometry), and where a centre has more pairs than a warp sorts in shared memory (150) it runs once they are known.
@pytest.mark.parametrize("entry,n", [("rascal_neighbours", 60), ("rascal_neighbours_noalloc", 60), ("rascal_neighbours", 151)])
def test_neighbour_fill_waits_for_the_counts(rg, entry, n):
    import ctypes as C

    import torch

    s = _cell(n, np.eye(3) * (11.0 if n == 60 else 2.2), 5.0 if n == 60 else 3.9, (1, 1, 1) if n == 60 else (0, 0, 0),
              **({} if n == 60 else dict(d_min=0.3)))
    ref = neighbour_list(s, s.hypers["r_cut"])
    P = len(ref["nbr_j"])
    calc = rg.SoapCalculator(**s.hypers)

    def call(system, capacity):
        ds = rg.DeviceSystem.from_numpy(system)
        off = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
        j = torch.full((P,), -5, dtype=torch.int32, device="cuda")
        sh = torch.full((P, 3), -5, dtype=torch.int32, device="cuda")
        rij = torch.full((P, 4), -5.0, device="cuda")
        sys_c, count = ds.c_struct(), C.c_int64(0)
        st = getattr(rg._lib.lib(), entry)(calc._ctx, C.byref(sys_c), capacity, *(C.c_void_p(t.data_ptr()) for t in (off, j, sh, rij)),
                                           C.byref(count))
        torch.cuda.synchronize()
        return st, count.value, j.cpu().numpy(), sh.cpu().numpy(), rij.cpu().numpy()

    calc._bind_stream()
    st, count, j, sh, rij = call(s, P - 1)
    assert st == rg._lib.RASCAL_E_CAPACITY and count == P and np.all(j == -5) and np.all(sh == -5) and np.all(rij == -5.0)
    same = s.positions.copy()
    same[1] = same[0]
    st, _, j, sh, rij = call(System(same, s.species, s.cells, s.pbc, s.struct_offsets, s.hypers), P)
    assert st == rg._lib.RASCAL_E_GEOMETRY and np.all(j == -5) and np.all(sh == -5) and np.all(rij == -5.0)
    st, count, j, sh, rij = call(s, P)
    assert st == 0 and count == P and np.array_equal(j, ref["nbr_j"]) and np.array_equal(sh, ref["shifts"])
    assert np.allclose(rij[:, :3], ref["rij"], rtol=0, atol=2e-6)


# Outputs of one 16-column tile, of half a 32-column slab, not a multiple of 4 (scalar stores), the most TMEM holds; batches
# of one, one short of and one past a tile, several tiles; with and without derivatives; nothing written past the last row.
# Bounds of the other inference test: 2e-2 (values) and 3e-2 (derivatives) of the largest, from the 16-bit operands.
@pytest.mark.parametrize("n_max,l_max", [(1, 0), (5, 2), (4, 3), (7, 6), (16, 12), (16, 15)])
def test_inference_tiles(rg, n_max, l_max):
    calc = rg.SoapCalculator(5.0, 0.5, n_max, l_max, [1], spline_intervals=64)
    F = n_max * (l_max + 1)
    p = mlp_initial_params(H, F)
    calc.mlp_set_params(p, np.ones(F, np.float32))
    rng = np.random.default_rng(59)
    r = rng.uniform(0.2, 5.0, 700).astype(np.float32)
    y, dy, _ = omlp.forward(_network(p, F), r.astype(np.float64) / 5.0, tangent=True)
    dy = dy / 5.0
    whole, dwhole = (t.cpu().numpy() for t in calc.mlp_eval(r, derivative=True))
    assert np.max(np.abs(whole - y)) <= 2e-2 * np.max(np.abs(y)) and np.max(np.abs(dwhole - dy)) <= 3e-2 * np.max(np.abs(dy))
    for n in (1, 127, 129, 700):
        v, d = (t.cpu().numpy() for t in calc.mlp_eval(r[:n], derivative=True))
        assert np.array_equal(v, whole[:n]) and np.array_equal(d, dwhole[:n])
        assert np.array_equal(calc.mlp_eval(r[:n]).cpu().numpy(), whole[:n])


# The fused call in the tensor-core precisions is the coefficients followed by the spectrum of stored coefficients, whatever
# the layout and the alignment of its outputs: Q = 1, 21, 24, 48, one species round and several, no atoms' worth of pairs.
@pytest.mark.parametrize("n_max,l_max,S,n", [(1, 0, 1, 9), (7, 5, 3, 70), (8, 6, 3, 70), (12, 9, 4, 70), (16, 7, 5, 40)])
@pytest.mark.parametrize("precision", ["bf16", "tf32x3"])
def test_fused_tensor_core_precisions(rg, n_max, l_max, S, n, precision):
    import torch

    calc = rg.SoapCalculator(4.5, 0.5, n_max, l_max, list(range(1, S + 1)), include_center=n_max > 1, spline_intervals=64)
    rng = np.random.default_rng(67)
    L = (n / 0.08) ** (1 / 3)
    s = System(np.concatenate([random_cell_atoms(n, np.eye(3) * L, 1.0, rng), [[0.0, 0.0, 60.0]]]),
               rng.integers(1, S + 1, n + 1).astype(np.int32), np.diag([L, L, 200.0])[None], np.array([[1, 1, 0]], np.int32),
               np.array([0, n + 1], np.int32), {})
    ds = rg.DeviceSystem.from_numpy(s)
    pairs = calc.neighbours(ds)
    c_ref = calc.spherical_expansion(ds, pairs)
    for layout in ("packed", "full"):
        p_ref = calc.power_spectrum(c_ref, precision=precision, layout=layout)
        for shift in range(0, 4, 1 + 2 * (layout == "full")):
            c = torch.full((c_ref.numel() + 8,), 7.0, device="cuda")
            p = torch.full((p_ref.numel() + 8,), 7.0, device="cuda")
            calc.soap(ds, pairs, layout=layout, precision=precision, coeffs=c[shift:], ps=p[3 - shift:])
            assert torch.equal(c[shift:shift + c_ref.numel()].view_as(c_ref), c_ref)
            assert torch.equal(p[3 - shift:3 - shift + p_ref.numel()].view_as(p_ref), p_ref)
            assert bool((c[:shift] == 7.0).all()) and bool((p[3 - shift + p_ref.numel():] == 7.0).all())
