"""How wide the sums are that lead from per-pair and per-centre terms to the FP64 outputs."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from synth import System  # noqa: E402
from tests.test_gpu_tiles import test_gradient_chunks as gradient_chunks  # noqa: E402


@pytest.fixture(scope="module")
def rg():
    import paper_2101_08814_gb300 as rg

    return rg


# A centre's force and virial are its pairs' terms (FP32) added beyond FP32: with at most one pair per lane, the same terms from
# calls with one pair each add up to the virial within the second-order error of compensated sums of 16 terms (15^2 2^-48 of the
# magnitudes; a plain FP32 sum is off by up to 2^-24 of them per addition), and to the force within its one rounding to FP32 on
# top. CTAs of 128 and of 256 threads, compiled and runtime shapes, both kinds of weights.
@pytest.mark.parametrize("linear", [True, False])
@pytest.mark.parametrize("n_max,l_max,S", [(8, 6, 2), (5, 3, 1), (10, 8, 3), (12, 9, 4), (11, 7, 4)])
@pytest.mark.parametrize("P", [1, 17, 32])
def test_centre_sums_are_wider_than_fp32(rg, n_max, l_max, S, linear, P):
    import torch

    calc = rg.SoapCalculator(6.0, 0.5, n_max, l_max, list(range(1, S + 1)), spline_intervals=64)
    rng = np.random.default_rng(71)
    N, Q, L1 = P + 1, S * n_max, l_max + 1
    s = System(np.zeros((N, 3)), rng.integers(1, S + 1, N).astype(np.int32), np.eye(3)[None] * 50, np.zeros((1, 3), np.int32),
               np.array([0, N], np.int32), {})
    ds = rg.DeviceSystem.from_numpy(s)
    d = rng.standard_normal((P, 3)) * 1.8
    rij = torch.tensor(np.column_stack([d, np.linalg.norm(d, axis=1)]), dtype=torch.float32, device="cuda")
    j = torch.arange(1, N, dtype=torch.int32, device="cuda")
    c = torch.tensor(rng.standard_normal((N, Q * L1 * L1)), dtype=torch.float32, device="cuda")
    rows = S if linear else N
    w = torch.tensor(rng.standard_normal((rows, L1 * Q * (Q + 1) // 2)), dtype=torch.float32, device="cuda")

    def call(a, b):  # pairs a..b of centre 0, none of the others
        off = torch.full((N + 1,), b - a, dtype=torch.int64, device="cuda")
        off[0] = 0
        pairs = rg.PairList(off, j[a:b].contiguous(), None, rij[a:b].contiguous())
        f, v = calc.gradients(ds, pairs, c, **(dict(weights=w) if linear else dict(grad_ps=w)))
        return f[0].cpu().numpy(), v[0].cpu().numpy()

    f, v = call(0, P)
    one = [call(k, k + 1) for k in range(P)]
    fs, vs = (np.array([o[k] for o in one]) for k in (0, 1))
    eps = 15 ** 2 * 2.0 ** -48
    assert np.all(np.abs(v - vs.sum(0)) <= eps * np.abs(vs).sum(0))
    assert np.all(np.abs(f - fs.sum(0)) <= 2.0 ** -24 * np.abs(fs.sum(0)) + 2 * eps * np.abs(fs).sum(0))


# The structure energies are the same bits in every call, one CTA to a structure and several (one structure of 25 000 atoms; a
# large and two small ones), and the FP64 sums of the atoms' energies. Those spread over 24 decades, so that FP64 sums round.
@pytest.mark.parametrize("sizes", [(25000,), (700, 650), (6000, 3, 300)])
def test_gpr_energies_repeat(rg, sizes):
    import torch

    N, F = sum(sizes), 20
    rng = np.random.default_rng(73)
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int32)
    n = len(sizes)
    s = System(rng.uniform(0, 20, (N, 3)), rng.choice([1, 6], N).astype(np.int32), np.tile(np.eye(3) * 20, (n, 1, 1)),
               np.ones((n, 3), np.int32), off, {})
    calc = rg.SoapCalculator(4.0, 0.5, 2, 1, [1, 6], spline_intervals=64)
    model = rg.GprModel(calc, rng.random((60, F)), np.repeat([1, 6], 30), rng.standard_normal(60), normalize=False)
    ds = rg.DeviceSystem.from_numpy(s)
    p = torch.tensor(rng.random((N, F)) * 10.0 ** rng.uniform(-6, 6, (N, 1)), dtype=torch.float32, device="cuda")
    e, ea, _ = model.predict(ds, p)
    for _ in range(40):
        assert torch.equal(model.predict(ds, p)[0], e)
    ea = ea.double().cpu().numpy()
    for k in range(n):
        atoms = ea[off[k]:off[k + 1]]
        assert abs(e[k].item() - atoms.sum()) <= len(atoms) * 2.0 ** -53 * np.abs(atoms).sum()


# The adjoint of a per-centre dE/dp with several sets of rows to a warp: all l staged at once and groups of three and of one, CTAs of
# 128 and of 256 threads, the compiled wide shape's neighbours; and wide bases of a few l, which read dE/dp from global memory. The
# check and its bound are those of the other chunks.
@pytest.mark.parametrize("n_max,l_max,S", [(16, 0, 3), (5, 3, 4), (9, 6, 4), (12, 2, 8), (12, 4, 8), (16, 8, 8), (16, 2, 8)])
def test_split_rows(rg, n_max, l_max, S):
    gradient_chunks(rg, n_max, l_max, S)
