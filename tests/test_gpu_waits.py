"""Bounded waits of the tcgen05 kernels that ordinary calls run, made to run out without faulting the GPU.

The hook (rascal_debug_wait_timeout) points a CTA's first completion wait at an mbarrier that nothing arrives at; it gives up
after a given number of polls. The kernel then reports a timeout, waits for what it has issued and frees its tensor memory:
with the hook off the same kernel gives the results that it gave before.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from oracle import soap as osoap  # noqa: E402
from synth import System, mlp_initial_params, random_cell_atoms  # noqa: E402
from tests.gpu_common import block_rel_err, ps_blocks  # noqa: E402


@pytest.fixture(scope="module")
def rg():
    import paper_2101_08814_gb300 as rg

    return rg


def _times_out(rg, calc, call):
    lib = rg._lib.lib()
    assert lib.rascal_debug_wait_timeout(calc._ctx, 1000) == rg._lib.RASCAL_OK
    call()
    with pytest.raises(rg.RascalError) as e:
        calc.sync()
    assert e.value.code == rg._lib.RASCAL_E_TIMEOUT
    assert lib.rascal_debug_wait_timeout(calc._ctx, 0) == rg._lib.RASCAL_OK


# one tile of 128 distances and many, with and without derivatives (all of an SM's tensor memory)
@pytest.mark.parametrize("derivative", [False, True])
@pytest.mark.parametrize("n", [100, 70001])
def test_inference(rg, n, derivative):
    calc = rg.SoapCalculator(5.0, 0.5, 8, 6, [1], spline_intervals=64)
    calc.mlp_set_params(mlp_initial_params(64, 56), np.ones(56, np.float32))
    r = np.random.default_rng(3).uniform(0.2, 5.0, n).astype(np.float32)

    def run():
        out = calc.mlp_eval(r, derivative=derivative)
        return [t.cpu().numpy() for t in (out if derivative else (out,))]

    before = run()
    _times_out(rg, calc, run)
    for a, b in zip(run(), before):
        assert np.array_equal(a, b)
    calc.sync()


# Kernel and gradient GEMM; fewer k-blocks than the pipeline has stages (nobody else waits) and more (the copies, norms and
# loads fill the stages and their own waits, bounded too, run out), 4-byte and 16-byte copies, tiles of 128 and 256 points
@pytest.mark.parametrize("N,F,points", [(140, 36, (3, 17)), (300, 301, (130, 40)), (260, 1040, (256, 48)), (39000, 40, (250, 30))])
def test_gpr(rg, N, F, points):
    import torch

    rng = np.random.default_rng(5)
    s = System(rng.uniform(0, 20, size=(N, 3)), rng.choice([1, 6], size=N).astype(np.int32), np.eye(3)[None] * 20,
               np.ones((1, 3), np.int32), np.array([0, N], np.int32), {})
    calc = rg.SoapCalculator(4.0, 0.5, 2, 1, [1, 6], spline_intervals=64)
    ds = rg.DeviceSystem.from_numpy(s)
    model = rg.GprModel(calc, rng.random((sum(points), F)), np.repeat([1, 6], points), rng.standard_normal(sum(points)))
    p = torch.tensor(rng.random((N, F)), dtype=torch.float32, device="cuda")

    def run():
        return [t.cpu().numpy() for t in model.predict(ds, p, grad=True)[1:]]

    before = run()
    _times_out(rg, calc, run)
    for a, b in zip(run(), before):
        assert np.array_equal(a, b)
    calc.sync()


# The tcgen05 form of the BF16 Gram serves bases whose FULL l blocks do not fit the spectrum kernel beside the coefficients
# (Q = 128, l_max 14). One launch that computes c and p, against the oracle: c 1e-5 per block, p the bars of the other BF16
# tests; and the same kernel, with the same bits, after its wait has run out.
@pytest.mark.parametrize("n_max,S,l_max", [(16, 8, 14), (12, 10, 14), (16, 8, 13)])
def test_bf16_gram_of_wide_bases(rg, n_max, S, l_max):
    rng = np.random.default_rng(7)
    species, n = list(range(1, S + 1)), 41
    s = System(np.concatenate([random_cell_atoms(n - 1, np.eye(3) * 8.0, 1.2, rng), [[4.0, 4.0, 60.0]]]),
               rng.integers(1, S + 1, n).astype(np.int32), np.diag([8.0, 8.0, 200.0])[None], np.array([[1, 1, 0]], np.int32),
               np.array([0, n], np.int32), dict(r_cut=4.5, sigma=0.5, n_max=n_max, l_max=l_max, smooth_width=0.5, species=species))
    calc = rg.SoapCalculator(**s.hypers)
    ds = rg.DeviceSystem.from_numpy(s)
    pairs = calc.neighbours(ds)

    def run():
        return [t.cpu().numpy() for t in calc.soap(ds, pairs, layout="full", precision="bf16")]

    launches = rg.launch_count()
    c, p = run()
    assert rg.launch_count() == launches + 1
    p_separate = calc.power_spectrum(calc.spherical_expansion(ds, pairs), layout="full", precision="bf16").cpu().numpy()
    h = osoap.Hypers(**s.hypers)
    sel = [0, 7, 23, n - 1]
    c_ref = osoap.spherical_expansion(s, h, centres=sel)
    ref = osoap.power_spectrum(c_ref, h, "full").reshape(len(sel), l_max + 1, -1)
    assert block_rel_err(c[sel], c_ref, 2) <= 1e-5
    for got in (p, p_separate):
        assert np.all(np.isfinite(got)) and np.all(got[-1] == 0.0)
        blocks = ps_blocks(got[sel], l_max)
        assert block_rel_err(blocks, ref, 2) <= 2.0 ** -7
        fro = np.sqrt(np.sum((blocks - ref) ** 2, axis=-1) / np.maximum(np.sum(ref ** 2, axis=-1), 1e-300))
        assert np.max(fro) <= 5e-3
    _times_out(rg, calc, run)
    for a, b in zip(run(), (c, p)):
        assert np.array_equal(a, b)
    calc.sync()
