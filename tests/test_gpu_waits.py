"""Bounded waits of the tcgen05 kernels that ordinary calls run, made to run out without faulting the GPU.

The hook (rascal_debug_wait_timeout) points a CTA's first completion wait at an mbarrier that nothing arrives at; it gives up
after a given number of polls. The kernel then reports a timeout, waits for what it has issued and frees its tensor memory:
with the hook off the same kernel gives the results that it gave before.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from synth import System, mlp_initial_params  # noqa: E402


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
