"""Bounded waits of the tcgen05 kernels that ordinary calls run, made to run out without faulting the GPU.

The hook (rascal_debug_wait_timeout) points a CTA's first completion wait at an mbarrier that nothing arrives at; it gives up
after a given number of polls. The kernel then reports a timeout, waits for what it has issued and frees its tensor memory:
with the hook off the same kernel gives the results that it gave before.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from synth import mlp_initial_params  # noqa: E402


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
