"""Launch plans of the stored-coefficient power spectrum, which depend on the number of centres."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


# Up to one, two and eight centres per SM and more; Q = 2 and 36 (rows of an edge tile), 60 (one l block per group, then several),
# 80, 128 (512 threads), 200 (one CTA to an SM). The products of a centre are summed in the same order whatever the plan: a centre's
# spectrum is the same bits in every batch. (The small batch against the oracle: test_power_spectrum_items.)
@pytest.mark.parametrize("n_max,S,l_max", [(2, 1, 15), (9, 4, 15), (12, 4, 9), (15, 4, 12), (15, 4, 15), (16, 5, 4), (16, 8, 9),
                                           (20, 10, 2)])
def test_every_batch_gives_the_same_bits(n_max, S, l_max):
    import torch

    import paper_2101_08814_gb300 as rg

    calc = rg.SoapCalculator(5.0, 0.5, n_max, l_max, list(range(1, S + 1)), basis="dvr", spline_intervals=64)
    rng = np.random.default_rng(83)
    base = torch.tensor(rng.standard_normal((7, S, n_max, (l_max + 1) ** 2)), dtype=torch.float32, device="cuda")
    for layout in ("packed", "full"):
        for precision in ("fp32", "tf32x3", "bf16"):
            try:
                p = calc.power_spectrum(base, precision=precision, layout=layout)
            except rg.RascalError as e:
                assert e.code == rg._lib.RASCAL_E_UNSUPPORTED and precision != "fp32"
                continue
            for n in (150, 301, 700, 1300):
                if n * p.shape[1] > 3e8:
                    continue
                i = torch.arange(n, device="cuda") % 7
                assert torch.equal(calc.power_spectrum(base[i].contiguous(), precision=precision, layout=layout), p[i])
