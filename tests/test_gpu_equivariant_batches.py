"""Forms of the equivariant kernel, which depend on the number of centres and on the room that a basis leaves on an SM."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from oracle import lambda_soap as ols  # noqa: E402
from oracle import soap as osoap  # noqa: E402
from tests.gpu_common import block_rel_err  # noqa: E402


# One or two CTAs to an SM (5 and 300 centres; Q = 80, l_max 15: every batch), up to six (700), more (1300); one and several
# chunks of a pair, scalar and 16-byte stores, pairs of few and of 31 m. The batch of five against the oracle with the bound of
# the other tests of these kernels (2e-6 of a block's largest entry); the products of a centre are summed in the same order in
# every form, so the larger batches hold the same bits.
@pytest.mark.parametrize("n_max,S,l_max,lam", [(2, 1, 15, 4), (9, 1, 10, 0), (6, 1, 10, 2), (12, 3, 2, 2), (5, 4, 4, 4), (10, 6, 1, 1),
                                               (10, 8, 15, 0), (16, 3, 5, 1)])
def test_batches_have_the_same_bits(n_max, S, l_max, lam):
    import torch

    import paper_2101_08814_gb300 as rg

    species = list(range(1, S + 1))
    calc = rg.SoapCalculator(5.0, 0.5, n_max, l_max, species, spline_intervals=64)
    h = osoap.Hypers(5.0, 0.5, n_max, l_max, species)
    c = np.random.default_rng(89).standard_normal((5, S, n_max, (l_max + 1) ** 2)).astype(np.float32)
    c[4] = 0.0
    base = torch.tensor(c, device="cuda")
    T = calc.lambda_soap(base, lam)
    assert block_rel_err(T.cpu().numpy(), ols.equivariants(c, h, lam), 2) <= 2e-6
    for n in (300, 700, 1300):
        if n * T[0].numel() > 4e8:
            continue
        i = torch.arange(n, device="cuda") % 5
        assert torch.equal(calc.lambda_soap(base[i].contiguous(), lam), T[i])
