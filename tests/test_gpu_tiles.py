"""Kernels at the sizes where their tiles can go wrong: remainders, single elements, the widest shapes they accept."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from oracle import lambda_soap as ols  # noqa: E402
from oracle import mlp as omlp  # noqa: E402
from oracle import soap as osoap  # noqa: E402
from synth import mlp_initial_params  # noqa: E402
from tests.gpu_common import block_rel_err  # noqa: E402

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
