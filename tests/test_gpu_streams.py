"""One context used from several CUDA streams."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from synth import System, config_large  # noqa: E402


@pytest.fixture(scope="module")
def rg():
    import paper_2101_08814_gb300 as rg

    return rg


def _lists(pairs):
    return [getattr(pairs, k).cpu().numpy() for k in ("offsets", "nbr_j", "shifts", "rij")]


def _search(rg, calc, ds, stream, capacity, noalloc=False):
    """The library's own call on the given stream; returns with the pair arrays possibly still being written."""
    import torch

    lib = rg._lib.lib()
    assert lib.rascal_set_stream(calc._ctx, C.c_void_p(stream.cuda_stream)) == 0
    out = [torch.empty(ds.n_atoms + 1, dtype=torch.int64, device="cuda"), torch.empty(capacity, dtype=torch.int32, device="cuda"),
           torch.empty((capacity, 3), dtype=torch.int32, device="cuda"), torch.empty((capacity, 4), device="cuda")]
    sys_c, P = ds.c_struct(), C.c_int64(0)
    st = (lib.rascal_neighbours_noalloc if noalloc else lib.rascal_neighbours)(
        calc._ctx, C.byref(sys_c), capacity, *(C.c_void_p(t.data_ptr()) for t in out), C.byref(P))
    return st, P.value, out


# A search returns before its pair arrays are written (about 170 us for 2.95 M pairs): work that the context puts on another
# stream afterwards waits for it, after a search that succeeds and with the no-allocation entry point.
@pytest.mark.parametrize("noalloc", [False, True])
def test_another_stream_waits_for_the_fill(rg, noalloc):
    import torch

    s = config_large()
    calc = rg.SoapCalculator(**s.hypers)
    ds = rg.DeviceSystem.from_numpy(s)
    ref = _lists(calc.neighbours(ds))
    n = len(ref[1])
    torch.cuda.synchronize()
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    st, P, out = _search(rg, calc, ds, a, n, noalloc)
    assert st == 0 and P == n
    assert rg._lib.lib().rascal_set_stream(calc._ctx, C.c_void_p(b.cuda_stream)) == 0
    b.synchronize()
    assert a.query()  # what the other stream waited for is done
    for got, want in zip(out, ref):
        assert np.array_equal(got.cpu().numpy(), want)


# Two searches of one context on two streams, the first one refused (capacity) or not: each has its own list.
@pytest.mark.parametrize("short", [0, 1])
def test_searches_on_two_streams(rg, short):
    import torch

    s = config_large()
    other = System(s.positions[:20000] + 0.25, s.species[:20000], s.cells, s.pbc, np.array([0, 20000], np.int32), s.hypers)
    calc = rg.SoapCalculator(**s.hypers)
    sets = [rg.DeviceSystem.from_numpy(x) for x in (s, other)]
    ref = [_lists(calc.neighbours(x)) for x in sets]
    torch.cuda.synchronize()
    streams = torch.cuda.Stream(), torch.cuda.Stream()
    for _ in range(3):
        got = [_search(rg, calc, ds, st, len(r[1]) - (short if k == 0 else 0))
               for k, (ds, st, r) in enumerate(zip(sets, streams, ref))]
        torch.cuda.synchronize()
        for k, ((st, P, out), r) in enumerate(zip(got, ref)):
            assert P == len(r[1]) and st == (rg._lib.RASCAL_E_CAPACITY if short and k == 0 else 0)
            if st == 0:
                for o, w in zip(out, r):
                    assert np.array_equal(o.cpu().numpy(), w)


def test_a_captured_stream_takes_no_wait(rg):
    import torch

    s = config_large()
    calc = rg.SoapCalculator(**s.hypers)
    ds = rg.DeviceSystem.from_numpy(s)
    pairs = calc.neighbours(ds)  # leaves a fill behind on the current stream
    c = calc.spherical_expansion(ds, pairs)
    out = torch.zeros_like(c)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        calc.spherical_expansion(ds, pairs, out=out)
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, c)
    calc.neighbours(ds)
    calc.sync()


# The no-allocation search's scratch is shared by all contexts of a device: a refused call leaves nothing queued that reads it, so
# that the next search, on another stream and of another context, meets no fill of the refused one.
def test_a_refused_search_leaves_nothing_behind(rg):
    import torch

    s = config_large()
    other = System(s.positions[:20000] + 0.25, s.species[:20000], s.cells, s.pbc, np.array([0, 20000], np.int32), s.hypers)
    calcs = [rg.SoapCalculator(**s.hypers) for _ in range(2)]
    sets = [rg.DeviceSystem.from_numpy(x) for x in (s, other)]
    ref = [_lists(c.neighbours(x)) for c, x in zip(calcs, sets)]
    torch.cuda.synchronize()
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    for _ in range(3):
        st, P, refused = _search(rg, calcs[0], sets[0], a, len(ref[0][1]) - 1, noalloc=True)
        refused_pairs = [t.clone() for t in refused[1:]]
        assert st == rg._lib.RASCAL_E_CAPACITY and P == len(ref[0][1]) and a.query()
        st, P, out = _search(rg, calcs[1], sets[1], b, len(ref[1][1]), noalloc=True)
        torch.cuda.synchronize()
        assert st == 0 and P == len(ref[1][1])
        for o, w in zip(out, ref[1]):
            assert np.array_equal(o.cpu().numpy(), w)
        assert all(torch.equal(x.view(torch.uint8), y.view(torch.uint8)) for x, y in zip(refused_pairs, refused[1:]))
