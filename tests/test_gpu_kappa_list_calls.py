"""Calls with a host line list neither wait for the GPU nor keep anything of the list: they
return while the stream is busy, however many are queued, and a captured call's replays read
the caller's arrays again, as a replayed copy does."""
import ctypes as ct

import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rt():
    import paper_cs_0703028_gb300 as m
    return m


def _spec(nT=1, kappa_min=0.0):
    return synth.Spectral(nu_min=2000.0, dnu=0.05, n_nu=777, cutoff=5.0, profile="voigt", nT=nT, T_min=500.0,
                          T_max=500.0 if nT == 1 else 900.0, kappa_min=kappa_min)


def _lines(n, key):
    return synth.make_lines(n, 1996.0, 2042.0, synth.rng_for(44, key))


# few (node, line) pairs, many, and windows of their own
@pytest.mark.parametrize("nT,kappa_min", [(1, 0.0), (40, 0.0), (2, 1e-3)])
def test_queued_builds_return_while_the_stream_is_busy(rt, nT, kappa_min):
    import torch
    spec = _spec(nT, kappa_min)
    lists = [_lines(400 + i, i) for i in range(12)]
    outs = [torch.empty(nT, spec.n_nu, device="cuda") for _ in lists]
    big = torch.ones(1 << 29, device="cuda")
    for l, o in zip(lists, outs):
        rt.build_kappa(l, spec, out=o)
    torch.cuda.synchronize()
    want = [o.clone() for o in outs]
    done = torch.cuda.Event()
    for _ in range(300):  # about 0.2 s of the GPU's time
        big.mul_(1.0)
    done.record()
    for l, o in zip(lists, outs):
        rt.build_kappa(l, spec, out=o)
    assert not done.query()
    torch.cuda.synchronize()
    for o, w in zip(outs, want):
        assert torch.equal(o, w)


@pytest.mark.parametrize("n", [3, 400, 501, 1001])
def test_replays_read_the_list_again(rt, n):
    import torch
    L = rt.lib()
    spec, lines = _spec(2), _lines(n, 100 + n)
    S = rt.make_spectral(spec)
    ls, keep = rt.make_lines(lines)
    out = torch.empty(2, spec.n_nu, device="cuda")

    def build(stream):
        assert L.rt_build_kappa(ct.byref(ls), ct.byref(S), out.data_ptr(), None, None, stream) == rt.RT_OK, L.rt_last_error()

    graph, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(graph, stream=side):
        build(ct.c_void_p(side.cuda_stream))
    for scale in (1.0, 3.0):
        keep[1][:] *= scale  # the intensities
        graph.replay()
        torch.cuda.synchronize()
        got = out.clone()
        build(None)
        torch.cuda.synchronize()
        assert torch.equal(got, out)


# the longest list a launch carries, one more, and either side of its half, for both ways to carry it
@pytest.mark.parametrize("n", [1, 499, 500, 501, 999, 1000, 1001])
@pytest.mark.parametrize("nT,kappa_min", [(1, 0.0), (9, 0.0), (2, 1e-3)])
def test_carried_list_equals_device_list(rt, n, nT, kappa_min):
    import torch
    lines, spec = _lines(n, 200 + n), _spec(nT, kappa_min)
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    a, b = (torch.zeros(1, dtype=torch.int64, device="cuda") for _ in range(2))
    got = rt.build_kappa(lines, spec, evals=a)
    want = rt.build_kappa(lines, spec, memory="device", status=st, evals=b)
    assert torch.equal(got, want) and int(a) == int(b)
