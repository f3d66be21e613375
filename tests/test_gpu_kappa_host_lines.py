"""Host line lists, copied through a host thread's pinned buffers or from where they are, give
bit for bit the table of the same list resident on the GPU: around the longest staged list, for
more calls than there are buffers while the stream is busy, and from several threads at once."""
import threading

import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rt():
    import paper_cs_0703028_gb300 as m
    return m


def _spec():
    return synth.Spectral(nu_min=2000.0, dnu=0.05, n_nu=777, cutoff=5.0, profile="voigt", nT=2, T_min=500.0, T_max=900.0)


@pytest.mark.parametrize("n", [1, 2047, 2048, 2049, 4097])
def test_host_list_equals_device_list(rt, n):
    import torch
    lines = synth.make_lines(n, 1996.0, 2042.0, synth.rng_for(41, n))
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    assert torch.equal(rt.build_kappa(lines, _spec()), rt.build_kappa(lines, _spec(), memory="device", status=st))


def test_lists_queued_behind_a_busy_stream(rt):
    # the host arrays are overwritten as soon as each call returns
    import torch
    lists = [synth.make_lines(300 + i, 1996.0, 2042.0, synth.rng_for(42, i)) for i in range(11)]
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    want = [rt.build_kappa(l, _spec(), memory="device", status=st).clone() for l in lists]
    big = torch.ones(1 << 28, device="cuda")
    for _ in range(20):
        big.mul_(1.0)
    got = []
    for l in lists:
        got.append(rt.build_kappa(l, _spec()))
        if l.n <= 2048:
            for a in (l.nu0, l.S_ref, l.gamma_ref, l.E_lower):
                a[:] = 1.0
    for g, w in zip(got, want):
        assert torch.equal(g, w)


def test_threads_have_their_own_buffers(rt):
    import torch
    torch.cuda.synchronize()
    bad = []

    def work(t):
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            st = torch.zeros(1, dtype=torch.int32, device="cuda")
            for i in range(6):
                lines = synth.make_lines(500 + 10 * t + i, 1996.0, 2042.0, synth.rng_for(43, 10 * t + i))
                a, b = rt.build_kappa(lines, _spec()), rt.build_kappa(lines, _spec(), memory="device", status=st)
                if not torch.equal(a, b):
                    bad.append((t, i))
            s.synchronize()

    threads = [threading.Thread(target=work, args=(t,)) for t in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad
