"""mg_cycle on device arrays: the first call emits the launches, the second
captures them, later ones replay the graph; the same bits from each, with the
graph off, from host arrays, from arrays at other addresses, for several
cycles per call, on a user's stream and inside a user's own capture."""
import numpy as np
import pytest
import torch

import synth
from gpu_util import cdt, lib_handle, rnd
from paper_2404_02493_gb300 import binding as B

pytestmark = pytest.mark.gpu


def handle(prec, **kw):
    insts = [synth.config_lognormal(n=n, omega=0.3 * (n + 1), seed=n) for n in (47, 100)]
    return insts, lib_handle(insts, prec, M=2, autotune=0, **kw)


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_cycle_calls_give_the_same_bits(prec):
    insts, h = handle(prec)
    _, h0 = handle(prec, use_graph=0)
    N = sum(I.n * I.n for I in insts)
    g = rnd((N,), 1, cdt(prec))
    u0 = rnd((N,), 2, cdt(prec))
    for ncyc in (1, 3):
        want = u0.copy()
        B.mg_cycle(h0, want, g, ncyc)                     # host arrays, plain launches
        gd = torch.from_numpy(g).cuda()
        for _ in range(3):
            ud = torch.from_numpy(u0).cuda()
            B.mg_cycle(h, ud, gd.clone(), ncyc)
            assert np.array_equal(ud.cpu().numpy(), want)
        s = torch.cuda.Stream()
        ud = torch.from_numpy(u0).cuda()
        torch.cuda.synchronize()
        B.mg_cycle(h, ud, gd, ncyc, stream=s)
        s.synchronize()
        assert np.array_equal(ud.cpu().numpy(), want)
        # an array that starts off the alignment of whole vectors
        big = torch.zeros(N + 1, dtype=ud.dtype, device="cuda")
        big[1:] = torch.from_numpy(u0).cuda()
        B.mg_cycle(h, big[1:], gd, ncyc)
        assert np.array_equal(big[1:].cpu().numpy(), want)
    B.mg_destroy(h)
    B.mg_destroy(h0)


def test_cycle_zero_count_and_user_capture():
    insts, h = handle("mixed")
    N = sum(I.n * I.n for I in insts)
    g = torch.from_numpy(rnd((N,), 1, np.complex64)).cuda()
    u = torch.from_numpy(rnd((N,), 2, np.complex64)).cuda()
    keep = u.clone()
    B.mg_cycle(h, u, g, 0)
    torch.cuda.synchronize()
    assert torch.equal(u, keep)
    want = keep.clone()
    B.mg_cycle(h, want, g, 1)
    B.mg_cycle(h, want.clone(), g, 1)
    torch.cuda.synchronize()
    # captured by the caller: plain launches inside the caller's graph
    s = torch.cuda.Stream()
    gr = torch.cuda.CUDAGraph()
    with torch.cuda.graph(gr, stream=s, capture_error_mode="thread_local"):
        B.mg_cycle(h, u, g, 1, stream=s)
    u.copy_(keep)
    gr.replay()
    torch.cuda.synchronize()
    assert torch.equal(u, want)
    B.mg_destroy(h)
