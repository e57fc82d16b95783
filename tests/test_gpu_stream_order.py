"""The first solve on a handle builds its graph by a run on the workspace, on a
stream of the handle: it must wait for the cycles that the caller's stream
still runs there.  Cycles on a side stream, the solve begun at once without a
synchronisation; the same bits as with one."""
import numpy as np
import pytest
import torch

import synth
from gpu_util import lib_handle, rnd
from paper_2404_02493_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("outer", ["fgmres", "ir"])
def test_first_solve_waits_for_cycles_of_the_stream(outer):
    I = synth.config_lognormal(n=511, omega=0.3 * 512, seed=5)
    g = torch.from_numpy(rnd((511 * 511,), 1, np.complex64)).cuda()
    b = torch.from_numpy(I.g.ravel()).cuda()
    out = {}
    for wait in (True, False):
        h = lib_handle([I], "mixed", M=2, autotune=0, outer=outer)
        u, x = torch.zeros_like(g), torch.zeros_like(b)
        s = torch.cuda.Stream()
        torch.cuda.synchronize()
        B.mg_cycle(h, u, g, 40, stream=s)
        if wait:
            s.synchronize()
        B.mg_solve_begin(h, x, b, stream=s)
        B.mg_solve_steps(h, 2, stream=s)
        B.mg_solve_end(h, x, stream=s)
        s.synchronize()
        out[wait] = (u.cpu().numpy(), x.cpu().numpy())
        B.mg_destroy(h)
    assert np.array_equal(out[True][0], out[False][0])
    assert np.array_equal(out[True][1], out[False][1])
