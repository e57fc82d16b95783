"""mg_cycle on device arrays where the capture of its graph fails (a stand-in for
the failing call, on the host): the plain launches serve the call and all later
ones, with the same bits."""
import pytest

from fake_runtime import run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("which", [1, 2, 3])
def test_plain_launches_where_the_capture_fails(tmp_path, which):
    out = run(tmp_path, """
        import numpy as np
        import torch
        import synth
        from gpu_util import lib_handle, rnd
        from paper_2404_02493_gb300 import binding as B

        I = synth.config_lognormal(n=100, omega=30.0, seed=3)
        g = torch.from_numpy(rnd((100 * 100,), 1, np.complex64)).cuda()
        h = lib_handle([I], "mixed", M=2, autotune=0)

        def cycle():
            u = torch.zeros_like(g)
            B.mg_cycle(h, u, g, 2)
            torch.cuda.synchronize()
            return u

        want = cycle()
        ctypes.c_int.in_dll(lib, "fake_capture").value = %d
        for _ in range(3):
            assert torch.equal(cycle(), want)
        ctypes.c_int.in_dll(lib, "fake_capture").value = 0
        assert torch.equal(cycle(), want)
        # refused once, not asked for again
        assert ctypes.c_int.in_dll(lib, "fake_captures_refused").value == 1
        B.mg_destroy(h)
        print("passed")
    """ % which)
    assert "passed" in out
