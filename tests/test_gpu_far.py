"""The node-parallel kernel's two forms of offsets: the last lattice whose planes hold 2^32
bytes, and one just beyond (64-bit offsets), in windows at both ends and in the middle."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Lx", [1 << 31, (1 << 31) + 4099])
def test_planes_of_4_gigabytes(Lx):
    import torch
    from paper_2203_01380_gb300 import binding as B

    if torch.cuda.mem_get_info()[0] < 60e9:
        pytest.skip("needs 60 GB of device memory")
    kw = dict(lattice=1, Lx=Lx, Ly=1, n0=30.0, amp=0.0, omega_eff=1.5, seed=4, replica=1)
    ref = O.Lattice(**kw)
    out = torch.empty(3 * Lx, dtype=torch.int16, device="cuda")
    with B.Lattice(**kw) as lat:
        lat.init()
        lat.set_step_kernel(2)
        lat.step(1)
        lat.step(2)
        lat.get_state_device(out.data_ptr(), out.numel())
    out = out.view(3, Lx)
    for x0 in (0, Lx // 2 - 100, (1 << 31) - 200, Lx - 200):
        got = out[:, x0:x0 + 200].cpu().numpy().view(np.uint16)
        assert np.array_equal(got, ref.window(x0, 0, 200, 1, 3)[:, 0]), x0
