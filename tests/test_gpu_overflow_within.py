"""An overflow in the middle of a launch of many steps, by every kernel that takes several steps per
launch and on D2Q5 and D2Q9: two beams meet at a crowded node some twenty steps in.  The call reports
it and leaves the state before that step; the steps before it alone give the same state."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kernel", [2, 6, 7, -1])
@pytest.mark.parametrize("lattice,Ly", [(2, 16), (2, 160), (3, 16), (3, 160)])
def test_overflow_within_a_launch(lattice, Ly, kernel):
    from paper_2203_01380_gb300 import binding as B

    kw = dict(lattice=lattice, Lx=256, Ly=Ly, n0=5.0, omega_eff=0.02, theta=0.01, seed=21, replica=2)
    ref = O.Lattice(**kw)
    s0 = np.full((5 if lattice == 2 else 9, Ly, 256), 3, np.uint16)
    s0[0, 7, 100], s0[1, 7, 80], s0[2, 7, 120] = 65400, 48000, 48000
    s, t = s0, 3
    with pytest.raises(OverflowError):
        while t < 60:
            s, t = ref.step(s, t), t + 1
    assert 10 < t < 40
    with B.Lattice(**kw) as lat:
        lat.set_state(s0, 3)
        lat.set_step_kernel(kernel)
        with pytest.raises(B.IlgError) as e:
            lat.step(50)
        assert e.value.status == B.ILG_E_OVERFLOW
        got, at = lat.get_state()
        assert at == t and np.array_equal(got, s)
        lat.set_state(s0, 3)
        lat.step(t - 3)
        got, at = lat.get_state()
        assert at == t and np.array_equal(got, s)
