"""The simple update on tensors of any scale: the weights are normalised and the
new tensors are isometries, so a common factor of the start tensors drops out.
Factors that bring the squares of Theta's Gram matrix past the exponent range;
weights of one Trotter step against the oracle on the unscaled tensors, to 1e-10
(the bound of the other simple-update tests)."""
import numpy as np
import pytest

from oracle import peps_oracle as O
from oracle import simple_update as SU

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [1e-60, 1e-45, 1e-30, 1e30, 1e45])
@pytest.mark.parametrize("D", [2, 4])
def test_su_weights_do_not_depend_on_the_scale(D, scale):
    from paper_1611_09467_gb300 import build
    from paper_1611_09467_gb300.peps import SimpleUpdate
    build.build()
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    Gam, lam = SU.init_state(2, 2, D, 81)
    h, v = O.nn_bonds(2, 2)
    s = SimpleUpdate(scale * Gam, np.stack([lam[b] for b in h + v]), 2, 2, D, J1=1.0, J2=0.5)
    SU.trotter_step(Gam, lam, 2, 2, 1.0, 0.5, 0.05, D)
    s.evolve(0.05, 1, measure=False)
    ref = np.stack([lam[b] for b in h + v])
    assert np.abs(s.lam.cpu().numpy() - ref).max() < 1e-10
    s.close()
