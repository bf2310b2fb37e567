"""The simple update's SVD at the edges of its lane layout: one T warp (D = 1, 2),
several (D = 7, 8), more than four, whose warps also rotate V (D = 9, 12); the
matrices in shared memory (D <= 7) and in the scratch slot.  One Trotter step
of 2x2, weights against the oracle to 1e-10 (the bound of the other
simple-update tests)."""
import numpy as np
import pytest

from oracle import peps_oracle as O
from oracle import simple_update as SU

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1611_09467_gb300 import build
    build.build()
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")


@pytest.mark.parametrize("D", [1, 2, 7, 8, 9, 12])
def test_su_weights_by_bond_dimension(D):
    from paper_1611_09467_gb300.peps import SimpleUpdate
    Gam, lam = SU.init_state(2, 2, D, 77)
    h, v = O.nn_bonds(2, 2)
    s = SimpleUpdate(Gam, np.stack([lam[b] for b in h + v]), 2, 2, D, J1=1.0, J2=0.5)
    SU.trotter_step(Gam, lam, 2, 2, 1.0, 0.5, 0.05, D)
    s.evolve(0.05, 1, measure=False)
    ref = np.stack([lam[b] for b in h + v])
    assert np.abs(s.lam.cpu().numpy() - ref).max() < 1e-10
    s.close()


def test_su_states_of_two_bond_dimensions():
    """A state of a smaller D made in between does not lower the shared memory
    that the first one's launches may ask for."""
    from paper_1611_09467_gb300.peps import SimpleUpdate
    h, v = O.nn_bonds(2, 2)
    states = []
    for D in (7, 2):
        Gam, lam = SU.init_state(2, 2, D, 78)
        s = SimpleUpdate(Gam, np.stack([lam[b] for b in h + v]), 2, 2, D, J1=1.0, J2=0.5)
        states.append((s, Gam, lam, D))
    for s, Gam, lam, D in states:
        s.evolve(0.05, 1, measure=False)
        SU.trotter_step(Gam, lam, 2, 2, 1.0, 0.5, 0.05, D)
        ref = np.stack([lam[b] for b in h + v])
        assert np.abs(s.lam.cpu().numpy() - ref).max() < 1e-10
        s.close()


def test_su_nan_tensors():
    """NaN tensors give NaN weights and leave the device usable."""
    from paper_1611_09467_gb300.peps import SimpleUpdate
    Gam, lam = SU.init_state(2, 2, 3, 79)
    h, v = O.nn_bonds(2, 2)
    lam0 = np.stack([lam[b] for b in h + v])
    s = SimpleUpdate(np.full_like(Gam, np.nan), lam0, 2, 2, 3, J1=1.0, J2=0.5)
    s.evolve(0.05, 1, measure=False)
    assert np.isnan(s.lam.cpu().numpy()).all()
    s.close()
