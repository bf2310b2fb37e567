"""E and Delta of a configuration do not depend, in any bit, on the size of the
batch it is evaluated in: models whose sandwiches run on a warp or on a CTA
according to the number of items, in batches on both sides of the lines, items
past the first wave included."""
import numpy as np
import pytest

from paper_1611_09467_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1611_09467_gb300 import build
    build.build()
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")


@pytest.mark.parametrize("Lx,Ly,D,Dc,prec", [
    (4, 4, 4, 8, "fp64"), (5, 2, 4, 8, "fp64"), (4, 4, 4, 7, "fp64"), (3, 4, 5, 6, "fp64"), (4, 3, 3, 10, "fp64"),
    (4, 4, 2, 16, "fp64"), (3, 4, 6, 5, "fp64"), (4, 4, 3, 6, "fp64"),
    (4, 4, 4, 7, "fp32"), (3, 4, 5, 6, "fp32"), (4, 3, 3, 10, "fp32"), (4, 4, 2, 16, "fp32"), (3, 4, 6, 5, "fp32"),
    (4, 4, 4, 5, "fp32"), (4, 4, 3, 6, "fp32"), (4, 4, 5, 2, "fp32"), (4, 4, 5, 5, "fp64"),
])
def test_results_do_not_depend_on_the_batch(Lx, Ly, D, Dc, prec):
    from paper_1611_09467_gb300.peps import PEPS
    n = 2100   # the two-row items of a batch of n pass the warps that are resident; four items an SM is the highest line
    A = inputs.near_product_tensors(Ly, Lx, D, 97)
    S = torch.from_numpy(inputs.pack_spins(inputs.random_sz0(n, Lx * Ly, 98)).view(np.int64)).cuda()
    m = PEPS(A, Lx, Ly, D, Dc, J1=1.0, J2=0.5, prec=prec)
    big = m.evaluate(S, eloc=True, O=True)
    keys = ("logabs", "sign", "eloc", "status", "O")
    big = {k: big[k].clone() for k in keys}
    for first, count in ((0, 1), (0, 9), (700, 9), (n - 9, 9), (n - 150, 150)):
        got = m.evaluate(S[first:first + count].contiguous(), eloc=True, O=True)
        torch.cuda.synchronize()
        for k in keys:
            assert torch.equal(got[k], big[k][first:first + count]), (k, first, count)
    m.close()
