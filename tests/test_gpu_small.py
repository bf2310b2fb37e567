"""The one-warp boundary sweeps (models with Dc D <= 32) against the CTA sweeps.

peps_amplitudes_static keeps the 256-thread row absorption for every model, so
it is the reference: in FP32 the one-warp sweep adds the same terms in the same
order and must agree bit for bit; in FP64 (another Sturm count and inverse
iteration) ln|psi| must agree to the FP64 bound of 1e-10.  Sizes: the smallest
and largest block, blocks that are not a multiple of four, K of one, odd Dc,
wide and narrow lattices, more sweeps than resident warps."""
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


@pytest.mark.parametrize("Lx,Ly,D,Dc,n", [
    (2, 2, 2, 1, 3), (4, 4, 2, 4, 64), (3, 4, 2, 16, 9), (7, 4, 2, 5, 33), (5, 4, 3, 6, 20), (6, 3, 3, 10, 12),
    (4, 6, 4, 8, 40), (3, 8, 4, 7, 17), (4, 4, 5, 6, 21), (6, 5, 6, 5, 10), (16, 2, 4, 8, 11), (4, 3, 4, 8, 2000),
])
def test_small_sweeps_equal_cta_sweeps(Lx, Ly, D, Dc, n):
    from paper_1611_09467_gb300.peps import PEPS, amplitudes_static
    A = inputs.near_product_tensors(Ly, Lx, D, 91)
    S = torch.from_numpy(inputs.pack_spins(inputs.random_sz0(n, Lx * Ly, 92)).view(np.int64)).cuda()
    for prec, real in (("fp32", torch.float32), ("fp64", torch.float64)):
        m = PEPS(A, Lx, Ly, D, Dc, prec=prec)
        la, sg, st = m.amplitudes(S)
        Ad = torch.from_numpy(A).reshape(Lx * Ly, 2, D ** 4).cuda().to(real)
        ra, rs, rt = amplitudes_static(Ad, S, Lx, Ly, D, Dc, prec=prec)
        torch.cuda.synchronize()
        assert torch.equal(sg, rs) and torch.equal(st, rt)
        if prec == "fp32":
            assert torch.equal(la, ra), (la - ra).abs().max()
        else:
            assert (la - ra).abs().max() <= 1e-10
        m.close()
