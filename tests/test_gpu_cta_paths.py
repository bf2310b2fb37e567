"""The kernels with a CTA per item for models that small.cuh does not take, the
one-warp correlations in FP32, models whose truncation matrix needs 200 to 212 KB
of shared memory, and amplitudes that vanish or overflow on the one-warp sweeps.

Bounds are those of the other tests of the same outputs: FP64 1e-10 for ln|psi| and
M^2, 1e-9 for the correlation sums; FP32 on near-product tensors 1e-5."""
import numpy as np
import pytest

from oracle import correlations as C
from oracle import peps_oracle as O
from paper_1611_09467_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1611_09467_gb300 import build
    build.build()
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")


def packed(spins):
    return torch.from_numpy(inputs.pack_spins(spins).view(np.int64)).cuda()


# 7/20 in FP64 and 10/20, 14/15 in FP32: the matrix and its buffers take 200 to 212 KB
CTA = [(4, 4, 5, 8, "fp64"), (4, 3, 6, 12, "fp64"), (4, 4, 7, 20, "fp64"), (5, 4, 5, 8, "fp32"), (4, 3, 6, 12, "fp32"),
       (4, 4, 10, 20, "fp32"), (4, 4, 14, 15, "fp32")]


@pytest.mark.parametrize("Lx,Ly,D,Dc,prec", CTA + [(4, 4, 3, 6, "fp32"), (4, 4, 4, 8, "fp32"), (4, 4, 5, 6, "fp32")])
def test_correlations(Lx, Ly, D, Dc, prec):
    from paper_1611_09467_gb300.peps import PEPS
    A = inputs.near_product_tensors(Ly, Lx, D, 601)
    spins = inputs.random_sz0(4, Lx * Ly, 602)
    sites = [Lx * y + x for y in range(1, Ly) for x in range(1, 3)]
    p = PEPS(A, Lx, Ly, D, Dc, J1=1.0, J2=0.5, prec=prec)
    r = p.correlations(packed(spins), sites)
    torch.cuda.synchronize()
    ref = np.stack([C.correlations(A, s, Ly, Lx, Dc, sites) for s in spins])
    eps = np.array([C.staggered_sign(i, Lx) for i in sites])
    m2 = np.einsum("npq,p,q->n", ref, eps, eps) / len(sites) ** 2
    tol_m2, tol_c = (1e-10, 1e-9) if prec == "fp64" else (1e-5, 1e-5)
    total = ref.sum(0)
    assert (r["status"] == 0).all()
    assert np.abs(r["m2"].cpu().numpy() - m2).max() < tol_m2
    assert np.abs(r["corr"].cpu().numpy() - total).max() < tol_c * max(1.0, np.abs(total).max())
    p.close()


@pytest.mark.parametrize("Lx,Ly,D,Dc,prec", [(4, 4, 7, 20, "fp64"), (4, 4, 10, 20, "fp32"), (4, 4, 14, 15, "fp32")])
def test_amplitudes_with_a_large_matrix_in_shared_memory(Lx, Ly, D, Dc, prec):
    """ln|psi| of the sweeps with and without stored environments: equal to each
    other bit for bit and to the oracle."""
    from paper_1611_09467_gb300.peps import PEPS, amplitudes_static
    A = inputs.near_product_tensors(Ly, Lx, D, 603)
    spins = inputs.random_sz0(3, Lx * Ly, 604)
    S = packed(spins)
    m = PEPS(A, Lx, Ly, D, Dc, prec=prec)
    la, sg, st = m.amplitudes(S)
    Ad = torch.from_numpy(A).reshape(Lx * Ly, 2, D ** 4).cuda().to(torch.float64 if prec == "fp64" else torch.float32)
    ra, rs, rt = amplitudes_static(Ad, S, Lx, Ly, D, Dc, prec=prec)
    torch.cuda.synchronize()
    assert torch.equal(la, ra) and torch.equal(sg, rs) and torch.equal(st, rt)
    ref = np.array([O.evaluate(A, s, Ly, Lx, Dc, 1.0, 0.0, want_O=False).logabs for s in spins])
    assert np.abs(la.cpu().numpy() - ref).max() < (1e-10 if prec == "fp64" else 1e-5)
    m.close()


@pytest.mark.parametrize("Lx,Ly,D,Dc,prec", [(4, 3, 5, 8, "fp64"), (4, 3, 7, 20, "fp64"), (4, 3, 10, 20, "fp32"),
                                             (4, 3, 14, 15, "fp32")])
def test_chains_replay_the_oracle(Lx, Ly, D, Dc, prec):
    from paper_1611_09467_gb300.peps import PEPS
    n = 2
    A = inputs.near_product_tensors(Ly, Lx, D, 605)
    spins = inputs.random_sz0(n, Lx * Ly, 606)
    S = packed(spins)
    m = PEPS(A, Lx, Ly, D, Dc, prec=prec)
    acc = m.mc_sweep(S, 1, seed=7).cpu().numpy()
    got = inputs.unpack_spins(S.cpu().numpy().view(np.uint64), Lx * Ly)
    for k in range(n):
        decisions = []
        s, a = O.mc_sweep(A, spins[k].copy(), Ly, Lx, Dc, 7, k, 0, decisions=decisions)
        # every decision is far enough from its threshold for FP32
        assert min(abs(ratio2 - u) for _, ratio2, u in decisions) > 1e-3
        assert np.array_equal(got[k], np.asarray(s, dtype=np.uint8)) and acc[k] == a
    m.close()


@pytest.mark.parametrize("D,Dc", [(2, 5), (4, 8), (5, 6)])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("case", ["zero", "overflow"])
def test_one_warp_sweeps_of_vanishing_and_overflowing_amplitudes(D, Dc, prec, case):
    """A site tensor that is zero for one spin makes the amplitudes of its
    configurations zero; entries whose squares overflow make their norms infinite.
    ln|psi|, sign and status equal those of the CTA sweeps, and the other
    configurations are not touched."""
    from paper_1611_09467_gb300.peps import PEPS, amplitudes_static
    Lx, Ly, n = 4, 3, 40
    A = inputs.near_product_tensors(Ly, Lx, D, 607)
    plain = A.copy()
    A[5, 0] = 0.0 if case == "zero" else A[5, 0] * (1e30 if prec == "fp32" else 1e250)
    spins = inputs.random_sz0(n, Lx * Ly, 608)
    S = packed(spins)
    Ad = torch.from_numpy(A).reshape(Lx * Ly, 2, D ** 4).cuda().to(torch.float64 if prec == "fp64" else torch.float32)
    m, q = PEPS(A, Lx, Ly, D, Dc, prec=prec), PEPS(plain, Lx, Ly, D, Dc, prec=prec)
    la, sg, st = m.amplitudes(S)
    ra, rs, rt = amplitudes_static(Ad, S, Lx, Ly, D, Dc, prec=prec)
    pa, ps, pt = q.amplitudes(S)
    torch.cuda.synchronize()
    hit = torch.from_numpy(spins[:, 5] == 0).cuda()
    assert hit.any() and not hit.all()
    assert torch.equal(st, rt) and torch.equal(sg, rs)
    assert torch.equal(la[~hit], pa[~hit]) and torch.equal(sg[~hit], ps[~hit]) and (st[~hit] == 0).all()
    if case == "zero":
        assert (st[hit] == 5).all() and (sg[hit] == 0).all() and torch.isneginf(la[hit]).all()
    assert torch.equal(torch.isfinite(la), torch.isfinite(ra))
    m.close()
    q.close()
