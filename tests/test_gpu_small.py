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


@pytest.mark.parametrize("Lx,Ly,D,Dc,n,prec", [
    (3, 3 + 1, 3, 6, 7, "fp64"), (4, 5, 2, 4, 3, "fp64"), (4, 4, 4, 8, 200, "fp64"), (4, 3, 4, 8, 3, "fp64"),
    (3, 4, 5, 6, 6, "fp64"), (4, 4, 3, 5, 5, "fp32"), (3, 4, 5, 6, 330, "fp32"), (3, 4, 6, 5, 330, "fp32"),
    (4, 4, 2, 16, 330, "fp32"), (2, 4, 2, 5, 4, "fp32"),
])
def test_small_sandwiches_match_the_oracle(Lx, Ly, D, Dc, n, prec):
    """E_loc and Delta of models with Dc D <= 32 against the oracle, for batches on
    both sides of the dispatch between a warp and a CTA per sandwich.  FP64 to
    1e-9 of the scale; FP32 to 1e-4 (the inputs are well conditioned: FP32 sums
    of a few thousand terms)."""
    from paper_1611_09467_gb300.peps import PEPS
    A = inputs.near_product_tensors(Ly, Lx, D, 93)
    S = torch.from_numpy(inputs.pack_spins(inputs.random_sz0(n, Lx * Ly, 94)).view(np.int64)).cuda()
    m = PEPS(A, Lx, Ly, D, Dc, J1=1.0, J2=0.5, prec=prec)
    got = m.evaluate(S, eloc=True, O=True)
    many = torch.cat([S] * 40)[: 40 * n] if n <= 10 else S
    same = m.evaluate(many, eloc=True)          # other dispatch of the same items
    torch.cuda.synchronize()
    from oracle import peps_oracle as O
    spins = inputs.unpack_spins(S.cpu().numpy().view(np.uint64), Lx * Ly)
    tol = 1e-9 if prec == "fp64" else 1e-4
    for k in range(min(n, 3)):
        ev = O.evaluate(A, spins[k], Ly, Lx, Dc, 1.0, 0.5)
        assert abs(got["eloc"][k].item() - ev.eloc) < tol * (1 + abs(ev.eloc))
        assert abs(same["eloc"][k].item() - ev.eloc) < tol * (1 + abs(ev.eloc))
        d = got["O"][k].cpu().numpy().reshape(ev.O.shape) - ev.O
        assert np.abs(d).max() < tol * np.abs(ev.O).max()
    m.close()


@pytest.mark.parametrize("D,Dc,prec", [(3, 6, "fp64"), (2, 5, "fp32"), (4, 8, "fp64"), (5, 6, "fp64")])
def test_small_chains_replay_the_oracle(D, Dc, prec):
    """One sweep of one-warp chains equals the oracle's decisions (no decision of
    these chains is within 1e-3 of its threshold in FP32)."""
    from oracle import peps_oracle as O
    from paper_1611_09467_gb300.peps import PEPS
    Lx, Ly, n = 4, 3, 4
    A = inputs.near_product_tensors(Ly, Lx, D, 95)
    spins = inputs.random_sz0(n, Lx * Ly, 96)
    S = torch.from_numpy(inputs.pack_spins(spins).view(np.int64)).cuda()
    m = PEPS(A, Lx, Ly, D, Dc, prec=prec)
    acc = m.mc_sweep(S, 1, seed=5).cpu().numpy()
    got = inputs.unpack_spins(S.cpu().numpy().view(np.uint64), Lx * Ly)
    for k in range(n):
        ref = O.mc_sweep(A, spins[k].copy(), Ly, Lx, Dc, 5, k, 0)
        s, a = ref[0], ref[1]
        assert np.array_equal(got[k], np.asarray(s, dtype=np.uint8)) and acc[k] == a
    m.close()
