"""The autotuner on models whose sweeps and sandwiches run on warps: it names what it
times, its boundary grids are of the kernel that runs, and no choice changes the
boundary sweeps' results."""
import numpy as np
import pytest

from paper_1611_09467_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D,Dc,prec", [(3, 7, "fp32"), (3, 7, "fp64"), (4, 8, "fp32")])
def test_names_and_grids(D, Dc, prec):
    from paper_1611_09467_gb300 import build
    from paper_1611_09467_gb300.peps import PEPS
    build.build()
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    L, n = 4, 1000
    A = inputs.near_product_tensors(L, L, D, 611)
    S = torch.from_numpy(inputs.pack_spins(inputs.random_sz0(n, L * L, 612)).view(np.int64)).cuda()
    m = PEPS(A, L, L, D, Dc, J1=1.0, J2=0.5, prec=prec)
    before = m.tuned_config()
    ref = m.evaluate(S, eloc=True)
    rep = m.autotune(S)
    print("\n" + rep)
    cfg = m.tuned_config()
    grids = [int(g.split()[0]) for g in rep.split("boundary grid:")[1].split("->")[0].replace(" ms", " ms,").split(",") if g.strip()]
    assert "warps" in rep.split("boundary grid:")[1]
    assert before["boundary_ctas"] == grids[0] and cfg["boundary_ctas"] in grids
    # nine warps or more of the smallest of these models share an SM: more than CTAs of any kind
    assert grids[0] > 4 * torch.cuda.get_device_properties(0).multi_processor_count
    if (D, Dc) == (3, 7):
        assert before["two_row_kernel"] == before["single_row_kernel"] == "one-warp"
        assert "one-warp" in rep.split("single-row kernel:")[0] and "one-warp" in rep.split("single-row kernel:")[1]
        assert "fused" not in rep
    else:
        assert before["two_row_kernel"] == before["single_row_kernel"] == "fused" and "one-warp" not in rep
    got = m.evaluate(S, eloc=True)
    torch.cuda.synchronize()
    assert torch.equal(got["logabs"], ref["logabs"]) and torch.equal(got["sign"], ref["sign"])
    m.close()
