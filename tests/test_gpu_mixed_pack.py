"""A pack with models on both sides of Dc D = 32: results equal the separate calls
(also when calls follow each other without a wait, and on the legacy stream), and
the two kinds of sweeps overlap."""
import numpy as np
import pytest

from paper_1611_09467_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def requests():
    from paper_1611_09467_gb300 import build
    from paper_1611_09467_gb300.peps import PEPS
    build.build()
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    reqs = []
    for L, D, Dc, n in ((8, 8, 16, 1), (10, 4, 8, 96)):
        m = PEPS(inputs.near_product_tensors(L, L, D, D), L, L, D, Dc, J1=1.0, J2=0.5, prec="fp32")
        reqs.append((m, torch.from_numpy(inputs.pack_spins(inputs.random_sz0(n, L * L, L)).view(np.int64)).cuda()))
    yield reqs
    for m, _ in reqs:
        m.close()


@pytest.mark.parametrize("own_stream", [False, True])
def test_results_equal_separate_calls(requests, own_stream):
    from paper_1611_09467_gb300.peps import Packer
    ref = [m.evaluate(S, eloc=True) for m, S in requests]
    torch.cuda.synchronize()
    with torch.cuda.stream(torch.cuda.Stream() if own_stream else torch.cuda.default_stream()):
        pk = Packer()
        # both orders, back to back: the second call's sweeps wait for the first call's readers
        calls = [pk.evaluate(r, eloc=True) for r in (requests, requests[::-1], requests)]
        torch.cuda.synchronize()
        pk.close()
    for outs, order in zip(calls, ((0, 1), (1, 0), (0, 1))):
        for o, i in zip(outs, order):
            for k in ("logabs", "sign", "eloc", "status"):
                assert torch.equal(o[k], ref[i][k]), (k, i)


def test_the_two_kinds_of_sweeps_overlap(requests):
    """One long sweep leaves nearly all SMs idle, so the small model's sweeps cost
    next to nothing beside it: the pack takes less than nine tenths of the two alone."""
    from paper_1611_09467_gb300.peps import Packer
    with torch.cuda.stream(torch.cuda.Stream()):
        pk = Packer()

        def ms(reqs):
            t = []
            for k in range(7):
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record()
                pk.evaluate(reqs, eloc=False)
                b.record()
                b.synchronize()
                t.append(a.elapsed_time(b))
            return sorted(t)[3]
        both, large, small = ms(requests), ms(requests[:1]), ms(requests[1:])
        pk.close()
    print(f"pack {both:.2f} ms, the large model alone {large:.2f}, the small one {small:.2f}")
    assert both < 0.9 * (large + small)
