"""Where and when the passes are launched must not change what they compute: steps
recorded into a caller's CUDA graph (dependent launches included) and ensembles
whose workspaces exceed what is let under way at once both equal direct steps."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
B = pytest.importorskip("paper_2012_04838_gb300.binding")


@pytest.fixture()
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch.device("cuda:0")


@pytest.mark.parametrize("N,prec", [(8, B.FP32_MIXED), (32, B.FP64), (64, B.FP32_MIXED), (128, B.FP32_MIXED),
                                    (192, B.FP32_MIXED)])
def test_steps_captured_by_the_caller_equal_direct_steps(dev, N, prec):
    p = B.Params(N=N, precision=prec, ic=B.IC_SPECTRUM_K4, nu=0.01, cfl=0.5, record_every=3,
                 forcing=B.FORCE_HOLD_ENERGY)
    st = torch.cuda.Stream(dev)
    a, b = B.Simulation(p, device=dev, stream=st), B.Simulation(p, device=dev)
    a.init_field()
    b.init_field()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        a.step(2)
    for _ in range(3):
        g.replay()
    torch.cuda.synchronize()
    b.step(6)
    assert torch.equal(a.get_state(), b.get_state())


def test_ensemble_larger_than_what_runs_at_once(dev):
    sizes = [128] * 3 + [96] * 6 + [64] * 4 + [32] * 3

    def boxes():
        out = []
        for i, N in enumerate(sizes):
            p = B.Params(N=N, precision=B.FP32_MIXED, ic=B.IC_SPECTRUM_K4, seed=60 + i, nu=0.01, cfl=0.5, record_every=2)
            out.append(B.Simulation(p, device=dev, stream=torch.cuda.Stream(dev)))
            out[-1].init_field()
        return out

    alone, mixed = boxes(), boxes()
    for s in alone:
        s.step(4)
    b = B.Batch(mixed)
    b.step(1)
    b.step(3)
    b.synchronize()
    for a, m in zip(alone, mixed):
        assert torch.equal(a.get_state(), m.get_state())
        assert a.time() == m.time()
    b.close()
