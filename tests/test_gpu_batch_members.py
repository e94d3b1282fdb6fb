"""Graph batches whose members differ in kind and size compute what each member computes
alone: one member by itself, members larger than the budget of what is let under way,
such members beside small ones, and FP64, phase-shift and convective members.  And steps
of the last two kinds that the caller captures, where the launches are dependent ones."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
B = pytest.importorskip("paper_2012_04838_gb300.binding")

F, D = dict(precision=B.FP32_MIXED), dict(precision=B.FP64)
PS = dict(precision=B.FP32_MIXED, dealias=B.DEALIAS_PHASE_SHIFT)
CV = dict(precision=B.FP32_MIXED, nonlinear_form=B.NL_CONVECTIVE)


@pytest.fixture()
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch.device("cuda:0")


def params(i, N, kw):
    return B.Params(N=N, ic=B.IC_SPECTRUM_K4, seed=80 + i, nu=0.01, cfl=0.5, record_every=2, **kw)


@pytest.mark.parametrize("members", [
    [(256, F)],
    [(192, F), (256, F), (192, F)],
    [(256, F)] + [(64, F)] * 5 + [(32, F)],
    [(256, F)] * 2 + [(192, F)] * 3 + [(128, F)] * 2 + [(96, F)] * 2 + [(64, F)] * 3,
    [(128, D), (96, PS), (128, CV), (64, PS), (48, D), (16, F)],
])
def test_batch_equals_members_alone(dev, members):
    alone, mixed = [[B.Simulation(params(i, N, kw), device=dev, stream=torch.cuda.Stream(dev))
                     for i, (N, kw) in enumerate(members)] for _ in range(2)]
    for s in alone + mixed:
        s.init_field()
    for s in alone:
        s.step(3)
    b = B.Batch(mixed)
    b.step(1)
    b.step(2)
    b.synchronize()
    for a, m in zip(alone, mixed):
        assert torch.equal(a.get_state(), m.get_state())
        assert a.time() == m.time()
    b.close()


@pytest.mark.parametrize("N,kw", [(12, PS), (64, PS), (128, PS), (16, CV), (96, CV), (128, CV)])
def test_captured_steps_of_the_other_forms(dev, N, kw):
    st = torch.cuda.Stream(dev)
    a, b = B.Simulation(params(0, N, kw), device=dev, stream=st), B.Simulation(params(0, N, kw), device=dev)
    a.init_field()
    b.init_field()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        a.step(2)
    for _ in range(2):
        g.replay()
    torch.cuda.synchronize()
    b.step(4)
    assert torch.equal(a.get_state(), b.get_state())
