"""The FP32 statistics add every point of a row to a compensated sum.  A field that takes
the values a, 0, -a, 0 along y and nothing else along x and z has exact values and, for
this a, an exact a^2 of 24 bits, so K_phys = a^2 / 4 to within the sum's own error:
at most n^2 2^-48 for a thread's n <= 512 terms of one size (1e-9).  Sixteen such terms
added plainly are off by 2.2e-7."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
B = pytest.importorskip("paper_2012_04838_gb300.binding")


@pytest.mark.parametrize("N", [64, 128, 256])
def test_sums_of_equal_terms(N):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    dev = torch.device("cuda:0")
    a = 1.79052734375  # 3667 / 2048
    sim = B.Simulation(B.Params(N=N, precision=B.FP32_MIXED, nu=1e-2, dt=1e-3), device=dev)
    shape = B.compact_shape(N)
    K = shape[3] - 1
    u = torch.zeros(shape, dtype=torch.complex64, device=dev)
    for ky in (-N // 4, N // 4):
        u[2, K, K + ky, 0] = 0.5 * a * N ** 3
    sim.set_state(u)
    rec = sim.stats()[0]
    sim.close()
    assert rec["K"] == pytest.approx(a * a / 4, rel=1e-6)
    assert abs(rec["K_phys"] - a * a / 4) <= 1e-9 * a * a / 4
