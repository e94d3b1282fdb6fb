"""The FP32 statistics and pressure X passes on staged rows (256^3, one warp for two
rows; 512^3, one for a row) against the FP64 path, which runs other kernels, on the
same state: the record's documented bounds (2e-5 relative, skewness and flatness
1e-4 absolute) and 2e-5 of the pressure's norm."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
B = pytest.importorskip("paper_2012_04838_gb300.binding")


@pytest.mark.parametrize("N", [256, 512])
def test_fp32_record_and_pressure_match_fp64(N):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    dev = torch.device("cuda:0")
    out = {}
    state = None
    for prec in (B.FP32_MIXED, B.FP64):
        sim = B.Simulation(B.Params(N=N, precision=prec, nu=2e-3, cfl=0.5, ic=B.IC_SPECTRUM_K4, seed=9), device=dev)
        if state is None:
            sim.init_field()
            sim.step(2)
            state = sim.get_state()
        else:
            sim.set_state(state.to(torch.complex128))
        out[prec] = (sim.stats()[0], sim.pressure())
        sim.close()
        del sim
    (a, pa), (b, pb) = out[B.FP32_MIXED], out[B.FP64]
    for k in ("K", "K_phys", "eps", "eps_phys", "chi", "chi_phys", "phi_var", "umax"):
        assert a[k] == pytest.approx(b[k], rel=2e-5), k
    for k in ("skew", "flat", "skew_phi", "flat_phi"):
        assert a[k] == pytest.approx(b[k], abs=1e-4), k
    assert float((pa.to(torch.complex128) - pb).norm()) <= 2e-5 * float(pb.norm())
