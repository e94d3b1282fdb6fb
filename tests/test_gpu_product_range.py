"""The quadratic terms of the right-hand side hold over the range of the precision:
without viscosity, forcing or mean gradient rhs(a x) = a^2 rhs(x), bit for bit when a
is a power of two and nothing overflows.  a = 2^48 makes |u||omega| about 2^100: well
inside FP32 with its N^3-fold sums, and beyond it where products are formed from
fields that are N^3 times too large."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
B = pytest.importorskip("paper_2012_04838_gb300.binding")


@pytest.mark.parametrize("N,form,dealias", [
    (64, B.NL_ROTATIONAL, B.DEALIAS_TWO_THIRDS), (96, B.NL_ROTATIONAL, B.DEALIAS_TWO_THIRDS),
    (128, B.NL_CONVECTIVE, B.DEALIAS_TWO_THIRDS), (192, B.NL_ROTATIONAL, B.DEALIAS_PHASE_SHIFT),
    (256, B.NL_ROTATIONAL, B.DEALIAS_TWO_THIRDS), (256, B.NL_CONVECTIVE, B.DEALIAS_TWO_THIRDS),
    (256, B.NL_ROTATIONAL, B.DEALIAS_PHASE_SHIFT)])
def test_products_keep_the_range_of_fp32(N, form, dealias):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    dev = torch.device("cuda:0")
    p = B.Params(N=N, precision=B.FP32_MIXED, nu=0.0, beta=0.0, dt=1e-3, forcing=B.FORCE_NONE, nonlinear_form=form,
                 dealias=dealias)
    g = torch.Generator(device=dev).manual_seed(N)
    x = torch.view_as_complex(torch.randn((*B.compact_shape(N, dealias), 2), generator=g, device=dev)) * float(N) ** 1.5
    x[:, :, :, 0] = 0  # keep the kx = 0 plane trivially Hermitian
    sim = B.Simulation(p, device=dev)
    r = sim.rhs(x)
    s = sim.rhs(x * 2.0 ** 48)
    sim.close()
    assert bool(torch.isfinite(torch.view_as_real(s)).all())
    assert torch.equal(s, r * 2.0 ** 96)
