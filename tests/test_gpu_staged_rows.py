"""The staged strided passes on rows the tensor maps do not describe as they are:
compact rows of odd length (128^3 and 512^3: the z-inverse copies its tile with
cp.async), padded stream rows, and the 520-point lines transformed by 26 lanes.
Every variant runs the same arithmetic per column as variant 0, so the
right-hand sides agree bit for bit."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

B = pytest.importorskip("paper_2012_04838_gb300.binding")


@pytest.mark.parametrize("N,dealias", [(128, B.DEALIAS_TWO_THIRDS), (128, B.DEALIAS_PHASE_SHIFT),
                                       (192, B.DEALIAS_PHASE_SHIFT), (512, B.DEALIAS_TWO_THIRDS),
                                       (520, B.DEALIAS_TWO_THIRDS), (520, B.DEALIAS_PHASE_SHIFT)])
def test_staged_variants_agree_bit_for_bit(monkeypatch, N, dealias):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    dev = torch.device("cuda:0")
    p = B.Params(N=N, precision=B.FP32_MIXED, nu=1e-3, dt=1e-3, dealias=dealias)
    g = torch.Generator(device=dev).manual_seed(N)
    x = torch.view_as_complex(torch.randn((*B.compact_shape(N, dealias), 2), generator=g, device=dev)) * 1e3
    x[:, :, :, 0] = 0  # keep the kx = 0 plane trivially Hermitian
    ref = None
    for v in ("0000", "2222", "3333", "4433"):
        monkeypatch.setenv("PSC_STRIDED_VARIANT", v)
        sim = B.Simulation(p, device=dev)
        try:
            assert all(sim.tile_staged().values()) == (v != "0000")
            r = sim.rhs(x)
        finally:
            sim.close()
        del sim
        if ref is None:
            ref = r
        else:
            assert torch.equal(r, ref), v
        torch.cuda.empty_cache()
