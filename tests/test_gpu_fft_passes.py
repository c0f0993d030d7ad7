"""The strided FFT passes at every line length: forward transform of a full random mesh, the
inverse of its spectrum, and the potential's two-transform pass (through the force).

References are torch's FFTs in 64 bits.  Tolerance: the rounding of a 3 log2(N)-level FP32
transform is about 6e-8 sqrt(3 log2 N) <= 3.5e-7 in relative RMS; three times that is allowed.
"""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

TOL = 1e-6


@pytest.fixture(scope="module")
def pm():
    import __graft_entry__ as g
    g.build()
    from paper_2007_13394_gb300 import pm as _pm
    return _pm


def _rel(a, b):
    return ((a - b).norm() / b.norm()).item()


@pytest.mark.parametrize("nmesh", [32, 64, 128, 256, 512, 1024])
def test_forward_and_inverse_of_a_random_mesh(pm, nmesh):
    ctx = pm.ParticleMesh(pm.RunConfig(box=100.0, nmesh=nmesh, nc=8))
    g = torch.Generator(device="cuda").manual_seed(nmesh)
    mesh = torch.randn((nmesh,) * 3, generator=g, device="cuda")
    out = torch.view_as_complex(ctx.fft_r2c(mesh))
    ref = torch.fft.rfftn(mesh.double())
    assert _rel(out, ref) < TOL
    back = ctx.fft_c2r(torch.view_as_real(ref.to(torch.complex64)).contiguous())
    ctx.sync()
    assert _rel(back.double() / nmesh ** 3, mesh.double()) < TOL
    ctx.close()


@pytest.mark.parametrize("nmesh", [32, 128, 256, 512])
@pytest.mark.parametrize("spectral", [False, True])
def test_green_function_pass(pm, nmesh, spectral):
    cfg = pm.RunConfig(box=100.0, nmesh=nmesh, nc=8, flags=pm.FLAG_SPECTRAL_KERNEL if spectral else 0)
    ctx = pm.ParticleMesh(cfg)
    g = torch.Generator(device="cuda").manual_seed(nmesh)
    mesh = torch.randn((nmesh,) * 3, generator=g, device="cuda")
    phi = torch.view_as_complex(ctx.potential(mesh))
    ctx.sync()
    n = torch.fft.fftfreq(nmesh, 1.0 / nmesh, dtype=torch.float64, device="cuda")
    half = torch.arange(nmesh // 2 + 1, dtype=torch.float64, device="cuda")
    k2 = (2 * torch.pi / cfg.box) ** 2 * ((n ** 2)[:, None, None] + (n ** 2)[None, :, None] + half ** 2)
    if spectral:
        w = torch.sinc(n / nmesh) ** 4
        k2 = k2 * w[:, None, None] * w[None, :, None] * torch.sinc(half / nmesh) ** 4
    k2[0, 0, 0] = float("inf")
    ref = torch.fft.rfftn(mesh.double()) * (-1.5 * cfg.omega_m / nmesh ** 3 / k2)
    assert _rel(phi, ref) < TOL
    ctx.close()
