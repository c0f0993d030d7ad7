"""The precision of the strided passes' radix-32 stages.

A transform of a white random mesh against torch's in 64 bits, relative rms error.  The bounds are
the errors of the same transforms in stages of radix 8 and 16 with factors rounded to FP32 (8-8-4
at 256, 8-8-8 at 512, 16-16-4 at 1024): 1.760e-7, 1.922e-7 and 2.134e-7, one per cent allowed for
the draw (four meshes differ by less).  Radix-32 stages with rounded factors have 1.851e-7 at
256^3 and 2.074e-7 at 512^3.
"""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.fixture(scope="module")
def pm():
    import __graft_entry__ as g
    g.build()
    from paper_2007_13394_gb300 import pm as _pm
    return _pm


@pytest.mark.parametrize("nmesh,bound", [(256, 1.760e-7), (512, 1.922e-7), (1024, 2.134e-7)])
def test_rounding_error_of_the_transforms(pm, nmesh, bound):
    ctx = pm.ParticleMesh(pm.RunConfig(box=100.0, nmesh=nmesh, nc=8, flags=pm.FLAG_TWO_MESH))
    g = torch.Generator(device="cuda").manual_seed(17)
    mesh = torch.randn((nmesh,) * 3, generator=g, device="cuda")
    ref = torch.fft.rfftn(mesh.double())
    out = torch.view_as_complex(ctx.fft_r2c(mesh))
    ctx.sync()
    assert ((out - ref).norm() / ref.norm()).item() < 1.01 * bound
    del out, mesh
    spectrum = ref.to(torch.complex64)
    del ref
    back = ctx.fft_c2r(torch.view_as_real(spectrum).contiguous())
    ctx.sync()
    ctx.close()
    exact = torch.fft.irfftn(spectrum.to(torch.complex128), s=(nmesh,) * 3)
    assert ((back.double() / nmesh ** 3 - exact).norm() / exact.norm()).item() < 1.01 * bound
