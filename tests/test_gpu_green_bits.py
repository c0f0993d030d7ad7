"""The Green's function of meshes up to 512^3, bit for bit: FP32 sums of the tabulated k^2 and one
correctly rounded division.

The mesh holds a single 1 at the origin, so every stage of the forward transform is exact and the
spectrum is 1 everywhere; phi_k is then the Green's function itself, which numpy's float32
arithmetic restates.
"""
import numpy as np
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


@pytest.mark.parametrize("nmesh", [32, 64, 128, 256, 512])
def test_green_function_is_correctly_rounded(pm, nmesh):
    cfg = pm.RunConfig(box=173.0, nmesh=nmesh, nc=8)
    ctx = pm.ParticleMesh(cfg)
    mesh = torch.zeros((nmesh,) * 3, device="cuda")
    mesh[0, 0, 0] = 1.0
    phi = ctx.potential(mesh).cpu().numpy()
    ctx.sync()
    ctx.close()
    i = np.arange(nmesh)
    k = 2.0 * np.pi / cfg.box * np.where(i < nmesh // 2, i, i - nmesh)
    ksq = (k * k).astype(np.float32)
    gcoef = np.float32(-1.5 * cfg.omega_m / float(nmesh) ** 3)
    k2 = (ksq[:, None, None] + ksq[None, :, None]) + ksq[None, None, :nmesh // 2 + 1]
    k2[0, 0, 0] = np.inf
    np.testing.assert_array_equal(phi[..., 0], gcoef / k2)
    assert not phi[..., 1].any()
