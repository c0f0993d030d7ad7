"""The VJP readouts where tiles are full: 512 threads a tile from a mean of 1000 particles a tile on,
and the staged readout of one mesh from 200 on, against the general forms.

* force VJP, default against PM_FLAG_TWO_MESH; with the learned factor against
  PM_FLAG_KSPACE_GRADIENT: both sides carry the rounding of FP32 transforms and of the stencil of an
  FP32 potential, a few 1e-6 in relative RMS; 2e-5 is allowed, 1e-4 for the factor's gradient.
* paint VJP: a mesh that is not 16-byte aligned takes the gathering form; the same sums of eight
  products up to fused multiply-adds, a few 1e-7; 1e-6 is allowed.
"""
import pytest

from paper_2007_13394_gb300 import inputs

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


def _particles(nmesh, n, seed):
    """n particles, a third of them in an octant, some on the tiles' last cells; shuffled ids."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    u = torch.randint(0, 2 ** 32, (3, n), generator=g, device="cuda", dtype=torch.int64)
    u[:, ::3] //= 2
    cell = 2 ** 32 // nmesh
    u[0, 1::5] = u[0, 1::5] // (16 * cell) * (16 * cell) + 15 * cell + u[0, 1::5] % cell
    u = ((u + 2 ** 31) % 2 ** 32 - 2 ** 31).to(torch.int32)
    ids = torch.randperm(nmesh ** 3, generator=g, device="cuda")[:n].to(torch.int32)
    lam = torch.randn((3, n), generator=g, device="cuda")
    return u, ids, lam


def _rel(a, b):
    return ((a.double() - b.double()).norm() / b.double().norm()).item()


@pytest.mark.parametrize("nmesh,n", [(32, 8 * 1000 - 1), (32, 8 * 1000), (32, 31003), (64, 64 * 1000), (64, 200003),
                                     (128, 512 * 1000 + 7)])
def test_force_vjp_of_full_tiles(pm, nmesh, n):
    out = []
    u, ids, lam = _particles(nmesh, n, n)
    for flags in (0, pm.FLAG_TWO_MESH):
        ctx = pm.ParticleMesh(pm.RunConfig(box=130.0, nmesh=nmesh, nc=nmesh, flags=flags))
        out.append(ctx.force_vjp(u, ids, lam))
        ctx.sync()
        ctx.close()
    assert _rel(out[0], out[1]) < 2e-5


@pytest.mark.parametrize("nmesh,n", [(32, 8 * 1000 - 1), (32, 8 * 1000), (64, 64 * 1000), (128, 512 * 1000 + 7)])
def test_learned_vjp_of_full_tiles(pm, nmesh, n):
    out = []
    u, ids, lam = _particles(nmesh, n, n)
    for flags in (0, pm.FLAG_KSPACE_GRADIENT):
        ctx = pm.ParticleMesh(pm.RunConfig(box=130.0, nmesh=nmesh, nc=nmesh, flags=flags))
        ctx.set_mlp(inputs.mlp_parameters(3, last_scale=0.3))
        ctx.set_force_time(0.7)
        out.append((ctx.force_vjp(u, ids, lam), ctx.mlp_grad()))
        ctx.sync()
        ctx.close()
    assert _rel(out[0][0], out[1][0]) < 2e-5
    assert _rel(out[0][1], out[1][1]) < 1e-4


@pytest.mark.parametrize("nmesh,n", [(32, 8 * 200 - 1), (32, 8 * 200), (32, 8 * 1000), (64, 64 * 200), (64, 64 * 1000 + 3)])
def test_paint_vjp_of_a_misaligned_mesh(pm, nmesh, n):
    u, ids, _ = _particles(nmesh, n, n)
    g = torch.Generator(device="cuda").manual_seed(1)
    mesh = torch.randn((nmesh,) * 3, generator=g, device="cuda")
    shifted = torch.empty(nmesh ** 3 + 1, device="cuda")[1:].view_as(mesh).copy_(mesh)
    assert mesh.data_ptr() % 16 == 0 and shifted.data_ptr() % 16 == 4
    ctx = pm.ParticleMesh(pm.RunConfig(box=130.0, nmesh=nmesh, nc=nmesh))
    a, b = ctx.paint_vjp(u, ids, mesh), ctx.paint_vjp(u, ids, shifted)
    ctx.sync()
    ctx.close()
    assert _rel(a, b) < 1e-6
