"""The force VJP's one-pass forms (three weights painted together, the staged readouts) against
the general forms behind the flags, over mesh sizes, particle orders and cotangent scales.

* default against PM_FLAG_TWO_MESH: one component at a time through the single-weight paint and
  the per-axis stencil; the same potentials up to FP32 rounding.
* learned factor, default against PM_FLAG_KSPACE_GRADIENT: three force meshes and a k-space sum.

Both sides carry the rounding of FP32 transforms and of the stencil of an FP32 potential, a few
1e-6 in relative RMS; 2e-5 is allowed, and 1e-4 for the factor's gradient (sums with cancellation).
"""
import numpy as np
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


def _particles(pm, cfg, n, seed):
    """n clustered particles (half of them in a few cells, some on tile faces), shuffled ids."""
    rng = np.random.default_rng(seed)
    u = inputs.uniform_positions(n, seed)
    half = n // 2
    cells = (rng.integers(0, cfg.nmesh, size=(3, 20))[:, rng.integers(0, 20, half)]).astype(np.uint64)
    cells[:, : half // 2] = cells[:, : half // 2] // 16 * 16 + 15
    u[:, :half] = (cells * (2 ** 32 // cfg.nmesh) + rng.integers(0, 2 ** 32 // cfg.nmesh, (3, half)).astype(np.uint64)) \
        .astype(np.uint32)
    ids = rng.permutation(cfg.n_particles())[:n].astype(np.uint32)
    return pm.as_u32_tensor(u), pm.as_u32_tensor(ids)


def _rel(a, b):
    return ((a.double() - b.double()).norm() / b.double().norm()).item()


CFG = dict(box=130.0, nc=24, nsites=4, nshell=3, nfib=1, m_nu=(0.1,) * 3)


@pytest.mark.parametrize("nmesh,n", [(32, 777), (64, 14001), (128, 14400), (256, 5000), (512, 3000)])
@pytest.mark.parametrize("scale", [1e-5, 1.0, 3e4])
def test_force_vjp_default_against_two_mesh(pm, nmesh, n, scale):
    out = []
    for flags in (0, pm.FLAG_TWO_MESH):
        cfg = pm.RunConfig(nmesh=nmesh, flags=flags, **CFG)
        ctx = pm.ParticleMesh(cfg)
        u, ids = _particles(pm, cfg, n, seed=n)
        g = torch.Generator(device="cuda").manual_seed(n)
        lam = torch.randn((3, n), generator=g, device="cuda") * scale
        out.append(ctx.force_vjp(u, ids, lam))
        ctx.sync()
        ctx.close()
    assert torch.isfinite(out[0]).all()
    assert _rel(out[0], out[1]) < 2e-5


@pytest.mark.parametrize("nmesh,n", [(32, 777), (64, 14001), (128, 14400), (256, 5000)])
def test_learned_vjp_default_against_kspace(pm, nmesh, n):
    out = []
    theta = inputs.mlp_parameters(3, last_scale=0.3)
    for flags in (0, pm.FLAG_KSPACE_GRADIENT):
        cfg = pm.RunConfig(nmesh=nmesh, flags=flags, **CFG)
        ctx = pm.ParticleMesh(cfg)
        ctx.set_mlp(theta)
        ctx.set_force_time(0.7)
        u, ids = _particles(pm, cfg, n, seed=n)
        g = torch.Generator(device="cuda").manual_seed(n)
        lam = torch.randn((3, n), generator=g, device="cuda")
        out.append((ctx.force_vjp(u, ids, lam), ctx.mlp_grad()))
        ctx.sync()
        ctx.close()
    assert _rel(out[0][0], out[1][0]) < 2e-5
    assert _rel(out[0][1], out[1][1]) < 1e-4


@pytest.mark.parametrize("scale", [2.0 ** -40, 1e-9, 0.3, 1.0, 77.0, 2.0 ** 20])
def test_signed_paint_is_the_exact_fixed_point_sum(pm, scale):
    """Weights from far below the 2^-32 resolution to beyond 32 bits of it, of both signs: the
    painted cells equal the 64-bit sums of the rounded contributions."""
    cfg = pm.RunConfig(box=10.0, nmesh=32, nc=16)
    ctx = pm.ParticleMesh(cfg)
    n = 4096
    u = inputs.uniform_positions(n, seed=5)
    u[:, : n // 2] = u[:, :8][:, np.arange(n // 2) % 8]          # many contributions to a few cells
    w = (np.random.default_rng(1).standard_normal(n) * scale).astype(np.float32)
    got = ctx.readout_T(pm.as_u32_tensor(u), torch.from_numpy(w).cuda()).cpu().numpy()
    ctx.sync()
    sums = np.zeros((32,) * 3, dtype=np.int64)
    cell = (u >> 27).astype(np.int64)
    f = ((u & 0x7ffffff).astype(np.float32) * np.float32(2.0 ** -27)).astype(np.float32)
    one = np.float32(1.0)
    for b in np.ndindex(2, 2, 2):
        c = [f[d] if b[d] else one - f[d] for d in range(3)]
        q = np.rint((c[0] * c[1] * c[2] * w * np.float32(2.0 ** 32)).astype(np.float64)).astype(np.int64)
        np.add.at(sums, tuple((cell[d] + b[d]) % 32 for d in range(3)), q)
    np.testing.assert_array_equal(got, sums.astype(np.float32) * np.float32(2.0 ** -32))
    ctx.close()
