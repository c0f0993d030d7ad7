"""Full tiles and large neutrino tails: the readout's node form (mean particles a tile from 1500
on, meshes from 256^3) and the gather through records (from 2^21 particles beyond the CDM block).

* Force against the k-space gradient path, whose readout interpolates three force meshes: the
  forms differ by the rounding of FP32 transforms, a few 1e-6; 1e-5 is allowed.
* The input order decides which particles go through records and nothing else: the same forces
  and the same states bit for bit.  A drifting readout equals steps one by one bit for bit.
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


def _cfg(pm, flags=0):
    # 64^3 CDM + 40^3 x 100 neutrinos: 6.66 M particles, 1626 a tile of the 256^3 mesh
    return pm.RunConfig(box=200.0, nmesh=256, nc=64, nsites=40, nshell=20, nfib=2, m_nu=(0.1,) * 3, flags=flags)


def _positions(cfg):
    n = cfg.n_particles()
    g = torch.Generator(device="cuda").manual_seed(2)
    u = torch.randint(-2 ** 31, 2 ** 31, (3, n), generator=g, device="cuda", dtype=torch.int64)
    u[:, ::3] = u[:, ::3] // 64                        # a dense corner across the periodic boundary
    u[0, 1::3] = u[0, 1::3] // 2 ** 28 * 2 ** 28 - 1   # the tiles' high x faces
    return u.to(torch.int32)


def test_node_form_matches_the_kspace_gradient(pm):
    cfg = _cfg(pm)
    u = _positions(cfg)
    out = []
    for flags in (0, pm.FLAG_KSPACE_GRADIENT):
        ctx = pm.ParticleMesh(_cfg(pm, flags))
        out.append(ctx.force(u).double())
        ctx.sync()
        ctx.close()
    assert ((out[0] - out[1]).norm() / out[1].norm()).item() < 1e-5


def test_input_order_changes_no_bit(pm):
    cfg = _cfg(pm)
    u = _positions(cfg)
    n = u.shape[1]
    ctx = pm.ParticleMesh(cfg)
    ids = torch.arange(n, dtype=torch.int32, device="cuda")
    F = ctx.force(u)
    order = torch.randperm(n, generator=torch.Generator(device="cuda").manual_seed(3), device="cuda")
    assert torch.equal(ctx.force(u, ids), F)
    assert torch.equal(ctx.force(u[:, order].contiguous(), ids[order].contiguous()), F[:, order])
    p = torch.randn((3, n), generator=torch.Generator(device="cuda").manual_seed(4), device="cuda")
    states = []
    for o in (torch.arange(n, device="cuda"), order):
        st = {"u": u[:, o].contiguous(), "p": p[:, o].contiguous(), "id": ids[o].contiguous(),
              "f": torch.zeros_like(p), "f_valid": 0}
        ctx.run(st, [(0.5, 0.51, 0.52), (0.52, 0.53, 0.54)])
        back = torch.argsort(st["id"].long())
        states.append([st[k][:, back] for k in ("u", "p", "f")])
    assert all(torch.equal(a, b) for a, b in zip(*states))
    st = {"u": u.clone(), "p": p.clone(), "id": ids.clone(), "f": torch.zeros_like(p), "f_valid": 0}
    ctx.step(st, 0.5, 0.51, 0.52)
    ctx.step(st, 0.52, 0.53, 0.54)
    back = torch.argsort(st["id"].long())
    assert all(torch.equal(st[k][:, back], a) for k, a in zip(("u", "p", "f"), states[0]))
    ctx.sync()
    ctx.close()
