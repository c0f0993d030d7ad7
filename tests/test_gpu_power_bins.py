"""Spectrum binning against a plain 64-bit binning of the same painted meshes.

Mode counts are integers: equal.  Mean wavenumbers: sums of at most 1e7 square roots in FP64,
1e-12.  P: white spectra (uniform random particles), so every mode carries the FP32 transform's
error of about 3.5e-7 of the rms amplitude, twice in a product; 1e-5 per bin.
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


def _reference(ra, rb, box, nbins):
    N = ra.shape[0]
    da, db = (torch.fft.rfftn(r.double() / r.double().mean()) for r in (ra, rb))
    n = torch.fft.fftfreq(N, 1.0 / N, dtype=torch.float64, device="cuda")
    half = torch.arange(N // 2 + 1, dtype=torch.float64, device="cuda")
    n2 = ((n ** 2)[:, None, None] + (n ** 2)[None, :, None] + half ** 2).reshape(-1)
    w = torch.sinc(n / N) ** -4
    P = (da * db.conj()).real * w[:, None, None] * w[None, :, None] * torch.sinc(half / N) ** -4
    mult = (1.0 + ((half > 0) & (half < N // 2)).double()).expand(N, N, -1).reshape(-1)
    b = torch.floor(torch.sqrt(n2) - 0.5).long()
    b = torch.where((n2 == 0) | (b >= nbins), torch.full_like(b, nbins), b)
    tot = lambda v: torch.zeros(nbins + 1, dtype=torch.float64, device="cuda").index_add(0, b, v)[:nbins].cpu().numpy()  # noqa: E731
    cnt = tot(mult)
    one = np.maximum(cnt, 1.0)
    return (tot(mult * torch.sqrt(n2)) / one * 2 * np.pi / box,
            tot(mult * P.reshape(-1)) / one * box ** 3 / float(N) ** 6, cnt.astype(np.int64))


@pytest.mark.parametrize("nmesh,nbins", [(32, 1), (32, 16), (32, 2048), (64, 31), (128, 64), (128, 111), (256, 200)])
@pytest.mark.parametrize("sa,sb", [(3, 3), (1, 2)])
def test_bins_match_a_64_bit_binning(pm, nmesh, nbins, sa, sb):
    cfg = pm.RunConfig(box=97.0, nmesh=nmesh, nc=20, nsites=6, nshell=3, nfib=1, m_nu=(0.1,) * 3)
    ctx = pm.ParticleMesh(cfg)
    u = pm.as_u32_tensor(inputs.uniform_positions(cfg.n_particles(), seed=nmesh + nbins))
    k, P, cnt = ctx.power(u, None, sa, sb, nbins=nbins)
    again = ctx.power(u, None, sa, sb, nbins=nbins)
    kr, Pr, cr = _reference(ctx.paint(u, None, sa), ctx.paint(u, None, sb), cfg.box, nbins)
    np.testing.assert_array_equal(cnt, cr)
    np.testing.assert_allclose(k, kr, rtol=1e-12)
    # relative to the white level: a cross spectrum has bins near zero
    level = np.abs(Pr[cr > 100]).mean() if (cr > 100).any() else np.abs(Pr).max()
    auto = [ctx.power(u, None, s, s, nbins=nbins)[1] for s in (sa, sb)]
    scale = np.sqrt(auto[0] * auto[1]) + 1e-30 if sa != sb else np.maximum(np.abs(Pr), 1e-30 * level + 1e-300)
    assert np.all(np.abs(P - Pr)[cr > 0] <= 1e-5 * scale[cr > 0])
    for x, y in zip((k, P, cnt), again):
        np.testing.assert_array_equal(x, y)   # fixed summation order
    ctx.close()


@pytest.mark.parametrize("nmesh,nbins", [(32, 16), (64, 64), (128, 20)])
def test_spectrum_gradient_weights(pm, nmesh, nbins):
    """sum_b w_b P_b moves with the particles as the gradient says (central difference along a
    random direction; FP32 spectra limit it to about 1e-3)."""
    cfg = pm.RunConfig(box=50.0, nmesh=nmesh, nc=16)
    ctx = pm.ParticleMesh(cfg)
    rng = np.random.default_rng(nmesh)
    u = inputs.uniform_positions(16 ** 3, seed=nmesh)
    w = rng.standard_normal(nbins)
    g = ctx.power_vjp(pm.as_u32_tensor(u), None, w).double().cpu().numpy()
    d = rng.standard_normal(u.shape) * 1e-3 * cfg.box / nmesh
    vals = []
    for sgn in (1.0, -1.0):
        step = np.rint(sgn * d * 2.0 ** 32 / cfg.box).astype(np.int64)
        v = ((u.astype(np.int64) + step) % 2 ** 32).astype(np.uint32)
        vals.append(float((ctx.power(pm.as_u32_tensor(v), None, nbins=nbins)[1] * w).sum()))
    scale = np.linalg.norm(g) * np.linalg.norm(d) / np.sqrt(g.size)
    assert abs((vals[0] - vals[1]) / 2 - (g * d).sum()) < 3e-2 * scale + 1e-6 * abs(vals[0])
    ctx.close()
