"""The radix sort at the edges of its tiles (4096 keys) and chunks (one per CTA, 456 of them),
for every digit width: the permutation equals torch's stable sort of the keys, exactly."""
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


def _keys(u, nmesh):
    c = (u.long() & 0xffffffff) * nmesh >> 32
    t, l = c // 16, c % 16
    nt = nmesh // 16
    cls = 4 * (l[0] == 15) + 2 * (l[1] == 15) + (l[2] == 15).long()
    return ((t[0] * nt + t[1]) * nt + t[2]) * 8 + cls


# 7-bit digits in one pass (32), 9 in one (64), 7 in two (128), 8 in two (256), 9 in two (512),
# 7 in three (1024)
@pytest.mark.parametrize("nmesh", [32, 64, 128, 256, 512, 1024])
@pytest.mark.parametrize("n", [1, 31, 4095, 4096, 4097, 3 * 4096 + 17, 456 * 4096, 456 * 4096 + 1, 2 * 456 * 4096 + 4097])
@pytest.mark.parametrize("clustered", [False, True])
def test_sort_is_the_stable_sort(pm, nmesh, n, clustered):
    ctx = pm.ParticleMesh(pm.RunConfig(box=1.0, nmesh=nmesh, nc=8, n_max=n))
    g = torch.Generator(device="cuda").manual_seed(n + nmesh)
    u = torch.randint(-2 ** 31, 2 ** 31, (3, n), generator=g, device="cuda", dtype=torch.int64)
    if clustered:  # nearly all in one tile, and its neighbours' faces
        u = torch.where(torch.rand((1, n), generator=g, device="cuda") < 0.9, (u % (2 ** 32 // nmesh * 17)), u)
        u = (u + 2 ** 31) % 2 ** 32 - 2 ** 31
    u = u.to(torch.int32)
    perm, keys = ctx.sort(u)
    ctx.sync()
    k, p = torch.sort(_keys(u, nmesh), stable=True)
    assert torch.equal(keys.long(), k)
    assert torch.equal(perm.long() & 0xffffffff, p)
    ctx.close()
