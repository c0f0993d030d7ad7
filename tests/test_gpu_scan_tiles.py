"""The re-sort's scan from one tile of 4096 words to many: one launch up to eight tiles, two launches
above.  A step whose state is in the last sort's order (it takes its bucket starts from the scan)
against the same step in a new context (sorted from scratch, starts by search in the sorted keys):
the same state in the same order, bit for bit.
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


# words of the scan 3 (8 (N / 16)^3 + 1): 195, 1539, 12291 (4 tiles), 98307 (25), 786435 (193),
# 6291459 (1537)
@pytest.mark.parametrize("nmesh,n", [(32, 5000), (64, 30011), (128, 200003), (256, 300007), (512, 100003), (1024, 70001)])
def test_near_sorted_step_equals_the_step_from_scratch(pm, nmesh, n):
    cfg = pm.RunConfig(box=100.0, nmesh=nmesh, nc=min(nmesh, 128), n_max=n, flags=pm.FLAG_TWO_MESH)
    g = torch.Generator(device="cuda").manual_seed(n)
    u = torch.randint(-2 ** 31, 2 ** 31, (3, n), generator=g, device="cuda", dtype=torch.int64)
    u[:, ::2] //= 8  # half of them in one corner
    p = torch.randn((3, n), generator=g, device="cuda") * 3.0
    st = {"u": u.to(torch.int32), "p": p, "id": torch.arange(n, dtype=torch.int32, device="cuda"),
          "f": torch.zeros_like(p), "f_valid": 0, "a": 0.3}
    near = pm.ParticleMesh(cfg)
    near.step(st, 0.3, 0.31, 0.32)
    near.sync()
    copy = {k: v.clone() if torch.is_tensor(v) else v for k, v in st.items()}
    near.step(st, 0.32, 0.33, 0.34)
    near.sync()
    fast, full, movers = near.sort_stats()
    assert (fast, full) == (2, 0) and 0 < movers < n
    near.close()
    scratch = pm.ParticleMesh(cfg)
    scratch.step(copy, 0.32, 0.33, 0.34)
    scratch.sync()
    assert scratch.sort_stats()[:2] == (0, 1)
    scratch.close()
    for k in ("u", "p", "id", "f"):
        assert torch.equal(st[k], copy[k]), k
