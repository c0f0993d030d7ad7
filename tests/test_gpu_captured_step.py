"""A captured step, replayed after another call of the same context has sorted more particles into
the array that holds the bucket starts of the state's order.

The state's n particles are the first n of the larger set in order, so the step takes the state
for near-sorted; its last bucket's range then ends beyond n and has to be cut there.  The replay
gives the eager step's state bit for bit.
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


@pytest.mark.parametrize("nmesh", [32, 64, 128])
def test_replay_after_a_larger_sort(pm, nmesh):
    n, extra = 20011, 5003
    cfg = pm.RunConfig(box=100.0, nmesh=nmesh, nc=32, n_max=n + extra)
    g = torch.Generator(device="cuda").manual_seed(nmesh)
    u = torch.randint(-2 ** 31, 2 ** 31, (3, n), generator=g, device="cuda", dtype=torch.int64).to(torch.int32)
    p = torch.randn((3, n), generator=g, device="cuda")
    st = {"u": u, "p": p, "id": torch.arange(n, dtype=torch.int32, device="cuda"), "f": torch.zeros_like(p),
          "f_valid": 0, "a": 0.3}
    ctx = pm.ParticleMesh(cfg)
    ctx.step(st, 0.3, 0.31, 0.32)
    ctx.sync()
    expected = {k: v.clone() if torch.is_tensor(v) else v for k, v in st.items()}
    other = pm.ParticleMesh(cfg)
    other.step(expected, 0.32, 0.33, 0.34)
    other.sync()
    other.close()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        ctx.step(st, 0.32, 0.33, 0.34)
    # the state, then particles of the last key (the last tile's last cell)
    tail = torch.full((3, extra), -1, dtype=torch.int32, device="cuda")
    ids = torch.arange(n + extra, dtype=torch.int32, device="cuda")
    ctx.force(torch.cat([st["u"], tail], dim=1), ids)
    ctx.sync()
    graph.replay()
    ctx.sync()
    fast, full, _ = ctx.sort_stats()
    assert (fast, full) == (2, 0)  # the replayed step took the near-sorted way
    for k in ("u", "p", "id", "f"):
        assert torch.equal(st[k], expected[k]), k
    ctx.close()
