"""Products launched back to back start while the one before drains: a chain
in which each reads what the last wrote gives the same bits as with a wait
after every product, and as the same chain replayed from a captured graph."""
import pytest

torch = pytest.importorskip("torch")

SIZES = [(5, 4), (69, 45), (513, 391), (5, 4, 6), (17, 17, 17), (33, 25, 29), (45, 47, 52)]


def _chain(pf, H, x, v, ys, fp32, wait):
    src = v
    for y in ys:
        if fp32:
            pf.hessvec(H, 0, x, src, y)
        else:
            pf.hessvec_lagged(H, 0, src, y)
        if wait:
            torch.cuda.synchronize()
        src = y
    return [y.clone() for y in ys]


@pytest.mark.gpu
@pytest.mark.parametrize("fp32", [True, False], ids=["fp32", "fp64"])
@pytest.mark.parametrize("n", SIZES, ids=lambda n: "x".join(map(str, n)))
def test_chain_of_products(n, fp32):
    import paper_2007_12908_gb300 as pf

    st = torch.cuda.Stream()
    g = torch.Generator(device="cuda").manual_seed(sum(n))
    dt = torch.float32 if fp32 else torch.float64
    with torch.cuda.stream(st):
        H = pf.mesh_hierarchy_create(len(n), list(n), 1, 1.0, E=1.0, nu=0.25, Gc=1.0, ls_over_h=2.0, stream=st)
        pf.pressure_set(H, 5e-4)
        x = torch.rand(H.ndof(), dtype=dt, device="cuda", generator=g) * 0.5
        v = torch.randn(H.ndof(), dtype=dt, device="cuda", generator=g)
        if not fp32:
            pf.hessvec_lag_set(H, 0, x)
        ys = [torch.empty_like(v) for _ in range(6)]
        want = _chain(pf, H, x, v, ys, fp32, wait=True)
        for y in ys:
            y.fill_(float("nan"))
        got = _chain(pf, H, x, v, ys, fp32, wait=False)
        st.synchronize()
        graph = torch.cuda.CUDAGraph()
        for y in ys:
            y.fill_(float("nan"))
        st.synchronize()
    with torch.cuda.graph(graph, stream=st):
        replayed = _chain(pf, H, x, v, ys, fp32, wait=False)
    graph.replay()
    torch.cuda.synchronize()
    for a, b, c in zip(want, got, replayed):
        assert torch.isfinite(a).all()
        assert torch.equal(a, b)
        assert torch.equal(a, c)
