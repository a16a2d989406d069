"""Calls that put FP32 coordinates in locality order first (permuted meshes from 2^18
nodes on): forward and backward against the scatter plan, the host pipeline's row ranges,
calls of several streams on one mesh, and capture.

The buffer of ordered coordinates belongs to the mesh, so calls on different streams
pass it on; a captured call takes X by node id.
"""
import numpy as np
import pytest

import meshgen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

GRID = (66, 64, 62)  # 67 x 65 x 63 nodes, just above 2^18


@pytest.fixture(scope="module")
def fem():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1501_04784_gb300 import fem as f
    return f


def dev(a, dtype):
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda", dtype)


@pytest.fixture(scope="module", params=["hex", "tet"])
def case(request):
    gen = meshgen.hex_grid if request.param == "hex" else meshgen.kuhn_tets
    m = gen(*GRID, jitter=0.2, permute_nodes=True, permute_elems=True)
    E, X = dev(m.E, torch.int32), dev(m.X, torch.float64)
    g = torch.Generator("cuda").manual_seed(3)
    # three sets of coordinates, far enough apart that a mixture of two is seen
    Xs = [(X * s).float().contiguous() for s in (1.0, 1.25, 0.75)]
    cs = [torch.rand(m.n_elems, device="cuda", generator=g) + 0.5 for _ in Xs]
    return m, E, X, Xs, cs


def launches(fem, call):
    fem.launch_count(reset=True)
    r = call()
    return fem.launch_count(), r


def test_forward_and_backward(fem, case):
    m, E, X, Xs, cs = case
    a = fem.Mesh(E, m.n_nodes, X=X, patch_entries=2816 if m.E.shape[1] == 8 else 1024)
    b = fem.Mesh(E, m.n_nodes, X=X, patch_entries=2816 if m.E.shape[1] == 8 else 1024, fp64_fused=1)
    a.pattern()
    b.pattern()
    assert a.info()["gather_lists"] == 1 and b.info()["gather_lists"] == 0
    G = torch.randn(a.nnz, device="cuda", generator=torch.Generator("cuda").manual_seed(5))
    for x, c in zip(Xs, cs):
        n, v = launches(fem, lambda: a.build_K(x, c, "mixed"))
        assert n == 2  # the coordinates, then the values
        assert torch.equal(v, b.build_K(x, c, "mixed"))
        for u, w in zip(a.vjp(x, c, G, "mixed"), b.vjp(x, c, G, "mixed")):
            # the two plans sum a node's contributions in orders of their own
            assert float((u - w).abs().max()) <= 4e-6 * float(w.abs().max())
    a.sync()


def test_host_ranges(fem, case):
    m, E, X, Xs, cs = case
    mesh = fem.Mesh(E, m.n_nodes, X=X, host_chunks=4)
    mesh.pattern()
    for x, c in zip(Xs[:2], cs):
        want = mesh.build_K(x, c, "mixed").cpu()
        assert torch.equal(mesh.build_K_host(x.cpu().pin_memory(), c.cpu().pin_memory(), "mixed"), want)


def test_streams(fem, case):
    """Builds and backward passes of three streams, one set of coordinates each."""
    m, E, X, Xs, cs = case
    mesh = fem.Mesh(E, m.n_nodes, X=X)
    mesh.pattern()
    want = [mesh.build_K(x, c, "mixed").clone() for x, c in zip(Xs, cs)]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in Xs]
    outs = [[torch.empty_like(want[0]) for _ in range(4)] for _ in Xs]
    torch.cuda.synchronize()
    for r in range(4):
        for s, x, c, o in zip(streams, Xs, cs, outs):
            mesh.build_K(x, c, "mixed", out=o[r], stream=s)
    torch.cuda.synchronize()
    for o, w in zip(outs, want):
        for v in o:
            assert torch.equal(v, w)
    # a backward pass on one stream beside builds on the others
    G = torch.randn(mesh.nnz, device="cuda", generator=torch.Generator("cuda").manual_seed(5))
    dX, dc = [t.clone() for t in mesh.vjp(Xs[0], cs[0], G, "mixed")]
    torch.cuda.synchronize()
    for o in outs[1] + outs[2]:
        o.zero_()
    torch.cuda.synchronize()
    with torch.cuda.stream(streams[0]):
        got = [mesh.vjp(Xs[0], cs[0], G, "mixed") for _ in range(3)]
    for r in range(4):
        for k in (1, 2):
            mesh.build_K(Xs[k], cs[k], "mixed", out=outs[k][r], stream=streams[k])
    torch.cuda.synchronize()
    for u, w in got:
        assert torch.equal(u, dX) and torch.equal(w, dc)
    for k in (1, 2):
        for v in outs[k]:
            assert torch.equal(v, want[k])


def test_capture(fem, case):
    """A captured build takes X by id: graphs replayed side by side share no buffer."""
    m, E, X, Xs, cs = case
    mesh = fem.Mesh(E, m.n_nodes, X=X)
    mesh.pattern()
    want = [mesh.build_K(x, c, "mixed").clone() for x, c in zip(Xs[:2], cs)]
    outs = [torch.zeros_like(w) for w in want]
    graphs = []
    for x, c, o in zip(Xs, cs, outs):
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            n, _ = launches(fem, lambda: mesh.build_K(x, c, "mixed", out=o))
        assert n == 1
        graphs.append(g)
    streams = [torch.cuda.Stream() for _ in graphs]
    torch.cuda.synchronize()
    for _ in range(4):
        for g, s in zip(graphs, streams):
            with torch.cuda.stream(s):
                g.replay()
    torch.cuda.synchronize()
    for o, w in zip(outs, want):
        assert torch.equal(o, w)
