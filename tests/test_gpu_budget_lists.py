"""Gather lists under a memory budget: what a plan may take and what later calls need."""
import numpy as np
import pytest

import meshgen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MB = 1 << 20


@pytest.fixture(scope="module")
def fem():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1501_04784_gb300 import fem as f
    return f


def dev(a, dtype):
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda", dtype)


@pytest.fixture(scope="module")
def case():
    m = meshgen.hex_grid(40, 40, 40, jitter=0.2, permute_nodes=True)
    return m, dev(m.E, torch.int32), dev(m.X, torch.float32), dev(m.c, torch.float32)


@pytest.mark.parametrize("room", [MB // 4, MB, 60 * MB, 200 * MB])
@pytest.mark.parametrize("prec", ["mixed", "fp64"])
def test_tuning_keeps_the_lists(fem, case, room, prec):
    """The tuner's scratch and the FP64 matrices are held while it plans: a plan made
    afterwards, with the defaults, is the one the mesh had before."""
    m, E, X, c = case
    dt = fem.value_dtype(prec)
    free = fem.Mesh(E, m.n_nodes, X=X)
    free.pattern()
    held = 256 * MB + (m.n_elems * 36 * 8 if prec == "fp64" else 0)
    mesh = fem.Mesh(E, m.n_nodes, X=X, mem_budget_bytes=free.info()["live_bytes"] + held + room)
    want = mesh.build_K(X.to(dt), c.to(dt), prec).clone()
    before = mesh.info()
    mesh.autotune(X.to(dt), c.to(dt), prec)
    mesh.set_tuning(0, 0)
    after = mesh.info()
    assert (after["n_patches"], after["n_groups"]) == (before["n_patches"], before["n_groups"])
    assert torch.equal(mesh.build_K(X.to(dt), c.to(dt), prec), want)
    mesh.sync()


@pytest.mark.parametrize("room", [0, MB, 12 * MB])
def test_lists_leave_room_for_staging(fem, case, room):
    """A budget that holds the scatter's plan and the call's staging is enough."""
    m, E, X, c = case
    Xh, ch = X.cpu(), c.cpu()  # pageable: K's values need device staging
    # planned for the scatter, its memory counted as under a budget (not in slabs)
    plain = fem.Mesh(E, m.n_nodes, X=X, fp64_fused=1, mem_budget_bytes=1 << 40)
    plain.pattern()
    want = plain.build_K_host(Xh, ch, "mixed", out=torch.empty(plain.nnz))
    X64, c64 = X.double(), c.double()
    G = torch.randn(plain.nnz, device="cuda", dtype=torch.float64)
    plain.vjp(X64, c64, G, "fp64")  # the in-row positions and the staged gradients (24 values a brick)
    budget = plain.info()["live_bytes"] + m.n_elems * (36 - 24) * 8 + room
    mesh = fem.Mesh(E, m.n_nodes, X=X, mem_budget_bytes=budget)
    mesh.pattern()
    assert mesh.info()["n_groups"] == 1
    v = mesh.build_K_host(Xh, ch, "mixed", out=torch.empty(mesh.nnz))
    assert float((v - want).abs().max()) <= 4e-6 * float(want.abs().max())
    # FP64 builds and backward passes run staged (two launches each), as without a budget
    mesh.build_K(X64, c64, "fp64")
    mesh.vjp(X64, c64, G, "fp64")
    for call in (lambda: mesh.build_K(X64, c64, "fp64"), lambda: mesh.vjp(X64, c64, G, "fp64")):
        fem.launch_count(reset=True)
        call()
        assert fem.launch_count() == 2
    assert mesh.info()["peak_bytes"] <= budget
    mesh.sync()


def test_ordered_coordinates_under_a_budget(fem):
    """A permuted mesh of 2^18 nodes: builds, then the first backward pass, within budgets
    that hold the scatter's plan and staging, and with lists where all of it fits."""
    m = meshgen.hex_grid(66, 64, 62, jitter=0.2, permute_nodes=True)
    E, X, c = dev(m.E, torch.int32), dev(m.X, torch.float32), dev(m.c, torch.float32)
    free = fem.Mesh(E, m.n_nodes, X=X)
    plain = fem.Mesh(E, m.n_nodes, X=X, fp64_fused=1, mem_budget_bytes=1 << 40)
    want, _ = free.build_K(X, c, "mixed"), plain.build_K(X, c, "mixed")
    G = torch.randn(free.nnz, device="cuda", generator=torch.Generator("cuda").manual_seed(5))
    dX, dc = free.vjp(X, c, G, "mixed")
    plain.vjp(X, c, G, "mixed")
    assert free.info()["gather_lists"] == 1 and plain.info()["gather_lists"] == 0
    seen = set()
    for extra in (0, 4, 16, 64, 1024):
        budget = plain.info()["peak_bytes"] + extra * MB
        mesh = fem.Mesh(E, m.n_nodes, X=X, mem_budget_bytes=budget)
        v = mesh.build_K(X, c, "mixed")
        assert float((v - want).abs().max()) <= 4e-6 * float(want.abs().max())
        for u, w in zip(mesh.vjp(X, c, G, "mixed"), (dX, dc)):
            assert float((u - w).abs().max()) <= 4e-6 * float(w.abs().max())
        fem.launch_count(reset=True)
        mesh.vjp(X, c, G, "mixed")
        assert fem.launch_count() in (2, 3)  # staged, the coordinates ordered or not
        info = mesh.info()
        assert info["n_groups"] == 1 and info["peak_bytes"] <= budget
        seen.add(info["gather_lists"])
        mesh.sync()
    assert seen == {0, 1}


def test_captured_calls_keep_their_plan(fem, case):
    """A captured build reads the plan it was captured with: calls that would need the
    lists' room afterwards do without."""
    m, E, X, c = case
    free = fem.Mesh(E, m.n_nodes, X=X, mem_budget_bytes=1 << 40)
    want = free.build_K(X, c, "mixed").clone()
    mesh = fem.Mesh(E, m.n_nodes, X=X, mem_budget_bytes=free.info()["peak_bytes"] + MB)
    out = torch.zeros_like(want)
    assert torch.equal(mesh.build_K(X, c, "mixed"), want) and mesh.info()["gather_lists"] == 1
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        mesh.build_K(X, c, "mixed", out=out)
    a = mesh.build_K(X.double(), c.double(), "fp64")  # 18 MB of matrices: fused instead
    b = free.build_K(X.double(), c.double(), "fp64")
    assert float((a - b).abs().max()) <= 1.6e-13 * float(b.abs().max())
    assert mesh.info()["gather_lists"] == 1
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, want)
    mesh.sync()
