"""Builds on gather lists against the colour-ordered scatter kernels.

A mesh with ``fp64_fused=1`` is planned for the scatter (accumulator targets); any
other scalar mesh for the gather lists.  Planned with the same patches, both sum an
entry's contributions in the same order and take every element matrix from the same arithmetic, so the mixed
values, and the assembly of given matrices, are equal bit for bit.  The sizes are
those where the lists have edges: one element, rows with nothing but their diagonal,
chunks that are not full, patches of a few rows, and patch sizes out of the gather
kernels' range.
"""
import numpy as np
import pytest

import meshgen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fem():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1501_04784_gb300 import fem as f
    return f


def dev(a, dtype):
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda", dtype)


def grid(kind, nx, ny, nz, **kw):
    gen = meshgen.hex_grid if kind == "hex" else meshgen.kuhn_tets
    return gen(nx, ny, nz, jitter=0.25, permute_nodes=True, permute_elems=True, **kw)


def pair(fem, m, n_nodes=None, **opts):
    opts.setdefault("patch_entries", 2816)  # the default differs between the two
    E, X = dev(m.E, torch.int32), dev(m.X, torch.float64)
    n = n_nodes or m.n_nodes
    return fem.Mesh(E, n, X=X, **opts), fem.Mesh(E, n, X=X, fp64_fused=1, **opts)


SHAPES = [(1, 1, 1), (2, 1, 1), (3, 5, 2), (9, 7, 11), (31, 17, 13)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("kind", ["hex", "tet"])
@pytest.mark.parametrize("opts", [{}, {"patch_entries": 40}, {"patch_entries": 900}, {"patch_entries": 16384},
                                  {"operator_kind": 1}, {"fp64_sums": 1, "valence_threshold": 3}],
                         ids=lambda o: "-".join(f"{k}{v}" for k, v in o.items()) or "default")
def test_mixed_builds_equal_the_scatter(fem, kind, shape, opts):
    m = grid(kind, *shape)
    a, b = pair(fem, m, **opts)
    for dt in (torch.float32, torch.float64):
        X, c = dev(m.X, dt), dev(m.c, torch.float32)
        assert torch.equal(a.build_K(X, c, "mixed"), b.build_K(X, c, "mixed"))
    for prec, dt in (("mixed", torch.float32), ("fp64", torch.float64)):
        ke = a.integrate_local(dev(m.X, dt), dev(m.c, dt), prec)
        assert torch.equal(a.assemble_csr(ke, prec), b.assemble_csr(ke, prec))
    a.sync()
    b.sync()


@pytest.mark.parametrize("every", [1, 7, 400])
def test_distorted_bricks(fem, every):
    """Elements past the distortion threshold, from one in a patch to all of them."""
    m = grid("hex", 13, 11, 12)
    X = m.X.copy()
    for e in range(0, m.n_elems, every):  # pull one corner most of the way to the opposite one
        n = m.E[e]
        X[n[6]] += 0.55 * (X[n[0]] - X[n[6]]) / (1 if every > 50 else 4)
    a, b = pair(fem, m)
    X32, c = dev(X, torch.float32), dev(m.c, torch.float32)
    assert torch.equal(a.build_K(X32, c, "mixed"), b.build_K(X32, c, "mixed"))
    a.sync()


def test_node_of_no_element(fem):
    """A node without elements has an empty row, which the lists do not represent: the
    mesh is planned for the scatter, also inside a batch."""
    m = grid("hex", 6, 5, 4)
    X = np.concatenate([m.X, [[0.5, 0.5, 0.5]]])  # inside the box: the other nodes keep their order
    E, X64 = dev(m.E, torch.int32), dev(X, torch.float64)
    lone = fem.Mesh(E, m.n_nodes + 1, X=X64, patch_entries=2816)
    full = fem.Mesh(E, m.n_nodes, X=dev(m.X, torch.float64), patch_entries=2816)
    Xa, Xb, c = dev(X, torch.float32), dev(m.X, torch.float32), dev(m.c, torch.float32)
    want = full.build_K(Xb, c, "mixed").clone()
    assert torch.equal(lone.build_K(Xa, c, "mixed"), want)
    full.pattern()
    for v in fem.build_K_batched([full, lone, full], [Xb, Xa, Xb], [c, c, c], "mixed"):
        assert torch.equal(v, want)
    assert torch.equal(full.build_K(Xb, c, "mixed"), want)


@pytest.mark.parametrize("kind", ["hex", "tet"])
@pytest.mark.parametrize("prec", ["mixed", "fp64"])
def test_batched_and_backward(fem, kind, prec):
    """Batches of meshes with and without lists, and the backward pass on either plan."""
    dt = torch.float32 if prec == "mixed" else torch.float64
    ms = [grid(kind, *s) for s in ((1, 1, 1), (7, 6, 9), (20, 3, 14))]
    a = [fem.Mesh(dev(m.E, torch.int32), m.n_nodes, X=dev(m.X, torch.float64)) for m in ms]
    X, c = [dev(m.X, dt) for m in ms], [dev(m.c, dt) for m in ms]
    for m in a:
        m.pattern()
    vals = fem.build_K_batched(a, X, c, prec)
    eps = 1e-6 if prec == "mixed" else 1e-14
    for m, x, k, v in zip(a, X, c, vals):
        ref = m.build_K(x, k, prec)
        if prec == "mixed":
            assert torch.equal(v, ref)
        else:  # fused in batches, staged alone: one rounding of the element sums apart
            assert float((v - ref).abs().max()) <= 16 * eps * float(ref.abs().max())
    b = fem.Mesh(dev(ms[2].E, torch.int32), ms[2].n_nodes, X=dev(ms[2].X, torch.float64), fp64_fused=1)
    G = torch.randn(a[2].nnz, dtype=dt, device="cuda", generator=torch.Generator("cuda").manual_seed(5))
    b.pattern()
    for u, w in zip(a[2].vjp(X[2], c[2], G, prec), b.vjp(X[2], c[2], G, prec)):
        assert float((u - w).abs().max()) <= 4 * eps * float(w.abs().max())


@pytest.mark.parametrize("kind", ["hex", "tet"])
@pytest.mark.parametrize("opts", [{}, {"patch_entries": 40}, {"patch_entries": 900}],
                         ids=lambda o: "-".join(f"{k}{v}" for k, v in o.items()) or "default")
def test_load_vectors_equal_the_scatter(fem, kind, opts):
    """The list form of the load vector (bricks) sums in the colour order too: equal bit for bit."""
    for shape in SHAPES:
        m = grid(kind, *shape)
        a, b = pair(fem, m, **opts)
        for prec, dt in (("mixed", torch.float32), ("mixed", torch.float64), ("fp64", torch.float64)):
            X, c = dev(m.X, dt), dev(m.c, dt)
            assert torch.equal(a.load_vector(X, c, prec), b.load_vector(X, c, prec))


@pytest.mark.parametrize("kind", ["hex", "tet"])
def test_patch_sizes_follow_the_route(fem, kind):
    """Lists and scatter have default patch sizes of their own: a mesh that cannot have
    lists is planned at the scatter's, and 4,096 entries bound the lists' default."""
    m = grid(kind, *((40, 40, 40) if kind == "hex" else (24, 24, 24)))
    E, X = dev(m.E, torch.int32), dev(m.X, torch.float64)
    c = dev(m.c, torch.float32)

    def planned(n=m.n_nodes, x=X, **opts):
        mesh = fem.Mesh(E, n, X=x, **opts)
        v = mesh.build_K(x.float(), c, "mixed")
        return mesh.info(), v

    lists, scatter = planned(), planned(fp64_fused=1)
    assert lists[0]["n_patches"] > scatter[0]["n_patches"]
    bound = planned(patch_entries=4096)
    assert bound[0]["n_patches"] == lists[0]["n_patches"] and torch.equal(bound[1], lists[1])
    far = torch.cat([X, X[:1]])  # one node of no element
    lone, other = planned(m.n_nodes + 1, far), planned(m.n_nodes + 1, far, fp64_fused=1)
    assert lone[0]["n_patches"] == other[0]["n_patches"] and torch.equal(lone[1], other[1])
    budget = int(0.7 * scatter[0]["plan_bytes"])
    tight, same = planned(mem_budget_bytes=budget), planned(mem_budget_bytes=budget, fp64_fused=1)
    assert tight[0]["n_groups"] == same[0]["n_groups"] and tight[0]["n_patches"] == same[0]["n_patches"]
    assert torch.equal(tight[1], same[1])
