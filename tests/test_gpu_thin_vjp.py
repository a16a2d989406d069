"""Backward pass of thin meshes planned for the scatter: their patches' closures hold so
many nodes that the coordinates take most of a block's shared memory."""
import numpy as np
import pytest

import meshgen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,dt", [("mixed", "float32"), ("mixed", "float64"), ("fp64", "float64")])
def test_thin_tetrahedra(prec, dt):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1501_04784_gb300 import fem
    m = meshgen.kuhn_tets(300, 300, 4, jitter=0.2, permute_nodes=True)
    E, X = torch.from_numpy(m.E).cuda().to(torch.int32), torch.from_numpy(m.X).cuda().to(getattr(torch, dt))
    c = torch.from_numpy(np.ascontiguousarray(m.c)).cuda().to(X.dtype)
    large, small = fem.Mesh(E, m.n_nodes, X=X), fem.Mesh(E, m.n_nodes, X=X, patch_entries=512)
    large.pattern()
    small.pattern()
    assert not large.info()["gather_lists"] and large.info()["max_patch_cnodes"] > 5000 > small.info()["max_patch_cnodes"]
    G = torch.randn(large.nnz, device="cuda", dtype=fem.value_dtype(prec),
                    generator=torch.Generator("cuda").manual_seed(5))
    eps = 1e-6 if prec == "mixed" else 1e-14
    for u, w in zip(large.vjp(X, c, G, prec), small.vjp(X, c, G, prec)):
        # the two plans sum a node's contributions in orders of their own
        assert float((u - w).abs().max()) <= 4 * eps * float(w.abs().max())


@pytest.mark.parametrize("grid", [(150, 150, 3), (512, 40, 40)])
def test_thin_meshes_are_planned_once(grid):
    """Closures out of the gather lists' range are found out before they are coloured and
    filled, and the plan is then the scatter's."""
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1501_04784_gb300 import fem
    m = meshgen.hex_grid(*grid, jitter=0.2, permute_nodes=True)
    E, X = torch.from_numpy(m.E).cuda().to(torch.int32), torch.from_numpy(m.X).cuda().float()
    c = torch.from_numpy(np.ascontiguousarray(m.c)).cuda().float()
    planned, launches = [], []
    for opts in ({}, {"fp64_fused": 1}):
        mesh = fem.Mesh(E, m.n_nodes, X=X, **opts)
        fem.launch_count(reset=True)
        mesh.pattern()
        launches.append(fem.launch_count())
        planned.append((mesh.info()["n_patches"], mesh.build_K(X, c, "mixed")))
    assert planned[0][0] == planned[1][0] and torch.equal(planned[0][1], planned[1][1])
    # the kernels up to the closures' node counts: eight of the global tables (a scan is
    # three), five of the closures' offsets, four of their elements, ranks and nodes
    assert launches[0] - launches[1] <= 8 + 5 + 4
