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
