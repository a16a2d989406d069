"""Batches that one launch cannot build: meshes with and without gather lists, and meshes
whose largest closures and node lists do not fit one launch's shared memory together."""
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


@pytest.mark.parametrize("kind", ["hex", "tet"])
@pytest.mark.parametrize("prec", ["mixed", "fp64"])
def test_mixed_batch_leaves_the_plans_alone(fem, kind, prec):
    """A mesh without lists (it has a node of no element) beside meshes with them."""
    gen = meshgen.hex_grid if kind == "hex" else meshgen.kuhn_tets
    ms = [gen(*g, jitter=0.2, permute_nodes=True) for g in ((24, 25, 26), (9, 8, 7), (21, 22, 20))]
    dt = torch.float32 if prec == "mixed" else torch.float64
    X = [dev(m.X, dt) for m in ms]
    X[1] = torch.cat([X[1], X[1].mean(0, keepdim=True)])
    c = [dev(m.c, dt) for m in ms]
    mesh = [fem.Mesh(dev(m.E, torch.int32), x.shape[0], X=x) for m, x in zip(ms, X)]
    for m in mesh:
        m.pattern()
    before = [m.info() for m in mesh]
    assert [i["gather_lists"] for i in before] == [1, 0, 1]
    want = [m.build_K(x, k, prec).clone() for m, x, k in zip(mesh, X, c)]
    order = [0, 1, 2, 1, 0]
    for _ in range(2):
        vals = fem.build_K_batched([mesh[i] for i in order], [X[i] for i in order], [c[i] for i in order], prec)
        for i, v in zip(order, vals):
            if prec == "mixed":
                assert torch.equal(v, want[i])
            else:  # fused in batches, staged alone: one rounding of the element sums apart
                assert float((v - want[i]).abs().max()) <= 1.6e-13 * float(want[i].abs().max())
    assert [m.info()["n_patches"] for m in mesh] == [i["n_patches"] for i in before]
    assert fem.batched_config([mesh[i] for i in order], prec)["grid"] > 0
    for m, x, k, w in zip(mesh, X, c, want):
        assert torch.equal(m.build_K(x, k, prec), w)
        m.sync()


def test_meshes_that_fit_alone_only(fem):
    """FP64: large closures of a cube's patches, long node lists of a chain's."""
    cube = meshgen.hex_grid(24, 24, 24, jitter=0.2)
    chain = meshgen.hex_grid(1, 1, 1000, jitter=0.1)
    chain.X[:, 2] *= 1000.0  # cells as long as wide: a patch is a run of the chain
    mesh, X, c = [], [], []
    for m, entries in ((cube, 4200), (chain, 9000), (cube, 4200)):
        X.append(dev(m.X, torch.float64))
        c.append(dev(m.c, torch.float64))
        mesh.append(fem.Mesh(dev(m.E, torch.int32), m.n_nodes, X=X[-1], patch_entries=entries))
        mesh[-1].pattern()
    info = [m.info() for m in mesh]
    # element matrices of the cube's closures and the chain's coordinates and ids alone
    # are more than the 227 KB a block can have
    need = 288 * max(i["max_patch_elems"] for i in info) + 28 * max(i["max_patch_cnodes"] for i in info)
    assert need > 205 << 10 and all(i["gather_lists"] for i in info)
    for m, x, k, v in zip(mesh, X, c, fem.build_K_batched(mesh, X, c, "fp64")):
        ref = m.build_K(x, k, "fp64")
        assert float((v - ref).abs().max()) <= 1.6e-13 * float(ref.abs().max())
