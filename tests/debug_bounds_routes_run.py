"""Child process of test_gpu_debug_bounds_routes.py: the bounds-check build on both routes
of the scalar builds, gather lists and the scatter.  Prints one JSON line.  Not a test
module by itself."""
import json
import os
import sys

import numpy as np
import torch

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))

import meshgen  # noqa: E402


def main():
    from paper_1501_04784_gb300 import _build
    assert _build.DEBUG_BOUNDS, "FEM_DEBUG_BOUNDS=1 must be set"
    _build.build()
    from paper_1501_04784_gb300 import abi, fem
    out = {"clean": {}, "planted": {}, "after": {}}

    def dev(a, dt):
        return torch.as_tensor(np.ascontiguousarray(a), device="cuda").to(dt)

    meshes = {"hex": meshgen.hex_grid(7, 5, 3, jitter=0.25, seed=5, permute_nodes=True, permute_elems=True),
              "tet": meshgen.kuhn_tets(6, 4, 3, jitter=0.3, seed=2, permute_nodes=True, permute_elems=True)}
    for name, m in meshes.items():
        E, X64 = dev(m.E, torch.int32), dev(m.X, torch.float64)
        for route, opts in (("lists", {}), ("scatter", {"fp64_fused": 1})):
            def make(**more):
                return fem.Mesh(E, m.n_nodes, X=X64, patch_entries=64, **opts, **more)

            for prec, dt in (("mixed", torch.float32), ("fp64", torch.float64)):
                X, c = dev(m.X, dt), dev(m.c, dt)
                a, b = make(), make()
                single = a.build_K(X, c, prec)
                b.pattern()
                assert a.info()["gather_lists"] == b.info()["gather_lists"] == (route == "lists")
                given = a.assemble_csr(a.integrate_local(X, c, prec), prec)
                batched = fem.build_K_batched([a, b], [X, X], [c, c], prec)
                a.load_vector(X, c, prec)
                G = torch.ones(a.nnz, dtype=dt, device="cuda")
                a.vjp(X, c, G, prec)
                a.sync()
                b.sync()
                top, eps = float(single.abs().max()), 1e-6 if prec == "mixed" else 1e-14
                out["clean"][f"{name}_{route}_{prec}"] = all(
                    float((v - single).abs().max()) <= 16 * eps * top for v in [given, *batched])
                # one planted out-of-range node id a patch: caught, skipped, reported once
                for how in ("single", "batched"):
                    if prec == "fp64" and route == "lists" and how == "single":
                        continue  # staged: the kernel reads element matrices, not coordinates
                    p = make(debug_stall=2)
                    p.pattern()
                    assert p.info()["gather_lists"] == (route == "lists")
                    if how == "single":
                        p.build_K(X, c, prec)
                    else:
                        fem.build_K_batched([p, p], [X, X], [c, c], prec)
                    try:
                        p.sync()
                        seen = "FEM_OK"
                    except abi.FemError as e:
                        seen = e.name
                    out["planted"][f"{name}_{route}_{prec}_{how}"] = seen
                    p.sync()
                out["after"][f"{name}_{route}_{prec}"] = torch.equal(a.build_K(X, c, prec), single)
                a.sync()
    print(json.dumps(out))


if __name__ == "__main__":
    main()
