"""The work this framework is used for, as cases that can be timed and compared.

A case names an operation of the public binding (``paper_1501_04784_gb300.fem``,
``autograd``), an element type, a grid, an operator, a precision and a numbering.
The meshes are those of the repository's own workloads: jittered brick grids on the
unit cube and the same grids with every cell cut into six tetrahedra, node and
element numbers permuted unless the case says otherwise, lognormal coefficients.

* ``build``:  values of K on a cached pattern (a time step, a Newton step).
* ``vjp``:    the backward pass for a given upstream gradient.
* ``train``:  forward and backward through autograd (shape or coefficient fitting).
* ``cold``:   a new mesh: handle, pattern, plan and first build (remeshing).
* ``batch``:  many uneven meshes in one call (data sets of small problems).
* ``step``:   mass matrix and load vector of a mesh (what a transient solve adds).
"""
import math

import torch

from paper_1501_04784_gb300 import autograd, fem

STIFFNESS, MASS, ELASTICITY = 0, 1, 2

# Corners of a cell as 4 z + 2 y + x bits: the brick's nodes in order, and the six
# tetrahedra around the main diagonal (odd permutations with nodes 1 and 2 swapped).
HEX = [[0, 1, 3, 2, 4, 5, 7, 6]]
TET = [[0, 1, 3, 7], [0, 5, 1, 7], [0, 3, 2, 7], [0, 2, 6, 7], [0, 4, 5, 7], [0, 6, 4, 7]]


def _case(do, kind, nx, ny, nz, op=STIFFNESS, prec="mixed", permute=True, jitter=0.2, sigma=0.5, meshes=1):
    return {"do": do, "kind": kind, "nx": nx, "ny": ny, "nz": nz, "op": op, "prec": prec, "permute": permute,
            "jitter": jitter, "sigma": sigma, "meshes": meshes}


def listed():
    def named(name, *a, **k):
        return {"name": name, **_case(*a, **k)}

    return [
        # the smallest real problem, rebuilt in FP64: launches and latency
        named("build_hex_8k_fp64", "build", "hex", 20, 20, 20, prec="fp64"),
        # the headline workload: a million bricks, mixed precision and FP64
        named("build_hex_1m_mixed", "build", "hex", 100, 100, 100, jitter=0.25, sigma=1.0),
        named("build_hex_1m_fp64", "build", "hex", 100, 100, 100, prec="fp64", jitter=0.25, sigma=1.0),
        # three million tetrahedra, the element of automatic meshers
        named("build_tet_3m_mixed", "build", "tet", 80, 80, 80, jitter=0.3),
        # the largest single mesh, in a mesher's natural numbering
        named("build_hex_27m_mixed", "build", "hex", 300, 300, 300, permute=False),
        # a data set of 512 small and medium problems in one call
        named("batch_hex_512_mixed", "batch", "hex", 60, 60, 60, permute=False, meshes=512),
        # sensitivities of a million-brick model with respect to geometry and material
        named("vjp_hex_1m_mixed", "vjp", "hex", 100, 100, 100, jitter=0.25, sigma=1.0),
        # one optimisation step on a tetrahedral mesh: K and both gradients
        named("train_tet_3m_mixed", "train", "tet", 80, 80, 80),
        # solid mechanics: the 3 x 3-block stiffness matrix of a million bricks
        named("build_elastic_hex_1m_mixed", "build", "hex", 100, 100, 100, op=ELASTICITY, jitter=0.25, sigma=1.0),
        # and its sensitivities on a smaller tetrahedral part
        named("vjp_elastic_tet_384k_mixed", "vjp", "tet", 40, 40, 40, op=ELASTICITY),
        # a new million-brick mesh: everything up to its first matrix
        named("cold_hex_1m_mixed", "cold", "hex", 100, 100, 100, jitter=0.25, sigma=1.0),
        # mass matrix and load vector of an odd-sized medium mesh
        named("step_hex_79k_mixed", "step", "hex", 53, 37, 41, op=MASS),
    ]


def _elements(case):
    return case["nx"] * case["ny"] * case["nz"] * (1 if case["kind"] == "hex" else 6)


def draw(rng):
    do = rng.choice(["build", "build", "build", "vjp", "train", "cold", "batch", "step"])
    kind = rng.choice(["hex", "hex", "tet"])
    prec = rng.choice(["mixed", "mixed", "fp64"])
    op = {"step": MASS, "batch": STIFFNESS}.get(do)
    if op is None:
        op = rng.choice([STIFFNESS, STIFFNESS, STIFFNESS, MASS, ELASTICITY])
    # tetrahedra are kept from degenerating, as any mesher keeps them
    jitter, sigma = rng.uniform(0.05, 0.3 if kind == "hex" else 0.2), rng.uniform(0.3, 1.0)
    if do == "batch":
        n = rng.randrange(10, 61)  # the largest grid edge of the batch
        most = (256 if kind == "hex" else 128) // (4 if prec == "fp64" else 1)
        meshes = int(math.exp(rng.uniform(math.log(8), math.log(most))))
        return _case(do, kind, n, n, n, op, prec, False, jitter, sigma, meshes)
    top = 3.0e6 / (3 if prec == "fp64" else 1) / (3 if op == ELASTICITY else 1)
    cells = math.exp(rng.uniform(math.log(1e3), math.log(top))) / (1 if kind == "hex" else 6)
    edge = max(4.0, cells ** (1 / 3))
    nx, ny = (max(3, round(edge * math.exp(rng.uniform(-0.4, 0.4)))) for _ in range(2))
    nz = max(3, round(edge ** 3 / (nx * ny)))
    return _case(do, kind, nx, ny, nz, op, prec, rng.random() < 0.7, jitter, sigma)


# ------------------------------------------------------------------- inputs
def _mesh(kind, nx, ny, nz, jitter, sigma, permute, dtype, op, gen):
    """X, E and c (elasticity: Lame parameters from a modulus and a Poisson ratio)."""
    dev = gen.device
    mx, my, mz = nx + 1, ny + 1, nz + 1
    n = mx * my * mz
    i = torch.arange(n, device=dev)
    ijk = torch.stack([i % mx, i // mx % my, i // (mx * my)], 1).double()
    size = torch.tensor([nx, ny, nz], dtype=torch.float64, device=dev)
    inside = ((ijk > 0) & (ijk < size)).all(1, keepdim=True)
    shift = (2 * torch.rand(n, 3, dtype=torch.float64, device=dev, generator=gen) - 1) * jitter
    X = (ijk + shift * inside) / size
    e = torch.arange(nx * ny * nz, device=dev)
    corner0 = e % nx + mx * (e // nx % ny + my * (e // (nx * ny)))
    at = [[(v & 1) + mx * (v >> 1 & 1) + mx * my * (v >> 2) for v in el] for el in (HEX if kind == "hex" else TET)]
    at = torch.tensor(at, device=dev)
    E = (corner0[:, None, None] + at).reshape(-1, at.shape[1])
    c = torch.exp(sigma * torch.randn(E.shape[0], dtype=torch.float64, device=dev, generator=gen))
    if permute:
        p = torch.randperm(n, device=dev, generator=gen)
        X[p] = X.clone()
        E = p[E][torch.randperm(E.shape[0], device=dev, generator=gen)]
    if op == ELASTICITY:
        nu = 0.1 + 0.35 * torch.rand(E.shape[0], dtype=torch.float64, device=dev, generator=gen)
        c = torch.stack([c * nu / ((1 + nu) * (1 - 2 * nu)), c / (2 * (1 + nu))], 1)
    return X.to(dtype).contiguous(), E.to(torch.int32).contiguous(), c.to(dtype).contiguous()


def _grids(case):
    """Grids of the case's meshes: one, or a batch's uneven shapes (element counts
    log-uniform up to the largest, edges from 10 cells)."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    if case["do"] != "batch":
        return [(nx, ny, nz)]
    r = torch.rand(case["meshes"], 3, dtype=torch.float64, generator=torch.Generator().manual_seed(17)).tolist()
    lo, grids = min(10, nx), []
    for a, b, t in r:
        gx, gy = lo + int(a * (nx - lo + 1)), lo + int(b * (nx - lo + 1))
        want = math.exp(math.log(lo ** 3) + t * math.log(max(1.0, min(2e5, nx ** 3) / lo ** 3)))
        grids.append((gx, gy, min(nx, max(lo, round(want / (gx * gy))))))
    return grids


def _inputs(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    dtype = fem.value_dtype(case["prec"])
    return [_mesh(case["kind"], *g, case["jitter"], case["sigma"], case["permute"], dtype, case["op"], gen)
            for g in _grids(case)], gen


def _upstream(nnz, dtype, gen):
    return torch.randn(nnz, dtype=dtype, device="cuda", generator=gen)


def _source(n_elems, dtype, gen):
    return torch.randn(n_elems, dtype=dtype, device="cuda", generator=gen)


def prepare(case, seed):
    parts, gen = _inputs(case, seed)
    dtype = fem.value_dtype(case["prec"])
    state = {"case": case, "parts": parts}
    if case["do"] == "cold":
        return state
    meshes = [fem.Mesh(E, X.shape[0], X=X, operator_kind=case["op"]) for X, E, c in parts]
    for m in meshes:
        m.pattern()
    state["meshes"] = meshes
    if case["do"] == "batch":
        # one buffer for every matrix of the batch, each starting on 256 bytes
        starts = [0]
        for m in meshes:
            starts.append(starts[-1] + -(-m.nnz // 64) * 64)
        state["flat"] = torch.zeros(starts[-1], dtype=dtype, device="cuda")
        state["out"] = [state["flat"][s:s + m.nnz] for s, m in zip(starts, meshes)]
    elif case["do"] in ("vjp", "train"):
        state["G"] = _upstream(meshes[0].nnz, dtype, gen)
    elif case["do"] == "step":
        state["src"] = _source(meshes[0].n_elems, dtype, gen)
    elif case["do"] == "build":
        state["out"] = torch.empty(meshes[0].nnz, dtype=dtype, device="cuda")
    return state


def run(state):
    case = state["case"]
    do, prec = case["do"], case["prec"]
    if do == "batch":
        X, c = [p[0] for p in state["parts"]], [p[2] for p in state["parts"]]
        fem.build_K_batched(state["meshes"], X, c, prec, out=state["out"])
        return state["flat"]
    X, E, c = state["parts"][0]
    if do == "cold":
        m = fem.Mesh(E, X.shape[0], X=X, operator_kind=case["op"])
        vals = m.build_K(X, c, prec)
        rowptr, col = m.get_pattern()
        return {"rowptr": rowptr, "col": col, "vals": vals}
    m = state["meshes"][0]
    if do == "build":
        return m.build_K(X, c, prec, out=state["out"])
    if do == "vjp":
        dX, dc = m.vjp(X, c, state["G"], prec)
        return {"dX": dX, "dc": dc}
    if do == "train":
        X, c = X.detach().requires_grad_(True), c.detach().requires_grad_(True)
        vals = autograd.build_K(m, X, c, prec)
        dX, dc = torch.autograd.grad(vals, (X, c), state["G"])
        return {"vals": vals.detach(), "dX": dX, "dc": dc}
    return {"M": m.build_K(X, c, prec), "F": m.load_vector(X, state["src"], prec)}


# ----------------------------------------------------------- work of one pass
# Floating-point operations of one element: matrix, then gradient.
FLOPS = {("hex", STIFFNESS): (1933, 4200), ("tet", STIFFNESS): (120, 300), ("hex", MASS): (520, 1500),
         ("tet", MASS): (60, 200), ("hex", ELASTICITY): (13700, 30000), ("tet", ELASTICITY): (700, 1700)}


def _nnz(kind, nx, ny, nz):
    """Entries of the node pattern's lower triangle: the diagonal and one entry for
    every neighbour offset of each opposite pair."""
    if kind == "hex":
        half = [(x, y, z) for x in (-1, 0, 1) for y in (-1, 0, 1) for z in (-1, 0, 1) if (z, y, x) > (0, 0, 0)]
    else:
        half = [(x, y, z) for x in (0, 1) for y in (0, 1) for z in (0, 1) if x + y + z]
    pairs = sum((nx + 1 - abs(x)) * (ny + 1 - abs(y)) * (nz + 1 - abs(z)) for x, y, z in half)
    return pairs + (nx + 1) * (ny + 1) * (nz + 1)


def work(case):
    s = 8 if case["prec"] == "fp64" else 4
    npe = 8 if case["kind"] == "hex" else 4
    total_bytes = total_flops = 0
    for g in _grids(case):
        nodes = (g[0] + 1) * (g[1] + 1) * (g[2] + 1)
        nel = _elements({**case, "nx": g[0], "ny": g[1], "nz": g[2]})
        nnz = _nnz(case["kind"], *g)
        rows = nodes
        if case["op"] == ELASTICITY:
            nnz, rows = 9 * nnz - 3 * nodes, 3 * nodes
        coef = nel * s * (2 if case["op"] == ELASTICITY else 1)
        inputs = 3 * nodes * s + 4 * npe * nel + coef
        gradients = 3 * nodes * s + coef
        f_mat, f_grad = FLOPS[case["kind"], case["op"]]
        do = case["do"]
        total_bytes += inputs + {"build": nnz * s, "batch": nnz * s, "vjp": nnz * s + gradients,
                                 "train": 2 * nnz * s + gradients, "cold": nnz * (s + 4) + 8 * (rows + 1),
                                 "step": nnz * s + nel * s + nodes * s}[do]
        total_flops += nel * {"vjp": f_grad, "train": f_mat + f_grad, "step": f_mat + 300}.get(do, f_mat)
    return {"bytes": total_bytes, "flops": total_flops}


# ------------------------------------------------- the same results in 64 bits
def _rule(kind, dev):
    """Quadrature weights [q], shape functions [q, a] and their derivatives [q, a, 3]."""
    if kind == "hex":
        at = torch.tensor([[v & 1, v >> 1 & 1, v >> 2] for v in HEX[0]], dtype=torch.float64, device=dev) * 2 - 1
        f = 0.5 + 0.5 * (at / math.sqrt(3.0))[:, None, :] * at[None]  # 1D factors (1 + xi xi_a) / 2
        d = 0.5 * at[None].expand_as(f)
        N = f.prod(2)
        dN = torch.stack([d[..., 0] * f[..., 1] * f[..., 2], f[..., 0] * d[..., 1] * f[..., 2],
                          f[..., 0] * f[..., 1] * d[..., 2]], 2)
        return torch.ones(8, dtype=torch.float64, device=dev), N, dN
    a, b = (5 + 3 * math.sqrt(5.0)) / 20, (5 - math.sqrt(5.0)) / 20  # exact for quadratics
    N = torch.full((4, 4), b, dtype=torch.float64, device=dev).fill_diagonal_(a)
    dN = torch.tensor([[-1, -1, -1], [1, 0, 0], [0, 1, 0], [0, 0, 1]], dtype=torch.float64, device=dev)
    return torch.full((4,), 1 / 24, dtype=torch.float64, device=dev), N, dN.expand(4, 4, 3)


def _element_matrices(case, x, c):
    """[e, n, n] (elasticity: [e, 3n, 3n]) of node coordinates x [e, n, 3] and c."""
    w, N, dN = _rule(case["kind"], x.device)
    J = torch.einsum("qai,eaj->eqij", dN, x)
    R = torch.linalg.cross(J[..., [1, 2, 0], :], J[..., [2, 0, 1], :])  # cofactor rows
    det = (J[..., 0, :] * R[..., 0, :]).sum(-1)
    wd = w * det.abs()
    if case["op"] == MASS:
        return torch.einsum("eq,qa,qb,e->eab", wd, N, N, c)
    B = torch.einsum("qai,eqij->eqaj", dN, R / det[..., None, None])
    if case["op"] == STIFFNESS:
        return torch.einsum("eq,eqai,eqbi->eab", wd, B, B) * c[:, None, None]
    P = torch.einsum("eq,eqai,eqbj->eaibj", wd, B, B)
    lam, mu = (c[:, k].reshape(-1, 1, 1, 1, 1) for k in (0, 1))
    eye = torch.eye(3, dtype=x.dtype, device=x.device).reshape(1, 1, 3, 1, 3)
    K = lam * P + mu * P.transpose(2, 4) + mu * eye * torch.einsum("eaibi->eab", P)[:, :, None, :, None]
    n = 3 * x.shape[1]
    return K.reshape(-1, n, n)


def _pattern(E, n, dofs):
    """Lower CSR of the mesh, and each element pair's position in it: pairs (a, b)
    of element degrees of freedom with the row from a."""
    if dofs == 3:
        E = (3 * E[:, :, None] + torch.arange(3, device=E.device)).reshape(E.shape[0], -1)
    keys = []
    rows = dofs * n
    for lo in range(0, E.shape[0], 1 << 20):
        e = E[lo:lo + (1 << 20)]
        k = e[:, :, None] * rows + e[:, None, :]
        keys.append(torch.unique(k[e[:, :, None] >= e[:, None, :]]))
    keys = torch.unique(torch.cat(keys))
    rowptr = torch.zeros(rows + 1, dtype=torch.int64, device=E.device)
    torch.cumsum(torch.bincount(keys // rows, minlength=rows), 0, out=rowptr[1:])
    return E, keys, rowptr, (keys % rows).to(torch.int32)


def _exact_matrix(case, X, E, c, G=None):
    """Values of the matrix; with G, also the gradients of sum G K."""
    n, dofs = X.shape[0], 3 if case["op"] == ELASTICITY else 1
    D, keys, rowptr, col = _pattern(E, n, dofs)
    vals = torch.zeros(keys.shape[0], dtype=torch.float64, device=X.device)
    dX, dc = torch.zeros_like(X), torch.zeros_like(c)
    for lo in range(0, E.shape[0], 1 << 17):
        e, d = E[lo:lo + (1 << 17)], D[lo:lo + (1 << 17)]
        x, ce = X[e].requires_grad_(G is not None), c[lo:lo + (1 << 17)].clone().requires_grad_(G is not None)
        K = _element_matrices(case, x, ce)
        lower = d[:, :, None] >= d[:, None, :]
        at = torch.searchsorted(keys, (d[:, :, None] * (dofs * n) + d[:, None, :])[lower])
        vals.index_add_(0, at, K[lower].detach())
        if G is not None:
            gx, gc = torch.autograd.grad((K[lower] * G[at]).sum(), (x, ce))
            dX.index_add_(0, e.reshape(-1), gx.reshape(-1, 3))
            dc[lo:lo + (1 << 17)] = gc
    return vals, rowptr, col, dX, dc


def exact(case, seed):
    if _elements(case) * case["meshes"] * (8 if case["op"] == ELASTICITY else 1) > 1.0e7 and case["do"] != "batch":
        return None
    parts, gen = _inputs(case, seed)
    if case["do"] == "batch":
        out = []
        for X, E, c in parts:
            v = _exact_matrix(case, X.double(), E.long(), c.double())[0]
            out += [v, v.new_zeros(-v.shape[0] % 64)]
        return torch.cat(out)
    X, E, c = parts[0]
    dtype = X.dtype
    X, E, c = X.double(), E.long(), c.double()
    if case["do"] in ("vjp", "train"):
        nnz = _nnz(case["kind"], case["nx"], case["ny"], case["nz"])
        if case["op"] == ELASTICITY:
            nnz = 9 * nnz - 3 * X.shape[0]
        vals, _, _, dX, dc = _exact_matrix(case, X, E, c, _upstream(nnz, dtype, gen).double())
        return {"dX": dX, "dc": dc} if case["do"] == "vjp" else {"vals": vals, "dX": dX, "dc": dc}
    vals, rowptr, col, _, _ = _exact_matrix(case, X, E, c)
    if case["do"] == "cold":
        return {"rowptr": rowptr, "col": col, "vals": vals}
    if case["do"] == "step":
        src = _source(E.shape[0], dtype, gen).double()
        f = _element_matrices(case, X[E], src).sum(2)  # int N_a = sum_b int N_a N_b
        return {"M": vals, "F": torch.zeros_like(X[:, 0]).index_add_(0, E.reshape(-1), f.reshape(-1))}
    return vals
