"""The assembly calls that a flow solver makes through this library, as measurable cases.

Meshes are generated on the GPU from a seed: boxes of hexes split into 6 linear tets (interior nodes
moved by up to 15% of the spacing, nodes in lexicographic or in random order), and a pipe of rings around a
polar axis whose layers thin towards the wall.  Velocities are three sinusoids per component plus 5% noise.
"""
import itertools
import math

import torch

import paper_2111_05651_gb300 as nsi

RHO, DT = 1.0, 1e-2
DEV = "cuda"


def _case(name, op, mesh, nx, ny, nz, numbering, precision, mu=1e-3, sizes=""):
    return {"name": name, "op": op, "mesh": mesh, "nx": nx, "ny": ny, "nz": nz, "numbering": numbering,
            "precision": precision, "mu": mu, "sizes": sizes}


def listed():
    return [
        # the smallest calls: a unit-test sized mesh assembled with the default arguments, where launches and
        # host work are the whole time
        _case("tiny_mixed64", "assemble", "box", 4, 4, 4, "natural", "mixed64"),
        # the plain FP64 verification mesh (8^3 hexes, 3072 tets)
        _case("cube8_fp64", "assemble", "box", 8, 8, 8, "natural", "fp64"),
        # one flow mesh of ordinary size, odd extents, float outputs
        _case("box_mixed32", "assemble", "box", 47, 61, 38, "random", "mixed32", 1e-2),
        # the benchmark mesh: 6 M tets in random node order, double outputs
        _case("cube100_mixed64", "assemble", "box", 100, 100, 100, "random", "mixed64"),
        # the accuracy reference on a mesh of ordinary size
        _case("box_fp64", "assemble", "box", 40, 33, 52, "random", "fp64"),
        # a pipe (the usual elbow benchmark's cross-section): thin wall layers, whose elements the mixed modes
        # take in double, and a polar axis, whose rows are longer than 32 entries
        _case("pipe_mixed64", "assemble", "pipe", 14, 40, 70, "natural", "mixed64"),
        # many independent meshes of uneven size in one captured launch, replayed every time step
        _case("batch_mixed64", "batch", "box", 0, 0, 0, "natural", "mixed64",
              sizes="10,34,17,28,21,12,36,25,31,14,19,23,11,30,16,27"),
        # a time step with cached geometry: the convection and right-hand side of one more velocity
        _case("step_mixed64", "step", "box", 81, 70, 66, "random", "mixed64", 1e-4),
        # the per-node outputs without the matrix
        _case("nodal_mixed64", "nodal", "box", 45, 52, 49, "natural", "mixed64"),
        # the stabilised 3x3 velocity block
        _case("stab_mixed64", "stab", "box", 64, 57, 60, "random", "mixed64"),
        # a Newton or adjoint iteration: the residual and its vector-Jacobian product
        _case("adjoint_mixed64", "adjoint", "box", 50, 50, 50, "natural", "mixed64"),
        _case("adjoint_fp64", "adjoint", "box", 30, 28, 33, "random", "fp64"),
    ]


#: hexes of the largest drawn case of an operation, below the largest listed case's time
_MOST = {("assemble", "fp64"): 80_000, ("assemble", "mixed64"): 950_000, ("assemble", "mixed32"): 950_000,
         ("step", "fp64"): 100_000, ("step", "mixed64"): 900_000, ("step", "mixed32"): 900_000,
         ("nodal", "fp64"): 150_000, ("nodal", "mixed64"): 900_000, ("nodal", "mixed32"): 900_000,
         ("stab", "fp64"): 15_000, ("stab", "mixed64"): 250_000, ("stab", "mixed32"): 300_000,
         ("adjoint", "fp64"): 40_000, ("adjoint", "mixed64"): 300_000, ("adjoint", "mixed32"): 300_000,
         ("batch", "mixed64"): 400_000, ("batch", "mixed32"): 400_000}


def draw(rng):
    op = rng.choice(["assemble", "assemble", "assemble", "pipe", "batch", "step", "nodal", "stab", "adjoint"])
    mu = rng.choice([1e-2, 1e-3, 1e-4])
    if op == "pipe":
        nr, nth = rng.randint(6, 18), rng.randint(17, 56)
        c = _case("", "assemble", "pipe", nr, nth, int(math.exp(rng.uniform(math.log(10), math.log(100)))),
                  rng.choice(["natural", "random"]), rng.choice(["mixed64", "mixed32"]), mu)
    elif op == "batch":
        precision = rng.choice(["mixed64", "mixed64", "mixed32"])
        sizes, left = [], _MOST[op, precision]
        for _ in range(rng.randint(3, 20)):
            n = int(math.exp(rng.uniform(math.log(3), math.log(40))))
            if n ** 3 <= left:
                left -= n ** 3
                sizes.append(n)
        c = _case("", "batch", "box", 0, 0, 0, "natural", precision, mu, ",".join(map(str, sizes)))
    else:
        precision = rng.choice(["mixed64", "mixed64", "mixed32", "fp64"])
        hexes = math.exp(rng.uniform(math.log(40), math.log(_MOST[op, precision])))
        a, b = math.exp(rng.uniform(-0.5, 0.5)), math.exp(rng.uniform(-0.5, 0.5))
        side = hexes ** (1 / 3)
        nx, ny = max(2, round(side * a)), max(2, round(side * b))
        c = _case("", op, "box", nx, ny, max(2, int(hexes / (nx * ny))), rng.choice(["natural", "random"]), precision, mu)
    del c["name"]
    return c


# ------------------------------------------------------------------- meshes --
def _kuhn(ids):
    """Tets [E, 4] of the hexes of a node grid ids [X, Y, Z]: the 6 paths of axis steps from a hex's first
    corner to its last (hexes in order of the last axis, then the middle, then the first)."""
    X, Y, Z = (s - 1 for s in ids.shape)
    tets = []
    for p in itertools.permutations(range(3)):
        at, path = [0, 0, 0], []
        for step in (None,) + p:
            if step is not None:
                at[step] += 1
            path.append(ids[at[0]:at[0] + X, at[1]:at[1] + Y, at[2]:at[2] + Z].permute(2, 1, 0).reshape(-1))
        tets.append(torch.stack(path, 1))
    return torch.stack(tets, 1).reshape(-1, 4)


def _oriented(coord, t):
    d = coord[t[:, 1:]] - coord[t[:, :1]]
    odd = (d[:, 0] * torch.linalg.cross(d[:, 1], d[:, 2])).sum(1) < 0
    t[odd] = t[odd][:, [0, 1, 3, 2]]
    return t


def _box(nx, ny, nz, gen):
    X, Y, Z = nx + 1, ny + 1, nz + 1
    h = 1.0 / max(nx, ny, nz)
    k, j, i = torch.meshgrid(*(torch.arange(s, device=DEV) for s in (Z, Y, X)), indexing="ij")
    coord = torch.stack([i, j, k], -1).reshape(-1, 3).double() * h
    inner = ((i > 0) & (i < nx) & (j > 0) & (j < ny) & (k > 0) & (k < nz)).reshape(-1, 1)
    coord += inner * (torch.rand(coord.shape, dtype=torch.float64, device=DEV, generator=gen) - 0.5) * (0.3 * h)
    ids = torch.arange(X * Y * Z, device=DEV).reshape(Z, Y, X).permute(2, 1, 0)
    return coord, _oriented(coord, _kuhn(ids))


def _pipe(nr, nth, nz, gen):
    """Rings r = 1..nr around an axis, each layer 0.82 times as thick as the one inside it (at most 12 times)."""
    thick = torch.tensor([0.82 ** min(r, 12) for r in range(nr)], dtype=torch.float64, device=DEV)
    radius = 0.5 * torch.cat([thick.new_zeros(1), torch.cumsum(thick, 0)]) / thick.sum()
    ring = 1 + nr * nth
    r, th, z = torch.meshgrid(*(torch.arange(s, device=DEV) for s in (nr + 1, nth + 1, nz + 1)), indexing="ij")
    ids = ring * z + torch.where(r == 0, 0, 1 + (r - 1) * nth + th % nth)
    ang = 2 * math.pi * th / nth
    coord = torch.empty(ring * (nz + 1), 3, dtype=torch.float64, device=DEV)
    coord[ids.reshape(-1)] = torch.stack([radius[r] * torch.cos(ang), radius[r] * torch.sin(ang), 0.1 * z], -1).reshape(-1, 3)
    coord[ring:-ring, 2] += (torch.rand(ring * (nz - 1), dtype=torch.float64, device=DEV, generator=gen) - 0.5) * 0.02
    t = _kuhn(ids)
    s = t.sort(1).values
    t = t[(s[:, 1:] != s[:, :-1]).all(1)]  # the cells at the axis are wedges: 3 of the 6 tets
    return coord, _oriented(coord, t)


def _mesh(c, gen, side=None):
    if c["mesh"] == "pipe":
        coord, t = _pipe(c["nx"], c["ny"], c["nz"], gen)
    else:
        coord, t = _box(*((side,) * 3 if side else (c["nx"], c["ny"], c["nz"])), gen)
    if c["numbering"] == "random":
        new = torch.randperm(coord.shape[0], device=DEV, generator=gen)
        moved = torch.empty_like(coord)
        moved[new] = coord
        coord, t = moved, new[t]
    return coord, t.to(torch.int32).contiguous()


def _velocity(coord, gen):
    u = torch.zeros(3, coord.shape[0], dtype=torch.float64, device=DEV)
    for k in range(3):
        for _ in range(3):
            kappa = torch.randint(1, 4, (3,), device=DEV, generator=gen).double()
            phase = torch.rand(1, dtype=torch.float64, device=DEV, generator=gen)
            u[k] += torch.sin(2 * math.pi * (coord @ kappa + phase))
    return u + 0.05 * torch.randn(u.shape, dtype=torch.float64, device=DEV, generator=gen)


def _counts(c):
    """(nodes, tets, CSR entries) of every mesh of the case."""
    if c["mesh"] == "pipe":
        nr, nth, nz = c["nx"], c["ny"], c["nz"]
        ring, flat = 1 + nr * nth, (3 * nr - 1) * nth  # nodes and edges of one cross-section
        n = ring * (nz + 1)
        return [(n, nz * nth * (6 * nr - 3), n + 2 * (ring * nz + flat * (2 * nz + 1)))]
    boxes = [(int(s),) * 3 for s in c["sizes"].split(",")] if c["sizes"] else [(c["nx"], c["ny"], c["nz"])]
    out = []
    for x, y, z in boxes:
        n = (x + 1) * (y + 1) * (z + 1)
        edges = 7 * x * y * z + 3 * (x * y + y * z + z * x) + x + y + z
        out.append((n, 6 * x * y * z, n + 2 * edges))
    return out


# -------------------------------------------------------------------- cases --
def _inputs(c, seed):
    gen = torch.Generator(DEV).manual_seed(int(seed))
    meshes, us = [], []
    for side in ([int(s) for s in c["sizes"].split(",")] if c["op"] == "batch" else [None]):
        coord, t = _mesh(c, gen, side)
        meshes.append((coord, t))
        us.append(_velocity(coord, gen).to(torch.float64 if c["precision"] == "fp64" else torch.float32))
    w = torch.randn(us[0].shape, dtype=torch.float64, device=DEV, generator=gen).to(us[0].dtype)
    return meshes, us, w


def prepare(case, seed):
    meshes, us, w = _inputs(case, seed)
    asms = [nsi.Assembler(coord, t, precision=case["precision"]) for coord, t in meshes]
    s = {"op": case["op"], "asm": asms[0], "u": us[0], "w": w, "mu": case["mu"]}
    if case["op"] == "step":
        s["A_static"], _ = asms[0].static_part(rho=RHO, mu=case["mu"], dt=DT)
    elif case["op"] == "batch":
        # the program keeps the meshes' outputs and the captured launch, and writes new velocities into `us`
        outs = [a.empty_outputs() for a in asms]
        call = dict(rho=RHO, mu=case["mu"], dt=DT, outs=outs)
        nsi.assemble_batched(asms, us, **call)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            nsi.assemble_batched(asms, us, **call)
        s.update(graph=graph, outs=outs, asms=asms, us=us)
    return s


def run(s):
    asm, u, mu, op = s["asm"], s["u"], s["mu"], s["op"]
    if op == "assemble":
        return asm.assemble(u, rho=RHO, mu=mu, dt=DT)
    if op == "step":
        return asm.assemble_convective(u, s["A_static"], rho=RHO, mu=mu, dt=DT)
    if op == "nodal":
        return asm.nodal(u, rho=RHO, dt=DT)
    if op == "stab":
        return asm.assemble_stabilized(u, rho=RHO, mu=mu, dt=DT)
    if op == "adjoint":
        R = asm.residual(u, rho=RHO, mu=mu, dt=DT)
        return (R,) + tuple(asm.vjp(u, s["w"], rho=RHO, mu=mu, dt=DT))
    s["graph"].replay()
    return s["outs"]


def work(case):
    """Connectivity, coordinates, velocities and the CSR pattern read once, the outputs written once."""
    real = 8 if case["precision"] == "fp64" else 4
    out = 4 if case["precision"] == "mixed32" else 8
    b = f = 0
    for n, E, nnz in _counts(case):
        read = 16 * E + n * (24 + 3 * real)
        pattern = 4 * (n + 1) + 4 * nnz
        if case["op"] in ("assemble", "batch"):
            b, f = b + read + pattern + out * (4 * nnz + 3 * n), f + 220 * E
        elif case["op"] == "step":
            b, f = b + read + pattern + out * (2 * nnz + 3 * n), f + 120 * E
        elif case["op"] == "nodal":
            b, f = b + read + out * 5 * n, f + 25 * E
        elif case["op"] == "stab":
            b, f = b + read + pattern + out * (12 * nnz + 3 * n), f + 600 * E
        else:
            b, f = b + 2 * read + real * 9 * n, f + 450 * E
    return {"bytes": b, "flops": f}


def tolerance(case):
    # About four times the distance from exact() over these ranges: FP64 2.4e-16 (6e-16 for the adjoint), the
    # mixed modes 9e-8 (float element terms and sums), their adjoint 5e-6 (the viscosity gradient is one sum of
    # terms of both signs over all elements, whose cancellation varies with the mesh).
    if case["precision"] == "fp64":
        return {"rel": 1e-14 if case["op"] == "adjoint" else 1e-15, "max": 1e-13}
    return {"rel": 5e-5} if case["op"] == "adjoint" else {"rel": 4e-7, "max": 2e-5}


# ------------------------------------------------------------------- exact --
def _geometry(coord, t):
    x = coord[t]
    d1, d2, d3 = x[:, 1] - x[:, 0], x[:, 2] - x[:, 0], x[:, 3] - x[:, 0]
    c = [None, torch.linalg.cross(d2, d3), torch.linalg.cross(d3, d1), torch.linalg.cross(d1, d2)]
    c[0] = -(c[1] + c[2] + c[3])
    det = (d1 * c[1]).sum(1)
    return [v / det[:, None] for v in c], det / 6  # shape gradients, volumes


def _pattern(t, n):
    """(keys, position) of the CSR pattern: sorted distinct row * n + column, and where a pair sits."""
    keys = torch.cat([t[:, a] * n + t[:, b] for a in range(4) for b in range(4)]).unique()
    return keys, lambda a, b: torch.searchsorted(keys, t[:, a] * n + t[:, b])


def _exact_matrix(coord, t, u, mu, stab):
    n = coord.shape[0]
    g, vol = _geometry(coord, t)
    keys, at = _pattern(t, n)
    nnz = keys.numel()
    ue = [u[:, t[:, a]].T for a in range(4)]
    S = ue[0] + ue[1] + ue[2] + ue[3]
    A = torch.zeros(9 if stab else 1, nnz, dtype=torch.float64, device=DEV)
    G = torch.zeros(3, nnz, dtype=torch.float64, device=DEV)
    rhs = torch.zeros(3, n, dtype=torch.float64, device=DEV)
    if stab:
        h = (6 * vol) ** (1 / 3)
        tau1 = 1 / (4 * mu / h ** 2 + 2 * RHO * (S / 4).norm(dim=1) / h)
        tau2 = h ** 2 / (4 * tau1)
    for a in range(4):
        m = RHO * vol / (4 * DT)
        rhs.index_add_(1, t[:, a], m * ue[a].T)
        for b in range(4):
            p = at(a, b)
            v = RHO * vol / 20 * ((S + ue[a]) * g[b]).sum(1) + mu * vol * (g[a] * g[b]).sum(1) + (m if a == b else 0)
            if stab:
                sg = (S * g[a]).sum(1) * (S * g[b]).sum(1)
                for w in ue:
                    sg = sg + (w * g[a]).sum(1) * (w * g[b]).sum(1)
                v = v + tau1 * RHO ** 2 * vol / 20 * sg
                for i in range(3):
                    for j in range(3):
                        k = mu * vol * g[a][:, j] * g[b][:, i] + tau2 * vol * g[a][:, i] * g[b][:, j]
                        A[3 * i + j].index_add_(0, p, k + v if i == j else k)
            else:
                A[0].index_add_(0, p, v)
            for d in range(3):
                G[d].index_add_(0, p, -vol / 4 * g[a][:, d])
    return (A if stab else A[0]), G, rhs


def _exact_adjoint(coord, t, u, w, mu):
    g, vol = _geometry(coord, t)
    u = u.clone().requires_grad_(True)
    m = torch.tensor(mu, dtype=torch.float64, device=DEV, requires_grad=True)
    ue = [u[:, t[:, a]].T for a in range(4)]
    S = ue[0] + ue[1] + ue[2] + ue[3]
    grad = sum(ue[b][:, :, None] * g[b][:, None, :] for b in range(4))  # du_k / dx_l
    R = torch.zeros_like(u)
    for a in range(4):
        conv = (grad * (S + ue[a])[:, None, :]).sum(2) * (RHO * vol / 20)[:, None]
        visc = (grad * g[a][:, None, :]).sum(2) * (m * vol)[:, None]
        mass = (RHO * vol / (4 * DT))[:, None] * (ue[a] - ue[a].detach())
        R = R.index_add(1, t[:, a], (conv + visc + mass).T)
    gu, gm = torch.autograd.grad((R * w).sum(), (u, m))
    return R.detach(), gu, gm.reshape(1)


def exact(case, seed):
    meshes, us, w = _inputs(case, seed)
    out = []
    for (coord, t), u in zip(meshes, us):
        t, u = t.long(), u.double()
        if case["op"] == "adjoint":
            return _exact_adjoint(coord, t, u, w.double(), case["mu"])
        if case["op"] == "nodal":
            vol = _geometry(coord, t)[1]
            mass = torch.zeros(coord.shape[0], dtype=torch.float64, device=DEV)
            for a in range(4):
                mass.index_add_(0, t[:, a], RHO * vol / 4)
            return mass / DT * u, mass / DT, mass
        A, G, rhs = _exact_matrix(coord, t, u, case["mu"], case["op"] == "stab")
        if case["op"] == "step":
            return A, rhs
        out.append((A, G, rhs))
    return out if case["op"] == "batch" else out[0]
