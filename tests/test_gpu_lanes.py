"""The row gather at the edges of its lane rule: meshes around the row count
where four lanes per row become two (and, in FP64, two one), and one whose groups are more than the
resident warps (every warp takes several), against the oracle; a batch that
mixes both kinds against the single calls, bit for bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import meshgen
import oracle
from tests._common import errors, vec_scaled_err

nsi = pytest.importorskip("paper_2111_05651_gb300")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")]
TOL = {"fp64": 1e-12, "mixed64": 1e-5, "mixed32": 1e-5}  # the library's stated bars


@pytest.mark.parametrize("precision,N", [(p, N) for p in ("fp64", "mixed64", "mixed32") for N in (20, 21, 36)] +
                         [("fp64", 49), ("fp64", 59)])  # 9,261, 10,648, 50,653, 125,000 and (one lane in FP64) 216,000 rows
def test_lanes_match_oracle(precision, N):
    mesh, u = meshgen.config_mesh(N=N, jitter=0.15, numbering="random", seed=300 + N)
    asm = nsi.Assembler(mesh.coord, mesh.lnods, precision=precision)
    ut = torch.as_tensor(u.T.copy())
    uo = u if precision == "fp64" else u.astype(np.float32).astype(np.float64)
    rp, _, oA, oG, orhs = oracle.assemble(mesh.coord, mesh.lnods, uo, None, 1.0, 1e-3, 1e-2)
    A, G, rhs = asm.assemble(ut, rho=1.0, mu=1e-3, dt=1e-2)
    got = [t.double().cpu().numpy() for t in (A, G, rhs)]
    assert max(errors(rp, *got, oA, oG, orhs).values()) <= TOL[precision]
    A_static, _ = asm.static_part(rho=1.0, mu=1e-3, dt=1e-2)
    A2, rhs2 = asm.assemble_convective(ut, A_static, rho=1.0, mu=1e-3, dt=1e-2)
    got = [A2.double().cpu().numpy(), oG, rhs2.double().cpu().numpy()]
    assert max(errors(rp, *got, oA, oG, orhs).values()) <= TOL[precision]
    alias = A_static.clone()
    asm.assemble_convective(ut, alias, rho=1.0, mu=1e-3, dt=1e-2, out=(alias, rhs2))
    assert torch.equal(alias, A2)
    onr, ondt, onm = oracle.nodal(mesh.coord, mesh.lnods, uo, 1.0, 1e-2)
    r3, dtr, mr = (t.double().cpu().numpy() for t in asm.nodal(ut, rho=1.0, dt=1e-2))
    assert max([vec_scaled_err(dtr, ondt), vec_scaled_err(mr, onm)] +
               [vec_scaled_err(r3[k], onr[k]) for k in range(3)]) <= TOL[precision]


@pytest.mark.parametrize("precision", ["fp64", "mixed64", "mixed32"])
def test_batch_of_both_kinds_equals_single(precision):
    asms, us = [], []
    for N in (3, 36, 20, 59, 22):
        mesh, u = meshgen.config_mesh(N=N, jitter=0.15, numbering="natural", seed=310 + N)
        asms.append(nsi.Assembler(mesh.coord, mesh.lnods, precision=precision))
        us.append(torch.as_tensor(u.T.copy()))
    single = [[t.clone() for t in a.assemble(v)] for a, v in zip(asms, us)]
    for s, b in zip(single, nsi.assemble_batched(asms, us)):
        for x, y in zip(s, b):
            assert torch.equal(x, y)


@pytest.mark.parametrize("precision", ["mixed64", "mixed32"])
@pytest.mark.parametrize("N", [1, 7, 22])  # four lanes per row (8 and 512 rows), two (12,167)
def test_flat_cube_rows_in_double(precision, N):
    """A cube 40 times flatter than wide: every element is badly shaped, every
    row is recomputed in double, so mixed64 is as exact as its inputs (the
    coordinates are kept as float pairs, 2^-48 of the domain against flat edges
    of 1/(40 N)) and mixed32 as its float outputs."""
    mesh, u = meshgen.config_mesh(N=N, jitter=0.1, numbering="random", seed=320 + N)
    coord = mesh.coord * np.array([1.0, 1.0, 1.0 / 40])
    asm = nsi.Assembler(coord, mesh.lnods, precision=precision)
    assert asm.info().exact_rows == mesh.n_nodes
    tol = 1e-10 if precision == "mixed64" else 3e-7
    ut = torch.as_tensor(u.T.copy())
    uo = u.astype(np.float32).astype(np.float64)
    rp, _, oA, oG, orhs = oracle.assemble(coord, mesh.lnods, uo, None, 1.0, 1e-3, 1e-2)
    got = [t.double().cpu().numpy() for t in asm.assemble(ut, rho=1.0, mu=1e-3, dt=1e-2)]
    assert max(errors(rp, *got, oA, oG, orhs).values()) <= tol
    A_static, _ = asm.static_part(rho=1.0, mu=1e-3, dt=1e-2)
    A2, rhs2 = asm.assemble_convective(ut, A_static, rho=1.0, mu=1e-3, dt=1e-2)
    got = [A2.double().cpu().numpy(), oG, rhs2.double().cpu().numpy()]
    assert max(errors(rp, *got, oA, oG, orhs).values()) <= 1e-5
    onr, ondt, onm = oracle.nodal(coord, mesh.lnods, uo, 1.0, 1e-2)
    r3, dtr, mr = (t.double().cpu().numpy() for t in asm.nodal(ut, rho=1.0, dt=1e-2))
    assert max([vec_scaled_err(dtr, ondt), vec_scaled_err(mr, onm)] +
               [vec_scaled_err(r3[k], onr[k]) for k in range(3)]) <= tol


@pytest.mark.parametrize("precision", ["fp64", "mixed64", "mixed32"])
def test_row_of_more_entries_than_a_block_has_threads(precision):
    mesh, u = meshgen.delaunay_hub(8, 300, seed=330)
    asm = nsi.Assembler(mesh.coord, mesh.lnods, precision=precision)
    assert asm.max_row > 256 and asm.info().long_rows > 0
    ut = torch.as_tensor(u.T.copy())
    uo = u if precision == "fp64" else u.astype(np.float32).astype(np.float64)
    rp, _, oA, oG, orhs = oracle.assemble(mesh.coord, mesh.lnods, uo, None, 1.0, 1e-3, 1e-2)
    got = [t.double().cpu().numpy() for t in asm.assemble(ut, rho=1.0, mu=1e-3, dt=1e-2)]
    assert max(errors(rp, *got, oA, oG, orhs).values()) <= TOL[precision]
    A_static, _ = asm.static_part(rho=1.0, mu=1e-3, dt=1e-2)
    A2, rhs2 = asm.assemble_convective(ut, A_static, rho=1.0, mu=1e-3, dt=1e-2)
    got = [A2.double().cpu().numpy(), oG, rhs2.double().cpu().numpy()]
    assert max(errors(rp, *got, oA, oG, orhs).values()) <= TOL[precision]


@pytest.mark.parametrize("precision,N,shapes", [("mixed64", 6, 1), ("mixed64", 22, 2), ("fp64", 6, 1), ("fp64", 59, 4)])
def test_launch_shapes_are_distinct(precision, N, shapes):
    """Four lanes per row fill a block of four warps by every name, two have two
    launches, one lane four; a name that repeats a launch is still accepted."""
    mesh, u = meshgen.config_mesh(N=N, jitter=0.15, numbering="natural", seed=340 + N)
    asm = nsi.Assembler(mesh.coord, mesh.lnods, precision=precision)
    assert asm.info().n_plans == shapes
    ut = torch.as_tensor(u.T.copy())
    ref = [t.clone() for t in asm.assemble(ut)]
    for rows in (128, 32, 96, 64):
        nsi.nsi_set_launch(asm.handle, nsi.NSI_SCATTER_GATHER, rows)
        assert asm.info().rows_per_block == rows
        for x, y in zip(ref, asm.assemble(ut)):
            assert torch.equal(x, y)
    for rows in (16, 48, 160):
        with pytest.raises(RuntimeError):
            nsi.nsi_set_launch(asm.handle, nsi.NSI_SCATTER_GATHER, rows)


def _errors_natural(precision, numbering, mu):
    """rms errors of G(i,i), C(u)(i,i) and A's off-diagonal entries, 30^3 cube (two lanes per row)."""
    mesh, u = meshgen.config_mesh(N=30, jitter=0.15, numbering=numbering, seed=71)
    uo = u.astype(np.float32).astype(np.float64)
    rp, ci, oA, oG, _ = oracle.assemble(mesh.coord, mesh.lnods, uo, None, 1.0, mu, 1e-2)
    oC = oA - oracle.assemble(mesh.coord, mesh.lnods, np.zeros_like(uo), None, 1.0, mu, 1e-2)[2]
    asm = nsi.Assembler(mesh.coord, mesh.lnods, precision=precision)
    ut = torch.as_tensor(u.T.copy())
    A, G, _ = (t.double().cpu().numpy() for t in asm.assemble(ut, rho=1.0, mu=mu, dt=1e-2))
    zero = torch.zeros(asm.nnz, dtype=asm.out_dtype, device="cuda")
    C = asm.assemble_convective(ut, zero, rho=1.0, mu=mu, dt=1e-2)[0].double().cpu().numpy()
    d = np.repeat(np.arange(mesh.n_nodes), np.diff(rp)) == ci
    return [np.linalg.norm(x - y) / np.linalg.norm(y) for x, y in ((G[:, d], oG[:, d]), (C[d], oC[d]), (A[~d], oA[~d]))]


def test_row_sums_of_opposite_slots():
    """The order of a row's sums is fixed, so are these errors: with a lane's slots
    taken in pairs from both ends of the row G(i,i) 2.26e-7 and mixed32's C(i,i)
    2.56e-7, with every second slot 2.75e-7 and 3.84e-7, with one lane's in order
    2.45e-7 and 3.09e-7; the bounds are the last's."""
    g, c, _ = _errors_natural("mixed32", "natural", 1e-3)
    assert g <= 2.45e-7 and c <= 3.09e-7


def test_velocities_are_not_rounded_before_the_sum():
    """A's off-diagonal entries where convection leads: 8.44e-8, with every
    staged velocity multiplied by rho/120 first 8.57e-8; the bound is what the
    product in the element's step gave with one lane per row."""
    assert _errors_natural("mixed64", "random", 1e-4)[2] <= 8.51e-8
