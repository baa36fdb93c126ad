"""grad_mu of weights that nearly cancel in it, in FP64 and to the bit: on a
mesh of one block of elements no atomic order enters, and a change of any
element term's rounding shows multiplied by the sum's condition (8e5 to 2e8),
so equality is the bound.  ALPHA and GRAD_MU were recorded with the sums over
every element entry (kernel comment at vjp_element)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import meshgen

nsi = pytest.importorskip("paper_2111_05651_gb300")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")]

# seed: (alpha of w = w0 - alpha w1, grad_mu)
RECORDED = {
    0: (-3.614126205444336, "0x1.887a090000000p-24"),
    1: (-5.9641008377075195, "-0x1.c23d44c800000p-21"),
    2: (-0.9533786773681641, "0x1.5a3fc71200000p-18"),
    3: (-1.9860973358154297, "-0x1.91267e0000000p-24"),
    4: (0.8253288269042969, "-0x1.c5bed6ae00000p-19"),
    5: (-0.24225234985351562, "0x1.610aca3e80000p-18"),
}


def inputs(seed):
    """3^3-hex cube (162 tets), coordinates, velocity and two weight fields with few bits."""
    rng = np.random.default_rng(seed)
    mesh = meshgen.kuhn_cube(3)
    coord = np.round(mesh.coord * 2**20) / 2**20
    inner = ((mesh.coord > 0) & (mesh.coord < 1)).all(axis=1)
    coord[inner] += rng.integers(-2**15, 2**15, (int(inner.sum()), 3)) / 2**20
    n = coord.shape[0]
    return coord, mesh.lnods, *(rng.integers(-2**19, 2**19, (3, n)) / 2**18 for _ in range(3))


@pytest.mark.parametrize("seed", sorted(RECORDED))
def test_grad_mu_of_cancelling_weights(seed):
    alpha, ref = RECORDED[seed]
    coord, lnods, u, w0, w1 = inputs(seed)
    asm = nsi.Assembler(coord, lnods, precision="fp64")
    w = torch.as_tensor(w0 - alpha * w1).cuda()  # (exact: 20-bit fields, alpha of 20 fraction bits)
    _, gmu = asm.vjp(torch.as_tensor(u).cuda(), w, rho=1.0, mu=1e-3, dt=1e-2)
    assert gmu.item() == float.fromhex(ref)


def test_grad_mu_of_one_cluster_repeats():
    """750 tets, three blocks, whose sums are added in one order: repeats are equal to the bit."""
    mesh, u = meshgen.config_mesh(N=5, jitter=0.15, numbering="random", seed=51)
    w = torch.as_tensor(np.random.default_rng(52).standard_normal(u.shape).T.copy()).cuda()
    asm = nsi.Assembler(mesh.coord, mesh.lnods, precision="fp64")
    ut = torch.as_tensor(u.T.copy()).cuda()
    assert len({asm.vjp(ut, w)[1].item() for _ in range(20)}) == 1


@pytest.mark.parametrize("precision", ["fp64", "mixed64"])
def test_vjp_in_a_captured_graph(precision):
    mesh, u = meshgen.config_mesh(N=9, jitter=0.15, numbering="random", seed=53)
    asm = nsi.Assembler(mesh.coord, mesh.lnods, precision=precision)
    ut = torch.as_tensor(u.T.copy()).cuda().to(asm.vel_dtype)
    w = torch.as_tensor(np.random.default_rng(54).standard_normal(u.shape).T.copy()).cuda().to(asm.vel_dtype)
    gu, gmu = asm.vjp(ut, w)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        gu2, gmu2 = asm.vjp(ut, w)
    graph.replay()
    torch.cuda.synchronize()
    # (grad_u's and grad_mu's atomic additions have no fixed order)
    tol = 1e-13 if precision == "fp64" else 1e-5
    assert (gu2 - gu).abs().max() <= tol * gu.abs().max()
    assert abs(gmu2.item() - gmu.item()) <= tol * max(abs(gmu.item()), 1.0)


def test_residual_on_coarse_meshes():
    """rms error of R in mixed64 over eight 9^3 cubes, whose neighbours' velocities
    lie far apart: 1.30e-7 with the velocity gradient summed over the element's four
    nodes, 1.31e-7 with every entry, 1.37e-7 by differences to the first node (each
    within 0.04e-7, the atomics' order); the bound lies between."""
    import oracle

    total = 0.0
    for seed in range(8):
        mesh, u = meshgen.config_mesh(N=9, jitter=0.15, numbering="random", seed=600 + seed)
        uo = u.astype(np.float32).astype(np.float64)
        rp, ci, A, _, rhs = oracle.assemble(mesh.coord, mesh.lnods, uo, None, 1.0, 1e-3, 1e-2)
        ref = oracle.residual((rp, ci, A), rhs, uo).T
        asm = nsi.Assembler(mesh.coord, mesh.lnods, precision="mixed64")
        got = asm.residual(torch.as_tensor(u.T.copy()), rho=1.0, mu=1e-3, dt=1e-2).double().cpu().numpy()
        total += (np.linalg.norm(got - ref) / np.linalg.norm(ref)) ** 2
    assert (total / 8) ** 0.5 <= 1.34e-7
