"""Short and narrow Krylov blocks: the dots and reductions at the edges of their row chunks.

Blocks below 16 columns run the plain Gram-Schmidt kernels: a block of 16 warps splits into
16 // nvec row slots per vector, one pass takes 16 rows per thread, and the grid holds only blocks
with rows.  The dots are checked against FP64 dots of the same FP32 vectors within the first-order
bound of their FP32 sums (16 rows per chunk, then FP64: (16 + 4) * 2^-24 * sum |v||w|).
"""
import numpy as np
import pytest

from oracle import assemble as asm
from oracle import solve
from phantom import EPS_MATCHING, kuhn_mesh

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n_cols", [1, 3, 8, 15])
@pytest.mark.parametrize("n_rows,nvec", [(1, 1), (63, 2), (64, 5), (65, 15), (1025, 16), (4097, 17), (13428, 1), (13428, 64)])
def test_narrow_dots_against_fp64(n_rows, nvec, n_cols):
    from paper_2311_05322_gb300 import mw
    rng = np.random.default_rng(n_rows + 100 * nvec + n_cols)
    n = n_rows * n_cols
    vstride = (n + 31) // 32 * 32

    def draw(k):
        return (rng.standard_normal(k, np.float32) + 1j * rng.standard_normal(k, np.float32)).astype(np.complex64)

    V, w = draw(nvec * vstride), draw(n)
    c = mw.Context(0)
    h = c.krylov_dots(torch.from_numpy(V).cuda(), torch.from_numpy(w).cuda(), nvec, vstride, n_rows, n_cols)
    c.close()
    w64 = w.astype(np.complex128).reshape(n_rows, n_cols)
    for i in range(nvec):
        v = V[i * vstride:i * vstride + n].astype(np.complex128).reshape(n_rows, n_cols)
        scale = np.sum(np.abs(v) * np.abs(w64), axis=0)
        assert np.all(np.abs(h[i] - np.sum(np.conj(v) * w64, axis=0)) <= 20 * 2.0 ** -24 * scale), i


@pytest.mark.parametrize("n_cols,restart,mode", [(1, 63, 0), (5, 63, 1), (17, 33, 0), (128, 31, 1)])
def test_long_cycles_reach_the_direct_solution(n_cols, restart, mode):
    """Unpreconditioned cycles run all their steps: the back substitution at triangles up to 63."""
    from paper_2311_05322_gb300 import mw
    m = kuhn_mesh(4, 3, 2, lo=(-0.02, -0.015, -0.01), hi=(0.02, 0.015, 0.01))
    eps = np.full(m.n_tet, EPS_MATCHING, dtype=complex)
    c = mw.Context(0)
    E = c.set_mesh(m.xyz, m.tets).n_edge
    c.assemble([1e9], np.stack([eps.real, eps.imag], 1), EPS_MATCHING)
    rng = np.random.default_rng(restart + n_cols)
    B = rng.normal(size=(n_cols, E)) + 1j * rng.normal(size=(n_cols, E))
    b = torch.from_numpy(B).cuda()
    x = torch.empty_like(b)
    st = c.solve_rhs(n_cols, b, x, mw.solve_opts(mode=mode, restart=restart, tol=1e-10, inner_tol=1e-2, max_it=20000,
                                                 max_outer=400, use_precond=0))
    c.close()
    assert st["n_converged"] == n_cols and st["max_relres"] <= 1e-10
    sysm = asm.build_system(m.xyz, m.tets)
    ref = solve.solve_direct(sysm, asm.assemble(sysm, eps, 1e9, EPS_MATCHING), B.T)
    assert np.linalg.norm(x.cpu().numpy().T - ref) <= 1e-6 * np.linalg.norm(ref)
