"""The sums of the dots' partials on both sides of the line between a warp per entry and eight entries per block
(512 entries), and of column norms at widths that split a warp into 1 to 32 rows.  FP64 reference; bars: dots as
sums of at most 16-row FP32 passes (20 * 2^-24 of the absolute sum, as for the narrow blocks; FP32 tile sums of
512 rows for 16 and more columns); norms of FP64 right-hand sides through the relative residual of a zero solution
(FP64 sums of n terms: n 2^-53, far below 1e-12)."""
import numpy as np
import pytest

from phantom import EPS_MATCHING, kuhn_mesh

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("nvec,n_cols", [(1, 1), (34, 15), (35, 15), (32, 16), (33, 16), (4, 128), (5, 128)])
def test_dots_around_the_entry_count(nvec, n_cols):
    from paper_2311_05322_gb300 import mw
    n_rows = 2111
    rng = np.random.default_rng(nvec * 1000 + n_cols)
    n = n_rows * n_cols
    vstride = (n + 31) // 32 * 32

    def draw(k):
        return (rng.standard_normal(k, np.float32) + 1j * rng.standard_normal(k, np.float32)).astype(np.complex64)

    V, w = draw(nvec * vstride), draw(n)
    c = mw.Context(0)
    h = c.krylov_dots(torch.from_numpy(V).cuda(), torch.from_numpy(w).cuda(), nvec, vstride, n_rows, n_cols)
    c.close()
    w64 = w.astype(np.complex128).reshape(n_rows, n_cols)
    bar = (20 if n_cols < 16 else 512) * 2.0 ** -24
    for i in range(nvec):
        v = V[i * vstride:i * vstride + n].astype(np.complex128).reshape(n_rows, n_cols)
        assert np.all(np.abs(h[i] - np.sum(np.conj(v) * w64, axis=0)) <= bar * np.sum(np.abs(v) * np.abs(w64), axis=0)), i


@pytest.mark.parametrize("n_cols", [1, 2, 3, 5, 9, 17, 32, 33, 65, 128])
@pytest.mark.parametrize("mode", [0, 1])
def test_column_norms_scale_with_the_column(n_cols, mode):
    """Columns that are powers of two times one vector: equal relative residuals after the same solve."""
    from paper_2311_05322_gb300 import mw
    m = kuhn_mesh(3, 3, 2, lo=(-0.02, -0.015, -0.01), hi=(0.02, 0.015, 0.01))
    eps = np.full(m.n_tet, EPS_MATCHING, dtype=complex)
    c = mw.Context(0)
    E = c.set_mesh(m.xyz, m.tets).n_edge
    c.assemble([1e9], np.stack([eps.real, eps.imag], 1), EPS_MATCHING)
    rng = np.random.default_rng(7)
    b0 = rng.normal(size=E) + 1j * rng.normal(size=E)
    s = 2.0 ** np.arange(n_cols).clip(max=20)
    b = torch.from_numpy(b0[None, :] * s[:, None]).cuda()
    x = torch.empty_like(b)
    st = c.solve_rhs(n_cols, b, x, mw.solve_opts(mode=mode, restart=20, tol=1e-9, inner_tol=1e-2, max_it=20000,
                                                 max_outer=400, use_precond=0))
    c.close()
    assert st["n_converged"] == n_cols
    xs = x.cpu().numpy() / s[:, None]
    assert np.linalg.norm(xs - xs[0]) <= 1e-12 * np.linalg.norm(xs)
    assert np.all(np.abs(st["relres"] - st["relres"].ravel()[0]) <= 1e-12)


@pytest.mark.parametrize("n_cols", [1, 2, 3, 5, 9, 17, 32, 33, 65, 128])
@pytest.mark.parametrize("mode", [0, 1])
def test_reported_residuals_of_unfinished_solves(n_cols, mode):
    """||b - A x|| / ||b|| of columns with different supports after a few steps, against norms formed from the
    returned x on the CPU.  A lost row or warp moves them by its share, far above the bars: FP64 sums 1e-10;
    mixed mode rounds each residual entry to FP32 and sums its square from there, 4 * 2^-24."""
    from paper_2311_05322_gb300 import mw
    m = kuhn_mesh(7, 6, 5, lo=(-0.03, -0.025, -0.02), hi=(0.03, 0.025, 0.02))
    c = mw.Context(0)
    E = c.set_mesh(m.xyz, m.tets).n_edge
    c.assemble([1e9], np.tile([EPS_MATCHING.real, EPS_MATCHING.imag], (m.n_tet, 1)), EPS_MATCHING)
    _, _, _, rp, ci = c.get_topology()
    A = torch.sparse_csr_tensor(torch.from_numpy(rp), torch.from_numpy(ci.astype(np.int64)),
                                torch.from_numpy(c.get_matrix(0)), (E, E)).to_dense().numpy()
    rng = np.random.default_rng(100 * n_cols + mode)
    B = rng.normal(size=(n_cols, E)) + 1j * rng.normal(size=(n_cols, E))
    for q in range(n_cols):                 # every (1 + q % 5)-th row from a place of its own
        keep = np.zeros(E, bool)
        keep[37 * q % (E // 2)::1 + q % 5] = True
        B[q, ~keep] = 0.0
    b = torch.from_numpy(B).cuda()
    x = torch.empty_like(b)
    st = c.solve_rhs(n_cols, b, x, mw.solve_opts(mode=mode, restart=4, tol=1e-12, inner_tol=1e-1, max_it=4, max_outer=1,
                                                 use_precond=0), allow_noconv=True)
    c.close()
    true = np.linalg.norm(B.T - A @ x.cpu().numpy().T, axis=0) / np.linalg.norm(B, axis=1)
    assert np.all(true > 1e-3) and len(np.unique(np.round(true, 9))) == n_cols
    assert np.all(np.abs(st["relres"].ravel() - true) <= (4 * 2.0 ** -24 if mode else 1e-10) * true)
