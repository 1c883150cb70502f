"""A mesh with many long rows: the records of a block of rows do not fit the staged product's shared memory, so the
row-per-warp product runs, and the mixed residual takes tiles of 16 rows.  Products against FP64 products of the
same FP32 values (2e-6: the parity tests' bar), the BF16 form bit for bit against the widened vector; the residual
that an unfinished mixed solve reports against the one of its x (entries rounded to FP32: 4 * 2^-24)."""
import numpy as np
import pytest
import scipy.sparse as sp

from phantom import EPS_MATCHING

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _suspension(a, b):
    """Every edge of a path of a edges on the axis with every edge of a ring of b around it: a b tets.  The ring's
    edges come last, b rows of 3 a + 3 terms side by side."""
    z = np.stack([np.zeros(a + 1), np.zeros(a + 1), np.linspace(-0.02, 0.02, a + 1)], 1)
    t = 2 * np.pi * np.arange(b) / b
    ring = np.stack([0.02 * np.cos(t), 0.02 * np.sin(t), np.zeros(b)], 1)
    i, j = (q.ravel() for q in np.meshgrid(np.arange(a), np.arange(b), indexing="ij"))
    return (np.concatenate([z, ring]),
            np.stack([i, i + 1, a + 1 + j, a + 1 + (j + 1) % b], 1).astype(np.int32))


@pytest.mark.parametrize("n_cols", [1, 3, 16, 31, 64, 100, 128])
def test_products_and_residual(n_cols):
    from paper_2311_05322_gb300 import mw
    xyz, tets = _suspension(158, 45)
    c = mw.Context(0)
    E = c.set_mesh(xyz, tets).n_edge
    rng = np.random.default_rng(n_cols)
    eps = EPS_MATCHING + rng.uniform(-6, 6, len(tets)) + 1j * rng.uniform(-4, 4, len(tets))
    c.assemble([1e9], np.stack([eps.real, eps.imag], 1), EPS_MATCHING)
    _, _, _, rp, ci = c.get_topology()
    win = lambda k: max(rp[min(r + k, E)] - rp[r] for r in range(0, E, k))
    assert 16 * win(16) > 48 * 1024 and win(32) > 10000      # neither staged form
    A = sp.csr_matrix((c.get_matrix(0), ci, rp), (E, E))
    xb = torch.randn((E, n_cols, 2), generator=torch.Generator().manual_seed(n_cols)).to(torch.bfloat16)
    x = torch.view_as_complex(xb.float().contiguous())
    ref = A @ x.numpy().astype(np.complex128)
    y = torch.empty((E, n_cols), dtype=torch.complex64, device="cuda")
    yb = torch.empty_like(y)
    c.apply_matrix(0, mw.MW_PREC_FP32, x.cuda(), y, n_cols)
    c.apply_matrix(0, 5, xb.cuda(), yb, n_cols)
    assert np.linalg.norm(y.cpu().numpy() - ref) <= 2e-6 * np.linalg.norm(ref)
    assert torch.equal(torch.view_as_real(y), torch.view_as_real(yb))
    B = rng.normal(size=(n_cols, E)) + 1j * rng.normal(size=(n_cols, E))
    b = torch.from_numpy(B).cuda()
    s = torch.empty_like(b)
    st = c.solve_rhs(n_cols, b, s, mw.solve_opts(mode=mw.MW_MODE_MIXED, restart=4, tol=1e-12, inner_tol=1e-1, max_it=4,
                                                 max_outer=1, use_precond=0), allow_noconv=True)
    c.close()
    true = np.linalg.norm(B.T - A @ s.cpu().numpy().T, axis=0) / np.linalg.norm(B, axis=1)
    assert np.all(true > 1e-3)
    assert np.all(np.abs(st["relres"].ravel() - true) <= 4 * 2.0 ** -24 * true)
