"""The staged FP32 products and residual at their edges: column counts around the packs and lane counts,
rows at the end of a block and very long rows, against FP64 products of the same FP32 values
(2e-6: the parity tests' bar) and, for the BF16 form, bit for bit against the widened vector."""
import numpy as np
import pytest

from phantom import EPS_MATCHING, kuhn_mesh

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _fan(n):
    """n tets around one edge: two rows of about 3 n nonzeros."""
    t = 2 * np.pi * np.arange(n) / n
    ring = np.stack([0.01 * np.cos(t), 0.01 * np.sin(t), 0.002 * np.sin(3 * t)], 1)
    xyz = np.concatenate([[[0, 0, -0.01], [0, 0, 0.01]], ring])
    i = np.arange(n)
    return xyz, np.stack([np.zeros(n, int), np.ones(n, int), 2 + i, 2 + (i + 1) % n], 1).astype(np.int32)


@pytest.mark.parametrize("mesh", ["box", "fan", "long"])
@pytest.mark.parametrize("n_cols", [1, 2, 6, 15, 16, 18, 32, 33, 34, 36, 63, 64, 66, 100, 127, 128])
def test_products_and_solve(mesh, n_cols):
    from paper_2311_05322_gb300 import mw
    if mesh == "box":
        m = kuhn_mesh(5, 4, 3, lo=(-0.02, -0.015, -0.01), hi=(0.02, 0.015, 0.01))
        xyz, tets = m.xyz, m.tets
    else:
        xyz, tets = _fan(40 if mesh == "fan" else 150)      # 150: one row of 451 terms (480 columns at most)
    c = mw.Context(0)
    E = c.set_mesh(xyz, tets).n_edge
    rng = np.random.default_rng(n_cols)
    eps = EPS_MATCHING + rng.uniform(-6, 6, len(tets)) + 1j * rng.uniform(-4, 4, len(tets))
    c.assemble([1e9], np.stack([eps.real, eps.imag], 1), EPS_MATCHING)
    _, _, _, rp, ci = c.get_topology()
    A = torch.sparse_csr_tensor(torch.from_numpy(rp), torch.from_numpy(ci.astype(np.int64)),
                                torch.from_numpy(c.get_matrix(0)), (E, E))
    xb = torch.randn((E, n_cols, 2), generator=torch.Generator().manual_seed(n_cols)).to(torch.bfloat16)
    x = torch.view_as_complex(xb.float().contiguous())
    ref = torch.matmul(A.to_dense(), x.to(torch.complex128))
    y = torch.empty((E, n_cols), dtype=torch.complex64, device="cuda")
    yb = torch.empty_like(y)
    c.apply_matrix(0, mw.MW_PREC_FP32, x.cuda(), y, n_cols)
    c.apply_matrix(0, 5, xb.cuda(), yb, n_cols)
    assert torch.linalg.norm(y.cpu() - ref) <= 2e-6 * torch.linalg.norm(ref)
    assert torch.equal(torch.view_as_real(y), torch.view_as_real(yb))
    if n_cols in (1, 15, 33, 64, 128):
        # the mixed solver's residual reports the true one: 1e-10 on unpreconditioned solves of x's products
        b = (ref / torch.linalg.norm(ref, dim=0)).T.contiguous().cuda()
        z = torch.empty_like(b)
        st = c.solve_rhs(n_cols, b, z, mw.solve_opts(mode=mw.MW_MODE_MIXED, tol=1e-10, restart=50, max_it=20000,
                                                     max_outer=400, use_precond=0))
        r = torch.linalg.norm(b.cpu().T - torch.matmul(A.to_dense(), z.cpu().T), dim=0)
        assert st["n_converged"] == n_cols and float(r.max()) <= 2e-10
    c.close()
