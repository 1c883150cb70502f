"""Mixed solves of 1 to 128 columns, odd and even, with the basis of the preconditioned vectors in FP32 and BF16:
the solution update handles pairs of columns, single ones, ragged last rows and columns that stop early, and its
double-float copy of x feeds the residual.  Bar: the requested relative residual, checked in FP64 on the CPU
(1e-10 asked, twice that allowed for the check's own rounding)."""
import subprocess
import sys

import numpy as np
import pytest

from conftest import ROOT
from oracle import assemble as asm
from phantom import EPS_MATCHING, box_partition, kuhn_mesh

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("bf16", [0, 1])
@pytest.mark.parametrize("n_cols", [1, 2, 3, 16, 31, 64, 127, 128])
def test_residuals_of_the_updated_solution(n_cols, bf16):
    from paper_2311_05322_gb300 import mw
    m = kuhn_mesh(5, 4, 3, lo=(-0.02, -0.015, -0.01), hi=(0.02, 0.015, 0.01))
    rng = np.random.default_rng(n_cols)
    eps = EPS_MATCHING + rng.uniform(-6, 6, m.n_tet) + 1j * rng.uniform(-4, 4, m.n_tet)
    c = mw.Context(0)
    E = c.set_mesh(m.xyz, m.tets).n_edge
    c.assemble([1e9], np.stack([eps.real, eps.imag], 1), EPS_MATCHING)
    c.setup_preconditioner(4, box_partition(m, (2, 2, 1)), 1, mw.MW_PREC_BF16)
    c.set_z_storage(bf16)
    sysm = asm.build_system(m.xyz, m.tets)
    A = sysm.csr(asm.assemble(sysm, eps, 1e9, EPS_MATCHING))
    B = rng.normal(size=(n_cols, E)) + 1j * rng.normal(size=(n_cols, E))
    B[0] = A @ np.eye(1, E, 3)[0]           # a column that needs another number of steps
    if n_cols > 2:
        B[2] = 0.0                          # and one that needs none
    b = torch.from_numpy(B).cuda()
    x = torch.empty_like(b)
    st = c.solve_rhs(n_cols, b, x, mw.solve_opts(mode=1, restart=30, tol=1e-10, inner_tol=1e-3, max_it=3000,
                                                 max_outer=50))
    c.close()
    assert st["n_converged"] == n_cols
    r = B - (A @ x.cpu().numpy().T).T
    nb = np.linalg.norm(B, axis=1)
    assert np.all(np.linalg.norm(r, axis=1) <= 2e-10 * nb)


STAGED_Y = """
import numpy as np, torch
from paper_2311_05322_gb300 import mw
from phantom import EPS_MATCHING, box_partition, kuhn_mesh
m = kuhn_mesh(5, 4, 3, lo=(-0.02, -0.015, -0.01), hi=(0.02, 0.015, 0.01))
c = mw.Context(0)
E = c.set_mesh(m.xyz, m.tets).n_edge
c.assemble([1e9], np.tile([EPS_MATCHING.real, EPS_MATCHING.imag], (m.n_tet, 1)), EPS_MATCHING)
c.setup_preconditioner(4, box_partition(m, (2, 2, 1)), 1, mw.MW_PREC_BF16)
c.set_z_storage(%d)
rng = np.random.default_rng(%d)
b = torch.from_numpy(rng.normal(size=(%d, E)) + 1j * rng.normal(size=(%d, E))).cuda()
x = torch.empty_like(b)
st = c.solve_rhs(%d, b, x, mw.solve_opts(mode=1, restart=%d, tol=1e-10, inner_tol=1e-3, max_outer=50))
assert st["n_converged"] == %d
"""


@pytest.mark.parametrize("bf16", [0, 1])
@pytest.mark.parametrize("restart,n_cols", [(48, 128), (52, 118), (59, 104), (62, 99)])
def test_coefficients_that_just_fit_48_kilobytes(restart, n_cols, bf16):
    """The coefficients take 8 restart n_cols bytes, here at most 48 KB but more with the kernel's static shared
    memory.  Each in a process of its own: an earlier, larger solve leaves the kernel's limit raised."""
    n = n_cols
    subprocess.run([sys.executable, "-c", STAGED_Y % (bf16, restart, n, n, n, restart, n)], check=True, cwd=ROOT)
