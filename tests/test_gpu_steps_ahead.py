"""Products launched ahead of a step that may not be taken: solves stop at the same step, with the same bits, as
captured cycles (which launch no product of a step that is not taken) and as cycles with profiled classes (which wait
for every step's count), also where max_it or the restart length ends the cycle."""
import numpy as np
import pytest

from phantom import EPS_MATCHING, box_partition, kuhn_mesh

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n_cols,restart,max_it,tol", [(1, 30, 500, 1e-10), (5, 3, 500, 1e-10), (8, 30, 2, 1e-10),
                                                       (8, 1, 500, 1e-6), (33, 20, 7, 1e-12), (16, 2, 500, 1e-9)])
def test_steps_and_bits(n_cols, restart, max_it, tol):
    from paper_2311_05322_gb300 import mw
    m = kuhn_mesh(5, 4, 3, lo=(-0.02, -0.015, -0.01), hi=(0.02, 0.015, 0.01))
    rng = np.random.default_rng(n_cols + restart)
    eps = EPS_MATCHING + rng.uniform(-6, 6, m.n_tet) + 1j * rng.uniform(-4, 4, m.n_tet)
    out = []
    for way in ("ahead", "profiled", "graphs"):
        c = mw.Context(0)
        E = c.set_mesh(m.xyz, m.tets).n_edge
        c.assemble([1e9], np.stack([eps.real, eps.imag], 1), EPS_MATCHING)
        c.setup_preconditioner(4, box_partition(m, (2, 2, 1)), 1, mw.MW_PREC_BF16)
        c.set_autotune(False)
        if way == "profiled":
            c.profile_enable(1 << mw.MW_K_SPMM)
        c.set_graphs(way == "graphs")
        g = torch.Generator().manual_seed(n_cols)
        b = torch.complex(*(torch.randn(n_cols, E, generator=g, dtype=torch.float64) for _ in range(2))).cuda()
        x = torch.empty_like(b)
        st = c.solve_rhs(n_cols, b, x, mw.solve_opts(mode=1, restart=restart, tol=tol, inner_tol=1e-3, max_it=max_it,
                                                     max_outer=200), allow_noconv=True)
        out.append((x.cpu(), st["arnoldi_steps"], np.array(st["iters"]), st["n_converged"]))
        c.close()
    for o in out[1:]:
        assert torch.equal(torch.view_as_real(o[0]), torch.view_as_real(out[0][0]))
        assert o[1] == out[0][1] and np.array_equal(o[2], out[0][2]) and o[3] == out[0][3]
