"""Dense subdomain inverses: sizes around the 32-wide pivot blocks and the 64 x 64 update tiles,
subdomains that own everything, little or nothing, against the oracle's exact subdomain solves (bars of the parity tests: 1e-11 FP64, 2e-5 FP32, 1e-2 BF16)."""
import numpy as np
import pytest

from oracle import assemble as asm
from oracle import oras
from phantom import EPS_MATCHING, kuhn_mesh

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _partition(m, kind):
    c = np.floor((m.centroids() - np.asarray(m.lo)) / np.asarray(m.h)).astype(int)
    if kind == "one":
        return 1, np.zeros(m.n_tet, np.int32)
    if kind == "slabs":                       # one cell layer each along x
        return m.nx, c[:, 0].astype(np.int32)
    if kind == "corner":                      # a single cell, the rest, and a subdomain of one tet
        p = np.where((c == 0).all(axis=1), 1, 0).astype(np.int32)
        p[-1] = 2
        return 3, p
    # interleaved columns: the last ones own no edge of their own
    return 4, ((c[:, 0] + 2 * c[:, 1]) % 4).astype(np.int32)


@pytest.mark.parametrize("kind", ["one", "slabs", "corner", "mixed"])
@pytest.mark.parametrize("cells,overlap", [((2, 1, 1), 0), ((3, 3, 2), 0), ((4, 3, 3), 1), ((5, 4, 3), 0), ((5, 5, 4), 2)])
def test_owned_rows_of_the_inverses(kind, cells, overlap):
    from paper_2311_05322_gb300 import mw
    m = kuhn_mesh(*cells, lo=(-0.02, -0.015, -0.01), hi=(0.02, 0.015, 0.01))
    rng = np.random.default_rng(sum(cells) + overlap)
    eps = EPS_MATCHING + rng.uniform(-6, 6, m.n_tet) + 1j * rng.uniform(-4, 4, m.n_tet)
    n_sub, part = _partition(m, kind)
    c = mw.Context(0)
    E = c.set_mesh(m.xyz, m.tets).n_edge
    c.assemble([1e9], np.stack([eps.real, eps.imag], 1), EPS_MATCHING)
    P = oras.ORAS(asm.build_system(m.xyz, m.tets), part, n_sub, overlap, eps, 1e9, EPS_MATCHING)
    X = rng.normal(size=(E, 5)) + 1j * rng.normal(size=(E, 5))
    ref = np.stack([P.apply(X[:, k]) for k in range(5)], 1)
    x = torch.from_numpy(X).cuda()
    z = torch.empty_like(x)
    for prec, bar in ((mw.MW_PREC_FP64, 1e-11), (mw.MW_PREC_FP32, 2e-5), (mw.MW_PREC_FP64_FROM_FP32, 2e-5),
                      (mw.MW_PREC_BF16, 1e-2)):
        c.setup_preconditioner(n_sub, part, overlap, prec)
        c.apply_preconditioner(0, x, z, 5)
        torch.cuda.synchronize()
        assert np.linalg.norm(z.cpu().numpy() - ref) <= bar * np.linalg.norm(ref), prec
    c.close()
