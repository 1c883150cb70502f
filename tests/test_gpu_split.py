"""The double-float split of FP64 vectors over its ranges: ordinary values, zeros, ties, and exponents whose
parts are near or below the smallest normal floats.  The double-float product (prec 3) is compared with
the FP64 one: 2^-44 of sum |a||x| per row for parts in the normal range (48-bit operands, 16 terms), and the
smallest float times sum |a| more where parts are denormal."""
import numpy as np
import pytest

from phantom import EPS_MATCHING, kuhn_mesh

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("scale", [1.0, 2.0 ** 60, 2.0 ** -60, 2.0 ** -89, 2.0 ** -91, 2.0 ** -120])
def test_split_product_against_fp64(scale):
    from paper_2311_05322_gb300 import mw
    m = kuhn_mesh(5, 4, 3, lo=(-2.0, -1.5, -1.0), hi=(2.0, 1.5, 1.0))
    c = mw.Context(0)
    E = c.set_mesh(m.xyz, m.tets).n_edge
    c.assemble([1e7], np.tile([EPS_MATCHING.real, EPS_MATCHING.imag], (m.n_tet, 1)), EPS_MATCHING)
    _, _, _, rp, ci = c.get_topology()
    A = torch.sparse_csr_tensor(torch.from_numpy(rp), torch.from_numpy(ci.astype(np.int64)),
                                torch.from_numpy(c.get_matrix(0)), (E, E)).to_dense()
    rng = np.random.default_rng(7)
    X = rng.standard_normal((E, 3)) + 1j * rng.standard_normal((E, 3))
    X[::5] = 0.0
    X[1::7, 1] = -(1 + 2.0 ** -24) + 1j * (1 + 3 * 2.0 ** -24)           # ties of the high part
    X[2::7, 2] = (2 - 2.0 ** -52) - 1j * (1 - 2.0 ** -53)                 # the high part rounds up to a power of two
    x = torch.from_numpy(X * scale)
    y = torch.empty((E, 3), dtype=torch.complex128, device="cuda")
    c.apply_matrix(0, 3, x.cuda(), y, 3)
    torch.cuda.synchronize()
    ref = A @ x
    bound = 2.0 ** -44 * (A.abs() @ x.abs()) + 2.0 ** -148 * A.abs().sum(1, keepdim=True)
    assert torch.all((y.cpu() - ref).abs() <= bound)
    c.close()


@pytest.mark.parametrize("exponent", [121, 122, 123, 124, 125, 126, 127])
def test_split_near_the_largest_floats(exponent):
    """Values of one binade up to the largest floats, on a mesh whose matrix entries are small enough for their
    products: both parts are ordinary floats, so the bound is the one above without its denormal term."""
    from paper_2311_05322_gb300 import mw
    h = 2.0 ** 30
    m = kuhn_mesh(5, 4, 3, lo=(-2 * h, -1.5 * h, -h), hi=(2 * h, 1.5 * h, h))
    c = mw.Context(0)
    E = c.set_mesh(m.xyz, m.tets).n_edge
    c.assemble([1e7 / h], np.tile([EPS_MATCHING.real, EPS_MATCHING.imag], (m.n_tet, 1)), EPS_MATCHING)
    _, _, _, rp, ci = c.get_topology()
    A = torch.sparse_csr_tensor(torch.from_numpy(rp), torch.from_numpy(ci.astype(np.int64)),
                                torch.from_numpy(c.get_matrix(0)), (E, E)).to_dense()
    rng = np.random.default_rng(exponent)
    part = lambda: rng.uniform(1.0, 1.99, (E, 3)) * rng.choice([-1.0, 1.0], (E, 3))
    x = torch.from_numpy((part() + 1j * part()) * 2.0 ** exponent)
    y = torch.empty((E, 3), dtype=torch.complex128, device="cuda")
    c.apply_matrix(0, 3, x.cuda(), y, 3)
    torch.cuda.synchronize()
    c.close()
    assert torch.all((y.cpu() - A @ x).abs() <= 2.0 ** -44 * (A.abs() @ x.abs()))
