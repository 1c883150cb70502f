"""Row stores of the tensor-core applies: 16-byte pieces where rows are whole, aligned pieces, single values
elsewhere.  Even and odd column counts, partial groups of 8 columns and buffers that start off a 16-byte
boundary give each column the value that it has in a block of 64 columns.

Bar: a column's sums hold the same BF16 products whatever the block's width, so dense applies differ by FP32
sums of at most 2 K <= 2000 terms (2000 * 2^-24 < 2^-12 of the row's absolute sum; 2^-7 leaves room for
cancellation); the sparse sweeps round to BF16 (2^-9) between heights.  A misplaced store gives O(1).
"""
import numpy as np
import pytest

from phantom import EPS_MATCHING, box_partition, kuhn_mesh

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _ctx(sparse):
    from paper_2311_05322_gb300 import mw
    m = kuhn_mesh(6, 5, 4, lo=(-0.03, -0.025, -0.02), hi=(0.03, 0.025, 0.02))
    rng = np.random.default_rng(2)
    eps = EPS_MATCHING + rng.uniform(-6, 6, m.n_tet) + 1j * rng.uniform(-4, 4, m.n_tet)
    c = mw.Context(0)
    E = c.set_mesh(m.xyz, m.tets).n_edge
    c.assemble([1e9], np.stack([eps.real, eps.imag], 1), EPS_MATCHING)
    c.setup_preconditioner(4, box_partition(m, (2, 2, 1)), 1, mw.MW_PREC_SPARSE_BF16 if sparse else mw.MW_PREC_BF16)
    g = torch.Generator(device="cuda").manual_seed(5)
    x = torch.complex(*(torch.randn(E, 64, device="cuda", generator=g) for _ in range(2)))
    return c, E, x


@pytest.mark.parametrize("sparse", [False, True])
@pytest.mark.parametrize("R", [1, 2, 3, 4, 6, 7, 8, 10, 17, 34, 40])
def test_columns_do_not_depend_on_the_block(sparse, R):
    c, E, x = _ctx(sparse)
    ref = torch.empty(E, 64, dtype=torch.complex128, device="cuda")
    c.apply_preconditioner(0, x.to(torch.complex128), ref, 64)
    xr = x[:, :R].contiguous()
    z = torch.empty(E, R, dtype=torch.complex128, device="cuda")
    c.apply_preconditioner(0, xr.to(torch.complex128), z, R)
    tol = 2.0 ** -7
    assert float((z - ref[:, :R]).norm() / ref[:, :R].norm()) <= tol
    if not sparse:
        for off in (0, 1):   # complex64 buffers on and off a 16-byte boundary
            xb, zb = (torch.zeros(E * R + 3, dtype=torch.complex64, device="cuda") for _ in range(2))
            xb[off:off + E * R] = xr.reshape(-1)
            zb[off + E * R] = 7.0
            c.apply_preconditioner_noalloc(0, xb[off:off + E * R], zb[off:off + E * R], R)
            assert float((zb[off:off + E * R].reshape(E, R) - ref[:, :R]).norm() / ref[:, :R].norm()) <= tol
            assert zb[off + E * R] == 7.0
    c.close()


@pytest.mark.parametrize("cells,parts,overlap,R", [((5, 4, 3), (2, 1, 1), 0, 3), ((10, 9, 8), (2, 2, 1), 3, 8),
                                                   ((24, 4, 2), (6, 1, 1), 2, 33), ((12, 10, 8), (1, 1, 1), 0, 16)])
def test_pruned_sweeps_against_all_rows(cells, parts, overlap, R):
    """The BF16 sweeps compute only rows that reach an owned dof; the FP32 sweeps compute all of them.  Bar: BF16
    tiles and operands (2^-9 each) compounded over the heights, 3e-2; a row left out by mistake gives O(1)."""
    from paper_2311_05322_gb300 import mw
    m = kuhn_mesh(*cells, lo=(-0.03, -0.025, -0.02), hi=(0.03, 0.025, 0.02))
    rng = np.random.default_rng(R)
    eps = EPS_MATCHING + rng.uniform(-6, 6, m.n_tet) + 1j * rng.uniform(-4, 4, m.n_tet)
    z = []
    for prec in (mw.MW_PREC_SPARSE, mw.MW_PREC_SPARSE_BF16):
        c = mw.Context(0)
        E = c.set_mesh(m.xyz, m.tets).n_edge
        c.assemble([1e9], np.stack([eps.real, eps.imag], 1), EPS_MATCHING)
        c.setup_preconditioner(int(np.prod(parts)), box_partition(m, parts), overlap, prec)
        g = torch.Generator(device="cuda").manual_seed(R)
        x = torch.complex(*(torch.randn(E, R, device="cuda", generator=g, dtype=torch.float64) for _ in range(2)))
        for persistent in (True, False):
            c.set_sweep_schedule(persistent)
            z.append(torch.empty_like(x))
            c.apply_preconditioner(0, x, z[-1], R)
        c.close()
    assert torch.equal(z[2], z[3])
    assert float((z[2] - z[0]).norm() / z[0].norm()) <= 3e-2
