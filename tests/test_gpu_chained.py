"""Chained launches keep the stream's order: long queues of short dependent calls give the bits of calls that are
separated by a synchronisation, also with another library's kernels in between, and under stream capture."""
import numpy as np
import pytest

from phantom import EPS_MATCHING, box_partition, kuhn_mesh

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _ctx(stream):
    from paper_2311_05322_gb300 import mw
    m = kuhn_mesh(6, 5, 4, lo=(-0.03, -0.025, -0.02), hi=(0.03, 0.025, 0.02))
    rng = np.random.default_rng(4)
    eps = EPS_MATCHING + rng.uniform(-6, 6, m.n_tet) + 1j * rng.uniform(-4, 4, m.n_tet)
    c = mw.Context(0, stream)
    E = c.set_mesh(m.xyz, m.tets).n_edge
    c.assemble([1e9], np.stack([eps.real, eps.imag], 1), EPS_MATCHING)
    c.setup_preconditioner(4, box_partition(m, (2, 2, 1)), 1, mw.MW_PREC_BF16)
    return c, E


@pytest.mark.parametrize("R", [1, 8, 32])
def test_queued_calls_have_the_bits_of_separate_calls(R):
    st = torch.cuda.Stream()
    c, E = _ctx(st.cuda_stream)
    torch.manual_seed(R)
    x = torch.randn(E, R, dtype=torch.complex64, device="cuda")

    def chain(sync):
        v, w, z = x.clone(), torch.empty_like(x), torch.empty_like(x)
        torch.cuda.synchronize()
        with torch.cuda.stream(st):
            for k in range(40):
                c.apply_matrix(0, 1, v, w, R)
                if sync:
                    torch.cuda.synchronize()
                c.apply_matrix(0, 1, w, v, R)
                if sync:
                    torch.cuda.synchronize()
                if k % 2:
                    v *= 2.0 ** -40   # another library's kernel between chained ones (an exact scaling)
                if k % 8 == 0:
                    c.apply_preconditioner_noalloc(0, v, z, R)
        torch.cuda.synchronize()
        return v, w, z

    for a, b in zip(chain(True), chain(False)):
        assert torch.equal(torch.view_as_real(a), torch.view_as_real(b)) and torch.isfinite(a.abs()).all()
    c.close()


def test_capture_replays_the_same_bits():
    st = torch.cuda.Stream()
    c, E = _ctx(st.cuda_stream)
    torch.manual_seed(3)
    x = torch.randn(E, 8, dtype=torch.complex64, device="cuda")
    y, z = torch.empty_like(x), torch.empty_like(x)
    torch.cuda.synchronize()
    with torch.cuda.stream(st):
        c.apply_matrix(0, 1, x, y, 8)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        c.apply_matrix(0, 1, x, z, 8)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(y, z)
    c.close()
