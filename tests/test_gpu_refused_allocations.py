"""Allocations refused one after the other: a memory cap that rises in small steps makes every allocation of a call
fail once.  A refused call reports MW_ENOMEM and keeps nothing; a smaller call between two refusals either does too or
gives the right result, and without the cap everything gives the results of a context that saw no refusal."""
import numpy as np
import pytest

from phantom import EPS_MATCHING, box_partition, kuhn_mesh

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
LIMIT = 3000   # steps of a climb: a call that kept buffers when it is refused would never get past its cap


def _used(c):
    """Bytes the context holds: the largest cap at which the self-test's 16 bytes are refused, less 15."""
    from paper_2311_05322_gb300 import mw
    lo, hi = 1, 1 << 34
    while lo < hi:
        mid = (lo + hi) // 2
        c.set_memory_cap(mid)
        try:
            c.selftest_bounded_wait(16)
            hi = mid
        except mw.MWError as e:
            assert e.status == mw.MW_ENOMEM
            lo = mid + 1
    c.set_memory_cap(0)
    return lo - 16


def _climb(c, call, between=lambda: None, step=1 << 16, start=1):
    """call() under a rising cap until it succeeds; between() after every refusal.  Returns the refusals; the cap
    that sufficed is start + refusals * step."""
    from paper_2311_05322_gb300 import mw
    for refused in range(LIMIT):
        c.set_memory_cap(start + refused * step)
        for f in (call, between):
            try:
                f()
                if f is call:
                    c.set_memory_cap(0)
                    return refused
            except mw.MWError as e:
                assert e.status == mw.MW_ENOMEM, e
    pytest.fail("the cap never sufficed")


def _context(prec, eps=None):
    from paper_2311_05322_gb300 import mw
    m = kuhn_mesh(5, 4, 3, lo=(-0.02, -0.015, -0.01), hi=(0.02, 0.015, 0.01))
    c = mw.Context(0)
    E = c.set_mesh(m.xyz, m.tets).n_edge
    c.assemble([1e9], np.tile([EPS_MATCHING.real, EPS_MATCHING.imag], (m.n_tet, 1)), EPS_MATCHING)
    if prec is not None:
        c.setup_preconditioner(4, box_partition(m, (2, 2, 1)), 1, prec)
    return mw, m, c, E


@pytest.mark.parametrize("what", ["matrix", "preconditioner", "dots", "grid", "tikhonov"])
def test_refused_calls_keep_nothing(what):
    """A cap that a climb of refused calls found sufficient is no larger than a fresh context needs."""
    def ready():
        from paper_2311_05322_gb300 import mw as lib
        mw, m, c, E = _context(lib.MW_PREC_FP32)
        x = torch.ones((E, 6), dtype=torch.complex128, device="cuda")
        y = torch.empty_like(x)
        v = torch.ones(4 * 6 * E, dtype=torch.complex64, device="cuda")
        call = {"matrix": lambda: c.apply_matrix(0, 3, x, y, 6),
                "preconditioner": lambda: c.apply_preconditioner(0, x, y, 6),
                "dots": lambda: c.krylov_dots(v, v, 3, 6 * E, E, 6),
                "grid": lambda: c.nn_grid_to_tets(np.ones((2, 32, 32, 32), np.float32), [-0.02] * 3 + [0.02] * 3),
                "tikhonov": lambda: c.tikhonov(np.ones((m.n_tet, 2)))}[what]
        return mw, c, call
    step = 1 << 13
    mw, c, call = ready()
    refused = _climb(c, call, step=step)
    assert refused > 0
    c.close()
    mw, c, call = ready()
    c.set_memory_cap(1 + (refused - 1) * step)
    with pytest.raises(mw.MWError) as e:
        call()
    assert e.value.status == mw.MW_ENOMEM
    c.set_memory_cap(1 + refused * step)
    call()
    c.close()


@pytest.mark.parametrize("prec", ["BF16", "SPARSE_BF16", "SPARSE", "FP32"])
def test_solver_workspace(prec):
    """Workspace and preconditioner scratch are recorded as present only when they are complete: a solve of fewer
    columns after a refused one used to take the record of the larger workspace for memory it did not have."""
    from paper_2311_05322_gb300 import mw as lib
    mw, m, c, E = _context(getattr(lib, "MW_PREC_" + prec))
    g = torch.Generator().manual_seed(3)
    b = torch.complex(*(torch.randn(6, E, generator=g, dtype=torch.float64) for _ in range(2))).cuda()
    o = mw.solve_opts(mode=1, restart=10, tol=1e-9, inner_tol=1e-2)
    c.set_autotune(False)
    want = torch.empty_like(b)
    c.solve_rhs(6, b, want, o)
    small_want = torch.empty_like(b[:2])
    c.solve_rhs(2, b[:2], small_want, o)
    z_want = torch.empty((E, 6), dtype=torch.complex128, device="cuda")
    r = b.T.contiguous()
    c.apply_preconditioner(0, r, z_want, 6)
    c.close()
    _, _, c, _ = _context(getattr(lib, "MW_PREC_" + prec))
    c.set_autotune(False)
    x, small, z = torch.empty_like(b), torch.empty_like(b[:2]), torch.empty_like(z_want)

    def between():
        small.zero_()
        c.solve_rhs(2, b[:2], small, o)
        assert torch.equal(torch.view_as_real(small), torch.view_as_real(small_want))

    assert _climb(c, lambda: c.solve_rhs(6, b, x, o), between) > 5
    assert torch.equal(torch.view_as_real(x), torch.view_as_real(want))
    _climb(c, lambda: c.apply_preconditioner(0, r, z, 6), step=1 << 14)
    assert torch.equal(torch.view_as_real(z), torch.view_as_real(z_want))
    c.solve_rhs(6, b, x, o)
    assert torch.equal(torch.view_as_real(x), torch.view_as_real(want))
    c.close()


def _data(n, nf=1):
    rng = np.random.default_rng(n)
    s = lambda: torch.from_numpy(rng.normal(size=(nf, n, n)) + 1j * rng.normal(size=(nf, n, n))).cuda()
    return s(), s()


@pytest.mark.parametrize("reciprocal", [False, True])
def test_fields_of_an_evaluation(reciprocal):
    """Forward and adjoint fields of several frequencies: an evaluation that was refused some of them leaves none."""
    from paper_2311_05322_gb300 import mw as lib
    pos = np.array([[0.012, 0.0, 0.002], [-0.012, 0.0, 0.002], [0.0, 0.01, 0.002]])
    freqs = [0.9e9, 1.0e9, 1.1e9]
    obs, emp = _data(3, 3)

    def ready():
        mw, m, c, E = _context(None)
        eps = np.tile([EPS_MATCHING.real, EPS_MATCHING.imag], (m.n_tet, 1))
        c.assemble(freqs, eps, EPS_MATCHING)
        c.set_sources(pos, np.tile([0.0, 0.0, 1.0], (3, 1)))
        c.setup_preconditioner(4, box_partition(m, (2, 2, 1)), 1, lib.MW_PREC_BF16)
        c.set_autotune(False)
        c.set_adjoint_mode(reciprocal)
        g = torch.zeros((m.n_tet, 2), dtype=torch.float64, device="cuda")
        o = mw.solve_opts(mode=1, restart=10, tol=1e-9, inner_tol=1e-2)
        return c, g, o, lambda: c.gradient_dev(obs, emp, g, 0.0, o)

    c, want, o, call = ready()
    J = call()
    S, _ = c.solve(o)
    c.close()
    c, g, o, call = ready()
    got = []

    def between():
        s, _ = c.solve(o)
        assert np.array_equal(s, S)

    _climb(c, lambda: got.append(call()), between, step=1 << 15)
    assert got[-1] == J and torch.equal(g, want)
    assert np.array_equal(c.solve(o)[0], S)
    c.close()


def test_matrices_of_several_frequencies():
    """An assembly that was refused a buffer leaves nothing assembled."""
    freqs = [0.9e9, 1.0e9, 1.1e9]
    mw, m, c, E = _context(None)
    eps = np.tile([EPS_MATCHING.real, EPS_MATCHING.imag], (m.n_tet, 1))
    c.assemble(freqs, eps, EPS_MATCHING)
    want = [c.get_matrix(f) for f in range(3)]
    c.close()
    mw, m, c, E = _context(None)
    x = torch.ones((E, 3), dtype=torch.complex64, device="cuda")
    y = torch.empty_like(x)

    def between():
        for call in (lambda: c.apply_matrix(0, mw.MW_PREC_FP32, x, y, 3), c.solve):
            with pytest.raises(mw.MWError) as e:
                call()
            assert e.value.status in (mw.MW_EINVAL, mw.MW_ESTATE)

    assert _climb(c, lambda: c.assemble(freqs, eps, EPS_MATCHING), between, step=1 << 14) > 10
    assert all(np.array_equal(c.get_matrix(f), want[f]) for f in range(3))
    c.close()


def test_sources():
    """Sources that were refused a table are no sources, and their vectors are freed once."""
    from paper_2311_05322_gb300 import mw as lib
    mw, m, c, E = _context(lib.MW_PREC_BF16)
    c.set_autotune(False)
    rng = np.random.default_rng(1)
    pos = rng.uniform(-0.009, 0.009, (40, 3))
    z = np.tile([0.0, 0.0, 1.0], (40, 1))
    o = mw.solve_opts(mode=1, restart=10, tol=1e-9, inner_tol=1e-2)
    c.set_sources(pos, z)
    want, _ = c.solve(o)
    c.set_sources(pos[:7], z[:7])           # drops the fields, which the tables would otherwise find room in
    seen = set()

    def between():
        with pytest.raises(mw.MWError) as e:
            c.solve(o)                      # no sources, or no memory for the fields of the old ones
        seen.add(e.value.status)
        if e.value.status == mw.MW_ESTATE:
            c.set_memory_cap(0)
            c.set_sources(pos[:7], z[:7])

    _climb(c, lambda: c.set_sources(pos, z), between, step=16, start=_used(c))
    assert seen == {mw.MW_ENOMEM, mw.MW_ESTATE}
    assert np.array_equal(c.solve(o)[0], want)
    c.close()


def test_network():
    """A network that was refused a buffer is none, and a batch that was refused one leaves no room for smaller ones."""
    from paper_2311_05322_gb300 import inversion, mw
    n_in, rng = 9, np.random.default_rng(2)
    th = inversion.he_init(n_in, 2)
    x = rng.normal(size=(24, n_in)).astype(np.float32)
    t = (0.1 * rng.normal(size=(24, 2, 32, 32, 32))).astype(np.float32)
    c = mw.Context(0)
    c.nn_init(n_in, th)
    want, small = c.nn_infer(x), c.nn_infer(x[:2])
    losses, _ = c.nn_train(x, t, batch=10, epochs=2, lr=1e-3, seed=1)
    params = c.nn_get_params()
    c.close()
    c = mw.Context(0)

    def none():
        with pytest.raises(mw.MWError) as e:
            c.nn_infer(x[:2])
        assert e.value.status == mw.MW_ESTATE

    assert _climb(c, lambda: c.nn_init(n_in, th), none, step=1 << 18) > 10
    assert np.array_equal(c.nn_infer(x[:2]), small)
    got = []
    between = lambda: np.testing.assert_array_equal(c.nn_infer(x[:2]), small)
    assert _climb(c, lambda: got.append(c.nn_infer(x)), between, step=1 << 18, start=_used(c)) > 5
    assert np.array_equal(got[-1], want)
    assert _climb(c, lambda: got.append(c.nn_train(x, t, batch=10, epochs=2, lr=1e-3, seed=1)), between, step=1 << 18,
                  start=_used(c)) > 5
    assert np.array_equal(got[-1][0], losses) and np.array_equal(c.nn_get_params(), params)
    c.close()


def test_ports():
    """Ports that were refused a buffer leave a boundary without classes: the matrix of an open boundary, no sources."""
    from paper_2311_05322_gb300 import mw
    from phantom import waveguide_section
    m, fv, lab, ps = waveguide_section((4, 2, 6), 0.02, 0.01, 0.03, 59.0 - 1.0j)
    eps = np.tile([59.0, -1.0], (m.n_tet, 1))
    c = mw.Context(0)
    c.set_mesh(m.xyz, m.tets)
    c.assemble([8e8], eps, EPS_MATCHING)
    open_ = c.get_matrix(0)
    ports = lambda: c.set_ports(ps.origin, ps.u, ps.v, ps.a, ps.eps_fill, fv, lab)
    ports()
    W, n = c.get_port_vectors()
    c.assemble([8e8], eps, EPS_MATCHING)
    closed = c.get_matrix(0)
    assert not np.array_equal(open_, closed)
    c.close()
    c = mw.Context(0)
    c.set_mesh(m.xyz, m.tets)
    ports()                                  # the ports that the refused ones replace

    def between():
        with pytest.raises(mw.MWError) as e:
            c.get_port_vectors()
        assert e.value.status == mw.MW_ESTATE
        c.set_memory_cap(0)
        c.assemble([8e8], eps, EPS_MATCHING)
        assert np.array_equal(c.get_matrix(0), open_)

    ports()
    start = _used(c) - 4096                  # the classes go first: refusals begin below what is held
    _climb(c, ports, between, step=256, start=start)
    W2, n2 = c.get_port_vectors()
    c.assemble([8e8], eps, EPS_MATCHING)
    assert np.array_equal(W, W2) and np.array_equal(n, n2) and np.array_equal(c.get_matrix(0), closed)
    c.close()


@pytest.mark.parametrize("prec", ["FP64", "FP32", "BF16", "SPARSE", "SPARSE_BF16"])
def test_mesh_and_preconditioner(prec):
    """A mesh or a preconditioner that was refused a buffer is none, and holds nothing."""
    from paper_2311_05322_gb300 import mw as lib
    mw, m, c, E = _context(None)
    part = box_partition(m, (2, 2, 1))
    code = getattr(lib, "MW_PREC_" + prec)
    held = _used(c)
    r = torch.ones((E, 3), dtype=torch.complex128, device="cuda")
    want, z = torch.empty_like(r), torch.empty_like(r)
    c.setup_preconditioner(4, part, 1, code)
    c.apply_preconditioner(0, r, want, 3)
    c.close()
    mw, m, c, E = _context(None)

    def between():
        with pytest.raises(mw.MWError) as e:
            c.apply_preconditioner(0, r, z, 3)
        assert e.value.status == mw.MW_ESTATE
        assert _used(c) == held

    assert _climb(c, lambda: c.setup_preconditioner(4, part, 1, code), between, step=1 << 14, start=held) > 5
    c.apply_preconditioner(0, r, z, 3)
    assert torch.equal(torch.view_as_real(z), torch.view_as_real(want))
    c.close()
    c = mw.Context(0)

    def none():
        with pytest.raises(mw.MWError) as e:
            c.assemble([1e9], np.tile([EPS_MATCHING.real, EPS_MATCHING.imag], (m.n_tet, 1)), EPS_MATCHING)
        assert e.value.status == mw.MW_ESTATE
        assert _used(c) == 0

    assert _climb(c, lambda: c.set_mesh(m.xyz, m.tets), none, step=1 << 13) > 5
    c.close()
