"""Products queued ahead of an Arnoldi step look at the device word of active columns: at zero every form of the FP32
product leaves its output alone, else all forms give the same bits.  The library's launchers are called directly (no
public call shows a product whose step is not taken); a window of nonzeros too large for shared memory selects the
row-per-warp form."""
import ctypes as C
import subprocess

import numpy as np
import pytest

from phantom import EPS_MATCHING, kuhn_mesh

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


class SpmmDev(C.Structure):
    _fields_ = [("n_block", C.c_int64), ("halo_max", C.c_int)] + [
        (k, C.c_void_p) for k in ("blk_row", "blk_halo", "halo", "rows", "rptr", "lcol", "src")]


@pytest.mark.parametrize("n_cols", [2, 3, 16, 34, 128])
@pytest.mark.parametrize("form", ["staged", "rows", "staged_bf16", "rows_bf16", "halo"])
def test_the_word_is_looked_at(form, n_cols):
    from paper_2311_05322_gb300 import mw
    if form == "halo" and n_cols % 2:
        pytest.skip("the halo-tiled product takes even column counts")
    lib = mw.load_library()
    name = {"rows": "8spmm_f32E", "rows_bf16": "11spmm_f32_bxE", "halo": "13spmm_halo_f32E"}
    name = name[{"staged": "rows", "staged_bf16": "rows_bf16"}.get(form, form)]
    symbols = subprocess.run(["nm", "-D", "--defined-only", lib._name], capture_output=True, text=True, check=True)
    fn = lib[next(q.split()[2] for q in symbols.stdout.splitlines() if "_ZN3mwk" + name in q)]
    m = kuhn_mesh(3, 3, 2)
    c = mw.Context(0)
    E = c.set_mesh(m.xyz, m.tets).n_edge
    c.assemble([1e9], np.tile([EPS_MATCHING.real, EPS_MATCHING.imag], (m.n_tet, 1)), EPS_MATCHING)
    _, _, _, rp, ci = c.get_topology()
    assert E <= 480 and rp[-1] <= 4096
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    A = dev(c.get_matrix(0).astype(np.complex64))
    drp, dci = dev(rp.astype(np.int64)), dev(ci.astype(np.int32))
    xb = torch.randn((E, n_cols, 2), generator=torch.Generator().manual_seed(1)).to(torch.bfloat16).cuda()
    x = torch.view_as_complex(xb.float().contiguous())
    ref = torch.empty((E, n_cols), dtype=torch.complex64, device="cuda")
    c.apply_matrix(0, mw.MW_PREC_FP32, x, ref, n_cols)
    ptr = lambda a: C.c_void_p(a.data_ptr())
    for word in (0, 1):
        go = torch.full((1,), word, dtype=torch.int32, device="cuda")
        y = torch.full_like(ref, 7.0)
        torch.cuda.synchronize()
        if form == "halo":
            one = [dev(np.array(q)) for q in ([0, E], [0, E], np.arange(E, dtype=np.int32), np.arange(E, dtype=np.int32),
                                              rp.astype(np.int64), ci.astype(np.uint16), np.arange(rp[-1], dtype=np.int32))]
            plan = SpmmDev(1, 480, *(ptr(q) for q in one))
            fn.restype = C.c_bool
            assert fn(C.byref(plan), ptr(A), ptr(x), ptr(y), C.c_int(n_cols), None, ptr(go))
        else:
            win = (C.c_int * 3)(*([1 << 20] * 3 if form.startswith("rows") else [int(rp[-1])] * 3))
            fn.restype = None
            fn(ptr(drp), ptr(dci), ptr(A), ptr(xb if form.endswith("bf16") else x), ptr(y), C.c_int64(E), C.c_int(n_cols),
               None, C.c_int(256), win, ptr(go))
        torch.cuda.synchronize()
        want = ref if word else torch.full_like(ref, 7.0)
        assert torch.equal(torch.view_as_real(y), torch.view_as_real(want))
    c.close()
