"""How many products share one float32 sum in the Gram-Schmidt reductions: a product of 2^24 swallows the ones that are
added to its sum after it (and rounds an odd sum before it to an even one), so the error of the whole counts them.
Never more than n / 155,648 work items (pairs, quads or elements, rounded up) go into one sum; the norm of an update is
summed in float64."""
import ctypes

import numpy as np
import pytest

from fm_inputs import make_workload

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SUMS = 152 * 1024
# (workload, precision): 83 k, 202 k and 979 k unknowns; 40,401 and 521,667 (odd: one component alone)
EVEN = [dict(nint=(24, 24, 8)), dict(nint=(30, 30, 13)), dict(nint=(60, 60, 16))]
ODD = [dict(nint=(22, 22, 2), basis=1, mode=2), dict(nint=(46, 46, 8), basis=1, mode=2)]
P, D, I, L, F = ctypes.c_void_p, ctypes.c_double, ctypes.c_int, ctypes.c_int64, ctypes.c_float


def _context(kw, precision):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2005_05398_gb300 as pkg
    ctx = pkg.Context(make_workload("He", 0, R=(30.0, 30.0), **kw), precision=precision, restart_m=2, ncv=3)

    def fn(name, *args):
        f = pkg.lib()[name]
        f.argtypes, f.restype = args, ctypes.c_int
        return f
    return pkg, ctx, fn


def _spots(n):
    return [0, 1, n // 3, n // 2, n - 1]


@pytest.mark.parametrize("kw", EVEN + ODD)
def test_first_pass_multi_dot(kw):
    pkg, ctx, fn = _context(kw, 0)
    f = fn("_ZN3fmi12dot_many_devEP6fm_ctxPKdliS3_S3_Pdb", P, P, L, I, P, P, P, ctypes.c_bool)
    n = ctx.n
    per = 1 if n % 2 else 2
    bound = per * -(-(n // per) // SUMS)
    for nv in (1, 9):
        for at in _spots(n):
            w = torch.ones(n, dtype=torch.float64, device="cuda")
            w[at] = 2.0 ** 12
            V = w.repeat(nv, 1).contiguous()
            h = torch.zeros(nv, dtype=torch.float64, device="cuda")
            assert f(ctx.h, V.data_ptr(), n, nv, w.data_ptr(), None, h.data_ptr(), True) == 0
            torch.cuda.synchronize()
            lost = 2.0 ** 24 + n - 1 - h.cpu().numpy()
            assert np.all(np.abs(lost) < bound), (at, lost, bound)
    ctx.close()


@pytest.mark.parametrize("kw", EVEN)
def test_float32_multi_dots_and_norm(kw):
    pkg, ctx, fn = _context(kw, 2)
    n = ctx.n
    dot = fn("_ZN3fmi10dot_many32EP6fm_ctxPKfliS3_Pd", P, P, L, I, P, P)
    gs = fn("_ZN3fmi10gs_cgs2_32EP6fm_ctxPKfiPfS4_PdS5_", P, P, I, P, P, P, P)
    upd = fn("_ZN3fmi16axpy_many_norm32EP6fm_ctxPKfliPKdfPfPd", P, P, L, I, P, F, P, P)
    slot = pkg.lib()["_ZN3fmi12tc_flag_slotEP6fm_ctx"]
    slot.argtypes, slot.restype = [P], P
    # the first coefficient of the first pass: 3 x 264 + 8 doubles before the wait flag
    class First:
        __cuda_array_interface__ = {"shape": (1,), "typestr": "<f8", "data": (slot(ctx.h) - 800 * 8, False), "version": 3}
    first = torch.as_tensor(First(), device="cuda")
    for at in _spots(n):
        w = torch.ones(n, dtype=torch.float32, device="cuda")
        w[at] = 2.0 ** 12
        want = 2.0 ** 24 + n - 1
        h = (ctypes.c_double * 1)()
        torch.cuda.synchronize()
        assert dot(ctx.h, w.data_ptr(), n, 1, w.data_ptr(), h) == 0
        assert abs(want - h[0]) < -(-n // SUMS), (at, want - h[0])
        v, out = w.clone(), torch.empty_like(w)
        hn = ctypes.c_double()
        torch.cuda.synchronize()
        assert gs(ctx.h, v.data_ptr(), 1, w.data_ptr(), out.data_ptr(), h, ctypes.byref(hn)) == 0
        assert abs(want - first.item()) < 4 * -(-(n // 4) // SUMS), (at, want - first.item())
        h[0] = 0.0
        torch.cuda.synchronize()
        assert upd(ctx.h, v.data_ptr(), n, 1, h, 1.0, v.data_ptr(), ctypes.byref(hn)) == 0
        assert hn.value == want
    ctx.close()
