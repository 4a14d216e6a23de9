"""V^(s) coupling with n_M known at run time and in double-float, through whole applications: float64 against the
oracle's matrices, float32 and double-float (the MIXED inner operators) against float64, on mirrored pairs (blocks that
end inside a pair's planes), unequal boxes (positions outside) and more than one pair of sources."""
import ctypes

import numpy as np
import pytest

from fm_inputs import make_workload, rand_vec

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# J, (n_x, n_y, n_z) intervals, basis, identical pair, component 3's grid: n_M = 1 .. 6 and 7 .. 12
CASES = [(0, (9, 7, 3), 0, 12, None), (1, (6, 5, 2), 0, 12, None), (2, (5, 4, 3), 0, 0, None), (3, (4, 5, 2), 0, 12, None),
         (5, (7, 5, 3), 0, 12, None), (6, (4, 3, 5), 0, 12, ((3, 5, 4), (4.0, 3.0))), (8, (3, 5, 2), 0, 0, None),
         (11, (3, 3, 6), 0, 12, None), (0, (3, 3, 2), 1, 12, None), (3, (2, 3, 1), 1, 12, ((3, 2, 2), (4.0, 3.0))),
         (5, (2, 3, 3), 1, 12, None), (7, (2, 2, 1), 1, 12, None)]


def _workload(J, n, basis, pair, g3):
    wl = make_workload("He", J, nint=n, R=(12.0, 11.0), basis=basis, identical_pair=pair)
    if g3:
        wl["grids"] = {1: {"nint": n, "R": (12.0, 11.0)}, 3: {"nint": g3[0], "R": g3[1]}}
    return wl


@pytest.fixture(scope="module")
def pkg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2005_05398_gb300 as p
    return p


@pytest.mark.parametrize("J,n,basis,pair,g3", CASES)
def test_float64_matches_the_oracle(pkg, J, n, basis, pair, g3):
    from oracle.system import FMSystem
    wl = _workload(J, n, basis, pair, g3)
    s = FMSystem(wl)
    v = rand_vec(s.N, 3)
    ref = s.H() @ v + 2.1 * (s.S() @ v)
    ctx = pkg.Context(wl, restart_m=2, ncv=3)
    x = torch.tensor(v, device="cuda")
    y = torch.full_like(x, 7.0)
    ctx.fm_apply(-2.1, x, y)
    torch.cuda.synchronize()
    assert np.linalg.norm(y.cpu().numpy() - ref) < 1e-12 * np.linalg.norm(ref)  # as the other comparisons of H
    ctx.close()


@pytest.mark.parametrize("J,n,basis,pair,g3", CASES)
@pytest.mark.parametrize("kind,eps", [("f32", 2.0 ** -24), ("dd", 2.0 ** -46)])
def test_low_precision_operators_match_float64(pkg, J, n, basis, pair, g3, kind, eps):
    wl = _workload(J, n, basis, pair, g3)
    ctx = pkg.Context(wl, precision=2, mixed_scheme=2 if kind == "dd" else 0, restart_m=2, ncv=3)
    v = rand_vec(ctx.n, 4).astype(np.float32)
    x = torch.tensor(v.astype(np.float64), device="cuda")
    ref = torch.empty_like(x)
    ctx.fm_apply(-2.1, x, ref)
    name = {"f32": "_ZN3fmi14launch_apply32EP6fm_ctxdPKfPfb", "dd": "_ZN3fmi15launch_apply_ddEP6fm_ctxdPKNS_2ddEPS2_b"}[kind]
    fn = pkg.lib()[name]
    fn.argtypes = [ctypes.c_void_p, ctypes.c_double, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_bool]
    if kind == "f32":
        a = torch.tensor(v, device="cuda")
        b = torch.full_like(a, 7.0)
    else:  # pairs (hi, lo)
        a = torch.tensor(np.stack([v, np.zeros_like(v)], axis=1), device="cuda")
        b = torch.full_like(a, 7.0)
    torch.cuda.synchronize()
    assert fn(ctx.h, -2.1, a.data_ptr(), b.data_ptr(), False) == 0
    torch.cuda.synchronize()
    got = b.double() if kind == "f32" else b.double().sum(dim=1)
    # the largest terms of an output set its size and its rounding: 1e3 roundings cover the r^3 n_M + 10 r of a point
    assert torch.linalg.norm(got - ref).item() < 1e3 * eps * torch.linalg.norm(ref).item()
    ctx.close()
