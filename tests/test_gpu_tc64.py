"""Float64 mode products on the tensor cores (digit splitting) against the float64 CUDA-core kernels: tile edges
of rows (128), columns (64 and 32), contraction blocks (64, 192 | 194, 256 | 258) and both component layouts."""
import numpy as np
import pytest

from fm_inputs import make_workload, rand_vec

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2005_05398_gb300 as p
    from paper_2005_05398_gb300 import build
    build.build()
    p.lib()
    return p


def _pair(pkg, wl, E, v, **opt):
    out = []
    for mma in (0, 1):  # tensor cores, CUDA cores
        ctx = pkg.Context(wl, mma=mma, restart_m=4, ncv=3, **opt)
        ctx.fm_set_shift(E)
        y = torch.full_like(v, 7.0)
        ctx.fm_precond_apply(v, y)
        torch.cuda.synchronize()
        out.append(y)
        ctx.close()
    return out


def _bound(wl):
    """Rounding of the two evaluations: n u, amplified by the condition numbers of the z and x eigenvector matrices
    (the z modes of fine grids come in nearly degenerate pairs, so theirs grow to 1e6 and more)."""
    from oracle.splines import Axis
    mx, _, mz = wl["maps"]
    az = Axis(mz, wl["nint"][2], -1.0, 1.0, dirichlet=False, basis=wl["basis"])
    ax = Axis(mx, wl["nint"][0], 0.0, wl["R"][0], dirichlet=True, basis=wl["basis"])
    z, x = az.pts, ax.pts
    kz = kx = 1.0
    for Mp in range(wl["J"] + 1):
        Dz = (1 - z * z)[:, None] * az.mat(2) - (2 * (Mp + 1) * z)[:, None] * az.mat(1) - Mp * (Mp + 1) * az.mat(0)
        kz = max(kz, np.linalg.cond(np.linalg.eig(np.linalg.solve(az.mat(0), Dz))[1]))
    for l in (0, wl["J"] + az.n - 1):
        A = -ax.mat(2) + ((l * (l + 1) / x ** 2) - 2 / x)[:, None] * ax.mat(0)
        kx = max(kx, np.linalg.cond(np.linalg.eig(np.linalg.solve(ax.mat(0), A))[1]))
    return 4 * max(az.n, ax.n) * np.finfo(float).eps * kz * kx


# interval counts (n_x = 2 N, n_y = 2 N, n_z = 2 N + 2; quintic 3 N + 1, 3 N + 1, 3 N + 3)
SIZES = [((1, 2, 1), 0, 0), ((8, 3, 3), 0, 0), ((31, 32, 2), 0, 1), ((32, 33, 4), 0, 0), ((33, 16, 3), 0, 2),
         ((64, 17, 2), 0, 0), ((65, 8, 3), 0, 1), ((96, 5, 3), 0, 0), ((97, 31, 2), 0, 0), ((128, 9, 2), 0, 0),
         ((129, 4, 2), 0, 0), ((6, 5, 31), 0, 0), ((5, 6, 9), 0, 3), ((21, 11, 2), 1, 0), ((7, 8, 3), 1, 2)]


@pytest.mark.parametrize("n,basis,J", SIZES)
def test_tensor_core_float64_equals_cuda_cores(pkg, n, basis, J):
    wl = make_workload("He", J, nint=n, R=(20.0, 17.0), basis=basis)
    N = pkg.Context(wl, restart_m=2, ncv=3).n
    v = torch.tensor(rand_vec(N, 11), device="cuda")
    a, b = _pair(pkg, wl, -2.4, v)
    assert (torch.linalg.norm(a - b) / torch.linalg.norm(b)).item() < _bound(wl)


def test_y_diagonalised_form(pkg):
    wl = make_workload("He", 0, nint=(17, 20, 4), R=(20.0, 17.0))
    N = pkg.Context(wl, restart_m=2, ncv=3).n
    v = torch.tensor(rand_vec(N, 12), device="cuda")
    a, b = _pair(pkg, wl, -2.4, v, y_solver=2)
    assert (torch.linalg.norm(a - b) / torch.linalg.norm(b)).item() < _bound(wl)


@pytest.mark.parametrize("scale", [1e-290, 1e-200, 1e200, 1e290])
def test_scales(pkg, scale):
    """The result is linear: a scaled input gives the scaled output, also beyond the splitting's exponent range."""
    wl = make_workload("He", 0, nint=(9, 7, 3), R=(20.0, 17.0))
    N = pkg.Context(wl, restart_m=2, ncv=3).n
    v = torch.tensor(rand_vec(N, 13), device="cuda")
    ref = _pair(pkg, wl, -2.4, v)[1]
    got = _pair(pkg, wl, -2.4, v * scale)[0] / scale
    assert (torch.linalg.norm(got - ref) / torch.linalg.norm(ref)).item() < _bound(wl)


def test_zero_and_non_finite_inputs(pkg):
    wl = make_workload("He", 0, nint=(9, 7, 3), R=(20.0, 17.0))
    N = pkg.Context(wl, restart_m=2, ncv=3).n
    z = torch.zeros(N, dtype=torch.float64, device="cuda")
    assert not _pair(pkg, wl, -2.4, z)[0].any().item()
    for bad in (np.inf, np.nan):
        v = torch.tensor(rand_vec(N, 14), device="cuda")
        v[5] = bad
        a, b = _pair(pkg, wl, -2.4, v)
        fa, fb = torch.isfinite(a), torch.isfinite(b)
        assert torch.equal(fa, fb)
        if fb.any():
            assert (torch.linalg.norm(a[fb] - b[fb]) / torch.linalg.norm(b[fb])).item() < _bound(wl)
