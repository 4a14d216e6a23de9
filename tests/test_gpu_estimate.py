"""fm_estimate_bytes is within a few percent of what a context holds, also where the two sources of a mirrored component
share their taps and where the float32 application needs no scratch planes (few Krylov vectors, so that the tables
count)."""
import pytest

from fm_inputs import make_workload

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 2])
@pytest.mark.parametrize("J,n,basis", [(0, (21, 21, 5), 1), (0, (32, 32, 10), 0), (1, (14, 14, 3), 1), (6, (16, 16, 6), 0)])
def test_estimate_within_five_percent(J, n, basis, precision):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2005_05398_gb300 as pkg
    from paper_2005_05398_gb300._lib import fm_estimate_bytes
    wl = make_workload("He", J, nint=n, R=(8.0, 8.0), basis=basis)
    est = fm_estimate_bytes(wl, restart_m=2, ncv=3, precision=precision)
    ctx = pkg.Context(wl, restart_m=2, ncv=3, precision=precision)
    ctx.fm_set_shift(-2.9)
    held = ctx.fm_stats()["device_bytes"]
    ctx.close()
    assert held <= est <= 1.05 * held, (held, est)
