"""An expired device wait (its flag set here by hand, between calls) is reported once, by the next call that reads it,
and does not condemn the context: the call after it gives what a fresh context gives."""
import ctypes

import pytest

from fm_inputs import make_workload, rand_vec

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
TIMEOUT = -10


def _flag(pkg, ctx):
    fn = pkg.lib()["_ZN3fmi12tc_flag_slotEP6fm_ctx"]
    fn.argtypes, fn.restype = [ctypes.c_void_p], ctypes.c_void_p

    class Slot:
        __cuda_array_interface__ = {"shape": (1,), "typestr": "<i4", "data": (fn(ctx.h), False), "version": 3}
    return torch.as_tensor(Slot(), device="cuda")


# precision, mma, call: the reader of the flag is the multi-dot, the end of the solve, or the preconditioner
CASES = [(0, 0, "solve"), (1, 0, "solve"), (1, 1, "solve"), (2, 0, "solve"), (0, 0, "eigs"), (1, 0, "eigs"), (1, 0, "precond")]


@pytest.mark.parametrize("precision,mma,call", CASES)
def test_reported_once(precision, mma, call):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2005_05398_gb300 as pkg
    wl = make_workload("He", 0, nint=(8, 8, 3), R=(20.0, 20.0))
    ctx = pkg.Context(wl, precision=precision, mma=mma)
    v = torch.tensor(rand_vec(ctx.n, 6), device="cuda")
    ctx.fm_set_shift(-2.95)

    def run():
        out = torch.zeros_like(v)
        if call == "solve":
            ctx.fm_solve(-2.95, v, out)
        elif call == "eigs":
            ctx.fm_eigs(-2.95, 1, v, out)
        else:
            ctx.fm_precond_apply(v, out)
        torch.cuda.synchronize()
        return out
    ref = run()
    _flag(pkg, ctx).fill_(1)
    torch.cuda.synchronize()
    with pytest.raises(pkg._lib.FMError) as e:
        run()
    assert e.value.code == TIMEOUT
    assert torch.equal(run(), ref)
    ctx.close()


def test_breakdown_of_an_expired_wait_is_a_timeout():
    """What an expired wait leaves is NaN: a solve that breaks down on it names the wait."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2005_05398_gb300 as pkg
    ctx = pkg.Context(make_workload("He", 0, nint=(8, 8, 3), R=(20.0, 20.0)))
    v = torch.full((ctx.n,), float("nan"), dtype=torch.float64, device="cuda")
    out = torch.zeros_like(v)
    _flag(pkg, ctx).fill_(1)
    torch.cuda.synchronize()
    with pytest.raises(pkg._lib.FMError) as e:
        ctx.fm_solve(-2.95, v, out)
    assert e.value.code == TIMEOUT
    with pytest.raises(pkg._lib.FMError) as e:
        out.zero_()
        ctx.fm_solve(-2.95, v, out)
    assert e.value.code == -5
    ctx.close()
