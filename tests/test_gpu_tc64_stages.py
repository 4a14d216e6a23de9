"""Each float64 digit stage by itself: z forward, z inverse, x forward and x inverse against sums of more than 53 bits,
no less accurate than the float64 multiply-add chain (which the kernel itself runs on columns scaled beyond its
exponent range: that also yields its matrices, from unit columns).  Inputs: white noise, and mode amplitudes as the
chain gives them (a smooth vector through the forward stage, high modes damped), at tile edges of both forms."""
import ctypes

import numpy as np
import pytest

from fm_inputs import make_workload

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# (n_x, n_y, n_z) intervals, basis, J, x box: contraction lengths 8 .. 256 on both sides of 64, 128 and 192
CASES = [((6, 9, 3), 0, 0, 20.0), ((8, 7, 8), 0, 2, 20.0), ((10, 6, 24), 0, 1, 20.0), ((6, 8, 12), 0, 10, 20.0),
         ((5, 6, 31), 0, 0, 20.0), ((5, 6, 32), 0, 1, 20.0), ((4, 4, 63), 0, 0, 20.0), ((3, 4, 8), 1, 4, 12.0),
         ((6, 4, 7), 1, 2, 20.0), ((33, 16, 1), 0, 0, 40.0), ((64, 12, 1), 0, 1, 80.0), ((96, 10, 1), 0, 0, 40.0),
         ((97, 9, 1), 0, 0, 40.0), ((128, 12, 1), 0, 0, 40.0), ((55, 6, 1), 1, 1, 45.0),
         ((9, 8, 33), 0, 1, (20.0, (10, 6, 4))), ((128, 5, 2), 0, 0, (40.0, (50, 7, 5)))]  # (component 3's own grid)


@pytest.fixture(scope="module")
def pkg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2005_05398_gb300 as p
    return p


class Stage:
    """One stage of every component: x, a list of [slab][K][N] arrays, to the same of products."""

    def __init__(self, pkg, ctx, stage):
        self.ctx, self.stage = ctx, stage
        self.fn = pkg.lib()["_ZN3fmi9f64_stageEP6fm_ctxiPKdPd"]
        self.fn.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_void_p, ctypes.c_void_p]
        self.fn.restype = ctypes.c_int
        self.shapes = [(ctx.nM, c["nz"], c["nx"] * c["ny"]) if stage < 2 else (ctx.nM * c["nz"], c["nx"], c["ny"])
                       for c in ctx.components]

    def __call__(self, xs):
        flat = [(x.swapaxes(1, 2) if self.stage == 3 else x).reshape(-1) for x in xs]
        a = torch.tensor(np.concatenate(flat), device="cuda")
        b = torch.full_like(a, 7.0)
        assert self.fn(self.ctx.h, self.stage, a.data_ptr(), b.data_ptr()) == 0
        torch.cuda.synchronize()
        out, off = [], 0
        for s, k, n in self.shapes:
            v = b[off:off + s * k * n].cpu().numpy()
            out.append(v.reshape(s, n, k).swapaxes(1, 2) if self.stage == 2 else v.reshape(s, k, n))
            off += s * k * n
        return out

    def matrices(self):
        """W of every slab, from unit columns of 2^700."""
        ws = [np.zeros((s, k, k)) for s, k, n in self.shapes]
        for p in range(max((k + n - 1) // n for s, k, n in self.shapes)):
            xs = []
            for s, k, n in self.shapes:
                x = np.zeros((s, k, n))
                for c in range(min(n, k - p * n)):
                    x[:, p * n + c, c] = 2.0 ** 700
                xs.append(x)
            for w, y, (s, k, n) in zip(ws, self(xs), self.shapes):
                cols = max(0, min(n, k - p * n))
                w[:, :, p * n:p * n + cols] = y[:, :, :cols] * 2.0 ** -700
        return ws

    def chain(self, xs):
        """The float64 chain: the same columns beyond the digits' exponent range."""
        return [y * 2.0 ** -800 for y in self([x * 2.0 ** 800 for x in xs])]


@pytest.mark.parametrize("n,basis,J,R", CASES)
def test_no_less_accurate_than_the_float64_chain(pkg, n, basis, J, R):
    R, n3 = R if isinstance(R, tuple) else (R, None)
    wl = make_workload("He", J, nint=n, R=(R, 17.0), basis=basis)
    if n3:
        wl["grids"] = {1: {"nint": n, "R": (R, 17.0)}, 3: {"nint": n3, "R": (9.0, 8.0)}}
    ctx = pkg.Context(wl, restart_m=2, ncv=3)
    rng = np.random.default_rng(sum(n) + J)
    stages = [Stage(pkg, ctx, s) for s in range(4)]
    W = [st.matrices() for st in stages]
    for fwd, inv in ((0, 1), (2, 3)):
        kinds = {}
        white = [rng.standard_normal(sh) for sh in stages[fwd].shapes]
        kinds["white"] = (white, white)
        smooth = [np.exp(-4.0 * np.arange(k) / k)[None, :, None] * (1.0 + 0.1 * rng.random((s, 1, c)))
                  for s, k, c in stages[fwd].shapes]
        modes = []
        for x, w in zip(smooth, W[fwd]):
            k = np.arange(x.shape[1])
            m = (w @ x) / (1.0 + k * (k + 1.0))[None, :, None]
            modes.append(m / np.exp2(np.floor(np.log2(np.abs(m).max(axis=1, keepdims=True)))))
        kinds["modes"] = (smooth, modes)
        for name, (xf, xi) in kinds.items():
            for s, xs in ((fwd, xf), (inv, xi)):
                got, chain = stages[s](xs), stages[s].chain(xs)
                for w, x, y, z in zip(W[s], xs, got, chain):
                    cols = np.unique(np.linspace(0, x.shape[2] - 1, 24).astype(int))
                    for b in range(len(x)):
                        ref = w[b].astype(np.longdouble) @ x[b][:, cols].astype(np.longdouble)
                        nrm = np.linalg.norm(ref.astype(float))
                        err = np.linalg.norm((y[b][:, cols] - ref).astype(float)) / nrm
                        e64 = np.linalg.norm((z[b][:, cols] - ref).astype(float)) / nrm
                        # one rounding beside the chain's error
                        assert err <= e64 + 2.0 ** -53, (name, s, b, err, e64)
    ctx.close()
