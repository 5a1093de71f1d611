"""The choice between packed pairs and 64 x 64 tiles in the FP64 formation (csrc/formation_fp64.cu).

Both give every entry by the same operations: d_k = 1 / (E_k - E), products w_jk d_k rounded, one chain of FMAs over
ascending poles from zero, the sum times 0.5 / a. Entries on both sides of the lines where the choice changes (and
of the edges of tiles, warp loads and chunks) are that chain, formed with the C library's fma, to the bit; the chosen
kernel's rate per stored entry at the widest sizes is within an eighth of the one at 256 channels (tiles and packed
pairs run at the FP64 pipe; their padding differs by at most a tenth between these sizes, and the wrong kernel is a
quarter slower)."""
import ctypes
import ctypes.util

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1909_07321_gb300 import rmgb, synth  # noqa: E402

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]

libm = ctypes.CDLL(ctypes.util.find_library("m"))
libm.fma.restype = ctypes.c_double
libm.fma.argtypes = [ctypes.c_double] * 3


@pytest.mark.parametrize("n", [32, 63, 64, 65, 128, 129, 320, 384, 439, 448, 449, 503, 512, 513, 577, 640, 641, 784, 785,
                               1024])
def test_every_route_is_one_chain(n):
    N, m = 21, 2
    pw = synth.random_pw(60 + n, n, N, z=1.0, a=15.0, sigma=0.1)
    rng = np.random.default_rng(n)
    E = rng.uniform(0.01, 3.0, m)
    with rmgb.Context() as ctx:
        ctx.load_pw(0, pw)
        R = torch.full((m, n, n), float("nan"), dtype=torch.float64, device="cuda")
        ctx.form_r(0, torch.tensor(E, device="cuda"), R)
        ctx.sync()
        R = R.cpu().numpy()
    assert np.isfinite(R).all()
    W = pw["W"]
    at = [(0, 0), (0, n - 1), (n - 1, n - 1), (n // 2, n // 2)] + [tuple(sorted(p)) for p in rng.integers(0, n, (200, 2))]
    for e in range(m):
        d = 1.0 / (pw["E_k"] - E[e])
        for i, j in at:
            acc = 0.0
            for k in range(N):
                acc = libm.fma(W[i, k], W[j, k] * d[k], acc)
            assert R[e, i, j] == R[e, j, i] == acc * (0.5 / pw["a"]), (e, i, j)


@pytest.mark.parametrize("n,m", [(640, 100), (768, 64), (1024, 40)])
def test_no_wide_size_takes_the_slower_kernel(n, m):
    def rate(n, m):
        E = torch.tensor(synth.midpoint_grid(0.01, 2.5, m), device="cuda")
        R = torch.empty((m, n, n), dtype=torch.float64, device="cuda")
        with rmgb.Context() as ctx:
            ctx.load_pw(0, synth.random_pw(n, n, 1000, z=2.0, a=15.0))
            best = np.inf
            for _ in range(4):
                ctx.profile_enable(True)
                ctx.form_r(0, E, R)
                best = min(best, ctx.profile_get(rmgb.RM_PH_FORM)[1])
        return m * n * (n + 1) / 2 / best

    assert rate(n, m) >= 0.875 * rate(256, 600)
