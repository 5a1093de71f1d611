"""FP64 formation of R (csrc/formation_fp64.cu) over the edges of its dispatch: one warp to several CTAs an
energy, 1 to 31 channels (quotients), the three chunk lengths, the tiled kernel above 1024 channels, pole
counts around a chunk. Every entry is a chain of N FMAs of terms with at most 4 roundings each, scaled once:
|R - exact| <= (N + 5) 2^-53 sum |w_i w_j d| / 2a."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1909_07321_gb300 import rmgb, synth  # noqa: E402

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]


@pytest.mark.parametrize("n,N,m", [(1, 1, 1), (2, 15, 3), (7, 16, 2), (8, 17, 2), (15, 33, 2), (16, 31, 2), (31, 100, 2),
                                   (32, 64, 2), (33, 47, 3), (64, 129, 2), (97, 40, 2), (256, 33, 1), (257, 25, 1),
                                   (512, 9, 1), (513, 21, 1), (1024, 18, 1), (1025, 18, 1)])
def test_against_extended_sums(n, N, m):
    pw = synth.random_pw(40 + n, n, N, z=1.0, a=15.0, sigma=0.1)
    E = np.random.default_rng(n).uniform(0.01, 3.0, m)
    with rmgb.Context() as ctx:
        ctx.load_pw(0, pw)
        R = torch.full((m, n, n), float("nan"), dtype=torch.float64, device="cuda")
        ctx.form_r(0, torch.tensor(E, device="cuda"), R)
        ctx.sync()
        R = R.cpu().numpy()
    W, a = pw["W"].astype(np.longdouble), np.longdouble(pw["a"])
    for e in range(m):
        d = 1 / (pw["E_k"].astype(np.longdouble) - np.longdouble(E[e]))
        ref, S = (W * d) @ W.T / (2 * a), (abs(W) * abs(d)) @ abs(W).T / (2 * a)
        assert np.array_equal(R[e], R[e].T)
        assert np.all(np.abs(R[e] - ref) <= (N + 5) * 2.0 ** -53 * S)
