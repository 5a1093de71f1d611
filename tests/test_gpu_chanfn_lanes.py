"""Channel functions without tables (four or eight lanes per pair, csrc/channel_functions.cu): a pair's values do not depend
on which pairs share its warp, its block or its list. All energies in one call against each alone, to the bit: pair
counts around a block of 32, ladder lengths around a chunk of four l, fractions of very different depths side by
side, pairs deep enough for the list, z = 0 on both sides of the distance from which its vanishing fractions are not
run; channel functions directly, and K of both modes."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1909_07321_gb300 import rmgb, synth  # noqa: E402

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]


@pytest.mark.parametrize("n,m,z,ls", [(1, 1, 1.0, [0]), (1, 33, 2.0, [3]), (3, 11, 2.0, [0, 1, 4]),
                                      (4, 8, 3.0, [5, 8, 3, 12]), (2, 17, 1.0, [9, 20]), (3, 13, 0.0, [0, 1, 5]),
                                      (5, 13, 2.0, [0, 2, 4, 6, 7])])
def test_alone_and_together(n, m, z, ls):
    pw = synth.random_pw(77, n, 20, z=z, a=15.0, e_max=1.5)
    pw["l"][:] = ls
    E = np.random.default_rng(n * m).uniform(0.02, 2.5, m)
    if m > 4:
        E[:4] = pw["e_thr"][-1] + np.array([3e-5, -3e-5, 1e-6, -4e-6])
    with rmgb.Context(channel_tables=0) as ctx:
        ctx.load_pw(0, pw)

        def functions(x):
            out = torch.zeros((x.size, n, 4), dtype=torch.float64, device="cuda")
            ctx.channel_functions(0, torch.tensor(x, device="cuda"), out)
            ctx.sync()
            return out.cpu().numpy()

        def k_matrices(x, mode):
            K = torch.zeros((x.size, n, n), dtype=torch.float64, device="cuda")
            ctx.solve_energies(0, x, mode, K_out=K)
            ctx.collision_strengths(reset=True)
            return K.cpu().numpy()

        for f in (functions, lambda x: k_matrices(x, 0), lambda x: k_matrices(x, 1)):
            whole = f(E)
            assert np.isfinite(whole).all() and whole.any()
            for e in range(m):
                assert np.array_equal(whole[e], f(E[e:e + 1])[0]), e


@pytest.mark.parametrize("z", [0.0, 2.0])
def test_eight_lanes_against_four(z):
    """More than 16384 pairs take four lanes each, fewer eight: the same bits either way."""
    n, m = 9, 2400
    pw = synth.random_pw(5, n, 30, z=z, a=15.0, e_max=1.5, l_max=12)
    E = np.sort(np.random.default_rng(1).uniform(0.02, 2.5, m))
    with rmgb.Context(channel_tables=0) as ctx:
        ctx.load_pw(0, pw)
        got = []
        for parts in (1, 2):
            K = torch.zeros((m, n, n), dtype=torch.float64, device="cuda")
            for mode in (0, 1):
                for x, k in zip(np.split(E, parts), torch.split(K, m // parts)):
                    ctx.solve_energies(0, x, mode, K_out=k)
                    ctx.collision_strengths(reset=True)
                got.append(K.cpu().numpy())
        assert np.array_equal(got[0], got[2]) and np.array_equal(got[1], got[3])
