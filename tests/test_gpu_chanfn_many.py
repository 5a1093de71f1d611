"""Channel functions without tables for very many pairs (csrc/channel_functions.cu): where the deep ones have a list of
their own, one thread a pair above 458752 pairs in direct mode and 720896 in the quantum-defect mode, four lanes
below: the same bits on both sides, in one call and in parts, with pairs near thresholds (deep fractions) among them.
And many pairs take the kernel of the higher rate: 2.1 million pairs of 64 channels in one launch take at most 0.7
times what they take in six (four lanes each) one after another (0.57 by the times of the two kernels, 0.83 if the
one launch is of four lanes as well)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1909_07321_gb300 import rmgb, synth  # noqa: E402

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]


def parts(z, mode, m, n_parts, n=24):
    pw = synth.random_pw(31, n, 30, z=z, a=15.0, e_max=1.5, l_max=9)
    E = np.sort(np.random.default_rng(2).uniform(0.02, 2.5, m))
    E[:n] = pw["e_thr"] + 4e-5 * np.where(np.arange(n) % 2, 1, -1) + 5e-4 * (np.arange(n) == 0)
    K = torch.zeros((m, n, n), dtype=torch.float64, device="cuda")
    st = torch.zeros(m, dtype=torch.int32, device="cuda")
    with rmgb.Context(channel_tables=0) as ctx:
        ctx.load_pw(0, pw)
        for x, k, s in zip(np.array_split(E, n_parts), torch.tensor_split(K, n_parts), torch.tensor_split(st, n_parts)):
            ctx.solve_energies(0, np.ascontiguousarray(x), mode, K_out=k, status_out=s)
            ctx.collision_strengths(reset=True)
    return K.cpu().numpy(), st.cpu().numpy()


@pytest.mark.parametrize("z", [1.0, 3.0])
@pytest.mark.parametrize("mode,m", [(0, 19114), (0, 19115), (1, 30037), (1, 30038)])
def test_one_thread_as_four_lanes(z, mode, m):
    whole, halves = parts(z, mode, m, 1), parts(z, mode, m, 2)
    assert whole[0].any() and np.isfinite(whole[0]).all()
    assert np.array_equal(whole[1], halves[1])
    assert np.array_equal(whole[0], halves[0])


def test_many_pairs_by_the_faster_kernel():
    n, m = 64, 32768
    E = synth.midpoint_grid(0.01, 2.5, m)
    with rmgb.Context(channel_tables=0) as ctx:
        ctx.load_pw(0, synth.random_pw(9, n, 10, z=2.0, a=15.0, e_max=2.0, l_max=8))

        def ms(n_parts):
            best = np.inf
            for _ in range(4):
                ctx.profile_enable(True)
                for x in np.array_split(E, n_parts):
                    ctx.solve_energies(0, np.ascontiguousarray(x))
                    ctx.collision_strengths(reset=True)
                best = min(best, ctx.profile_get(rmgb.RM_PH_CHANFN)[1])
            return best

        assert ms(1) <= 0.7 * ms(6)
