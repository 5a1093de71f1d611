"""FP32 global-memory solver (csrc/dense_global_f32.cuh) at the edges of its dispatch (panel rows per thread,
threads, strip and tile remainders, operand forms of the widest systems) against the same solve in FP64 from the
same R (FP64 formation in both contexts).

The FP32 elimination is backward stable (partial pivoting) and the sweep inverts a matrix whose Hermitian part is
the identity, so per energy Omega differs by a modest multiple of n 2^-24 in the median; the bound taken is
n 2^-18 of the row's norm for at least half of the energies (a wrong entry, strip or permutation is an error of
order one at every energy)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1909_07321_gb300 import rmgb, synth  # noqa: E402

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]


def omega(pw, E, sp, mode):
    with rmgb.Context(precision=rmgb.RM_FP64, solve_precision=sp, solver=rmgb.RM_SOLVER_LARGE) as ctx:
        ctx.load_pw(0, pw)
        st = torch.zeros(E.size, dtype=torch.int32, device="cuda")
        ctx.solve_energies(0, E, mode, status_out=st)
        om = ctx.collision_strengths()
        assert not st.cpu().numpy().any()
        return om


@pytest.mark.parametrize("n,m,mode", [(1, 3, 0), (2, 3, 0), (31, 4, 0), (33, 4, 1), (64, 4, 0), (97, 4, 0), (127, 4, 1),
                                      (129, 4, 0), (256, 3, 0), (257, 3, 0), (511, 2, 0), (513, 2, 0), (1025, 2, 0),
                                      (1510, 2, 0)])
def test_against_fp64_solve(n, m, mode):
    # thresholds over most of the energy range: open and closed channels in every number
    pw = synth.random_pw(900 + n, n, max(8, 2 * n if n < 600 else 200), z=2.0, a=15.0, e_max=1.5, sigma=0.1)
    E = np.linspace(0.11, 1.61, m) + 0.003
    ref, got = omega(pw, E, rmgb.RM_FP64, mode), omega(pw, E, rmgb.RM_FP32, mode)
    off = np.linalg.norm(got - ref, axis=1) / np.linalg.norm(ref, axis=1)
    assert np.isfinite(off).all()
    assert np.median(off) <= max(n, 16) * 2.0 ** -18, off


@pytest.mark.parametrize("n", [5, 97, 128, 257, 300, 448])
def test_many_energies_as_few(n):
    """More energies than fit at once take smaller CTAs (up to 128 and 448 channels): the same bits."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    m = 2 * ((2 * sms if n <= 128 else sms) // 2 + 4)
    pw = synth.random_pw(700 + n, n, n + 20, z=2.0, a=15.0, e_max=1.5, sigma=0.1)
    E = np.linspace(0.11, 1.61, m) + 0.003
    Ks, oms = [], []
    for parts in (1, 2):
        with rmgb.Context(precision=rmgb.RM_FP64, solve_precision=rmgb.RM_FP32, solver=rmgb.RM_SOLVER_LARGE) as ctx:
            ctx.load_pw(0, pw)
            K = torch.zeros((m, n, n), dtype=torch.float64, device="cuda")
            om = []
            for x, k in zip(np.split(E, parts), torch.split(K, m // parts)):
                ctx.solve_energies(0, x, 0, K_out=k)
                om.append(ctx.collision_strengths(reset=True))
            Ks.append(K.cpu().numpy())
            oms.append(np.concatenate(om))
    assert np.array_equal(Ks[0], Ks[1])
    assert np.array_equal(oms[0], oms[1])
