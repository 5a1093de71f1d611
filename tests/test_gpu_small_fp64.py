"""FP64 quantum-defect solves: the shared-memory solver (its elimination now shares the direct mode's layout), the
global-memory solver and the coarse-mesh interpolation with every energy a node are three routes to the same Omega.

Each route is backward stable (partial pivoting), so Omega agrees to a modest multiple of n 2^-52 except where a
narrow resonance amplifies rounding: at least half of the energies to 1e-10 (a wrong entry is an error of order
one at every energy that has an eliminated channel)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1909_07321_gb300 import rmgb, synth  # noqa: E402

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]


def run(pw, E, solver=rmgb.RM_SOLVER_AUTO, iqdt=0):
    with rmgb.Context(solver=solver) as ctx:
        ctx.load_pw(0, pw)
        st = torch.zeros(E.size, dtype=torch.int32, device="cuda")
        if iqdt:
            ctx.solve_energies_qdt(0, E, -1, iqdt=iqdt, status_out=st)
        else:
            ctx.solve_energies(0, E, rmgb.RM_MQDT, status_out=st)
        return ctx.collision_strengths(), st.cpu().numpy()


@pytest.mark.parametrize("n", [1, 2, 3, 31, 32, 33, 64, 84, 95, 96])
def test_three_routes(n):
    pw = synth.random_pw(500 + n, n, 3 * n + 20, z=2.0, a=15.0, e_max=1.2, l_max=4)
    E = np.sort(np.random.default_rng(n).uniform(0.3, 1.4, 25))
    ref, st = run(pw, E, solver=rmgb.RM_SOLVER_LARGE)
    routes = [run(pw, E)]
    if n <= 84:   # the interpolation's complex system fits shared memory
        routes += [run(pw, E, iqdt=1), run(pw, E, iqdt=2)]
    for got, st2 in routes:
        ok = (st == 0) & (st2 == 0)
        assert ok.sum() >= 20
        off = np.linalg.norm(got[ok] - ref[ok], axis=1) / np.linalg.norm(ref[ok], axis=1)
        assert np.median(off) <= 1e-10, off
