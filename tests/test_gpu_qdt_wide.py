"""K-matrix interpolation (iqdt = 2) of 85 to 96 channels, past the size that the S-matrix form takes: with every energy
a node it is the quantum-defect solve, here of the global-memory solver. Both are backward stable, so Omega agrees to a
modest multiple of n 2^-52 except where a narrow resonance amplifies rounding: at least four fifths of the energies to
1e-10 (a wrong entry is an error of order one at every energy that has an eliminated channel)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1909_07321_gb300 import rmgb, synth  # noqa: E402

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]


@pytest.mark.parametrize("n", [84, 85, 91, 95, 96])
def test_every_energy_a_node(n):
    pw = synth.random_pw(500 + n, n, 3 * n + 20, z=2.0, a=15.0, e_max=1.2, l_max=4)
    E = np.sort(np.random.default_rng(n).uniform(0.3, 1.4, 25))
    got = {}
    for solver in (rmgb.RM_SOLVER_LARGE, rmgb.RM_SOLVER_AUTO):
        with rmgb.Context(solver=solver) as ctx:
            ctx.load_pw(0, pw)
            st = torch.zeros(E.size, dtype=torch.int32, device="cuda")
            if solver == rmgb.RM_SOLVER_LARGE:
                ctx.solve_energies(0, E, rmgb.RM_MQDT, status_out=st)
            else:
                ctx.solve_energies_qdt(0, E, -1, iqdt=2, status_out=st)
            got[solver] = ctx.collision_strengths(), st.cpu().numpy()
    (ref, st), (om, st2) = got[rmgb.RM_SOLVER_LARGE], got[rmgb.RM_SOLVER_AUTO]
    ok = (st == 0) & (st2 == 0)
    assert ok.sum() >= 20
    off = np.linalg.norm(om[ok] - ref[ok], axis=1) / np.linalg.norm(ref[ok], axis=1)
    assert np.quantile(off, 0.8) <= 1e-10, off
