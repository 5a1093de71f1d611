"""One context per host thread, both on one device: the shared-memory limit that a launch needs belongs to the kernel in
the whole process, so a smaller wave in one thread must not take it from a larger one in another between its being
set and the launch (that launch then fails). Two sizes of every solver and formation that share a kernel, in a tight
loop; the results of both threads are those of each alone, to the bit."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1909_07321_gb300 import rmgb, synth  # noqa: E402

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]

FP64 = dict()
FP32 = dict(solve_precision=rmgb.RM_FP32)
# context options, the two channel counts, what is called
CASES = [("form", FP64, (24, 31)), ("form", FP64, (300, 400)), ("form", dict(precision=rmgb.RM_BF16X3), (20, 60)),
         (rmgb.RM_DIRECT, FP64, (40, 64)), (rmgb.RM_MQDT, FP64, (40, 64)),
         (rmgb.RM_DIRECT, dict(solver=rmgb.RM_SOLVER_LARGE), (30, 120)),
         (rmgb.RM_DIRECT, FP32, (70, 90)), (rmgb.RM_DIRECT, dict(FP32, solver=rmgb.RM_SOLVER_LARGE), (20, 100)),
         ("prop", FP64, (4, 12)), ("prop", FP64, (20, 30)), ("qdt", FP64, (10, 24))]
CALLS = {"form": 4000}   # else 400


@pytest.mark.parametrize("what,opts,sizes", CASES)
def test_two_threads(what, opts, sizes):
    E = np.array([0.41, 0.83, 1.27])
    Ed = torch.tensor(E, device="cuda")
    waves = [synth.random_pw(300 + n, n, 8, z=2.0, a=15.0) for n in sizes]
    rng = np.random.default_rng(1)
    A = [rng.normal(0.0, 0.1, (1, n, n)) for n in sizes]
    A = [0.5 * (x + x.transpose(0, 2, 1)) for x in A]

    def work(i, calls):
        """The results of the last call and of the errors' count."""
        n = sizes[i]
        out = torch.zeros((3, n, n), dtype=torch.float64, device="cuda")
        with rmgb.Context(stream=0, **opts) as ctx:
            ctx.load_pw(0, waves[i])
            if what == "prop":
                ctx.set_multipoles(0, A[i], waves[i]["a"] + 1.0, 2)
            gate.wait()
            for _ in range(calls):
                if what == "form":
                    ctx.form_r(0, Ed, out)
                elif what == "qdt":
                    ctx.solve_energies_qdt(0, E, -1)
                else:
                    ctx.solve_energies(0, Ed, rmgb.RM_DIRECT if what == "prop" else what, K_out=out)
                if what != "form" and _ + 1 < calls:
                    ctx.reset_omega()
            ctx.sync()
            return out.cpu().numpy(), None if what == "form" else ctx.collision_strengths(reset=True)

    def run(i, calls, res):
        try:
            res[i] = work(i, calls)
        except Exception as e:   # noqa: BLE001 - reported below
            res[i] = e

    alone, got = {}, {}
    for i in (0, 1):
        gate = threading.Barrier(1)
        run(i, 1, alone)
        assert not isinstance(alone[i], Exception), alone[i]
    gate = threading.Barrier(2)
    threads = [threading.Thread(target=run, args=(i, CALLS.get(what, 400), got)) for i in (0, 1)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for i in (0, 1):
        assert not isinstance(got[i], Exception), got[i]
        assert np.array_equal(got[i][0], alone[i][0])
        if what != "form":
            assert np.array_equal(got[i][1], alone[i][1])
