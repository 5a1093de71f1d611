"""Omega read out in pieces while later pieces are solved (rm_collision_strengths after a solve of more than 64 MB of
rows) against the streamed read-out, which copies after everything: the same bits, for one and for several solves on
the grid, after a reset, for solves in several blocks of energies, the interpolation, pageable and page-locked
output, and on a lane."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1909_07321_gb300 import rmgb, synth  # noqa: E402

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]

M = 6100   # 64 levels: 101 MB of rows, three pieces


def wave():
    pws, _ = synth.workload_64ch(2)
    return pws[0]


@pytest.mark.parametrize("kw,mode", [(dict(precision=2, solve_precision=1), 0), (dict(precision=2, solve_precision=1), 1),
                                     (dict(precision=2, solve_precision=1, mem_budget=40 << 20), 0),
                                     (dict(precision=2, solve_precision=1), "qdt")])
def test_same_as_whole_copy(kw, mode):
    E = synth.midpoint_grid(0.01, 2.5, M)
    with rmgb.Context(**kw) as ctx:
        ctx.load_pw(0, wave())
        ctx.load_pw(1, dict(wave(), g=2.5))
        tri = 64 * 65 // 2

        def solve(w):
            if mode == "qdt":
                ctx.solve_energies_qdt(w, E, -30)
            else:
                ctx.solve_energies(w, E, mode)

        def whole(*waves):
            out = torch.empty((M, tri), dtype=torch.float64, pin_memory=True).numpy()
            for w in waves:
                solve(w)
            ctx.collision_strengths_async(out, reset=True)
            ctx.sync()
            return out

        def parts(out, *waves):
            for w in waves:
                solve(w)
            return ctx.collision_strengths(out, reset=True)

        one, two = whole(0), whole(0, 1)
        assert not np.array_equal(one, two)
        pinned = torch.empty((M, tri), dtype=torch.float64, pin_memory=True).numpy()
        pageable = np.full((M, tri), np.nan)
        assert np.array_equal(parts(pinned, 0), one)
        assert np.array_equal(parts(pageable, 0), one)
        assert np.array_equal(parts(pinned, 0, 1), two)
        # read without reset, then more on top, then a reset of the accumulator alone
        solve(0)
        assert np.array_equal(ctx.collision_strengths(pinned), one)
        solve(1)
        assert np.array_equal(ctx.collision_strengths(pinned), two)
        ctx.reset_omega()
        assert not ctx.collision_strengths(pinned).any()
        solve(0)
        assert np.array_equal(ctx.collision_strengths(pinned, reset=True), one)
        # a smaller grid afterwards
        ctx.solve_energies(0, E[:10], 0)
        assert ctx.collision_strengths(reset=True).shape == (10, tri)


def test_on_a_lane():
    E = synth.midpoint_grid(0.01, 2.5, M)
    tri = 64 * 65 // 2
    with rmgb.Context(precision=2, solve_precision=1, lanes=2, stream=0) as ctx:
        ctx.load_pw(0, wave())
        got = [np.empty((M, tri)) for _ in range(2)]
        for lane in (0, 1):
            ctx.lane_solve_energies(lane, 0, E)
        for lane in (1, 0):
            ctx.lane_collision_strengths(lane, got[lane], reset=True)
        assert np.array_equal(got[0], got[1])
        ctx.solve_energies(0, E)
        out = torch.empty((M, tri), dtype=torch.float64, pin_memory=True).numpy()
        ctx.collision_strengths_async(out, reset=True)
        ctx.sync()
        assert np.array_equal(out, got[0])
