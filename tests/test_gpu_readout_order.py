"""rm_collision_strengths is ordered after everything on the context's stream: what the caller enqueues there between a
solve and the read-out (the stream is torch's by default, or was asked for with rm_lane_stream) runs before a byte of
omega_out is written, and what it adds to Omega is in it. The reference is the streamed read-out or a second context
that nothing was enqueued between. Solves of several pieces' size and solves in several blocks of energies."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1909_07321_gb300 import rmgb, synth  # noqa: E402

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]

TRI = 64 * 65 // 2
MIXED = dict(precision=rmgb.RM_BF16X3, solve_precision=rmgb.RM_FP32)
# 101 MB of rows in one block; 25 MB (and 101 MB) in several
SIZES = [(6100, {}), (1500, dict(mem_budget=8 << 20)), (6100, dict(mem_budget=40 << 20))]


def load(ctx):
    pw = synth.workload_64ch(2)[0][0]
    ctx.load_pw(0, pw)
    ctx.load_pw(1, dict(pw, g=2.5))


def solve(ctx, kind, w, E):
    if kind == "qdt":
        ctx.solve_energies_qdt(w, E, -30)
    else:
        ctx.solve_energies(w, E, kind)


def pinned(m):
    return torch.empty((m, TRI), dtype=torch.float64, pin_memory=True)


def expected(m, more, kind, waves):
    """Omega of the waves on a context of its own, read out by the streamed call (None: not at all)."""
    E = synth.midpoint_grid(0.01, 2.5, m)
    out = pinned(m).numpy()
    with rmgb.Context(stream=0, **MIXED, **more) as ctx:
        load(ctx)
        for w in waves:
            solve(ctx, kind, w, E)
        ctx.collision_strengths_async(out, reset=True)
        ctx.sync()
    return out


@pytest.mark.parametrize("kind", [rmgb.RM_DIRECT, rmgb.RM_MQDT, "qdt"])
@pytest.mark.parametrize("handed_out", [False, True])
@pytest.mark.parametrize("m,more", SIZES)
def test_upload_of_the_last_rows_before_the_read_out(m, more, kind, handed_out):
    """A loop that sends the rows it read last time back to the device, on the same stream, after it has enqueued the
    next solve: the upload takes the old rows, the read-out brings the new ones."""
    E = synth.midpoint_grid(0.01, 2.5, m)
    new = expected(m, more, kind, [0])
    with rmgb.Context(**(dict(stream=0) if handed_out else {}), **MIXED, **more) as ctx:
        load(ctx)
        s = torch.cuda.ExternalStream(ctx.lane_stream(0)) if handed_out else torch.cuda.current_stream()
        omega = pinned(m)
        dev = torch.empty((m, TRI), dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        got = []
        for old in (-1.0, -2.0):   # the lane's first solve and one after a blocking read-out
            omega.fill_(old)
            solve(ctx, kind, 0, E)
            with torch.cuda.stream(s):
                dev.copy_(omega, non_blocking=True)
            ctx.collision_strengths(omega.numpy(), reset=True)
            got.append((int((dev != old).any(dim=1).sum()), int((omega.numpy() != new).any(axis=1).sum())))
        del omega, dev   # while the stream they were used on is there
        torch.cuda.synchronize()
    assert got == [(0, 0), (0, 0)]   # rows of the upload, of the read-out, that are not what they should be


@pytest.mark.parametrize("m,more", SIZES)
def test_replay_of_a_captured_solve_before_the_read_out(m, more):
    """A solve that the caller captured on the context's stream and replays adds its wave to what is read out."""
    Eh = synth.midpoint_grid(0.01, 2.5, m)
    one, two = expected(m, more, 0, [0]), expected(m, more, 0, [0, 1])
    assert not np.array_equal(one, two)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s), rmgb.Context(**MIXED, **more) as ctx:
        load(ctx)
        E = torch.tensor(Eh, device="cuda")
        omega = pinned(m).numpy()
        for w in (0, 1):   # workspaces and operands of both waves
            ctx.solve_energies(w, E)
        s.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            ctx.solve_energies(1, E)
        ctx.collision_strengths(omega)
        for _ in range(2):
            ctx.reset_omega()
            ctx.solve_energies(0, E)
            graph.replay()
            assert np.array_equal(ctx.collision_strengths(omega), two)
        ctx.reset_omega()
        ctx.solve_energies(0, E)
        assert np.array_equal(ctx.collision_strengths(omega), one)
        del graph


@pytest.mark.parametrize("kind", [rmgb.RM_DIRECT, rmgb.RM_MQDT, "qdt"])
@pytest.mark.parametrize("m,more", SIZES)
def test_on_a_stream_of_the_contexts_own(m, more, kind):
    """Nothing of the caller's can lie between: blocking read-outs (first, after another, after further waves, page-
    locked and pageable, as one call and as two) bring the rows of the streamed one."""
    E = synth.midpoint_grid(0.01, 2.5, m)
    one, two = expected(m, more, kind, [0]), expected(m, more, kind, [0, 1])
    with rmgb.Context(stream=0, **MIXED, **more) as ctx:
        load(ctx)
        outs = [pinned(m).numpy(), np.full((m, TRI), np.nan)]
        for out in outs:
            solve(ctx, kind, 0, E)
            assert np.array_equal(ctx.collision_strengths(out, reset=True), one)
            solve(ctx, kind, 0, E)
            assert np.array_equal(ctx.collision_strengths(out), one)
            solve(ctx, kind, 1, E)
            assert np.array_equal(ctx.collision_strengths(out), two)
            assert np.array_equal(ctx.collision_strengths(out, reset=True), two)


def test_rows_beside_the_solve_only_into_page_locked_memory():
    """Pageable memory takes many small copies several times more slowly than one, so a solve after a read-out into it
    is not cut up: on the context's own stream it has the launches that it has on a caller's, and so once the stream
    was asked for; after a read-out into page-locked memory it has more."""
    m = 6100
    E = synth.midpoint_grid(0.01, 2.5, m)
    locked, pageable = pinned(m).numpy(), np.empty((m, TRI))

    def launches(ctx, out):
        """of the solve after a read-out into `out`"""
        ctx.solve_energies(0, E)
        ctx.collision_strengths(out, reset=True)
        before = ctx.launch_count()
        ctx.solve_energies(0, E)
        n = ctx.launch_count() - before
        ctx.collision_strengths(out, reset=True)
        return n

    with rmgb.Context(**MIXED) as ctx:
        load(ctx)
        whole = launches(ctx, locked)
        assert launches(ctx, pageable) == whole
    want = locked.copy()
    with rmgb.Context(stream=0, **MIXED) as ctx:
        load(ctx)
        assert launches(ctx, pageable) == whole
        assert np.array_equal(pageable, want)
        assert launches(ctx, locked) > whole
        assert np.array_equal(locked, want)
        assert launches(ctx, pageable) == whole
        ctx.lane_stream(0)
        assert launches(ctx, locked) == whole
        assert np.array_equal(locked, want)
