"""FP32 global-memory solver (csrc/dense_global_f32.cuh): every energy, not the middle one.

LU: where all channels are open, K is the solution of A K = B with A and B from the channel functions and R of the
same context; its residual stays below n 2^-24 (|A| |K| + |B|) in the Frobenius norm at every energy (elimination
with partial pivoting is backward stable; the constant n is the textbook's without its growth factor, some
hundred times what rounding gives in practice, and a wrong column, row or tile leaves a residual of order 1 / n).
Sweep: Omega from the K that the solve itself returned, W = (1 - iK)^{-1} in 64 bits; the error of W is at most
4 n 2^-24 times its condition number and size, whatever K is, at every energy and every number of open channels."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1909_07321_gb300 import rmgb, synth  # noqa: E402

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]

U = 2.0 ** -24


def solve(pw, E):
    n, m = pw["W"].shape[0], E.size
    with rmgb.Context(solve_precision=rmgb.RM_FP32, solver=rmgb.RM_SOLVER_LARGE) as ctx:
        ctx.load_pw(0, pw)
        Ed = torch.tensor(E, device="cuda")
        K = torch.zeros((m, n, n), dtype=torch.float64, device="cuda")
        no = torch.zeros(m, dtype=torch.int32, device="cuda")
        st = torch.zeros(m, dtype=torch.int32, device="cuda")
        ctx.solve_energies(0, E, 0, K_out=K, n_open_out=no, status_out=st)
        om = ctx.collision_strengths(reset=True)
        R = torch.zeros((m, n, n), dtype=torch.float64, device="cuda")
        f = torch.zeros((m, n, 4), dtype=torch.float64, device="cuda")
        ctx.form_r(0, Ed, R)
        ctx.channel_functions(0, Ed, f)
        ctx.sync()
    assert not st.cpu().numpy().any()
    return K.cpu().numpy(), no.cpu().numpy(), om, R.cpu().numpy(), f.cpu().numpy()


def check_omega(K, no, om, n, g):
    for e in range(len(no)):
        k = no[e]
        Ks = 0.5 * (K[e, :k, :k] + K[e, :k, :k].T)
        Z = np.eye(k) - 1j * Ks
        W = np.linalg.inv(Z)
        cond = np.linalg.norm(Z, 2) * np.linalg.norm(W, 2)
        ref = np.zeros((n, n))
        ref[:k, :k] = 4.0 * g * abs(W - np.eye(k)) ** 2
        ref = ref[np.triu_indices(n)]
        bound = 8.0 * g * np.linalg.norm(W - np.eye(k)) * 4.0 * k * U * cond * np.linalg.norm(W, 2)
        assert np.linalg.norm(om[e] - ref) <= bound, (e, k)


@pytest.mark.parametrize("n", [1, 5, 33, 63, 66, 97, 126, 129, 150, 190, 203, 257, 320, 331, 449, 513])
def test_all_open(n):
    pw = synth.random_pw(800 + n, n, n + 30, z=2.0, a=15.0, e_max=1.0, sigma=0.1)
    E = np.linspace(1.1, 2.6, 7) + 0.003
    K, no, om, R, f = solve(pw, E)
    assert (no == n).all()
    a, b = pw["a"], pw["b"]
    for e in range(E.size):
        s, sp, c, cp = f[e].T
        A, B = np.diag(c) - R[e] * (a * cp - b * c), R[e] * (a * sp - b * s) - np.diag(s)
        res = np.linalg.norm(A @ K[e] - B)
        assert res <= n * U * (np.linalg.norm(A) * np.linalg.norm(K[e]) + np.linalg.norm(B)), (e, res)
    check_omega(K, no, om, n, pw["g"])


@pytest.mark.parametrize("n", [40, 130, 260])
def test_every_number_of_open_channels(n):
    pw = synth.random_pw(860 + n, n, n + 30, z=2.0, a=15.0, e_max=1.5, sigma=0.1)
    thr = np.sort(pw["e_thr"])
    E = 0.5 * (thr[:-1] + thr[1:])
    E = E[np.diff(thr) > 1e-4][:: max(1, n // 65)]
    K, no, om, R, f = solve(pw, E)
    assert np.array_equal(no, (E[:, None] > thr[None]).sum(1))
    check_omega(K, no, om, n, pw["g"])
