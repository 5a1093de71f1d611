"""Elementwise kernels of the wide mixed path.

pe_reduce (csrc/formation_tc_energy.cu) sums the pole segments' floats exactly where their exponents allow and
plainly where not; both ways give the plain FP64 sum in segment order, which no entry point shows by itself, so R is
checked against 64-bit sums at 1 to 9 segments: the bound stated for the mixed formation (1e-4 of the sum of
magnitudes), on inputs whose segments differ by up to 2^60 (the plain branch), hold zeros, or are alike.
Assembly, classification, extraction and the collision-strength sums at row and column remainders of their 32 x 32
tiles, with open, eliminated and decaying channels in every number and levels of one to four channels: Omega
against the FP64 solver of the same formation, half of the energies within n 2^-18 (the FP32 solve's own error)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1909_07321_gb300 import rmgb, synth  # noqa: E402

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]


@pytest.mark.parametrize("N", [300, 4100, 8300, 30100, 33000])
@pytest.mark.parametrize("kind", ["alike", "spread", "zeros"])
def test_segment_sums(N, kind):
    n, a = 6, 15.0
    pw = synth.random_pw(N, n, N, z=2.0, a=a, sigma=0.05, pole_lo=-5.0, pole_hi=200.0)
    if kind == "spread":
        pw["W"] *= 2.0 ** np.repeat(np.linspace(0.0, 30.0, -(-N // 4096)).round(), 4096)[None, :N]
    elif kind == "zeros":
        pw["W"][:, : N // 2] = 0.0
        pw["W"][2] = 0.0
    E = np.array([0.3, 1.7, 5.0])
    with rmgb.Context(precision=rmgb.RM_BF16X3, formulation=rmgb.RM_FORM_ENERGY) as ctx:
        ctx.load_pw(0, pw)
        R = torch.zeros((3, n, n), dtype=torch.float64, device="cuda")
        ctx.form_r(0, torch.tensor(E, device="cuda"), R)
        ctx.sync()
        R = R.cpu().numpy()
    for e in range(3):
        d = 1.0 / (pw["E_k"] - E[e])
        ref, S = (pw["W"] * d) @ pw["W"].T / (2 * a), (abs(pw["W"]) * abs(d)) @ abs(pw["W"]).T / (2 * a)
        assert np.all(np.abs(R[e] - ref) <= 1e-4 * S)


@pytest.mark.parametrize("n,per,mode", [(97, 1, 0), (97, 4, 1), (127, 3, 1), (160, 2, 0), (193, 4, 1)])
def test_omega_against_fp64_solver(n, per, mode):
    pw = synth.random_pw(700 + n, n, 2 * n, z=2.0, a=15.0, e_max=1.5)
    level = (np.arange(n) // per).astype(np.int32)
    pw.update(level=level, n_levels=int(level[-1]) + 1, e_thr=pw["e_thr"][per * level])
    E = np.linspace(0.05, 1.7, 9)
    got = {}
    for sp in (rmgb.RM_FP64, rmgb.RM_FP32):
        with rmgb.Context(precision=rmgb.RM_BF16X3, solve_precision=sp) as ctx:
            ctx.load_pw(0, pw)
            no = torch.zeros(E.size, dtype=torch.int32, device="cuda")
            st = torch.zeros(E.size, dtype=torch.int32, device="cuda")
            ctx.solve_energies(0, E, mode, n_open_out=no, status_out=st)
            got[sp] = ctx.collision_strengths()
            assert not st.cpu().numpy().any()
            assert np.array_equal(no.cpu().numpy(), (E[:, None] > pw["e_thr"][None]).sum(1))
    ref, om = got[rmgb.RM_FP64], got[rmgb.RM_FP32]
    assert np.array_equal(ref == 0.0, om == 0.0)
    off = np.linalg.norm(om - ref, axis=1) / np.linalg.norm(ref, axis=1)
    assert np.median(off) <= n * 2.0 ** -18, off


@pytest.mark.parametrize("n", [1, 127, 128, 129, 255, 256, 257, 383, 385])
@pytest.mark.parametrize("prec", [rmgb.RM_BF16X3, rmgb.RM_FP32])
def test_formation_tiles(n, prec):
    """Per-energy formation where its 128 x 256 tiles are computed by halves: every entry within the mixed
    formation's bound (a half left out is an error of order one)."""
    pw = synth.random_pw(n, n, 2 * n + 70, z=2.0, a=15.0, sigma=0.05)
    E = np.array([0.3, 0.9, 2.2])
    with rmgb.Context(precision=prec, formulation=rmgb.RM_FORM_ENERGY) as ctx:
        ctx.load_pw(0, pw)
        R = torch.full((3, n, n), float("nan"), dtype=torch.float64, device="cuda")
        ctx.form_r(0, torch.tensor(E, device="cuda"), R)
        ctx.sync()
        R = R.cpu().numpy()
    for e in range(3):
        d = 1.0 / (pw["E_k"] - E[e])
        ref, S = (pw["W"] * d) @ pw["W"].T / 30.0, (abs(pw["W"]) * abs(d)) @ abs(pw["W"]).T / 30.0
        assert np.all(np.abs(R[e] - ref) <= 1e-4 * S)
