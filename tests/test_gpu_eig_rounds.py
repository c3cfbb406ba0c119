"""The eigen-steps' further rounds are taken where they are needed, and reported (rpca_plan_eig_rounds)."""
import numpy as np
import pytest

from oracle import rpca_oracle as O
from paper_2506_10257_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2506_10257_gb300 import rpca
    rpca.load()
    return rpca


def low_noise(T, m, noise):
    rng = np.random.Generator(np.random.PCG64(T))
    t = np.linspace(0, 1, T)
    X = rng.rayleigh(size=m) * (1 + 0.02 * t[:, None]) + 0.01 * rng.rayleigh(size=m) * np.cos(np.pi * t)[:, None]
    return (X + noise * rng.standard_normal((T, m))).astype(np.float32)


@pytest.mark.parametrize("T", [6, 20, 32, 50, 100])
def test_nearly_low_rank_windows_take_further_rounds(rp, T):
    # (all singular values count in the first step of a solve whose first mu is large)
    F = low_noise(T, 4096, 3e-4)
    mu0 = 1.25 / np.linalg.norm(F.astype(np.float64), 2)
    X = torch.from_numpy(F).cuda()
    plan = rp.Plan(4096, T, mu_init=1e5 * mu0)
    L, S, res = plan.solve(X)
    rounds = plan.eig_rounds()
    plan.close()
    assert rounds["further"] >= 1 and rounds["unfinished"] == 0
    # L + S = X to the solve's tolerance
    assert float(torch.linalg.norm((X - L - S).double())) <= 2e-7 * float(np.linalg.norm(F))


@pytest.mark.parametrize("T", [8, 20, 29, 32, 50, 100, 132])
def test_no_step_of_an_ordinary_window_runs_out_of_rounds(rp, T):
    w = synth.make_window(seed=T, ny=72, nx=61, T=T, n_bound=12, n_free=20).frames
    plan = rp.Plan(w.shape[1], T)
    assert plan.eig_rounds() == {"further": 0, "unfinished": 0}  # before the first solve
    _, _, res = plan.solve(torch.from_numpy(w).cuda())
    rounds = plan.eig_rounds()
    plan.close()
    assert res["iters"] == pytest.approx(O.rpca_frames(w).iters, abs=1)
    assert rounds["unfinished"] == 0 and rounds["further"] <= 2 * (res["iters"] + 1)


@pytest.mark.parametrize("noise", [1e-3, 3e-4, 1e-4])
@pytest.mark.parametrize("T", [20, 50, 100])
def test_nearly_low_rank_windows_keep_fp32_rounding(rp, T, noise):
    # a first mu at which all singular values count, though the Gram's FP32 sums leave it indefinite; bar: twice the FP32
    # rounding of the two T-term products (sqrt(T) u) and of the stored S, Y and L (4 u), relative to ||X||
    F = low_noise(T, 2048, noise)
    mu = 1e3 * 1.25 / np.linalg.norm(F.astype(np.float64), 2)
    plan = rp.Plan(2048, T, mu_init=mu)
    L, S, res = plan.solve(torch.from_numpy(F).cuda())
    plan.close()
    ref = O.rpca_frames(F, mu_init=mu, max_iter=res["iters"], tol=1e-30)
    bar = 2 * (np.sqrt(T) + 4) * 2.0 ** -24 * np.linalg.norm(F)
    eL, eS = np.linalg.norm(L.cpu().numpy() - ref.L), np.linalg.norm(S.cpu().numpy() - ref.S)
    assert eL <= bar and eS <= bar, (eL / bar, eS / bar)


@pytest.mark.parametrize("T", [40, 50, 100, 132])
def test_first_wide_step_resolves_what_its_gram_holds(rp, T):
    # singular values that span 1e4 in the first, unrotated Gram, all of them above tau: G, H and Gp need more than FP32
    # there (bar: the reduced precisions' 1e-4 of ||X||; in FP32 3e-4)
    F = low_noise(T, 2048, 1e-3)
    mu = 1e5 * 1.25 / np.linalg.norm(F.astype(np.float64), 2)
    plan = rp.Plan(2048, T, mu_init=mu)
    L, S, res = plan.solve(torch.from_numpy(F).cuda())
    plan.close()
    ref = O.rpca_frames(F, mu_init=mu, max_iter=res["iters"], tol=1e-30)
    eL = np.linalg.norm(L.cpu().numpy() - ref.L)
    assert eL <= 1e-4 * np.linalg.norm(F), (eL / np.linalg.norm(F), res["iters"])


def test_eig_rounds_checks_its_arguments(rp):
    assert rp.load().rpca_plan_eig_rounds(None, None, None) == rp.ERR_ARG
