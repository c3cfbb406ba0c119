"""The first mu of a warm solve that resumes from the plan's previous solve (mu_prev_scale), on windows whose first
eigen-step needs more than one round: frames that are nearly of low rank, all of whose singular values count because
the resumed mu is large."""
import numpy as np
import pytest

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
    bg = rng.rayleigh(size=m)
    t = np.linspace(0, 1, T)
    X = bg * (1 + 0.02 * t[:, None]) + 0.01 * rng.rayleigh(size=m) * np.cos(np.pi * t)[:, None]
    return (X + noise * rng.standard_normal((T, m))).astype(np.float32)


@pytest.mark.parametrize("noise", [1e-3, 3e-4, 1e-4])
@pytest.mark.parametrize("T", [6, 20, 32, 50, 100])
def test_warm_solve_starts_at_the_scaled_previous_mu(rp, T, noise):
    m, scale = 4096, 1e5
    X = torch.from_numpy(low_noise(T, m, noise)).cuda()
    plan = rp.Plan(m, T, warm_start=1, mu_prev_scale=scale, max_iter=1)
    L, S = torch.zeros_like(X), torch.zeros_like(X)
    _, _, first = plan.solve(X, L=L, S=S)  # no previous solve: the schedule's first mu
    L.zero_()
    S.zero_()
    _, _, second = plan.solve(X, L=L, S=S)
    plan.close()
    s1 = np.linalg.norm(X.cpu().numpy().astype(np.float64), 2)
    # 1.25 / ||X||_2, the norm from the FP32 Gram (relative error of its entries: at most m products' rounding)
    assert abs(first["mu"] * s1 / 1.25 - 1) <= 1e-5
    assert first["iters"] == second["iters"] == 1
    assert abs(second["mu"] / (scale * first["mu"]) - 1) <= 1e-12
