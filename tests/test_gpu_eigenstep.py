"""The eigen-steps at the frame counts where their tiles and blocks end (blocks of
four columns, 16-row column lengths, an odd number of blocks, one frame), and on
Grams that a Cholesky factor alone could not take: repeated, zero and exactly
low-rank frames.

Bar: relative Frobenius error of L and S against the CPU FP64 oracle at the same
iteration count, 1e-5 as for every FP32 solve; where S is (nearly) zero the error
is taken relative to ||X||.
"""
import numpy as np
import pytest

from oracle import rpca_oracle as O
from paper_2506_10257_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-5


@pytest.fixture(scope="module")
def rp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2506_10257_gb300 import rpca
    rpca.load()
    return rpca


def check(rp, frames, rel_to_x=False):
    T, m = frames.shape
    plan = rp.Plan(m, T)
    L, S, res = plan.solve(torch.from_numpy(frames).cuda())
    L, S = L.cpu().numpy().astype(np.float64), S.cpu().numpy().astype(np.float64)
    plan.close()
    ref = O.rpca_frames(frames)
    if not rel_to_x:  # (the residual of a nearly exact split can sit at rounding level for many iterations)
        assert abs(res["iters"] - ref.iters) <= 1
    if res["iters"] != ref.iters:
        ref = O.rpca_frames(frames, max_iter=res["iters"], tol=1e-30)
    nL, nS = (np.linalg.norm(frames),) * 2 if rel_to_x else (np.linalg.norm(ref.L), np.linalg.norm(ref.S))
    eL, eS = np.linalg.norm(L - ref.L) / nL, np.linalg.norm(S - ref.S) / nS
    assert eL <= TOL and eS <= TOL, (eL, eS, res["iters"], ref.iters)


@pytest.mark.parametrize("T", [1, 2, 3, 4, 5, 8, 13, 15, 16, 17, 20, 24, 25, 28, 29, 31, 32])
def test_narrow_frame_counts(rp, T):
    check(rp, synth.make_window(seed=T, ny=40, nx=33, T=T, n_bound=6, n_free=10).frames)


@pytest.mark.parametrize("T", [6, 20, 32])
@pytest.mark.parametrize("kind", ["repeated", "zero frames", "rank two", "tiny", "large"])
def test_degenerate_grams(rp, T, kind):
    w = synth.make_window(seed=7, ny=32, nx=32, T=T, n_bound=5, n_free=8).frames.copy()
    if kind == "repeated":
        w[:] = w[0]
    elif kind == "zero frames":
        w[1::3] = 0.0
    elif kind == "rank two":
        w[:] = (np.linspace(1, 2, T)[:, None] * w[0] + np.cos(np.arange(T))[:, None] * w[1]).astype(np.float32)
    elif kind == "tiny":
        w *= np.float32(2.0 ** -40)
    else:
        w *= np.float32(2.0 ** 40)
    check(rp, w, rel_to_x=True)


@pytest.mark.parametrize("T", [33, 36, 47, 48, 49, 63, 64, 65, 81, 97, 112, 113, 128, 129, 145, 160, 161, 193, 209, 224])
def test_wide_frame_counts(rp, T):
    check(rp, synth.make_window(seed=T, ny=72, nx=61, T=T, n_bound=12, n_free=20).frames)


@pytest.mark.parametrize("T", [40, 100])
@pytest.mark.parametrize("kind", ["zero frames", "rank two", "tiny", "large"])
def test_wide_degenerate_grams(rp, T, kind):
    test_degenerate_grams(rp, T, kind)


def test_batch_runs_the_wide_step_on_every_column_count(rp):
    # one CTA per step and larger product tiles than a plan's cluster
    shapes = [(9, 900), (33, 1200), (50, 1100), (100, 2000), (132, 2500), (224, 4400)]
    ws = [synth.make_window(seed=T, ny=m // 20, nx=20, T=T, n_bound=8, n_free=12).frames for T, m in shapes]
    b = rp.Batch([(w.shape[1], w.shape[0]) for w in ws])
    Ls, Ss, res = b.solve([torch.from_numpy(w).cuda() for w in ws])
    b.close()
    for w, L, S, r in zip(ws, Ls, Ss, res):
        ref = O.rpca_frames(w, max_iter=r["iters"], tol=1e-30)
        eL = np.linalg.norm(L.cpu().numpy() - ref.L) / np.linalg.norm(ref.L)
        eS = np.linalg.norm(S.cpu().numpy() - ref.S) / np.linalg.norm(ref.S)
        assert eL <= TOL and eS <= TOL, (w.shape, eL, eS, r["iters"])
