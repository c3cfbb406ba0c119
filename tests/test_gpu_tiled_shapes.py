"""Tiled passes and their eigen-steps at column counts that no other test reaches: complex windows whose real columns
fall into the 96-, 192- and 256-column tiles, as plans and as batches (there with the rows of i Z apart from Z's), with
ragged pixel counts; and at most 32 real columns, which take the narrow eigen-step on the tiled path.

Bar: twice what FP32 rounding of the two T-term products (sqrt(T) u, u = 2^-24, in quadrature) and of the stored S, Y
and L (4 u together) leaves, relative to ||X||; T counts real columns.
"""
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


def window(T, ny, nx, cplx=True):
    return synth.make_window(seed=ny + T, ny=ny, nx=nx, T=T, n_bound=8, n_free=14, complex_iq=cplx).frames


def check(w, L, S, res, rp, bar=None):
    assert res["status"] == rp.OK
    ref = O.rpca_frames(w)
    assert abs(res["iters"] - ref.iters) <= 1
    if res["iters"] != ref.iters:
        ref = O.rpca_frames(w, max_iter=res["iters"], tol=1e-30)
    cols = w.shape[0] * (2 if np.iscomplexobj(w) else 1)
    bar = (bar or 2 * (np.sqrt(cols) + 4) * 2.0 ** -24) * np.linalg.norm(w)
    L, S = L.cpu().numpy().astype(ref.L.dtype), S.cpu().numpy().astype(ref.S.dtype)
    eL, eS = np.linalg.norm(L - ref.L), np.linalg.norm(S - ref.S)
    assert eL <= bar and eS <= bar, (eL / bar, eS / bar, res["iters"], ref.iters)


@pytest.mark.parametrize("T,ny,nx", [(33, 41, 39), (40, 50, 33), (48, 64, 40), (65, 45, 50), (75, 61, 37), (96, 64, 48),
                                     (97, 63, 51), (111, 57, 60)])
def test_complex_plans(rp, T, ny, nx):
    w = window(T, ny, nx)
    plan = rp.Plan(w.shape[1], T, dtype=rp.C64)
    L, S, res = plan.solve(torch.from_numpy(w).cuda())
    plan.close()
    check(w, L, S, res, rp)


def test_complex_batch_of_every_tile_width(rp):
    ws = [window(T, ny, nx) for T, ny, nx in ((9, 33, 30), (25, 41, 39), (45, 50, 33), (60, 40, 45), (80, 45, 50),
                                              (112, 57, 60))]
    b = rp.Batch([(w.shape[1], w.shape[0]) for w in ws], dtype=rp.C64)
    Ls, Ss, res = b.solve([torch.from_numpy(w).cuda() for w in ws])
    b.close()
    for w, L, S, r in zip(ws, Ls, Ss, res):
        check(w, L, S, r, rp)


@pytest.mark.parametrize("T", [4, 12, 20, 29, 32, 36, 52, 100, 132, 224])
def test_real_plans_reach_fp32_rounding(rp, T):
    w = window(T, 72, 61, cplx=False)
    plan = rp.Plan(w.shape[1], T)
    L, S, res = plan.solve(torch.from_numpy(w).cuda())
    plan.close()
    check(w, L, S, res, rp)


@pytest.mark.parametrize("drive", ["GRAPH", "HOST", "STREAM"])
@pytest.mark.parametrize("T,ny,nx", [(2, 30, 31), (3, 33, 30), (4, 64, 64), (8, 47, 45), (15, 41, 39), (16, 50, 33), (17, 50, 33)])
def test_complex_plans_of_few_frames(rp, T, ny, nx, drive):
    w = window(T, ny, nx)
    plan = rp.Plan(w.shape[1], T, dtype=rp.C64, drive=getattr(rp, "DRIVE_" + drive))
    L, S, res = plan.solve(torch.from_numpy(w).cuda())
    plan.close()
    check(w, L, S, res, rp)


@pytest.mark.parametrize("precision", ["TF32X3", "BF16X3"])
@pytest.mark.parametrize("T", [3, 8, 16])
def test_complex_plans_of_few_frames_on_tensor_cores(rp, T, precision):
    # (the eigen-step also writes the passes' operand images; bar: the reduced precisions' 1e-4)
    w = window(T, 50, 44)
    plan = rp.Plan(w.shape[1], T, dtype=rp.C64, precision=getattr(rp, "PREC_" + precision))
    L, S, res = plan.solve(torch.from_numpy(w).cuda())
    plan.close()
    check(w, L, S, res, rp, bar=1e-4)


@pytest.mark.parametrize("cplx", [False, True])
def test_batches_of_short_and_long_windows(rp, cplx):
    ws = [window(T, ny, nx, cplx) for T, ny, nx in ((2, 30, 31), (5, 33, 30), (8, 41, 39), (16, 50, 33), (20, 40, 45), (32, 45, 50),
                                                    (33, 47, 41))]
    kw = {"dtype": rp.C64} if cplx else {}
    b = rp.Batch([(w.shape[1], w.shape[0]) for w in ws], **kw)
    Ls, Ss, res = b.solve([torch.from_numpy(w).cuda() for w in ws])
    b.close()
    for w, L, S, r in zip(ws, Ls, Ss, res):
        check(w, L, S, r, rp)


def test_a_warm_complex_plan_of_few_frames(rp):
    # warm start: the first step after the extra Gram pass keeps the basis
    w = window(8, 40, 41)
    X = torch.from_numpy(w).cuda()
    plan = rp.Plan(w.shape[1], 8, dtype=rp.C64, warm_start=1)
    L, S = torch.zeros_like(X), torch.zeros_like(X)
    L, S, res = plan.solve(X, L=L, S=S)
    plan.close()
    check(w, L, S, res, rp)
