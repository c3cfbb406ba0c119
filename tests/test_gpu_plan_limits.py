"""Plans of different sizes side by side: what one plan sets on a kernel that plans share must not stop another.

The tiled pass kernels serve all frame counts of a column bucket and the wide eigen-step all of them, each plan
launching with the shared memory its own frame count needs.  Host- and stream-driven solves launch them anew at every
solve, so they see what was set last.
"""
import numpy as np
import pytest

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


def frames(T, cplx=False):
    return synth.make_window(seed=T, ny=40, nx=32, T=T, n_bound=6, n_free=10, complex_iq=cplx).frames


# (frames of the first plan, of the one made after it): the same column bucket, and different ones
@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("drive", ["HOST", "STREAM"])
@pytest.mark.parametrize("first,later", [(64, 33), (128, 97), (160, 130), (200, 40)])
def test_a_smaller_plan_made_later_leaves_a_larger_one_working(rp, first, later, drive, cplx):
    if cplx:
        first, later = first // 2, later // 2
    w = frames(first, cplx)
    kw = {"drive": getattr(rp, "DRIVE_" + drive)}
    if cplx:
        kw["dtype"] = rp.C64
    X = torch.from_numpy(w).cuda()
    big = rp.Plan(w.shape[1], first, **kw)
    small = rp.Plan(w.shape[1], later, **kw)
    b = rp.Batch([(w.shape[1], later), (w.shape[1], later)], **({"dtype": rp.C64} if cplx else {}))
    L, S, res = big.solve(X)
    Xs = torch.from_numpy(frames(later, cplx)).cuda()
    _, _, res_s = small.solve(Xs)
    L2, S2, res2 = big.solve(X)
    for p in (big, small, b):
        p.close()
    assert res["status"] == rp.OK and res_s["status"] == rp.OK and res2["status"] == rp.OK
    # the same kernels on the same data
    assert torch.equal(L, L2) and torch.equal(S, S2) and res["iters"] == res2["iters"]
    e = torch.linalg.norm((X - L - S).to(torch.complex128 if cplx else torch.float64))
    assert float(e) <= 2e-7 * float(np.linalg.norm(w))
