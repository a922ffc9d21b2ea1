"""Statistics of a solution against numpy on the per-observation residuals: sizes around one block's sums, around the
number of blocks that the final sum takes in one pass (256) and the largest grid (1024 blocks of 256)."""
import numpy as np
import pytest

from paper_2003_03134_gb300 import build, gbp, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    gbp.lib()


@pytest.mark.parametrize("n_kf,n_lm,precision", [(8, 30, 0), (20, 60, 2), (60, 7600, 0), (120, 30000, 0)])
def test_stats_are_the_residuals_statistics(n_kf, n_lm, precision):
    """The sums are FP64 over the same values in another order: 1e-12 relative."""
    p = synth.make_walk(5, n_kf=n_kf, n_lm=n_lm)
    with gbp.Graph(p, huber_nsigma=2.0, precision_mode=precision) as g:
        g.iterate(5)
        kf, lm = g.beliefs()
        e = g.residuals()
        st = g.stats()
        are, n, hub = g.problem_are()
        g.set_reference(p.kf_Rt_true, p.lm_true)
        ref = g.stats()["are_ref"]
    ok = e >= 0
    assert st["n_are"] == n[0] == ok.sum() and st["huber_count"] == hub[0] == (e[ok] > 2.0).sum()
    assert abs(st["are"] - e[ok].mean()) <= 1e-12 * e[ok].mean()
    assert abs(are[0] - e[ok].mean()) <= 1e-12 * e[ok].mean()

    def project(Rt, X):
        q = np.einsum("nij,nj->ni", Rt[p.obs_kf, :9].reshape(-1, 3, 3), X[p.obs_lm]) + Rt[p.obs_kf, 9:]
        return q[:, 2], np.stack([p.fx * q[:, 0] / q[:, 2] + p.cx, p.fy * q[:, 1] / q[:, 2] + p.cy], 1)

    z0, a = project(kf, lm)
    z1, b = project(p.kf_Rt_true, p.lm_true)
    both = ok & (z1 >= 0.05)
    # FP32 projections of ~500 px: 1e-4 px each
    assert abs(ref - np.linalg.norm(a - b, axis=1)[both].mean()) <= 1e-3 + 1e-4 * ref
