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


@pytest.mark.parametrize("n_lm", [40, 5381, 5382, 9000])
@pytest.mark.parametrize("precision", [0, 2])
def test_world_beliefs_are_the_chart_means(n_lm, precision):
    """Read-backs just below and above the size that goes through pinned memory (16384 doubles: 20 x 12 + 3 x 5381 is
    one less).  Points are lref + dl exactly; poses Exp(dw) Rref and t = -R c carry a few roundings of entries below
    20: 1e-13."""
    from scipy.spatial.transform import Rotation

    p = synth.make_walk(7, n_kf=20, n_lm=n_lm)
    with gbp.Graph(p, huber_nsigma=2.0, precision_mode=precision) as g:
        g.iterate(6)
        kf, lm = g.beliefs()
        mk, ml = g.means()
    assert np.array_equal(lm, p.lm_init + ml)
    R0 = p.kf_Rt_init[:, :9].reshape(-1, 3, 3)
    c = -np.einsum("nji,nj->ni", R0, p.kf_Rt_init[:, 9:]) + mk[:, :3]
    R = Rotation.from_rotvec(mk[:, 3:]).as_matrix() @ R0
    assert np.abs(kf[:, :9].reshape(-1, 3, 3) - R).max() <= 1e-13
    assert np.abs(kf[:, 9:] + np.einsum("nij,nj->ni", R, c)).max() <= 1e-13


def test_residuals_follow_the_observation_order_after_a_keyframe_is_added():
    init, steps = synth.make_stream(3, n_kf=14, n_lm=220, start_kf=10)
    with gbp.Graph(init, huber_nsigma=2.0) as g:
        g.iterate(5)
        assert g.residuals().shape == (init.n_obs,)
        ok, ol, uv = [init.obs_kf], [init.obs_lm], [init.obs_uv]
        for s in steps[:3]:
            k = g.add_keyframe(s.obs_lm, s.obs_uv, n_new_lm=s.n_new_lm)
            g.iterate(5)
            ok.append(np.full(len(s.obs_lm), k)), ol.append(s.obs_lm), uv.append(s.obs_uv)
            kf, lm = g.beliefs()
            a, b, z = np.concatenate(ok), np.concatenate(ol), np.concatenate(uv)
            q = np.einsum("nij,nj->ni", kf[a, :9].reshape(-1, 3, 3), lm[b]) + kf[a, 9:]
            h = np.stack([init.fx * q[:, 0] / q[:, 2] + init.cx, init.fy * q[:, 1] / q[:, 2] + init.cy], 1)
            e, want = g.residuals(), np.linalg.norm(z - h, axis=1)
            far = q[:, 2] > 0.5                     # FP32 projections: ~1e-6 relative of up to 1000 px and depth
            assert np.abs(e - want)[far].max() <= 0.05 + 1e-4 * want[far].max()


def test_reference_solution_through_precision_switches_and_added_keyframes():
    """The reference projections are replaced after the layout was rebuilt for another precision, and the freed
    buffers' addresses serve later layouts: the distance to the reference is that of a graph made afresh."""
    p = synth.make_walk(4, n_kf=20, n_lm=250)
    init, steps = synth.stream_plan(p, 16)
    with gbp.Graph(init, huber_nsigma=2.0) as g:
        for precision in (2, 0):
            g.set_reference(init.kf_Rt_true, init.lm_true)
            g.set_params(precision_mode=precision)
            g.set_reference(init.kf_Rt_true, init.lm_true)
            g.set_params(prior_anneal_iters=12)
            g.iterate(10)
            with gbp.Graph(init, huber_nsigma=2.0, precision_mode=precision, prior_anneal_iters=12) as f:
                f.set_reference(init.kf_Rt_true, init.lm_true)
                f.iterate(10)
                assert g.stats()["are_ref"] == f.stats()["are_ref"] > 0
                if precision == 0:
                    for st in steps:
                        for h in (f, g):
                            h.add_keyframe(st.obs_lm, st.obs_uv, n_new_lm=st.n_new_lm)
                            h.iterate(4)
                    for a, b in zip(f.means(), g.means()):
                        assert np.array_equal(a, b)


@pytest.mark.parametrize("n_lm", [300, 6000])
def test_beliefs_with_covariances_are_those_without(n_lm):
    """Poses and points read beside the covariances (one wait for both; up to 16384 doubles of them through pinned
    memory) are those read alone."""
    p = synth.make_walk(6, n_kf=24, n_lm=n_lm)
    with gbp.Graph(p, huber_nsigma=2.0) as g:
        g.iterate(15)
        kf, lm = g.beliefs()
        kf2, lm2, kc, lc = g.beliefs(covariances=True)
        g.iterate(1)
        assert not np.array_equal(g.beliefs()[0], kf)
        assert np.array_equal(kf, kf2) and np.array_equal(lm, lm2)
        for c in (kc, lc):
            assert (np.linalg.eigvalsh(c) > 0).all()
