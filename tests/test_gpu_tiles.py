"""The deferring factor kernel against the general factor phase at the edges of its tiles: landmarks with 31, 32, 33 and
more factors (split across tiles), tiles of one factor, landmarks without factors, relinearisations in every iteration
(beta = 0, interval 1) and none (linear)."""
import ctypes
import dataclasses

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


def _problem(counts):
    """A ring of 64 keyframes whose i-th landmark keeps counts[i] of its observations (0: none)."""
    p = synth.make_circle(11, n_kf=64, n_lm=len(counts), obs_range=(max(counts), max(counts)))
    rank = np.arange(p.n_obs) - np.searchsorted(p.obs_lm, p.obs_lm)
    keep = rank < np.asarray(counts)[p.obs_lm]
    return dataclasses.replace(p, obs_kf=p.obs_kf[keep], obs_lm=p.obs_lm[keep], obs_uv=p.obs_uv[keep],
                               obs_outlier=p.obs_outlier[keep])


@pytest.mark.parametrize("counts", [[31, 32, 33, 0, 1, 32, 40, 2, 3, 0], [1] * 70, [32] * 9, [4, 5, 6, 7, 8, 9, 10] * 12])
@pytest.mark.parametrize("params", [{}, {"linear": 1}, {"relin_beta": 0.0, "relin_interval": 3}])
def test_deferring_kernel_gives_the_general_phase_bits(counts, params):
    p = _problem(counts)
    got = []
    for mode, shape in ((2, 0), (2, 4), (2, 5), (1, 0)):
        with gbp.Graph(p, huber_nsigma=2.0, launch_mode=mode, factor_shape=shape, **params) as g:
            for n in (1, 9, 2, 13):
                g.iterate(n)
            got.append([*g.means(), g.relin_iters()])
    for other in got[1:]:
        for a, b in zip(got[0], other):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("n_problems", [1, 15, 16, 34, 36, 60])
@pytest.mark.parametrize("params", [{}, {"fp64_pivot_ratio": 1.0}, {"conv_tol": 1e-3, "check_every": 3}])
def test_persistent_launch_gives_the_per_phase_bits(n_problems, params):
    """Rings of 10 keyframes and ~17 tiles each as one graph: fewer and more keyframes than blocks (152), one and two
    tiles per factor warp's SM share (608 tiles), up to the size that the resident kernel takes; several calls, so that
    each starts from the state the last one left."""
    problems = [synth.make_circle(s) for s in range(n_problems)]
    got = []
    for mode in (1, 2):
        with gbp.Graph(problems, huber_nsigma=2.0, launch_mode=mode, **params) as g:
            done = [g.iterate(n) for n in (1, 2, 9, 20)]
            st = g.stats()
            got.append([np.array(done), *g.means(), g.relin_iters(),
                        np.array([st[k] for k in ("iterations", "max_dmu", "fp64_fallbacks", "relinearisations",
                                                  "held_messages", "fp64_resums")])])
    for a, b in zip(*got):
        assert np.array_equal(a, b)


def test_a_stream_that_outgrows_the_resident_kernel():
    """Automatic launches of a graph that grows from a few keyframes past 1216 tiles (~37k factors): the launch
    configuration changes on the way, the bits are those of per-phase launches throughout."""
    init, steps = synth.make_stream(5, n_kf=60, n_lm=6000, start_kf=4)
    got = []
    for mode in (0, 2):
        with gbp.Graph(init, huber_nsigma=2.0, launch_mode=mode) as g:
            g.iterate(3)
            used = [g.stats()["launch_mode"]]
            for s in steps:
                g.add_keyframe(s.obs_lm, s.obs_uv, n_new_lm=s.n_new_lm,
                               new_lm_xyz=s.new_lm_true if s.n_new_lm else None)
                g.iterate(2)
            used.append(g.stats()["launch_mode"])
            got.append((used, *g.means(), g.relin_iters()))
    assert got[0][0] == [1, 2], got[0][0]
    for a, b in zip(got[0][1:], got[1][1:]):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("scale,anneal", [(1e-30, 20), (1e-30, 60), (1e-12, 60), (1e-37, 90)])
@pytest.mark.parametrize("precision", [0, 1])
def test_divergence_ends_the_convergence_loop_at_the_next_check(scale, anneal, precision):
    """Points with one observation, whose prior all but vanishes: their beliefs stop being positive definite in the
    middle of a solve to a tolerance.  Persistent and per-phase launches leave at the same check, and at the first
    one of a later call, also when the error came from iterations that were not checked."""
    p = _problem([1, 4, 5, 6] * 30)
    got = []
    for mode in (1, 2):
        params = dict(launch_mode=mode, prior_final_scale=scale, prior_anneal_iters=anneal, precision_mode=precision)
        with gbp.Graph(p, conv_tol=1e-12, check_every=5, **params) as g, gbp.Graph(p, **params) as h:
            rec = []
            for n in (300, 12):
                done = ctypes.c_int32(-1)
                rec.append((gbp.lib().gbp_iterate(g.h, n, ctypes.byref(done)), done.value))
            assert h.iterate(100) == 100   # nothing is read back
            h.set_params(conv_tol=1e-12, check_every=7)
            done = ctypes.c_int32(-1)
            rec.append((gbp.lib().gbp_iterate(h.h, 50, ctypes.byref(done)), done.value))
            got.append(rec)
    assert got[0] == got[1]
    assert got[0][0][0] == gbp.GBP_EDIVERGED and 0 < got[0][0][1] < 300
    assert got[0][1:] == [(gbp.GBP_EDIVERGED, 5), (gbp.GBP_EDIVERGED, 7)]
