"""Graphs on streams that the legacy default stream is not ordered against (torch's side streams are created
non-blocking): every call's device work stays on the graph's own stream."""
import numpy as np
import pytest

from paper_2003_03134_gb300 import build, gbp, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    t = pytest.importorskip("torch")
    if not t.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    gbp.lib()
    return t


def _add_then_reset(torch, problem, start_kf, precision, stream, between):
    """A graph that grows to the whole problem and goes back to iteration 0 right after the last keyframe."""
    init, steps = synth.stream_plan(problem, start_kf)
    with gbp.Graph(init, stream=stream, huber_nsigma=2.0, precision_mode=precision, launch_mode=2) as g:
        g.iterate(7)
        for s in steps:
            g.add_keyframe(s.obs_lm, s.obs_uv, n_new_lm=s.n_new_lm,
                           new_lm_xyz=s.new_lm_true + 0.05 if s.n_new_lm else None)
            between()
        g.reset()
        between()
        g.iterate(12)
        return [*g.means(), g.relin_iters()]


@pytest.mark.parametrize("precision", [0, 2])
def test_reset_right_after_an_added_keyframe_on_a_side_stream(torch, precision):
    """gbp_add_keyframe leaves its upload (births among it) queued; a reset that follows at once, with the copy
    engines busy on another stream, starts every variable at iteration 0 as one on an idle device does."""
    p = synth.make_walk(3, n_kf=14, n_lm=150)
    want = _add_then_reset(torch, p, 8, precision, 0, torch.cuda.synchronize)
    side, other = torch.cuda.Stream(), torch.cuda.Stream()
    host = torch.empty(256 << 20, dtype=torch.uint8, pin_memory=True)
    dev = torch.empty_like(host, device="cuda")

    def busy():
        with torch.cuda.stream(other):
            dev.copy_(host, non_blocking=True)

    for _ in range(3):
        got = _add_then_reset(torch, p, 8, precision, side.cuda_stream, busy)
        torch.cuda.synchronize()
        for a, b in zip(want, got):
            assert np.array_equal(a, b)
