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


def test_calls_that_only_queue_work_can_be_captured(torch):
    """The allocation-free error, the network's forward pass and its training step, recorded into a CUDA graph with a
    copy in front of each and replayed on other inputs: the bits of the calls themselves."""
    n = 5000
    rng = np.random.default_rng(5)
    p = synth.make_walk(5, n_kf=20, n_lm=300)
    X = torch.from_numpy(rng.normal(size=(2, n, 16)).astype(np.float32)).cuda()
    t = torch.from_numpy(rng.uniform(0.0, 0.9, (2, n)).astype(np.float32)).cuda()
    params = (0.1 * rng.normal(size=gbp.GBP_MLP_NPARAM)).astype(np.float32)
    kf = torch.from_numpy(np.stack([p.kf_Rt_init, p.kf_Rt_true])).cuda()
    lm = torch.from_numpy(p.lm_true).cuda()
    ok, ol = torch.from_numpy(p.obs_kf).cuda(), torch.from_numpy(p.obs_lm).cuda()
    uv = torch.from_numpy(p.obs_uv).cuda()
    torch.cuda.synchronize()

    def run(net, stream, Xw, tw, kfw, y, err):
        gbp.gbp_reprojection_error_noalloc(p.intrinsics(), 0.05, p.n_kf, kfw.data_ptr(), p.n_lm, lm.data_ptr(), p.n_obs,
                                           ok.data_ptr(), ol.data_ptr(), uv.data_ptr(), err.data_ptr(), stream=stream)
        net.train_step(Xw.data_ptr(), tw.data_ptr(), n, 1e-3)
        net.train_step(Xw.data_ptr(), tw.data_ptr(), n // 2, 1e-3)
        net.forward(Xw.data_ptr(), n, y.data_ptr())

    def buffers():
        return (torch.empty_like(X[0]), torch.empty_like(t[0]), torch.empty_like(kf[0]),
                torch.empty(n, device="cuda"), torch.empty(2, dtype=torch.float64, device="cuda"))

    def fill(b, i):
        for dst, src in zip(b, (X[i], t[i], kf[i])):
            dst.copy_(src)

    side = torch.cuda.Stream()
    want = []
    with torch.cuda.stream(side):
        net = gbp.DampingNet(params, stream=side.cuda_stream)
        b = buffers()
        for i in (0, 1):
            net.set_params(params)   # the step count is the host's: a replay repeats the recorded ones
            fill(b, i)
            run(net, side.cuda_stream, *b)
            side.synchronize()
            want.append([b[3].cpu().numpy(), b[4].cpu().numpy(), net.params])
        net.set_params(params)
        graph = torch.cuda.CUDAGraph()
        src, b = buffers(), buffers()
        side.synchronize()
    with torch.cuda.graph(graph, stream=side):
        for dst, s in zip(b[:3], src):
            dst.copy_(s)
        run(net, side.cuda_stream, *b)
    with torch.cuda.stream(side):
        for i in (0, 1, 0):
            net.set_params(params)
            fill(src, i)
            graph.replay()
            side.synchronize()
            for w, got in zip(want[i], (b[3].cpu().numpy(), b[4].cpu().numpy(), net.params)):
                assert np.array_equal(w, got)
    net.close()
