"""The automatic launch mode's choices: what gbp_autotune measured is what runs, a choice holds for the graphs it was
made for, and every way leads to the bits of per-phase launches."""
import ctypes
import dataclasses
import glob
import os
import subprocess
import threading

import numpy as np
import pytest

from paper_2003_03134_gb300 import build, gbp, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def torch():
    t = pytest.importorskip("torch")
    if not t.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    gbp.lib()
    return t


def test_autotune_puts_the_shape_it_measured_in_use():
    """A graph large enough that its first iterations took a shape by size: each explicit timing that follows
    replaces it by the fastest shape of that timing."""
    p = synth.make_loop(0, n_kf=400, n_lm=36000)
    with gbp.Graph(p, huber_nsigma=2.0) as g:
        g.iterate(2)
        t = g.tuning()
        assert (t["launch_mode"], t["factor_shape"], t["n_candidates"]) == (2, 4, 1)
        for _ in range(8):
            chosen, _, _ = g.autotune(4)
            t = g.tuning()
            ms = {c["shape"]: c["ms"] for c in t["candidates"] if c["launch_mode"] == 2 and c["ms"] > 0}
            assert chosen == t["launch_mode"] == 2
            assert ms[t["factor_shape"]] == min(ms.values()), t


def _growing(seed, n_kf, n_lm, start):
    """A walk's first `start` keyframes with the points that two of them see, and the later keyframes' observations of
    those points: (problem, [(obs_lm, obs_uv), ...])."""
    p = synth.make_walk(seed, n_kf=n_kf, n_lm=n_lm)
    early = p.obs_kf < start
    keep = np.bincount(p.obs_lm[early], minlength=p.n_lm) >= 2
    index = np.cumsum(keep) - 1
    on = keep[p.obs_lm]
    sel = early & on
    init = dataclasses.replace(p, kf_Rt_true=p.kf_Rt_true[:start], kf_Rt_init=p.kf_Rt_init[:start],
                               lm_true=p.lm_true[keep], lm_init=p.lm_init[keep], obs_kf=p.obs_kf[sel],
                               obs_lm=index[p.obs_lm[sel]].astype(np.int32), obs_uv=p.obs_uv[sel],
                               obs_outlier=p.obs_outlier[sel])
    return init, [(index[p.obs_lm[on & (p.obs_kf == k)]].astype(np.int32), p.obs_uv[on & (p.obs_kf == k)])
                  for k in range(start, n_kf)]


def test_a_stream_returns_to_the_resident_kernel():
    """A point that nobody sees for one keyframe takes the graph off the resident kernel, to per-phase launches in the
    shape of its size without a timing; its first observation brings it back.  The bits are those of per-phase
    launches."""
    init, steps = _growing(9, 18, 400, 10)
    out = []
    for mode in (0, 2):
        used, records = [], []
        with gbp.Graph(init, huber_nsigma=2.0, launch_mode=mode) as g:
            g.iterate(6)
            used.append(g.stats()["launch_mode"])
            for i, (obs_lm, obs_uv) in enumerate(steps[:6]):
                n_lm = gbp.gbp_get_sizes(g.h)[1]
                unseen = i in (1, 4)
                if i in (2, 5):
                    obs_lm = np.append(obs_lm, n_lm - 1).astype(np.int32)
                    obs_uv = np.concatenate([obs_uv, [[320.0, 240.0]]])
                g.add_keyframe(obs_lm, obs_uv, n_new_lm=int(unseen),
                               new_lm_xyz=init.lm_true[:1] + 0.3 if unseen else None)
                g.iterate(6)
                used.append(g.stats()["launch_mode"])
                if unseen:
                    records.append(g.tuning())
            out.append((used, records, *g.means(), g.relin_iters()))
    used, records = out[0][:2]
    assert used == [1, 1, 2, 1, 1, 2, 1]
    for r in records:
        assert (r["n_candidates"], r["factor_shape"], r["candidates"][0]["ms"]) == (1, 0, 0.0)
    for a, b in zip(out[0][2:], out[1][2:]):
        assert np.array_equal(a, b)


def test_a_choice_is_not_handed_to_a_graph_the_resident_kernel_does_not_take():
    """Two graphs of the same numbers of keyframes, points, factors and tiles, one with a point that nobody sees: what
    the timing of the first chose (the resident kernel among its candidates) is not what the second starts with."""
    p = synth.make_circle(4, n_kf=12, n_lm=64, obs_range=(4, 4))
    other = p.obs_lm.copy()
    other[p.obs_lm == 63] = 62   # point 62 now has 8 observations, point 63 none
    q = dataclasses.replace(p, obs_lm=other)
    with gbp.Graph(p, huber_nsigma=2.0) as a, gbp.Graph(q, huber_nsigma=2.0) as b, \
            gbp.Graph(q, huber_nsigma=2.0, launch_mode=2) as c:
        a.autotune(4)
        for g in (a, b, c):
            g.iterate(9)
        assert a.tuning()["n_candidates"] == b.tuning()["n_candidates"] == 7
        assert a.tuning()["candidates"] != b.tuning()["candidates"]
        for x, y in zip(b.means(), c.means()):
            assert np.array_equal(x, y)


def test_a_timed_choice_is_reused_for_a_graph_of_the_same_shape():
    """Graphs whose candidates are timed (FP64 mode, and the FP32 path between the sizes that a rule covers): a second
    graph of the same sizes takes the first one's choice and its record, times included."""
    for p, params in ((synth.make_walk(7, n_kf=30, n_lm=300), {"precision_mode": 2}),
                      (synth.make_loop(2, n_kf=200, n_lm=6000), {})):
        with gbp.Graph(p, **params) as a, gbp.Graph(p, **params) as b:
            a.iterate(12)
            ta = a.tuning()
            assert ta["n_candidates"] > 1 and all(c["ms"] > 0 for c in ta["candidates"])
            b.iterate(12)
            assert b.tuning() == ta
            for x, y in zip(a.means(), b.means()):
                assert np.array_equal(x, y)


def _repeat_points(p, n):
    """The problem with its points, and their observations, n times over."""
    return dataclasses.replace(p, lm_true=np.tile(p.lm_true, (n, 1)), lm_init=np.tile(p.lm_init, (n, 1)),
                               obs_kf=np.tile(p.obs_kf, n), obs_uv=np.tile(p.obs_uv, (n, 1)),
                               obs_lm=(np.tile(p.obs_lm, n) + np.repeat(np.arange(n), p.n_obs) * p.n_lm).astype(np.int32),
                               obs_outlier=np.tile(p.obs_outlier, n))


@pytest.mark.parametrize("per_sm,shape", [(8, 0), (12, 1), (16, 0)])
def test_the_factor_shape_by_size_at_the_edges_of_its_waves(torch, per_sm, shape):
    """Per-phase launches that were never timed: shape 0 holds 8 tiles an SM at a time, shape 1 12; the one that needs
    fewer waves is taken, on both sides of each edge."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    ring = synth.make_circle(3, n_kf=10, n_lm=8, obs_range=(4, 4))
    assert ring.n_obs == 32   # a full tile
    for tiles, want in ((per_sm * sms, shape), (per_sm * sms + 1, 1 - shape)):
        p = _repeat_points(ring, tiles)
        with gbp.Graph(p, huber_nsigma=2.0, launch_mode=2) as g:
            assert g.tuning()["factor_shape"] == want
            g.iterate(5)
            got = g.means()
        with gbp.Graph(p, huber_nsigma=2.0, launch_mode=2, factor_shape=5) as g:
            g.iterate(5)
            for a, b in zip(got, g.means()):
                assert np.array_equal(a, b)


FAKE_LAUNCH = """
#include <stddef.h>
typedef struct { unsigned x, y, z; } dim3;
int fake_refuse_above = 1 << 30;   /* threads a block; a launch with more is refused */
int __real_cudaLaunchCooperativeKernel(const void*, dim3, dim3, void**, size_t, void*);
int __wrap_cudaLaunchCooperativeKernel(const void* f, dim3 grid, dim3 block, void** args, size_t shared, void* stream) {
    if ((int)block.x > fake_refuse_above) return 720;   /* cudaErrorCooperativeLaunchTooLarge */
    return __real_cudaLaunchCooperativeKernel(f, grid, block, args, shared, stream);
}
"""


@pytest.fixture
def refusing_lib(tmp_path, monkeypatch):
    """The library linked with a cooperative launch that the test can have refused on the host, as the driver refuses
    one that does not fit the SMs a stream may use.  Sets the number of threads a block above which it is refused."""
    objs = sorted(glob.glob(os.path.join(build.BUILD_DIR, "*.o")))
    if not objs:
        build.build(force=True)
        objs = sorted(glob.glob(os.path.join(build.BUILD_DIR, "*.o")))
    (tmp_path / "fake.c").write_text(FAKE_LAUNCH)
    subprocess.check_call(["gcc", "-c", "-fPIC", "-o", str(tmp_path / "fake.o"), str(tmp_path / "fake.c")])
    path = str(tmp_path / "libgbp_refusing.so")
    subprocess.check_call([build.nvcc(), *build.ARCH, "-shared", "-o", path, *objs, str(tmp_path / "fake.o"),
                           "-Xlinker", "--wrap=cudaLaunchCooperativeKernel"])
    monkeypatch.setattr(gbp, "LIB_PATH", path)
    monkeypatch.setattr(gbp, "_lib", None)
    return ctypes.c_int.in_dll(gbp.lib(), "fake_refuse_above")


def test_a_refused_cooperative_launch_is_replaced(refusing_lib):
    """Automatic launches of a graph for which a rule takes the resident kernel (256 threads a block) untried, and
    forced persistent launches: refused, the first run per phase and the second on the tile-walking kernel (128
    threads); with that refused too the forced launch reports the error, as it always did.  Same bits throughout."""
    p = synth.make_circle(5)

    def solve(mode):
        with gbp.Graph(p, huber_nsigma=2.0, launch_mode=mode, conv_tol=1e-30) as g:
            assert [g.iterate(n) for n in (3, 20)] == [3, 20]
            return g.stats()["launch_mode"], [*g.means(), g.relin_iters()]

    mode, want = solve(0)
    assert mode == 1   # nothing refused yet
    for limit in (128, 0):
        refusing_lib.value = limit
        for launch_mode in (0, 2) + ((1,) if limit else ()):
            mode, got = solve(launch_mode)
            if launch_mode or not limit:
                assert mode == (launch_mode or 2)
            for a, b in zip(want, got):
                assert np.array_equal(a, b)
    with pytest.raises(gbp.GBPError) as e:
        solve(1)
    assert e.value.status == gbp.GBP_ECUDA


def test_graphs_on_several_streams_leave_the_resident_kernel_when_they_do_not_fit(torch):
    """Resident launches run beside each other while all their blocks (one a keyframe here) fit the SMs; a graph whose
    blocks and those of other streams' graphs do not, launches per phase until there is room again."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    big = synth.make_walk(2, n_kf=sms // 2 + 10, n_lm=400)
    small = synth.make_circle(2)
    s1, s2 = torch.cuda.Stream().cuda_stream, torch.cuda.Stream().cuda_stream

    def graph(p, stream):
        return gbp.Graph(p, stream=stream, huber_nsigma=2.0)

    def run(g):
        g.iterate(8)
        return g.stats()["launch_mode"]

    a = graph(big, s1)
    assert run(a) == 1
    with graph(big, s2) as tuned_beside:   # timed where it does not fit, whatever that says is its own
        tuned_beside.autotune(4)
    same, beside, b = graph(big, s1), graph(small, s2), graph(big, s2)
    assert run(same) == 1 and run(beside) == 1 and run(a) == 1   # one stream; room for both
    assert [run(b), run(a), run(same), run(b)] == [2, 2, 2, 2]
    a.close()
    assert run(b) == 2
    same.close()
    assert run(b) == 1
    for x, y in zip(b.means(), _means_after(big, 4)):
        assert np.array_equal(x, y)
    b.close()
    beside.close()


def _means_after(problem, calls):
    with gbp.Graph(problem, huber_nsigma=2.0, launch_mode=2) as r:
        for _ in range(calls):
            r.iterate(8)
        return r.means()


def test_solves_in_threads_on_their_own_streams_give_the_same_bits(torch):
    """Four host threads make, solve and close graphs of different sizes at the same time, each on its own stream."""
    problems = [synth.make_walk(6, n_kf=100, n_lm=500), synth.make_circle(6), synth.make_walk(8, n_kf=60, n_lm=700)]
    want = [_means_after(p, 3) for p in problems]
    bad = []

    def work(i):
        try:
            stream = torch.cuda.Stream().cuda_stream
            for r in range(6):
                j = (i + r) % len(problems)
                with gbp.Graph(problems[j], stream=stream, huber_nsigma=2.0) as g:
                    for _ in range(3):
                        g.iterate(8)
                    if not all(np.array_equal(x, y) for x, y in zip(g.means(), want[j])):
                        bad.append((i, r))
        except Exception as e:   # a thread's exception does not fail the test by itself
            bad.append((i, repr(e)))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad
