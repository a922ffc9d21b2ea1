"""Performance cases: the work a user of this library has it do, each case one call
sequence through the public entry points (``paper_2003_03134_gb300.gbp``).

Kinds
  solve    a resident graph solved again from its initial estimate: ``reset``,
           ``iterate``, ``beliefs`` (what every example and experiment does)
  batch    the same for independent problems in one graph
  e2e      host arrays in, poses and points out: create, solve to a tolerance,
           read the beliefs, close
  stream   incremental SLAM (Sec. 9.2): a small graph, then one keyframe after
           another with 20 iterations each
  report   quality of a solution: statistics and every observation's residual
  are      the allocation-free average reprojection error of device arrays
  train    Adam steps of the damping network on recorded rows
  predict  the damping network evaluated over recorded rows

Solutions of the FP32 path are handed on in float32 (the precision they are
held in), those of the FP64 path in float64.  ``exact`` restates the method in
64 bits with plain torch operations.
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_2003_03134_gb300 import gbp, learned, synth

FX = FY = 500.0
CX, CY, WIDTH, HEIGHT = 320.0, 240.0, 640, 480
HUBER = 2.0               # Huber threshold of the benchmark's problems (sigmas)
MEAN_OBS = {"circle": 4.5, "walk": 9.1, "map": 9.0}   # observations per point of the generators


# ---------------------------------------------------------------------------
# the cases

def listed():
    return [
        # the smallest problem of the tests and of smoke(): latency of one small solve
        dict(name="circle_solve", kind="solve", gen="circle", n_kf=10, n_lm=100, iters=200),
        # the benchmark's problem (125 keyframes, 1919 points, ~17.5k observations) at the
        # library's default iteration count
        dict(name="walk_solve", kind="solve", gen="walk", n_kf=125, n_lm=1919, iters=200),
        # the benchmark's end-to-end figure: create, solve to 1e-6 or 1000 iterations, read back
        dict(name="walk_e2e", kind="e2e", gen="walk", n_kf=125, n_lm=1919, iters=1000),
        # the full-precision mode that references are computed with
        dict(name="walk_fp64", kind="solve", gen="walk", n_kf=125, n_lm=1919, iters=40, precision=2),
        # the learned damping schedule with the shipped network
        dict(name="walk_learned", kind="solve", gen="walk", n_kf=125, n_lm=1919, iters=100, learned=True),
        # independent problems of uneven size in one graph (basin and outlier experiments, batches)
        dict(name="batch_solve", kind="batch", gen="map", n_problems=32, iters=60),
        # one large map: the largest problem of the benchmark and the tests
        dict(name="loop_solve", kind="solve", gen="map", n_kf=2000, n_lm=200_000, iters=30),
        # a tracking session of 50 added keyframes
        dict(name="stream", kind="stream", n_kf=60, n_lm=960, start=10, iters=20),
        # quality report of a map of ~1M observations
        dict(name="map_report", kind="report", gen="map", n_kf=1000, n_lm=100_000, iters=12),
        # error of an application's own device arrays, at the entry point's largest size
        dict(name="device_are", kind="are", n_kf=1000, n_lm=100_000, n_obs=1 << 20),
        # the training loop's minibatch size (4096 rows), 50 Adam steps
        dict(name="net_train", kind="train", rows=1 << 20, batch=4096, steps=50),
        # held-out rows put through the network
        dict(name="net_predict", kind="predict", rows=4_000_000),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "batch", "e2e", "stream", "report", "are", "train", "predict"])
    if kind == "solve":
        c = dict(kind="solve", iters=rng.randint(20, 200))
        size = rng.choice(["circle", "walk", "walk", "map"])
        if size == "circle":
            c.update(gen="circle", n_kf=rng.randint(8, 24), n_lm=_log(rng, 60, 400))
        elif size == "walk":
            c.update(gen="walk", n_kf=_log(rng, 16, 200), n_lm=_log(rng, 200, 5000))
            option = rng.choice(["", "", "fp64", "learned"])
            if option == "fp64":
                c.update(precision=2, iters=rng.randint(10, 40))
            elif option == "learned":
                c.update(learned=True, iters=rng.randint(20, 100))
        else:
            c.update(gen="map", n_kf=_log(rng, 200, 1800), iters=rng.randint(12, 30))
            c["n_lm"] = c["n_kf"] * rng.randint(60, 100)
        return c
    if kind == "batch":
        return dict(kind="batch", gen="map", n_problems=rng.randint(3, 31), iters=rng.randint(20, 60))
    if kind == "e2e":
        return dict(kind="e2e", gen="walk", n_kf=_log(rng, 16, 200), n_lm=_log(rng, 200, 5000), iters=_log(rng, 50, 900))
    if kind == "stream":
        n_kf = rng.randint(24, 90)
        return dict(kind="stream", n_kf=n_kf, n_lm=16 * n_kf, start=rng.randint(8, 16), iters=rng.choice([10, 20]))
    if kind == "report":
        n_kf = _log(rng, 110, 1000)
        return dict(kind="report", gen="map", n_kf=n_kf, n_lm=n_kf * rng.randint(40, 99), iters=12)
    if kind == "are":
        return dict(kind="are", n_kf=_log(rng, 10, 1000), n_lm=_log(rng, 1000, 100_000), n_obs=_log(rng, 4000, 1 << 20))
    if kind == "train":
        return dict(kind="train", rows=_log(rng, 50_000, 1 << 20), batch=_log(rng, 256, 8192), steps=rng.randint(5, 50))
    return dict(kind="predict", rows=_log(rng, 5000, 3_900_000))


# ---------------------------------------------------------------------------
# inputs

def _map_problem(rng, n_kf, n_lm):
    """A map along two laps of a circle (an arc for fewer than 105 keyframes; 0.19 m
    between keyframes), vectorised: each point lies in front of a home keyframe and
    is seen by 5-15 of the keyframes around it on either lap; 1 px noise, 2 % outlier
    pixels, the benchmark's initial errors (0.05 rad, 0.1 m)."""
    step = min(4.0 * np.pi / n_kf, 0.12)
    radius = 0.19 / step
    a = step * np.arange(n_kf)
    wob = np.cumsum(rng.normal(0.0, 0.02, (n_kf, 3)), axis=0) * np.exp(-np.arange(n_kf) / 400.0)[:, None]
    c = np.stack([radius * np.cos(a), radius * np.sin(a), np.full(n_kf, 1.5)], 1) + np.clip(wob, -0.6, 0.6)
    yaw = a + 0.5 * np.pi + rng.normal(0.0, 0.03, n_kf)
    z = np.stack([np.cos(yaw), np.sin(yaw), np.zeros(n_kf)], 1)
    y = np.tile([0.0, 0.0, -1.0], (n_kf, 1))
    R = np.stack([np.cross(y, z), y, z], 1)

    def project(R, c, X):
        p = np.einsum("...ij,...j->...i", R, X - c)
        with np.errstate(all="ignore"):
            return p[..., 2], FX * p[..., 0] / p[..., 2] + CX, FY * p[..., 1] / p[..., 2] + CY

    offs = np.concatenate([np.arange(-20, 9), n_kf // 2 + np.arange(-20, 9)])
    pts, seen, n, tries = [], [], 0, 0
    while n < n_lm:
        tries += 1
        if tries > 400:
            raise RuntimeError("points seen often enough were not found")
        m = min(40_000, int(1.5 * (n_lm - n)) + 64)
        home = rng.integers(0, n_kf, m)
        d = rng.uniform(1.5, 12.0, m)
        p = np.stack([(rng.uniform(0, WIDTH, m) - CX) / FX * d, (rng.uniform(0, HEIGHT, m) - CY) / FY * d, d], 1)
        X = np.einsum("nji,nj->ni", R[home], p) + c[home]
        cand = home[:, None] + offs
        k = cand % n_kf
        dep, u, v = project(R[k], c[k], X[:, None])
        vis = (dep > 1.0) & (dep < 25.0) & (u >= 0) & (u < WIDTH) & (v >= 0) & (v < HEIGHT)
        if n_kf < 2 * offs.size:   # a keyframe may appear twice among the candidates: keep its first
            order = np.argsort(k, axis=1, kind="stable")
            ks = np.take_along_axis(k, order, 1)
            dup = np.zeros_like(vis)
            np.put_along_axis(dup, order[:, 1:], ks[:, 1:] == ks[:, :-1], 1)
            vis &= ~dup
        want = np.minimum(rng.integers(5, 16, m), vis.sum(1))
        key = np.where(vis, rng.random(vis.shape), 2.0)
        rank = np.argsort(np.argsort(key, axis=1), axis=1)
        take = (rank < want[:, None]) & vis
        ok = np.flatnonzero(vis.sum(1) >= min(5, n_kf))[: n_lm - n]
        rows, cols = np.nonzero(take[ok])
        pts.append(X[ok])
        seen.append((rows + n, k[ok][rows, cols]))
        n += ok.size
    X = np.concatenate(pts)
    ol = np.concatenate([s[0] for s in seen])
    ok = np.concatenate([s[1] for s in seen])
    _, u, v = project(R[ok], c[ok], X[ol])
    uv = np.stack([u, v], 1) + rng.normal(0.0, 1.0, (ol.size, 2))
    out = rng.random(ol.size) < 0.02
    uv[out] = rng.random((int(out.sum()), 2)) * [WIDTH, HEIGHT]
    w = rng.normal(0.0, 0.05, (n_kf, 3))
    ci = c + rng.normal(0.0, 0.1, c.shape)
    w[0], ci[0] = 0.0, c[0]
    Ri = np.stack([torch.stack(r, -1).numpy() for r in _so3(torch.from_numpy(w).T)[0]], 1) @ R
    Xi = X + rng.normal(0.0, 0.1, X.shape)
    keep = np.flatnonzero(project(Ri[ok], ci[ok], Xi[ol])[0] > 0.1)
    keep = np.sort(rng.permutation(keep)[: int(n_lm * MEAN_OBS["map"])])   # the count follows from the sizes alone
    Rt = np.concatenate([Ri.reshape(-1, 9), -np.einsum("nij,nj->ni", Ri, ci)], 1)
    return SimpleNamespace(kf_Rt_init=Rt, lm_init=Xi, obs_kf=ok[keep].astype(np.int32), obs_lm=ol[keep].astype(np.int32),
                           obs_uv=uv[keep], anchor_kf=np.zeros(1, np.int32),
                           intrinsics=lambda: (FX, FY, CX, CY, WIDTH, HEIGHT))


def _batch_sizes(case):
    """Uneven sizes, the benchmark's upper range: 20-200 keyframes, 100-5000 points each."""
    rng = np.random.Generator(np.random.PCG64(case["n_problems"]))
    return [(int(rng.integers(20, 201)), int(rng.integers(100, 5001))) for _ in range(case["n_problems"])]


def _problems(case, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    if case["kind"] == "batch":
        return [_map_problem(rng, n_kf, n_lm) for n_kf, n_lm in _batch_sizes(case)]
    if case["gen"] == "circle":
        return [synth.make_circle(seed, n_kf=case["n_kf"], n_lm=case["n_lm"])]
    if case["gen"] == "walk":
        return [synth.make_walk(seed, n_kf=case["n_kf"], n_lm=case["n_lm"])]
    return [_map_problem(rng, case["n_kf"], case["n_lm"])]


def _rows(case, seed):
    """Feature rows and damping targets with the shape of recorded ones: features in
    [0, 1], cosines in [-1, 1], targets in [0, 0.9] that depend on them."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    X = torch.rand((case["rows"], gbp.GBP_MLP_NFEAT), generator=gen, device="cuda")
    X[:, [7, 11]] = 2.0 * X[:, [7, 11]] - 1.0
    X[:, 1] = torch.where(X[:, 1] < 0.8, torch.ones_like(X[:, 1]), X[:, 1])
    T = (0.45 - 0.35 * X[:, 7] + 0.2 * (X[:, 4] - X[:, 8]) + 0.1 * torch.randn(case["rows"], generator=gen, device="cuda"))
    return X, T.clamp_(0.0, 0.9), gen


def prepare(case, seed):
    kind = case["kind"]
    s = SimpleNamespace(case=case, torch_stream=torch.cuda.current_stream().cuda_stream)
    if kind in ("solve", "batch", "report", "e2e"):
        s.problems = _problems(case, seed)
        s.options = dict(huber_nsigma=HUBER, precision_mode=case.get("precision", 0),
                         damping_mode=1 if case.get("learned") else 0)
        if kind == "e2e":
            return s
        s.graph = gbp.Graph(s.problems if kind == "batch" else s.problems[0], stream=s.torch_stream, **s.options)
        if case.get("learned"):
            s.net = gbp.DampingNet(learned.trained_params(), stream=s.torch_stream)
            s.graph.set_damping_model(s.net)
        if kind == "report":
            s.graph.iterate(case["iters"])
    elif kind == "stream":
        s.init, s.steps = synth.make_stream(seed, n_kf=case["n_kf"], n_lm=case["n_lm"], start_kf=case["start"])
        rng = np.random.Generator(np.random.PCG64(seed + 1))
        # new points start where a front end would have triangulated them
        s.new_lm = [st.new_lm_true + rng.normal(0.0, 0.05, st.new_lm_true.shape) for st in s.steps]
    elif kind == "are":
        rng = np.random.Generator(np.random.PCG64(seed))
        n_kf, n_lm, n = case["n_kf"], case["n_lm"], case["n_obs"]
        w = torch.from_numpy(rng.normal(0.0, 0.1, (3, n_kf)))
        R = torch.stack([torch.stack(r, -1) for r in _so3(w)[0]], 1).reshape(n_kf, 9)
        t = torch.from_numpy(rng.normal(0.0, 0.5, (n_kf, 3)) + [0.0, 0.0, 4.0])
        s.kf = torch.cat([R, t], 1).cuda()
        s.lm = torch.from_numpy(rng.uniform(-2.0, 2.0, (n_lm, 3))).cuda()
        s.obs_kf = torch.from_numpy(rng.integers(0, n_kf, n).astype(np.int32)).cuda()
        s.obs_lm = torch.from_numpy(rng.integers(0, n_lm, n).astype(np.int32)).cuda()
        gen = torch.Generator(device="cuda").manual_seed(seed)
        uv = torch.rand((n, 2), dtype=torch.float64, device="cuda", generator=gen)
        s.uv = uv * torch.tensor([WIDTH, HEIGHT], dtype=torch.float64, device="cuda")
        s.out = torch.zeros(2, dtype=torch.float64, device="cuda")
    else:
        s.X, s.T, gen = _rows(case, seed)
        s.params = learned.init_params(seed % 1000) if kind == "train" else learned.trained_params()
        s.net = gbp.DampingNet(s.params, stream=s.torch_stream)
        if kind == "train":
            s.idx = torch.randint(0, case["rows"], (case["steps"], case["batch"]), dtype=torch.int32, device="cuda",
                                  generator=gen)
        else:
            s.y = torch.empty(case["rows"], dtype=torch.float32, device="cuda")
    return s


# ---------------------------------------------------------------------------
# one pass

def _handed_on(case, arrays):
    return list(arrays) if case.get("precision") == 2 else [a.astype(np.float32) for a in arrays]


def run(s):
    case, kind = s.case, s.case["kind"]
    if kind in ("solve", "batch"):
        s.graph.reset()
        s.graph.iterate(case["iters"])
        return _handed_on(case, s.graph.beliefs())
    if kind == "e2e":
        with gbp.Graph(s.problems[0], stream=s.torch_stream, conv_tol=1e-6, iterations=case["iters"], check_every=25,
                       **s.options) as g:
            g.iterate()
            return _handed_on(case, g.beliefs())
    if kind == "stream":
        with gbp.Graph(s.init, stream=s.torch_stream, huber_nsigma=HUBER) as g:
            g.iterate(case["iters"])
            for st, new in zip(s.steps, s.new_lm):
                g.add_keyframe(st.obs_lm, st.obs_uv, n_new_lm=st.n_new_lm, new_lm_xyz=new if st.n_new_lm else None)
                g.iterate(case["iters"])
            return _handed_on(case, g.beliefs())
    if kind == "report":
        st = s.graph.stats()
        return dict(residuals=s.graph.residuals().astype(np.float32), are=st["are"], n_are=st["n_are"],
                    huber=st["huber_count"])
    if kind == "are":
        gbp.gbp_reprojection_error_noalloc((FX, FY, CX, CY, WIDTH, HEIGHT), 0.05, case["n_kf"], s.kf.data_ptr(),
                                           case["n_lm"], s.lm.data_ptr(), case["n_obs"], s.obs_kf.data_ptr(),
                                           s.obs_lm.data_ptr(), s.uv.data_ptr(), s.out.data_ptr(), s.torch_stream)
        return s.out
    if kind == "train":
        s.net.set_params(s.params)
        for idx in s.idx:
            s.net.train_step(s.X.data_ptr(), s.T.data_ptr(), case["batch"], 1e-3, idx_ptr=idx.data_ptr())
        return s.net.params
    s.net.forward(s.X.data_ptr(), case["rows"], s.y.data_ptr())
    return s.y


# ---------------------------------------------------------------------------
# what a pass cannot do without

def work(case):
    kind = case["kind"]
    if kind in ("train", "predict"):
        rows = case["rows"] if kind == "predict" else case["steps"] * case["batch"]
        mac = 16 * 64 + 64 * 64 + 64
        if kind == "predict":
            return dict(bytes=rows * 68 + 4 * gbp.GBP_MLP_NPARAM, flops=2 * mac * rows)
        return dict(bytes=rows * 72 + 2 * 4 * gbp.GBP_MLP_NPARAM, flops=6 * mac * rows)
    if kind == "are":
        return dict(bytes=24 * case["n_obs"] + 96 * case["n_kf"] + 24 * case["n_lm"] + 16, flops=60 * case["n_obs"])
    if kind == "batch":
        n_kf, n_lm = (sum(n) for n in zip(*_batch_sizes(case)))
    elif kind == "stream":   # the graph grows linearly: its mean size
        n_kf, n_lm = (case["n_kf"] + case["start"]) / 2, case["n_lm"] / 2
    else:
        n_kf, n_lm = case["n_kf"], case["n_lm"]
    n_f = n_lm * MEAN_OBS[case.get("gen", "walk")]
    real = 8 if case.get("precision") == 2 else 4
    if kind == "report":
        return dict(bytes=n_f * (16 + 2 * real + 8) + n_kf * 6 * real + n_lm * 3 * real, flops=200 * n_f)
    iters = case["iters"] * (case["n_kf"] - case["start"] + 1 if kind == "stream" else 1)
    # per iteration and factor: both messages (3 + 2 numbers each) read and written, the
    # linearisation read; per variable: belief and mean read and written, prior read
    per = n_f * real * (4 * 5 + 15) + n_kf * real * (2 * 33 + 6) + n_lm * real * (2 * 12 + 3)
    return dict(bytes=iters * per, flops=iters * 700 * n_f)


# ---------------------------------------------------------------------------
# the same in 64 bits: plain torch, one tensor per matrix entry over all factors

def _so3(w):
    """Exp(w) and the left Jacobian, as 3 x 3 nested lists of tensors."""
    th2 = (w[0] * w[0] + w[1] * w[1] + w[2] * w[2]).clamp_min(1e-30)
    th = th2.sqrt()
    small = th2 < 1e-6
    a = torch.where(small, 1 - th2 / 6, th.sin() / th)
    b = torch.where(small, 0.5 - th2 / 24, 2 * (0.5 * th).sin() ** 2 / th2)
    c = torch.where(small, 1.0 / 6 - th2 / 120, (th - th.sin()) / (th2 * th))
    zero = torch.zeros_like(th)
    K = [[zero, -w[2], w[1]], [w[2], zero, -w[0]], [-w[1], w[0], zero]]
    K2 = [[w[i] * w[j] - (th2 if i == j else 0) for j in range(3)] for i in range(3)]
    eye = [[1.0 if i == j else 0.0 for j in range(3)] for i in range(3)]
    return ([[eye[i][j] + a * K[i][j] + b * K2[i][j] for j in range(3)] for i in range(3)],
            [[eye[i][j] + b * K[i][j] + c * K2[i][j] for j in range(3)] for i in range(3)])


def _cholesky(A):
    n = len(A)
    L = [[None] * n for _ in range(n)]
    for j in range(n):
        L[j][j] = (A[j][j] - sum(L[j][p] * L[j][p] for p in range(j))).sqrt()
        for i in range(j + 1, n):
            L[i][j] = (A[i][j] - sum(L[i][p] * L[j][p] for p in range(j))) / L[j][j]
    return L


def _forward(L, b):
    x = []
    for i in range(len(L)):
        x.append((b[i] - sum(L[i][p] * x[p] for p in range(i))) / L[i][i])
    return x


def _backward(L, b):
    n, x = len(L), [None] * len(L)
    for i in reversed(range(n)):
        x[i] = (b[i] - sum(L[p][i] * x[p] for p in range(i + 1, n))) / L[i][i]
    return x


def _dot(a, b):
    return sum(x * y for x, y in zip(a, b))


class _Exact:
    """GBP on one problem in 64 bits: full messages, Schur complements through the
    2 x 2 form of the matrix inversion lemma, the schedule of Sec. 8."""

    def __init__(self, p, huber):
        dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")
        self.huber = huber
        Rt, X = dev(p.kf_Rt_init).double(), dev(p.lm_init).double()
        self.k, self.m = dev(p.obs_kf).long(), dev(p.obs_lm).long()
        self.z = list(dev(p.obs_uv).double().T)
        self.R0 = Rt[:, :9].reshape(-1, 3, 3)
        self.c0, self.X0 = -torch.einsum("nji,nj->ni", self.R0, Rt[:, 9:]), X
        self.n = [Rt.shape[0], X.shape[0]]
        self.x0 = [torch.zeros_like(self.z[0]) for _ in range(9)]
        self.tlin = torch.zeros_like(self.k)
        self.mu = [[torch.zeros(c, dtype=torch.float64, device="cuda") for _ in range(d)]
                   for c, d in zip(self.n, (6, 3))]
        self.J, self.y, self.W, _, _ = self.linearise(self.x0, 0.0)
        D = []
        for side, idx, cols in ((0, self.k, range(6)), (1, self.m, range(6, 9))):
            deg = self.sum(side, torch.ones_like(self.W), idx).clamp_min(1)
            d = torch.stack([self.sum(side, self.J[0][j] ** 2 + self.J[1][j] ** 2, idx) / deg for j in cols])
            top = d.max(0).values
            D.append(list(torch.where(top > 0, torch.maximum(d, 1e-9 * top), torch.ones_like(d))))
        self.D = D
        self.anchor = torch.zeros(self.n[0], dtype=torch.float64, device="cuda")
        self.anchor[dev(p.anchor_kf).long()] = 1000.0
        self.J, self.y, self.W, _, _ = self.linearise(self.x0, huber)
        self.msg = [([[torch.zeros_like(self.W) for _ in range(i + 1)] for i in range(d)],
                     [torch.zeros_like(self.W) for _ in range(d)]) for d in (6, 3)]
        self.t = 0
        self.beliefs()

    def sum(self, side, v, idx):
        return torch.zeros(self.n[side], dtype=torch.float64, device="cuda").index_add_(0, idx, v)

    def linearise(self, x, huber):
        E, Jw = _so3(x[3:6])
        Rk = [[self.R0[self.k, i, j] for j in range(3)] for i in range(3)]
        R = [[_dot(E[i], [Rk[q][j] for q in range(3)]) for j in range(3)] for i in range(3)]
        d = [(self.X0[self.m, i] - self.c0[self.k, i]) + (x[6 + i] - x[i]) for i in range(3)]
        p = [_dot(R[i], d) for i in range(3)]
        front = p[2] >= 0.05
        iz = 1.0 / torch.where(front, p[2], torch.ones_like(p[2]))
        u, v = FX * p[0] * iz, FY * p[1] * iz
        r = [self.z[0] - (u + CX), self.z[1] - (v + CY)]
        zero = torch.zeros_like(u)
        q = [[FX * iz, zero, -u * iz], [zero, FY * iz, -v * iz]]
        J = []
        for a in range(2):
            l = [_dot(q[a], [R[i][j] for i in range(3)]) for j in range(3)]
            x_ = [q[a][1] * p[2] - q[a][2] * p[1], q[a][2] * p[0] - q[a][0] * p[2], q[a][0] * p[1] - q[a][1] * p[0]]
            w = [-_dot(x_, [Jw[i][j] for i in range(3)]) for j in range(3)]
            J.append([torch.where(front, e, zero) for e in [-e for e in l] + w + l])
        err = (r[0] ** 2 + r[1] ** 2).sqrt()
        W = torch.ones_like(err)
        if huber > 0:
            M = err.clamp_min(huber)
            W = torch.where(err > huber, 2 * huber / M - (huber / M) ** 2, W)
        y = [torch.where(front, r[a] + _dot(J[a], x), zero) for a in range(2)]
        return J, y, torch.where(front, W, zero), err, front

    def beliefs(self):
        s = 0.01 ** (min(self.t, 10) / 10)
        self.bel = []
        for side, idx, d in ((0, self.k, 6), (1, self.m, 3)):
            lam, eta = self.msg[side]
            A = [[self.sum(side, lam[i][j], idx) for j in range(i + 1)] for i in range(d)]
            e = [self.sum(side, eta[i], idx) for i in range(d)]
            for i in range(d):
                A[i][i] = A[i][i] + s * self.D[side][i] + (self.anchor * self.D[0][i] if side == 0 else 0)
            L = _cholesky(A)
            self.bel.append((A, e))
            self.mu[side] = _backward(L, _forward(L, e))

    def step(self):
        t, x = self.t, [v[self.k] for v in self.mu[0]] + [v[self.m] for v in self.mu[1]]
        cav = []
        for side, idx, d in ((0, self.k, 6), (1, self.m, 3)):
            (A, e), (lam, eta) = self.bel[side], self.msg[side]
            L = _cholesky([[A[i][j][idx] - lam[i][j] for j in range(i + 1)] for i in range(d)])
            cav.append((L, [e[i][idx] - eta[i] for i in range(d)]))
        move = sum((a - b) ** 2 for a, b in zip(x, self.x0)).sqrt()
        take = (t - self.tlin >= 10) & (move > 0.01)
        self.tlin = torch.where(take, torch.full_like(self.tlin, t), self.tlin)
        self.x0 = [torch.where(take, a, b) for a, b in zip(x, self.x0)]
        if t >= 10:
            J, y, W, _, _ = self.linearise(self.x0, self.huber)
            self.J = [[torch.where(take, a, b) for a, b in zip(J[r], self.J[r])] for r in range(2)]
            self.y = [torch.where(take, a, b) for a, b in zip(y, self.y)]
            self.W = torch.where(take, W, self.W)
        keep = torch.where(t - self.tlin >= 8, 0.4, 0.0).double()
        cols, new = (range(6), range(6, 9)), []
        for side in (0, 1):
            L, q = cav[1 - side]
            B = [_forward(L, [self.J[a][j] for j in cols[1 - side]]) for a in range(2)]
            f, W = _forward(L, q), self.W
            a00, a01, a11 = 1 + W * _dot(B[0], B[0]), W * _dot(B[0], B[1]), 1 + W * _dot(B[1], B[1])
            det = a00 * a11 - a01 * a01
            M = [[W * a11 / det, -W * a01 / det], [-W * a01 / det, W * a00 / det]]
            e = [self.y[a] - _dot(B[a], f) for a in range(2)]
            g = [_dot(M[a], e) for a in range(2)]
            Ja = [[self.J[a][j] for j in cols[side]] for a in range(2)]
            d = len(cols[side])
            MJ = [[_dot([M[a][0], M[a][1]], [Ja[0][j], Ja[1][j]]) for j in range(d)] for a in range(2)]
            lam = [[Ja[0][i] * MJ[0][j] + Ja[1][i] * MJ[1][j] for j in range(i + 1)] for i in range(d)]
            eta = [(1 - keep) * (Ja[0][i] * g[0] + Ja[1][i] * g[1]) + keep * self.msg[side][1][i] for i in range(d)]
            new.append((lam, eta))
        self.msg = new
        self.t += 1
        self.beliefs()

    def world(self):
        E, _ = _so3(self.mu[0][3:6])
        R = torch.stack([torch.stack(r, -1) for r in E], 1) @ self.R0
        c = self.c0 + torch.stack(self.mu[0][:3], 1)
        Rt = torch.cat([R.reshape(-1, 9), -torch.einsum("nij,nj->ni", R, c)], 1)
        return Rt.cpu().numpy(), (self.X0 + torch.stack(self.mu[1], 1)).cpu().numpy()


def _exact_train(case, seed):
    X, T, gen = _rows(case, seed)
    W = torch.from_numpy(learned.init_params(seed % 1000)).cuda().double()
    idx = torch.randint(0, case["rows"], (case["steps"], case["batch"]), dtype=torch.int32, device="cuda", generator=gen)
    m, v = torch.zeros_like(W), torch.zeros_like(W)
    for t, rows in enumerate(idx, 1):
        w = W.clone().requires_grad_(True)
        loss = ((_network(w, X[rows.long()].double()) - T[rows.long()].double()) ** 2).mean()
        g, = torch.autograd.grad(loss, w)
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        W = W - 1e-3 * (m / (1 - 0.9 ** t)) / ((v / (1 - 0.999 ** t)).sqrt() + 1e-8)
    return W.cpu().numpy()


def _network(w, X):
    h = torch.relu(X @ w[:1024].reshape(16, 64) + w[1024:1088])
    h = torch.relu(h @ w[1088:5184].reshape(64, 64) + w[5184:5248])
    return 0.9 * torch.sigmoid(h @ w[5248:5312] + w[5312])


def exact(case, seed):
    kind = case["kind"]
    if kind == "train":
        return _exact_train(case, seed)
    if kind == "predict":
        w = torch.from_numpy(learned.trained_params()).cuda().double()
        return torch.cat([_network(w, x.double()) for x in _rows(case, seed)[0].split(1 << 18)])
    if kind == "are":
        s = prepare(case, seed)
        Rt, X = s.kf[s.obs_kf.long()], s.lm[s.obs_lm.long()]
        p = torch.einsum("nij,nj->ni", Rt[:, :9].reshape(-1, 3, 3), X) + Rt[:, 9:]
        ok = p[:, 2] >= 0.05
        uv = torch.stack([FX * p[:, 0] / p[:, 2] + CX, FY * p[:, 1] / p[:, 2] + CY], 1)
        err = torch.linalg.norm(s.uv - uv, dim=1)[ok]
        return torch.stack([err.mean(), ok.sum().double()])
    if kind == "stream" or case.get("learned"):
        return None   # the schedules of added variables and of the network are not restated here
    if kind == "e2e":
        return None   # where the iteration stops depends on the last digits of the mean change
    kf, lm = [], []
    for p in _problems(case, seed):
        g = _Exact(p, HUBER)
        for _ in range(case["iters"]):
            g.step()
        if kind == "report":
            x = [v[g.k] for v in g.mu[0]] + [v[g.m] for v in g.mu[1]]
            _, _, _, err, front = g.linearise(x, 0.0)
            return dict(residuals=torch.where(front, err, torch.full_like(err, -1.0)), are=float(err[front].mean()),
                        n_are=None, huber=None)
        a, b = g.world()
        kf.append(a)
        lm.append(b)
    return [np.concatenate(kf), np.concatenate(lm)]
