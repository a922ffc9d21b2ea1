"""The automatic launch mode's choices: what gbp_autotune measured is what runs, a choice holds for the graphs it was
made for, and every way leads to the bits of per-phase launches."""
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
