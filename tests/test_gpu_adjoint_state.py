"""After the reverse pass the handle stands where `iters` iterations from p leave it: further iterations
continue bit for bit, whatever the checkpoint interval, and a second pass on the same handle (whose
memory is kept) gives the first one's gradient."""
import numpy as np
import pytest

from paper_1504_07028_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B(lib):
    from paper_1504_07028_gb300 import binding
    return binding


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("g4", ["affine", "simplex"])
@pytest.mark.parametrize("iters,every", [(1, 1), (7, 7), (7, 3), (8, 4), (20, 50), (40, 17)])
def test_backward_leaves_the_final_state(B, prec, g4, iters, every):
    H, W, K = 19, 23, 5
    dt = np.float64 if prec == "fp64" else np.float32
    sc = synth.scene(H, W, K, S=4, gap=2.0, noise_std=1.0, wrong_frac=0.0, seed=iters)
    logp = np.log(sc.p).astype(dt)
    zbar = synth.random_field((K, H, W), seed=2).astype(dt)
    hs = []
    for _ in range(2):
        s = B.Solver(B.make_params(H, W, K, M=1, sigma=0.5, lam=1.2, mu=1.1, precision=prec))
        s.set_g4(g4)
        s.set_log_probs(logp)
        hs.append(s)
    a, b = hs
    g = a.backward(iters, zbar, every)
    g2 = a.backward(iters, zbar, every)
    assert np.array_equal(g[0], g2[0]) and g[1] == g2[1] and np.array_equal(g[2], g2[2])
    b.solve(iters)
    assert a.get_iteration() == iters
    sa, sb = a.get_state(), b.get_state()
    for k in sa:
        assert np.array_equal(sa[k], sb[k]), k
    a.solve(21)
    b.solve(21)
    assert np.array_equal(a.get_z(), b.get_z())
    for s in hs:
        s.close()
