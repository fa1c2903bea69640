"""Autotuning images whose weights rule out the pixel-domain z-update: a tiling tuned for the Gaussian
weights is not handed to them, their own one is cached, and their solves match the oracle (the 1e-4
of the parity tests)."""
import numpy as np
import pytest

from oracle import segsalsa_str_oracle as O
from paper_1504_07028_gb300 import synth
from tests.helpers import max_abs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B(lib):
    from paper_1504_07028_gb300 import binding
    return binding


def test_larger_weights_have_their_own_tilings(B):
    sizes, K = [(72, 64), (66, 75)], 5
    om = 1.5 * O.gaussian_weights(1, 0.5)
    make = lambda w: [B.make_params(H, W, K, sigma=0.5, lam=1.2, mu=1.0, weights=w) for H, W in sizes]
    b = B.Batch(make(None))
    b.autotune(2)
    b.close()
    fresh = B.Batch(make(om))
    for i, (H, W) in enumerate(sizes):
        s = B.Solver(make(om)[i])
        assert fresh.image(i).tiling() == s.tiling()
        s.close()
    chosen = fresh.autotune(2)
    fresh.close()
    b = B.Batch(make(om))
    assert [b.image(i).tiling() for i in range(len(sizes))] == chosen
    sc = [synth.scene(H, W, K, S=6, gap=2.0, noise_std=1.0, wrong_frac=0.0, seed=H) for H, W in sizes]
    for i, s in enumerate(sc):
        b.image(i).set_probs(s.p.astype(np.float32))
    b.solve(25)
    for i, s in enumerate(sc):
        ref, _ = O.solve(s.p.astype(np.float32).astype(np.float64), 1, 0.5, 1.2, 1.0, 1, 25, omega=om)
        assert max_abs(b.image(i).get_z(), ref.z) < 1e-4
        assert b.image(i).kernel_stats()["column_solve"][0] > 0
    b.close()
