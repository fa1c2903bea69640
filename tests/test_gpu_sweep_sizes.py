"""The fused sweep at the edges of its CTA sizes: images that take CTAs of 64 threads (the narrowest
that do, tiles off the column count, idle lanes and columns) and their neighbours that take 256,
against the oracle."""
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


@pytest.mark.parametrize("H,W,K,M,sp,g4,prec", [
    (9, 8, 16, 1, 1, "affine", "fp32"),       # two tiles of four columns
    (9, 7, 16, 1, 1, "affine", "fp32"),       # one column too few: 256 threads
    (13, 9, 11, 1, 2, "affine", "fp32"),      # idle lanes, three uneven tiles
    (12, 17, 8, 2, np.inf, "affine", "fp64"), # 5x5 patch, tiles of five and six columns
    (16, 15, 8, 2, 1, "simplex", "fp32"),
    (21, 33, 3, 1, np.inf, "affine", "fp64"), # class scalars shared by lanes, one idle
    (10, 40, 4, 0, 1, "simplex", "fp64"),
    (20, 24, 20, 1, np.inf, "affine", "fp32"),  # 32 lanes: 256 threads only
    (40, 61, 2, 2, 2, "affine", "fp64"),
    (64, 150, 13, 2, 1, "affine", "fp32"),
])
def test_solve_against_oracle(B, H, W, K, M, sp, g4, prec):
    sc = synth.scene(H, W, K, S=5, gap=2.0, noise_std=1.0, wrong_frac=0.0, seed=H * W + K)
    dt = np.float64 if prec == "fp64" else np.float32
    p = sc.p.astype(dt)
    s = B.Solver(B.make_params(H, W, K, M=M, sigma=max(0.5, M / 2), lam=1.2, mu=1.3, schatten_p=sp,
                               precision=prec))
    s.set_g4(g4)
    s.set_probs(p)
    tr = s.solve(15, trace_every=5)
    ref, rtr = O.solve(p.astype(np.float64), M, max(0.5, M / 2), 1.2, 1.3, sp, 15, trace_every=5, g4=g4)
    # the parity tests' tolerances: FP32 solves within 1e-4 of the oracle, FP64 within 1e-9
    assert max_abs(s.get_z(), ref.z) < (1e-9 if prec == "fp64" else 1e-4)
    assert np.allclose(np.asarray(tr)[:, 1:4], np.asarray(rtr)[:, 1:4], rtol=1e-9 if prec == "fp64" else 2e-3,
                       atol=1e-5 if prec == "fp32" else 1e-9)
    s.close()
