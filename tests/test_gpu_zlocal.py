"""The pixel-domain z-update (FP32, sum of squared weights at most 1) against the FP64 solve of eq.
(12) and against the three-launch form, at the sizes where its two kernels can go wrong: tile and
strip edges, images smaller than the halo, class counts off the quads, unaligned buffers.

Tolerance: an update x <- w g S + (1 - w) x + w b makes at most 6 roundings (u = 6e-8) and passes on
at most 4 w g + |1 - w| <= 0.73 of the errors before it, so the error stays below 6 u / 0.27 = 1.4e-6
of max |z|; truncation and halo add 3e-8."""
import numpy as np
import pytest

from oracle import segsalsa_str_oracle as O
from paper_1504_07028_gb300 import synth
from tests.helpers import hwk_to_khw, khw_to_hwk, max_abs

pytestmark = pytest.mark.gpu

TOL = 1.5e-6


@pytest.fixture(scope="module")
def B(lib):
    from paper_1504_07028_gb300 import binding
    return binding


def _check(z, rhs, om, M):
    ref = O.linear_solve(rhs.astype(np.float64), om, M)
    assert max_abs(z, ref) <= TOL * np.abs(ref).max()


@pytest.mark.parametrize("H,W,K,M,scale", [
    (2, 2, 2, 0, 1.0), (4, 5, 3, 1, 1.0), (13, 11, 5, 1, 1.0),   # smaller than the halo
    (1, 40, 4, 0, None), (64, 64, 4, 1, 1.0), (25, 103, 7, 1, 1.0), (145, 145, 16, 1, 1.0),
    (96, 104, 32, 1, 0.5), (30, 600, 2, 1, 1.0),                 # block form
    (610, 340, 9, 2, 1.0), (300, 313, 16, 1, 1.0), (512, 208, 17, 1, 1.0),   # streaming form
    (700, 105, 31, 1, 0.7), (40, 40, 6, 1, 0.0)])                # 0.0: the operator 3 I
def test_linear_solve(B, H, W, K, M, scale):
    if scale is None:                       # below the smallest image: still refused
        with pytest.raises(B.SegsalsaError):
            B.Solver(B.make_params(H, W, K, M=M))
        return
    om = scale * O.gaussian_weights(M, 0.5 + 0.5 * M)
    rhs = synth.random_field((K, H, W), seed=H + 7 * W).astype(np.float32)
    s = B.Solver(B.make_params(H, W, K, M=M, weights=om))
    z = hwk_to_khw(s.linear_solve(khw_to_hwk(rhs)))
    assert s.kernel_stats()["zupdate_fused"][0] == 1
    s.close()
    _check(z, rhs, om, M)


@pytest.mark.parametrize("H,W,K", [(64, 64, 4), (40, 70, 6), (300, 313, 16)])
@pytest.mark.parametrize("off", [1, 2])
def test_unaligned_buffers(B, H, W, K, off):
    """A caller's rhs and z that are only element-aligned give the aligned buffers' values."""
    import torch
    rhs = torch.from_numpy(khw_to_hwk(synth.random_field((K, H, W), seed=3)).astype(np.float32)).cuda()
    n = rhs.numel()
    a, z = torch.zeros(n + off, device="cuda"), torch.zeros(n + off, device="cuda")
    a[off:] = rhs.flatten()
    s = B.Solver(B.make_params(H, W, K))
    torch.cuda.synchronize()
    s.linear_solve(a[off:].view(H, W, K), z[off:].view(H, W, K))
    ref = s.linear_solve(rhs)
    torch.cuda.synchronize()
    assert torch.equal(z[off:].view(H, W, K), ref) and float(z[:off].abs().max()) == 0.0
    s.close()


@pytest.mark.parametrize("H,W,K,M", [(33, 47, 5, 1), (145, 145, 16, 1), (90, 61, 9, 2), (20, 24, 32, 0),
                                     (310, 330, 18, 1), (610, 340, 9, 2)])
def test_solve_matches_three_launches(B, H, W, K, M):
    """The sweep's partials in class quads, read by either kernel, against the transforms."""
    sc = synth.scene(H, W, K, S=12, gap=2.0, noise_std=1.0, wrong_frac=0.0, seed=H + W)
    out = []
    for zf in (0, 1):
        s = B.Solver(B.make_params(H, W, K, M=M), tiling=B.make_tiling(zfuse=zf))
        s.set_probs(sc.p.astype(np.float32))
        s.solve(20, trace_every=5)
        out.append((s.get_z(), s.get_state()["rhs"]))
        s.close()
    for a, b in zip(*out):
        assert max_abs(a, b) <= 2e-5 * np.abs(b).max()


def test_weights_switch_the_form_mid_solve(B):
    """set_weights across the limit: the partials of the last sweep change their layout's reader."""
    H, W, K = 50, 61, 6
    sc = synth.scene(H, W, K, S=6, gap=2.0, noise_std=1.0, wrong_frac=0.0, seed=9)
    om = O.gaussian_weights(1, 0.5)
    out = []
    for zf in (0, 1):
        s = B.Solver(B.make_params(H, W, K, weights=om), tiling=B.make_tiling(zfuse=zf))
        s.set_probs(sc.p.astype(np.float32))
        for f in (1.0, 1.5, 1.0, 0.8):
            s.set_weights(f * om)
            s.solve(19)
        out.append(s.get_z())
        s.close()
    assert max_abs(*out) < 1e-5
