"""linear_solve with a z that overlaps its rhs (the same buffer, or views of one buffer shifted by a
pixel or by half an image) gives the separate buffers' values bit for bit in every form of the
z-update, and touches nothing outside z."""
import numpy as np
import pytest

from oracle import segsalsa_str_oracle as O
from paper_1504_07028_gb300 import synth
from tests.helpers import khw_to_hwk

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B(lib):
    from paper_1504_07028_gb300 import binding
    return binding


@pytest.mark.parametrize("H,W,K,prec,zfuse,wscale", [
    (145, 145, 16, "fp32", 0, 1.0), (64, 64, 4, "fp32", 0, 1.0), (31, 90, 7, "fp32", 0, 1.0),  # block form
    (610, 340, 9, "fp32", 0, 1.0), (300, 313, 16, "fp32", 0, 1.0),                 # streaming form
    (145, 145, 16, "fp32", 0, 1.5), (610, 340, 9, "fp32", 1, 1.0),                 # three launches
    (145, 145, 16, "fp64", 0, 1.0), (610, 340, 9, "fp64", 0, 1.0),
    (64, 64, 4, "fp32", 8, 1.0), (64, 64, 6, "fp32", 3, 1.0), (48, 50, 5, "fp64", 3, 1.0)])
def test_overlapping_buffers(B, H, W, K, prec, zfuse, wscale):
    import torch
    n = H * W * K
    dt = np.float64 if prec == "fp64" else np.float32
    rhs = torch.from_numpy(khw_to_hwk(synth.random_field((K, H, W), seed=H + W)).astype(dt)).cuda()
    s = B.Solver(B.make_params(H, W, K, precision=prec, weights=wscale * O.gaussian_weights(1, 0.5)),
                 tiling=B.make_tiling(zfuse=zfuse))
    ref = torch.empty_like(rhs)
    torch.cuda.synchronize()
    s.linear_solve(rhs, ref)
    half = (H // 2) * W * K
    for at_r, at_z in ((0, 0), (0, half), (half, 0), (0, K), (K, 0), (0, 1)):
        buf = torch.full((n + half,), 7.0, dtype=rhs.dtype, device="cuda")
        buf[at_r:at_r + n] = rhs.flatten()
        want = buf.clone()
        want[at_z:at_z + n] = ref.flatten()
        torch.cuda.synchronize()
        s.linear_solve(buf[at_r:at_r + n].view(H, W, K), buf[at_z:at_z + n].view(H, W, K))
        torch.cuda.synchronize()
        assert torch.equal(buf, want), (at_r, at_z)
    host = rhs.cpu().numpy()
    s.linear_solve(host, host)
    assert np.array_equal(host, ref.cpu().numpy())
    s.close()


@pytest.mark.parametrize("H,W,K", [(145, 145, 16), (300, 313, 16), (64, 96, 5)])
def test_static_overlapping_buffers(B, H, W, K):
    """The handle-free call on overlapping buffers: the transforms, for any weights. Tolerance: that of
    the FP32 transforms against 64 bits in the parity tests."""
    import torch
    n, half = H * W * K, (H // 2) * W * K
    rhs_np = synth.random_field((K, H, W), seed=H + 3 * W).astype(np.float32)
    ref = khw_to_hwk(O.linear_solve(rhs_np.astype(np.float64), O.gaussian_weights(1, 0.5), 1))
    rhs = torch.from_numpy(khw_to_hwk(rhs_np)).cuda()
    for at_r, at_z in ((0, 0), (half, 0), (0, half)):
        buf = torch.zeros(n + half, device="cuda")
        buf[at_r:at_r + n] = rhs.flatten()
        torch.cuda.synchronize()
        z = buf[at_z:at_z + n].view(H, W, K)
        assert B.segsalsa_str_linear_solve_static(buf[at_r:at_r + n].view(H, W, K), z) == B.SEGSALSA_OK
        torch.cuda.synchronize()
        assert np.abs(z.cpu().numpy() - ref).max() <= 2e-5 * np.abs(ref).max()
