"""The FP32 transform passes of the z-update, which run for weights whose squares sum to more than 1.0005
and where a tiling asks for them: the row lengths that only they depend on, the handle-free call
with its tables, and whole solves. Tolerances are those of the same comparisons in the parity, full-size
and allocation-free tests."""
import numpy as np
import pytest

from oracle import segsalsa_str_oracle as O
from paper_1504_07028_gb300 import synth
from tests.helpers import hwk_to_khw, khw_to_hwk, label_agreement, max_abs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B(lib):
    from paper_1504_07028_gb300 import binding
    return binding


def _ran_passes(s, n):
    st = s.kernel_stats()
    return (st["row_fft_forward"][0], st["column_solve"][0], st["row_fft_inverse"][0],
            st["zupdate_fused"][0]) == (n, n, n, 0)


@pytest.mark.parametrize("H,W,K,M", [
    (64, 64, 4, 1), (145, 145, 16, 1), (37, 50, 5, 2), (97, 509, 4, 1), (256, 256, 8, 1), (61, 2048, 3, 1),
    (33, 17, 32, 1), (40, 143, 4, 1), (24, 121, 3, 1), (18, 546, 5, 1), (20, 206, 4, 1), (30, 127, 3, 1),
    (12, 1999, 4, 1), (12, 2047, 4, 1)])
@pytest.mark.parametrize("zfuse,wscale", [(1, 1.0), (0, 1.5)])
def test_linear_solve(B, H, W, K, M, zfuse, wscale):
    """Direct prime stages, their radix-7 and radix-3 tails and Bluestein lengths, by an explicit tiling
    and by the weights."""
    om = wscale * O.gaussian_weights(M, 0.5 + 0.5 * M)
    s = B.Solver(B.make_params(H, W, K, M=M, sigma=0.5 + 0.5 * M, weights=om), tiling=B.make_tiling(zfuse=zfuse))
    rhs = synth.random_field((K, H, W), seed=H * 1000 + W).astype(np.float32)
    z = hwk_to_khw(s.linear_solve(khw_to_hwk(rhs)))
    assert _ran_passes(s, 1)
    s.close()
    ref = O.linear_solve(rhs.astype(np.float64), om, M)
    assert max_abs(z, ref) <= 2e-5 * np.abs(ref).max()


def test_static_geometries_chained(B):
    """Geometries and weights A, B, C, A on one non-default stream with no synchronisation: every call
    rebuilds the tables in the static array and the row pass that follows must see them."""
    import torch
    om1, om2 = 1.5 * O.gaussian_weights(1, 0.5), np.ones(9)
    calls = [(96, 80, 8, om1), (61, 127, 4, om1), (61, 127, 4, om2), (96, 80, 8, om1)]
    rhs_np = [synth.random_field((H, W, K), 300 + j).astype(np.float32) for j, (H, W, K, _) in enumerate(calls)]
    rhs = [torch.from_numpy(r).cuda() for r in rhs_np]
    outs = [torch.full_like(r, float("nan")) for r in rhs]
    refs = []
    for (H, W, K, om), r in zip(calls, rhs):
        s = B.Solver(B.make_params(H, W, K, M=1, weights=om))
        refs.append(s.linear_solve(r).cpu().numpy())
        assert _ran_passes(s, 1)
        s.close()
    torch.cuda.synchronize()
    st = torch.cuda.Stream()
    for (H, W, K, om), r, o in zip(calls, rhs, outs):
        assert B.segsalsa_str_linear_solve_static(r, o, c_omega=float(np.sum(om ** 2)),
                                                  stream=st.cuda_stream) == B.SEGSALSA_OK
    st.synchronize()
    for j, (o, ref) in enumerate(zip(outs, refs)):
        z = o.cpu().numpy()
        assert np.abs(z - ref).max() <= 1e-6 * np.abs(ref).max(), j
        zo = np.moveaxis(O.linear_solve(np.moveaxis(rhs_np[j].astype(np.float64), -1, 0), calls[j][3], 1), 0, -1)
        assert np.abs(z - zo).max() <= 2e-5 * np.abs(zo).max(), j


def test_solve_fused_and_three_launch_agree(B):
    """Whole 145 x 145, K = 16 solves with the z-update over 8-CTA clusters and in three launches."""
    sc = synth.scene(145, 145, 16, S=40, gap=2.0, noise_std=1.5, wrong_frac=0.05, seed=2)
    out = []
    for zf in (8, 1):
        s = B.Solver(B.make_params(145, 145, 16, M=1, sigma=0.5, lam=1.5, mu=1.0, schatten_p=1,
                                   precision="fp32"), tiling=B.make_tiling(zfuse=zf))
        s.set_probs(sc.p.astype(np.float32))
        s.solve(60)
        assert _ran_passes(s, 59) if zf == 1 else s.kernel_stats()["zupdate_fused"][0] == 59
        out.append(s.get_z())
        s.close()
    ref, _ = O.solve(sc.p, 1, 0.5, 1.5, 1.0, 1, 60)
    for z in out:
        assert max_abs(z, ref.z) < 1e-4
    assert max_abs(out[0], out[1]) < 1e-5


@pytest.mark.parametrize("H,W,K,sp", [(1021, 1999, 16, 1), (1499, 2047, 8, 2)])
def test_large_rows_against_fp64(B, H, W, K, sp):
    """Rows of a Bluestein length and of two direct primes on large images, 30 iterations."""
    sc = synth.scene(H, W, K, S=24, gap=2.0, noise_std=1.0, wrong_frac=0.05, seed=H + W)
    z = {}
    for prec, dt in (("fp32", np.float32), ("fp64", np.float64)):
        s = B.Solver(B.make_params(H, W, K, M=1, sigma=0.5, lam=1.5, mu=1.0, schatten_p=sp, precision=prec),
                     tiling=B.make_tiling(zfuse=1))
        s.set_probs(sc.p.astype(dt))
        s.solve(30, trace_every=10)
        z[prec] = s.get_z()
        s.close()
    assert max_abs(z["fp32"], z["fp64"]) < 1e-4
    assert label_agreement(z["fp32"], z["fp64"])[0]
