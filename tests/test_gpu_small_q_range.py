"""Small-|Q| points of a shape so small, and at |Q| so large, that Q as a float overflows: the transform scales,
F(s v, Q/s) = s^3 F(v, Q), and s = 2^-133 scales these vertices exactly (FP32 denormals), Q r_max staying
below 1/4.  Both calls evaluate the same FP64 series on numbers that differ by powers of two; only roundings of
the radius in units of 2^-149 differ, which the series does not see, and sums of a few terms: held to 1e-13."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

S = 2.0 ** -133


@pytest.mark.parametrize("n_small", [1, 20, 33, 100])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_scaled(n_small, precision):
    torch = pytest.importorskip("torch")
    import paper_2104_08309_gb300 as pft
    v = np.array([[0, 0, 0], [16, 0, 0], [0, 8, 0], [0, 0, 24]], dtype=np.float64) / 32.0
    f = np.array([[0, 2, 1], [0, 1, 3], [0, 3, 2], [1, 2, 3]], dtype=np.int32)
    q = np.random.default_rng(n_small).uniform(-1, 1, (n_small, 3))
    q *= np.exp2(-3) / np.linalg.norm(q, axis=1, keepdims=True)      # |Q| r_max = 0.06
    assert (np.abs(q / S).max(axis=1) > np.finfo(np.float32).max).any()
    assert (np.float64(np.float32(v * S)) == v * S).all()
    def call(vv, qq):
        a = [torch.from_numpy(x).cuda() for x in (vv.astype(np.float32), f, qq)]
        return pft.pft3d_mesh(*a, options={"precision": precision}, check_status=True).cpu().numpy()
    got, ref = call(v * S, q / S), call(v, q)
    assert np.abs(got * S ** -3 - ref).max() <= 1e-13 * np.abs(ref).max()
