"""Small-|Q| points of shapes of few faces, which the finishing kernel sums over the faces itself (up to 256 faces and
3,000 units of a point and 32 faces), and the Q-gradient's line between direct sums and moments, at the edges of
both rules, against the series in numpy.  Tolerance as for the small-|Q| pass: 1e-12 of the largest value."""
import numpy as np
import pytest

from paper_2104_08309_gb300 import synth

pytestmark = pytest.mark.gpu
K = 16


def _series(v, f, q, c):
    """S(Q) = sum det sum_k i^k h_k(x) / (k + 3)! over the tetrahedra (c, face), times e^{iQ.c}, and its gradient in Q
    by central differences of the 64-bit series (step 1e-4 of the radius' inverse: 1e-8 relative)."""
    P = v[f].astype(np.float64) - c
    det = np.linalg.det(P)
    w = np.cumprod(1.0 / np.r_[6.0, np.arange(4, K + 4)]) * 1j ** np.arange(K + 1)
    out = np.zeros(q.shape[0], dtype=complex)
    for m in range(P.shape[0]):
        x = q @ P[m].T
        h = np.zeros((q.shape[0], K + 1))
        h[:, 0] = 1.0
        for j in range(3):
            for k in range(1, K + 1):
                h[:, k] += x[:, j] * h[:, k - 1]
        out += det[m] * (h @ w)
    return out * np.exp(1j * (q @ c))


def _case(n_faces, n_small, n_big, seed):
    v, f = synth.perturbed_icosphere(2, seed=5)
    f = f[:n_faces]                                   # an open surface is a signed sum of cones as well
    v = (v + np.float32(0.5)).astype(np.float32)
    c = 0.5 * (v.min(0).astype(np.float64) + v.max(0))
    radius = np.linalg.norm(v[f].reshape(-1, 3) - c, axis=1).max()
    rng = np.random.default_rng(seed)
    d = rng.normal(size=(n_small, 3))
    q = d / np.linalg.norm(d, axis=1, keepdims=True) * (0.2499 * rng.uniform(0.01, 1, (n_small, 1))) / radius
    return v, np.ascontiguousarray(f), c, q, rng.normal(size=(n_big, 3)) * 9.0 / radius


@pytest.mark.parametrize("n_faces,n_small,n_big", [(1, 1, 0), (12, 33, 0), (12, 3000, 0), (12, 3001, 0), (31, 40, 7),
                                                   (32, 500, 0), (33, 1500, 0), (33, 1501, 0), (255, 375, 0),
                                                   (256, 375, 0), (256, 376, 0), (257, 33, 0), (257, 20, 9),
                                                   (64, 300, 20000), (64, 20, 70000)])
def test_forward(n_faces, n_small, n_big):
    torch = pytest.importorskip("torch")
    import paper_2104_08309_gb300 as pft
    v, f, c, q, big = _case(n_faces, n_small, n_big, n_faces + n_small)
    ref = _series(v, f, q, c)
    a = [torch.from_numpy(x).cuda() for x in (v, f, np.concatenate([q, big]))]
    out = pft.pft3d_mesh(*a, check_status=True).cpu().numpy()
    assert np.isfinite(out).all()
    assert np.abs(out[:n_small, 0] + 1j * out[:n_small, 1] - ref).max() <= 1e-12 * np.abs(ref).max()


@pytest.mark.parametrize("n_faces,n_small", [(12, 33), (12, 666), (12, 667), (80, 312), (80, 313), (320, 108), (320, 109)])
def test_q_gradient(n_faces, n_small):
    """Against the other side of the rule: the points one by one in calls of up to 32, which are always direct."""
    torch = pytest.importorskip("torch")
    import paper_2104_08309_gb300 as pft
    v, f, c, q, _ = _case(n_faces, n_small, 0, n_faces)
    g = np.random.default_rng(1).normal(size=(n_small, 2))
    a = [torch.from_numpy(x).cuda() for x in (v, f, q, g)]
    got = pft.pft3d_mesh_qgrad(*a, check_status=True)
    ref = torch.cat([pft.pft3d_mesh_qgrad(a[0], a[1], a[2][i:i + 32], a[3][i:i + 32]) for i in range(0, n_small, 32)])
    assert (got - ref).abs().max().item() <= 1e-12 * ref.abs().max().item()
