"""The small-|Q| pass of the 3D forward calls (|Q| r_max < 1/4): up to 32 such points are evaluated one
by one, more of them from the shape's moments.  Both against the oracle, at the edges of that rule, of
the batches of 32 faces and of the face chunks, with larger Q points among them.

Tolerance: the FP64 bar of the other tests, 1e-12 of F(0) (the pass runs in FP64; its truncation and its
FP32 part stay below 1e-16 of it)."""
import numpy as np
import pytest

import oracle
from paper_2104_08309_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_dev():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2104_08309_gb300 import build as pbuild
    pbuild.build()
    return torch, torch.device("cuda:0")


@pytest.mark.parametrize("n_small", [1, 32, 33, 700])
@pytest.mark.parametrize("level,keep,shift,scale", [(0, None, 0.0, 1.0), (1, 65, 3.0, 1e6), (4, None, 0.5, 1e-6)])
def test_small_q_against_the_oracle(torch_dev, n_small, level, keep, shift, scale):
    torch, dev = torch_dev
    import paper_2104_08309_gb300 as pft
    v, f = synth.perturbed_icosphere(level, seed=2)
    f = f[:keep]                                      # an open surface is a signed sum of cones as well
    v = ((v + np.float32(shift)) * np.float32(scale)).astype(np.float32)
    c = 0.5 * (v.min(0).astype(np.float64) + v.max(0))
    radius = np.linalg.norm(v - c, axis=1).max()
    rng = np.random.default_rng(n_small)
    d = rng.normal(size=(n_small, 3))
    q = d / np.linalg.norm(d, axis=1, keepdims=True) * (10 ** rng.uniform(-6, np.log10(0.2499), (n_small, 1))) / radius
    big = rng.normal(size=(37, 3)) * 3.0 / radius
    q = rng.permutation(np.concatenate([q, big, np.zeros((2, 3))]))
    small = np.linalg.norm(q, axis=1) * radius < 0.25
    assert small.sum() >= n_small + 2
    # centred on the bounding box: the volume at Q = 0 of an open surface depends on the apex
    if keep is None:
        ref = oracle.ft3d(v, f, q)
    else:
        ref = np.empty(q.shape[0], dtype=complex)
        P = v[f].astype(np.float64) - c
        det = np.linalg.det(P)
        for i, Q in enumerate(q):
            x = P @ Q
            h = np.zeros((x.shape[0], 21))
            h[:, 0] = 1.0
            for j in range(3):
                for k in range(1, 21):
                    h[:, k] += x[:, j] * h[:, k - 1]
            w = np.cumprod(1.0 / np.r_[6.0, np.arange(4, 24)])
            ref[i] = np.sum(det * (h @ (w * 1j ** np.arange(21)))) * np.exp(1j * Q @ c)
    scale_f = np.abs(ref[small]).max()
    for precision in ("fp32", "fp64"):
        out = pft.pft3d_mesh(torch.from_numpy(v).to(dev), torch.from_numpy(f).to(dev), torch.from_numpy(q).to(dev),
                             options={"precision": precision}, check_status=True).cpu().numpy()
        got = out[:, 0] + 1j * out[:, 1]
        assert np.abs(got - ref)[small].max() <= 1e-12 * scale_f
        if keep is None:
            assert np.abs(got - ref).max() <= (1e-5 if precision == "fp32" else 1e-12) * scale_f


@pytest.mark.parametrize("n_small", [1, 24, 25, 33, 400])
@pytest.mark.parametrize("level,shift,scale", [(0, 0.0, 1.0), (2, 2.0, 1e5), (4, 0.5, 1e-5)])
def test_small_q_gradients_against_the_oracle(torch_dev, n_small, level, shift, scale):
    """Vertex gradient (up to 24 small points one by one, more through the polynomial of their sum) and
    Q-gradient (up to 32 one by one, more through the moments), small points only.  The vertex gradient
    is rounded to float32 once: 6e-8 of a value, held to 2e-7 of the largest; the Q-gradient to 1e-9
    of max|g| V max|r|."""
    torch, dev = torch_dev
    import paper_2104_08309_gb300 as pft
    v, f = synth.perturbed_icosphere(level, seed=4)
    v = ((v + np.float32(shift)) * np.float32(scale)).astype(np.float32)
    c = 0.5 * (v.min(0).astype(np.float64) + v.max(0))
    radius = np.linalg.norm(v - c, axis=1).max()
    rng = np.random.default_rng(n_small)
    d = rng.normal(size=(n_small, 3))
    q = d / np.linalg.norm(d, axis=1, keepdims=True) * (10 ** rng.uniform(-3, np.log10(0.2499), (n_small, 1))) / radius
    q[0] = 0.0
    g = rng.normal(size=(n_small, 2))
    vd, fd, qd, gd = (torch.from_numpy(np.ascontiguousarray(a)).to(dev) for a in (v, f, q, g))
    got = pft.pft3d_mesh_backward(vd, fd, qd, gd, check_status=True).cpu().numpy().astype(np.float64)
    ref = oracle.grad3d(v, f, q, g[:, 0] + 1j * g[:, 1])
    assert np.abs(got - ref).max() <= 2e-7 * np.abs(ref).max()
    got = pft.pft3d_mesh_qgrad(vd, fd, qd, gd, check_status=True).cpu().numpy()
    ref = oracle.qgrad3d(v, f, q, g[:, 0] + 1j * g[:, 1])
    bar = np.abs(g).max() * abs(oracle.ft3d(v, f, np.zeros((1, 3)))[0]) * np.abs(v).max()
    assert np.abs(got - ref).max() <= 1e-9 * bar
