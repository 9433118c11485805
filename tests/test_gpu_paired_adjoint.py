"""The paired 3D vertex adjoint (two faces a thread, 256 a block, tiles of 128 Q points) at the edges of
its blocks and tiles and in each of its forms, against the oracle: 1e-4 of max |grad| as for every FP32
gradient."""
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


def _points(n, scale, seed):
    rng = np.random.default_rng(seed)
    d = rng.normal(size=(n, 3))
    return d / np.linalg.norm(d, axis=1, keepdims=True) * scale * rng.uniform(0.6, 1.0, (n, 1)), rng.normal(size=(n, 2))


# a level-3 icosphere's faces have phase spreads of about 0.1 |Q|: short series, k <= 9, k <= 11, k <= 17, edge sum
@pytest.mark.parametrize("scale", [2.0, 8.0, 14.0, 25.0, 70.0])
@pytest.mark.parametrize("tau", [1.0, 3.0, 6.0])
def test_forms(torch_dev, scale, tau):
    torch, dev = torch_dev
    import paper_2104_08309_gb300 as pft
    v, f = synth.perturbed_icosphere(3, seed=12)
    q, g = _points(200, scale, int(scale))
    a = [torch.from_numpy(x).to(dev) for x in (v, f, q, g)]
    got = pft.pft3d_mesh_backward(*a, options={"face_series_tau": tau}, check_status=True).cpu().numpy()
    ref = oracle.grad3d(v, f, q, g[:, 0] + 1j * g[:, 1])
    assert np.abs(got - ref).max() <= 1e-4 * np.abs(ref).max()


@pytest.mark.parametrize("n_faces", [1, 2, 63, 64, 65, 255, 256, 257, 700])
@pytest.mark.parametrize("n_q", [1, 127, 128, 129, 700])
def test_sizes(torch_dev, n_faces, n_q):
    """An open surface is a signed sum of faces: its adjoint against the whole mesh's one is not defined
    by the oracle (boundary terms), so each size runs as a closed mesh plus the same faces taken twice
    with opposite orientation, whose sum is the mesh's gradient."""
    torch, dev = torch_dev
    import paper_2104_08309_gb300 as pft
    v, f = synth.perturbed_icosphere(1, seed=3)
    rng = np.random.default_rng(n_faces)
    pick = f[rng.integers(0, f.shape[0], n_faces)]
    both = np.concatenate([pick, f, pick[:, [0, 2, 1]]]).astype(np.int32)
    q, g = _points(n_q, 6.0, n_q)
    a = [torch.from_numpy(np.ascontiguousarray(x)).to(dev) for x in (v, both, q, g)]
    got = pft.pft3d_mesh_backward(*a, check_status=True).cpu().numpy()
    ref = oracle.grad3d(v, f, q, g[:, 0] + 1j * g[:, 1])
    # the cancelling faces' own rounding: 1e-6 of each of their terms, which are at most the mesh's largest
    per_vertex = 1.0 + np.bincount(pick.reshape(-1), minlength=v.shape[0]).max()
    assert np.abs(got - ref).max() <= 1e-4 * np.abs(ref).max() + 2e-6 * per_vertex * np.abs(ref).max()
