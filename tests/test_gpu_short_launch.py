"""Short launches: k_fwd_group in 3D and the smaller launch shapes in 2D against the same call with the
launch shape asked for (k_fwd).  Both add the same FP32 tile sums; only the FP64 sum over chunks may be
grouped differently, a few 1e-16 of the largest partial sum: held to 1e-12 of F(0)."""
import numpy as np
import pytest

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


@pytest.mark.parametrize("n_faces", [1, 3, 31, 33, 128, 129, 300, 1280])
@pytest.mark.parametrize("n_q", [1, 32, 33, 128, 129, 511, 513, 1200])
def test_mesh(torch_dev, n_faces, n_q):
    torch, dev = torch_dev
    import paper_2104_08309_gb300 as pft
    v, f = synth.perturbed_icosphere(3, seed=6)
    rng = np.random.default_rng(n_q)
    f = f[rng.permutation(f.shape[0])[:n_faces]]
    q = rng.normal(size=(n_q, 3)) * 10 ** rng.uniform(-1, 1.8, (n_q, 1))     # series of every length, edge sums
    q[::7] *= 1e-3                                                            # small |Q| among them
    a = [torch.from_numpy(np.ascontiguousarray(x)).to(dev) for x in (v, f, q)]
    for tau in (6.0, 1.0):
        short = pft.pft3d_mesh(*a, options={"face_series_tau": tau}, check_status=True)
        given = pft.pft3d_mesh(*a, options={"face_series_tau": tau, "q_per_thread": 4, "block_threads": 128},
                               check_status=True)
        assert (short - given).abs().max().item() <= 1e-12 * 4.2


@pytest.mark.parametrize("n", [3, 64, 300, 5000])
@pytest.mark.parametrize("n_q", [1, 100, 5000, 70000])
def test_loop(torch_dev, n, n_q):
    torch, dev = torch_dev
    import paper_2104_08309_gb300 as pft
    rng = np.random.default_rng(n_q)
    p, q = synth.star_polygon(n, seed=n), rng.normal(size=(n_q, 2)) * 20.0
    a = [torch.from_numpy(x).to(dev) for x in (p, q)]
    short = pft.pft2d_polygons(*a, check_status=True)
    given = pft.pft2d_polygons(*a, options={"q_per_thread": 4, "block_threads": 256}, check_status=True)
    assert (short - given).abs().max().item() <= 1e-12 * 4.2
