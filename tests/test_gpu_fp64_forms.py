"""The FP64 path's series forms, edge sum, sinc ranges and sincos ranges against the oracle.

Tolerance: 1e-12 of F(0) as in the other FP64 tests where phases are ordinary; for phases of 1e9 and more
the phase itself is only known to its own rounding, so an error of 16 half-ulps of the largest phase on
every term is allowed."""
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


# |Q| chosen so that a level-2 icosphere's faces (spread ~ 0.3 |Q|) fall in each series form, between
# them and in the edge sum with |u| below and above 2
@pytest.mark.parametrize("qmax", [0.5, 1.0, 2.0, 3.0, 4.5, 6.0, 8.0, 12.0, 40.0, 400.0])
@pytest.mark.parametrize("tau", [0.0, 1.0, 6.0])
def test_mesh_forms(torch_dev, qmax, tau):
    torch, dev = torch_dev
    import paper_2104_08309_gb300 as pft
    v, f = synth.perturbed_icosphere(2, seed=9)
    rng = np.random.default_rng(int(qmax * 10))
    d = rng.normal(size=(161, 3))
    q = d / np.linalg.norm(d, axis=1, keepdims=True) * qmax * rng.uniform(0.9, 1.0, (161, 1))
    q[:32] = q[0]                                    # a whole warp at one point
    q[40] = np.cross(v[f[5, 1]] - v[f[5, 0]], v[f[5, 2]] - v[f[5, 0]]) * 300.0   # along a face normal
    ref = oracle.ft3d(v, f, q)
    opts = {"precision": "fp64"}
    if tau:
        opts["face_series_tau"] = tau
    for r in (1, 2):
        out = pft.pft3d_mesh(torch.from_numpy(v).to(dev), torch.from_numpy(f).to(dev), torch.from_numpy(q).to(dev),
                             options={**opts, "q_per_thread": r}, check_status=True).cpu().numpy()
        assert np.abs(out[:, 0] + 1j * out[:, 1] - ref).max() <= 1e-12 * 4.2


@pytest.mark.parametrize("n", [3, 40, 257])
def test_loop_ranges(torch_dev, n):
    torch, dev = torch_dev
    import paper_2104_08309_gb300 as pft
    p = synth.star_polygon(n, seed=n)
    rng = np.random.default_rng(n)
    q = rng.normal(size=(700, 2)) * 10 ** rng.uniform(-1, 3.5, (700, 1))
    ref = oracle.ft2d(p, q)
    out = pft.pft2d_polygons(torch.from_numpy(p).to(dev), torch.from_numpy(q).to(dev),
                             options={"precision": "fp64"}, check_status=True).cpu().numpy()
    assert np.abs(out[:, 0] + 1j * out[:, 1] - ref).max() <= 1e-12 * 4.0


def test_huge_phases(torch_dev):
    torch, dev = torch_dev
    import paper_2104_08309_gb300 as pft
    p = synth.star_polygon(5, seed=3)
    rng = np.random.default_rng(0)
    d = rng.normal(size=(64, 2))
    q = d / np.linalg.norm(d, axis=1, keepdims=True) * 10 ** rng.uniform(8.5, 10, (64, 1))
    ref = oracle.ft2d(p, q)
    out = pft.pft2d_polygons(torch.from_numpy(p).to(dev), torch.from_numpy(q).to(dev),
                             options={"precision": "fp64"}, check_status=True).cpu().numpy()
    edge = np.roll(p, -1, 0).astype(np.float64) - p
    w = np.abs(q[:, :1] * edge[:, 1] - q[:, 1:] * edge[:, 0])
    u = np.abs(q @ edge.T) / 2
    qn = np.linalg.norm(q, axis=1)
    terms = (w / np.maximum(u, 1.0)).sum(1) / qn ** 2
    tol = 16 * 2.0 ** -53 * qn * np.abs(p).max() * 2 * terms
    assert np.all(np.abs(out[:, 0] + 1j * out[:, 1] - ref) <= tol)
