"""How the 3D vertex adjoint deals faces to threads: one a thread where pairs would leave the GPU idle and in a
warp's last 32 faces, else two a thread; and its runs of edge sums.  Face counts at the edges of the warps' 32 and
64 faces and of the blocks' 128 and 256, odd ones included, against the oracle: 1e-4 of max |grad| as for every
FP32 gradient.  A closed mesh has an even number of faces; degenerate ones (i, i, i), whose share is exactly
zero, fill it up in front, so that the last slot holds a real face."""
import numpy as np
import pytest

import oracle
from paper_2104_08309_gb300 import synth

pytestmark = pytest.mark.gpu
GTOL = 1e-4


def _filled(level, total, seed=3):
    v, f = synth.perturbed_icosphere(level, seed=seed)
    i = np.random.default_rng(total).integers(0, v.shape[0], (total - f.shape[0], 1))
    return v, f, np.concatenate([np.repeat(i, 3, axis=1), f]).astype(np.int32)


def _points(n, scales, seed):
    """Points of several magnitudes, in stretches: the series forms, the edge sum, and changes between them."""
    rng = np.random.default_rng(seed)
    d = rng.normal(size=(n, 3))
    scale = np.repeat(np.asarray(scales), -(-n // len(scales)))[:n, None]
    return d / np.linalg.norm(d, axis=1, keepdims=True) * scale * rng.uniform(0.6, 1.0, (n, 1)), rng.normal(size=(n, 2))


def _check(v, f, full, q, g):
    torch = pytest.importorskip("torch")
    import paper_2104_08309_gb300 as pft
    a = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (v, full, q, g)]
    got = pft.pft3d_mesh_backward(*a, check_status=True).cpu().numpy()
    ref = oracle.grad3d(v, f, q, g[:, 0] + 1j * g[:, 1])
    assert np.abs(got - ref).max() <= GTOL * np.abs(ref).max()


@pytest.mark.parametrize("level,total", [(0, 20), (0, 31), (0, 32), (0, 33), (0, 63), (0, 64), (0, 65), (1, 97), (1, 127),
                                         (1, 128), (1, 129), (1, 255), (1, 256), (1, 257), (1, 511), (1, 513)])
@pytest.mark.parametrize("n_q", [1, 17, 129, 700])
def test_one_face_a_thread(level, total, n_q):
    v, f, full = _filled(level, total)
    _check(v, f, full, *_points(n_q, [2.0, 40.0, 3.0, 70.0, 9.0, 50.0, 50.0], n_q))


@pytest.mark.parametrize("total", [1281, 1311, 1312, 1313, 1343, 1345, 1535, 1536, 1537])
def test_two_faces_a_thread(total):
    v, f, full = _filled(3, total)
    _check(v, f, full, *_points(13057, [2.0, 14.0, 25.0, 70.0, 90.0, 8.0, 60.0], total))


@pytest.mark.parametrize("n_meshes,n_q,lists", [(3, 200, False), (40, 2100, False), (3, 90, True), (300, 40, True),
                                               (40, 2100, True)])
def test_batches(n_meshes, n_q, lists):
    """Meshes of 80 + 0 .. 260 faces, most of them odd, on both sides of the rule."""
    torch = pytest.importorskip("torch")
    import paper_2104_08309_gb300 as pft
    rng = np.random.default_rng(n_meshes)
    vs, fs, off, closed, n = [], [], [0], [], 0
    for i in range(n_meshes):
        v, f, full = _filled(1, 80 + int(rng.integers(0, 130)) * 2 + i % 2, seed=i)
        v = (v * np.float32(0.4) + rng.uniform(-1, 1, 3).astype(np.float32)).astype(np.float32)
        vs.append(v)
        fs.append(full + n)
        closed.append((v, f))
        off.append(off[-1] + full.shape[0])
        n += v.shape[0]
    rows = n_meshes * n_q if lists else n_q
    q, _ = _points(rows, [2.0, 40.0, 90.0, 10.0, 60.0], n_q)
    g = rng.normal(size=(n_meshes, n_q, 2))
    a = [torch.from_numpy(np.ascontiguousarray(x)).cuda()
         for x in (np.concatenate(vs), np.concatenate(fs).astype(np.int32))]
    got = pft.pft3d_meshes_batched_backward(
        *a, np.asarray(off), torch.from_numpy(q).cuda(), torch.from_numpy(g.reshape(-1, 2) if lists else g).cuda(),
        np.arange(n_meshes + 1) * n_q if lists else None, check_status=True).cpu().numpy().reshape(n_meshes, -1, 3)
    for i in sorted({0, 1, n_meshes // 2, n_meshes - 1}):
        qi = q[i * n_q:(i + 1) * n_q] if lists else q
        ref = oracle.grad3d(*closed[i], qi, g[i, :, 0] + 1j * g[i, :, 1])
        assert np.abs(got[i] - ref).max() <= GTOL * np.abs(ref).max(), i
