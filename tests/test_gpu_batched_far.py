"""Batched adjoints of shapes far from the origin: the phase Q.c of k_bbq as a float pair, and in FP64 beyond 2^20
radians, rows on both sides of that line, in each of its block sizes (few shapes; many, with few and with many
rows).  Against the oracle at the same float32 vertices; the reduced phase carries 1.2e-7 rad, far below the 1e-4
of max |grad| to which every FP32 gradient is held."""
import numpy as np
import pytest

import oracle
from paper_2104_08309_gb300 import synth

pytestmark = pytest.mark.gpu
GTOL = 1e-4


def _cuda(*a):
    import torch
    return [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in a]


def _inputs(shape, n, rows, seed):
    """n copies of a shape about centres at 1e3 and at 7e4, and Q points up to 25 in each coordinate."""
    rng = np.random.default_rng(seed)
    dim = shape.shape[1]
    c = np.where(np.arange(n)[:, None] % 2 == 0, 1e3, 7e4) * rng.choice([-1.0, 1.0], (n, dim)) * rng.uniform(0.5, 1, (n, dim))
    v = (shape[None] * rng.uniform(0.5, 0.8, (n, 1, 1)) + c[:, None]).astype(np.float32)
    q = rng.uniform(-25, 25, (rows, dim))
    q[::6] *= 0.01
    if n > 1:
        ph = np.abs(q[:200] @ c[:2].T)
        assert (ph > 2 ** 20).any() and (ph < 2 ** 20).any()
    return v, q, rng.normal(size=(n, rows, 2))


def _sample(n):
    return sorted({0, 1, 2, n // 2 + 1, n - 1} & set(range(n)))


@pytest.mark.parametrize("n,rows", [(4, 150), (640, 20), (640, 130)])
def test_polygons(n, rows):
    pytest.importorskip("torch")
    import paper_2104_08309_gb300 as pft
    k = 9
    t = 2 * np.pi * np.arange(k) / k
    v, q, g = _inputs(np.stack([np.cos(t), np.sin(t)], axis=-1), n, rows, n + rows)
    got = pft.pft2d_polygons_batched_backward(*_cuda(v.reshape(-1, 2)), np.arange(n + 1) * k, *_cuda(q, g),
                                              check_status=True).cpu().numpy().reshape(n, -1, 2)
    for i in _sample(n):
        ref = oracle.grad2d(v[i], q, g[i, :, 0] + 1j * g[i, :, 1])
        assert np.abs(got[i] - ref).max() < GTOL * np.abs(ref).max(), i


@pytest.mark.parametrize("n,rows", [(4, 150), (640, 20), (640, 130)])
def test_meshes(n, rows):
    pytest.importorskip("torch")
    import paper_2104_08309_gb300 as pft
    u, f0 = synth.icosphere(0)
    v, q, g = _inputs(u.astype(np.float64), n, rows, n + rows)
    f = (f0[None] + u.shape[0] * np.arange(n)[:, None, None]).reshape(-1, 3).astype(np.int32)
    got = pft.pft3d_meshes_batched_backward(*_cuda(v.reshape(-1, 3), f), np.arange(n + 1) * f0.shape[0], *_cuda(q, g),
                                            check_status=True).cpu().numpy().reshape(n, -1, 3)
    for i in _sample(n):
        ref = oracle.grad3d(v[i], f0, q, g[i, :, 0] + 1j * g[i, :, 1])
        assert np.abs(got[i] - ref).max() < GTOL * np.abs(ref).max(), i
