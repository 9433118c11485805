"""Adjoints of batches of many small shapes (the launch shapes that take over from some 600 shapes and from 8,192),
against the oracle on a sample of the shapes: 1e-4 of max |grad| as for every FP32 gradient."""
import numpy as np
import pytest

import oracle
from paper_2104_08309_gb300 import synth

pytestmark = pytest.mark.gpu
GTOL = 1e-4


def _sample(n):
    return sorted({0, 1, n // 3, n // 2, n - 2, n - 1})


def _complex(rng, *n):
    return rng.normal(size=n) + 1j * rng.normal(size=n)


def _cuda(*a):
    import torch
    return [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in a]


def _parts(z):
    return np.stack([z.real, z.imag], axis=-1)


@pytest.mark.parametrize("n", [700, 8200])
@pytest.mark.parametrize("lists", [False, True])
def test_meshes(n, lists):
    pytest.importorskip("torch")
    import paper_2104_08309_gb300 as pft
    rng = np.random.default_rng(n)
    u, f0 = synth.icosphere(0)
    v = u[None] * (0.3 + 0.2 * rng.random((n, u.shape[0], 1))) + rng.uniform(-1, 1, (n, 1, 3))
    v = v.astype(np.float32)
    f = (f0[None] + (np.arange(n) * u.shape[0])[:, None, None]).reshape(-1, 3).astype(np.int32)
    off = np.arange(n + 1, dtype=np.int64) * f0.shape[0]
    per = 9
    q = rng.uniform(-12, 12, (n * per if lists else per, 3))
    q[::5] *= 0.01
    q_off = np.arange(n + 1, dtype=np.int64) * per if lists else None
    g = _complex(rng, n, per)
    got = pft.pft3d_meshes_batched_backward(*_cuda(v.reshape(-1, 3), f), off, *_cuda(q, _parts(g).reshape(-1, 2)
                                            if lists else _parts(g)), q_off, check_status=True).cpu().numpy()
    got = got.reshape(n, -1, 3)
    for i in _sample(n):
        ref = oracle.grad3d(v[i], f0, q[i * per:(i + 1) * per] if lists else q, g[i])
        assert np.abs(got[i] - ref).max() < GTOL * np.abs(ref).max(), i


@pytest.mark.parametrize("n", [700, 8200])
@pytest.mark.parametrize("lists", [False, True])
def test_polygons(n, lists):
    pytest.importorskip("torch")
    import paper_2104_08309_gb300 as pft
    rng = np.random.default_rng(n)
    k = 11
    t = 2 * np.pi * np.arange(k) / k
    v = np.stack([np.cos(t), np.sin(t)], axis=-1)[None] * (0.6 + 0.4 * rng.random((n, k, 1))) + rng.uniform(-1, 1, (n, 1, 2))
    v = v.astype(np.float32)
    off = np.arange(n + 1, dtype=np.int64) * k
    per = 9
    q = rng.uniform(-20, 20, (n * per if lists else per, 2))
    q[::5] *= 0.005
    q_off = np.arange(n + 1, dtype=np.int64) * per if lists else None
    g = _complex(rng, n, per)
    got = pft.pft2d_polygons_batched_backward(*_cuda(v.reshape(-1, 2)), off, *_cuda(q, _parts(g).reshape(-1, 2)
                                              if lists else _parts(g)), q_off, check_status=True).cpu().numpy()
    got = got.reshape(n, -1, 2)
    for i in _sample(n):
        ref = oracle.grad2d(v[i], q[i * per:(i + 1) * per] if lists else q, g[i])
        assert np.abs(got[i] - ref).max() < GTOL * np.abs(ref).max(), i
