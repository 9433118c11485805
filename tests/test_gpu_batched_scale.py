"""Batched adjoints of shapes so small that |Q|^2 leaves the FP32 range while |Q| r_max stays below 1/4: the
transform scales, F(s v, Q/s) = s^D F(v, Q), so the vertex gradients scale with s^(D-1).  s = 2^-66 scales every
coordinate exactly; the small-|Q| terms run in FP64 and the gradients are rounded to float32 once: 2^-24 of a value,
held to 2e-7 of the largest.  (The output gradients are scaled up, so that the vertex gradients are no denormals.)"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

S = 2.0 ** -66


def _cuda(*a):
    import torch
    return [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in a]


def _points(rng, n, dim, radius):
    d = rng.normal(size=(n, dim))
    q = d / np.linalg.norm(d, axis=1, keepdims=True) * rng.uniform(0.1, 0.24, (n, 1)) / radius
    assert ((q / S) ** 2).sum(axis=1).max() > np.finfo(np.float32).max
    return q


@pytest.mark.parametrize("lists", [False, True])
def test_polygons(lists):
    pytest.importorskip("torch")
    import paper_2104_08309_gb300 as pft
    rng = np.random.default_rng(1)
    n, k, n_q = 3, 7, 20
    t = 2 * np.pi * np.arange(k) / k
    v = (0.4 * np.stack([np.cos(t), np.sin(t)], axis=-1)[None] * (0.7 + 0.3 * rng.random((n, k, 1)))).astype(np.float32)
    q = _points(rng, n * n_q if lists else n_q, 2, 0.41)
    g = rng.normal(size=(n * n_q, 2) if lists else (n, n_q, 2))
    q_off = np.arange(n + 1) * n_q if lists else None

    def call(vv, qq, gg):
        return pft.pft2d_polygons_batched_backward(*_cuda(vv.reshape(-1, 2).astype(np.float32)), np.arange(n + 1) * k,
                                                   *_cuda(qq, gg), q_off, check_status=True).cpu().numpy().astype(np.float64)
    ref, got = call(v, q, g), call(v * S, q / S, g / S)
    assert np.abs(got - ref).max() <= 2e-7 * np.abs(ref).max()


@pytest.mark.parametrize("lists", [False, True])
def test_meshes(lists):
    pytest.importorskip("torch")
    import paper_2104_08309_gb300 as pft
    rng = np.random.default_rng(2)
    n, n_q = 3, 20
    u = np.array([[0, 0, 0], [1, 0, 0], [0, 1, 0], [0, 0, 1]], dtype=np.float64)
    f0 = np.array([[0, 2, 1], [0, 1, 3], [0, 3, 2], [1, 2, 3]], dtype=np.int32)
    v = ((u[None] - 0.4) * (0.3 + 0.2 * rng.random((n, 4, 3)))).astype(np.float32)
    f = (f0[None] + 4 * np.arange(n)[:, None, None]).reshape(-1, 3).astype(np.int32)
    q = _points(rng, n * n_q if lists else n_q, 3, 0.5)
    g = rng.normal(size=(n * n_q, 2) if lists else (n, n_q, 2))
    q_off = np.arange(n + 1) * n_q if lists else None

    def call(vv, qq, gg):
        return pft.pft3d_meshes_batched_backward(*_cuda(vv.reshape(-1, 3).astype(np.float32), f), np.arange(n + 1) * 4,
                                                 *_cuda(qq, gg), q_off, check_status=True).cpu().numpy().astype(np.float64)
    ref, got = call(v, q, g), call(v * S, q / S, g / S ** 2)
    assert np.abs(got - ref).max() <= 2e-7 * np.abs(ref).max()
