"""Batches of tiny shapes take policies of their own (up to 16 segments a polygon, up to 32 faces a mesh, on
average): the same shapes with a large one beside them, whose average is beyond the line, give the same results
bit for bit, for every launch shape that has such a policy."""
import numpy as np
import pytest

from paper_2104_08309_gb300 import synth

pytestmark = pytest.mark.gpu


def _cuda(*a):
    import torch
    return [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in a]


def _lists(rng, n, per, dim):
    q = rng.uniform(-40, 40, (n * per, dim))
    q[::9] *= 1e-3
    return q, np.arange(n + 1, dtype=np.int64) * per


@pytest.mark.parametrize("k", [3, 16])
@pytest.mark.parametrize("lists", [False, True])
def test_polygons(k, lists):
    torch = pytest.importorskip("torch")
    import paper_2104_08309_gb300 as pft
    rng = np.random.default_rng(k)
    n, per = 50, 77
    v = rng.uniform(-1, 1, (n * k, 2)).astype(np.float32)          # long segments: large sincs
    big = synth.star_polygon(3000, 5)
    off = np.arange(n + 1, dtype=np.int64) * k
    q, q_off = _lists(rng, n + 1, per, 2)
    if not lists:
        q, q_off = q[:1500], None                                  # fewer than fill the 512-thread shape
    qo = (lambda m: None if q_off is None else q_off[:m + 1])
    rows = (lambda m: q if q_off is None else q[:q_off[m]])
    few = pft.pft2d_polygons_batched(*_cuda(v), off, *_cuda(rows(n)), qo(n), check_status=True)
    both = pft.pft2d_polygons_batched(*_cuda(np.concatenate([v, big])), np.append(off, off[-1] + 3000), *_cuda(rows(n + 1)),
                                      qo(n + 1), check_status=True)
    assert torch.isfinite(few).all()
    assert torch.equal(few, both[:few.shape[0]])


@pytest.mark.parametrize("shape", ["lists", "shared", "shared512", "two points"])
def test_meshes(shape):
    torch = pytest.importorskip("torch")
    import paper_2104_08309_gb300 as pft
    rng = np.random.default_rng(4)
    n, per = 40, 33
    u, f0 = synth.icosphere(0)
    v = (u[None] * rng.uniform(0.3, 1.0, (n, 1, 1)) + rng.uniform(-1, 1, (n, 1, 3))).reshape(-1, 3).astype(np.float32)
    f = (f0[None] + u.shape[0] * np.arange(n)[:, None, None]).reshape(-1, 3).astype(np.int32)
    off = np.arange(n + 1, dtype=np.int64) * f0.shape[0]
    bv, bf = synth.icosphere(4)
    q, q_off = _lists(rng, n + 1, per, 3)
    if shape == "shared512":
        q = rng.uniform(-40, 40, (2500, 3))
    if shape != "lists":
        q_off = None
    opts = {"q_per_thread": 2, "block_threads": 128} if shape == "two points" else None
    qo = (lambda m: None if q_off is None else q_off[:m + 1])
    rows = (lambda m: q if q_off is None else q[:q_off[m]])
    few = pft.pft3d_meshes_batched(*_cuda(v, f), off, *_cuda(rows(n)), qo(n), options=opts, check_status=True)
    both = pft.pft3d_meshes_batched(*_cuda(np.concatenate([v, bv]).astype(np.float32), np.concatenate([f, bf + v.shape[0]]).astype(np.int32)),
                                    np.append(off, off[-1] + bf.shape[0]), *_cuda(rows(n + 1)), qo(n + 1), options=opts,
                                    check_status=True)
    assert torch.isfinite(few).all()
    assert torch.equal(few, both[:few.shape[0]])
