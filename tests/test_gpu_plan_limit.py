"""The forward planner around the allocation-free call's 32 MiB limit: meshes just under it get chunks as fine as
meshes just over it, and the allocation-free call still gives the workspace call's result bit for bit, with chunk sums
beyond the limit too."""
import ctypes

import numpy as np
import pytest

from paper_2104_08309_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2104_08309_gb300 import _capi
    return _capi.load()


@pytest.mark.parametrize("n_q", [241, 1000])
def test_chunks_do_not_depend_on_the_limit(lib, n_q):
    """Chunks from the workspace's size: 16 bytes a chunk and Q point, beside 48 bytes a face (the rest, below a
    hundredth of that, bounds the error).  An SM runs one block of each Q tile and chunk after the other, so the
    chunks of a launch of so few Q points are of the order of a thousand, whatever the faces."""
    for n_faces in (600_000, 640_000, 660_000, 680_000, 700_000, 720_000):
        need = lib.pft3d_workspace_size(n_faces // 2, n_faces, n_q, None)
        assert (need - 1.01 * 48 * n_faces) / (16 * n_q) > 700, n_faces


@pytest.mark.parametrize("n_faces,n_q", [(640_000, 1000), (330_000, 2000), (690_000, 241), (100_000, 5000)])
def test_noalloc_is_the_workspace_call(lib, n_faces, n_q):
    import torch
    v, f = synth.icosphere(8)
    q = np.random.default_rng(n_q).uniform(-20, 20, (n_q, 3))
    q[:40] *= 1e-3
    vd, fd, qd = (torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (v, f[:n_faces], q))
    need = lib.pft3d_workspace_size(v.shape[0], n_faces, n_q, None)
    assert need > 32 << 20
    ws = torch.empty(need, dtype=torch.uint8, device="cuda")
    ref = torch.empty(n_q, 2, dtype=torch.float64, device="cuda")
    out = torch.full_like(ref, float("nan"))
    stream = torch.cuda.current_stream().cuda_stream
    a = (vd.data_ptr(), v.shape[0], fd.data_ptr(), n_faces, qd.data_ptr(), n_q)
    assert lib.pft3d_mesh(*a, ref.data_ptr(), ws.data_ptr(), need, None, stream) == 0
    assert lib.pft_status(ws.data_ptr(), stream) == 0
    assert lib.pft3d_mesh_noalloc(*a, out.data_ptr(), None, stream) == 0
    torch.cuda.synchronize()
    assert torch.isfinite(out).all() and torch.equal(out, ref)


def test_noalloc_refuses_what_no_plan_fits(lib):
    """720,000 records are 33 MiB by themselves."""
    fake = ctypes.c_void_p(256)          # never dereferenced: the size check comes first
    assert lib.pft3d_mesh_noalloc(fake, 3, fake, 720_000, fake, 10, fake, None, None) == 9
