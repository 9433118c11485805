"""A few faces against many Q points, on both sides of the line between k_fwd_group and k_fwd (6 blocks of 512 Q points a
face, and 20), against the same call with k_fwd's launch shape asked for: the same FP32 tile sums, one tile, so the
FP64 sum over chunks has one term and the results are the same bit for bit."""
import numpy as np
import pytest

from paper_2104_08309_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_faces", [1, 4, 12, 20, 33])
@pytest.mark.parametrize("over", [-512, 0, 1, 513])
def test_line(n_faces, over):
    torch = pytest.importorskip("torch")
    import paper_2104_08309_gb300 as pft
    v, f = synth.perturbed_icosphere(1, seed=6)
    n_q = (6 * n_faces + 20) * 512 + over
    q = np.random.default_rng(n_q).normal(size=(n_q, 3)) * 12.0
    q[::1001] *= 1e-3                                    # small |Q| among them
    a = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (v, f[:n_faces], q)]
    short = pft.pft3d_mesh(*a, check_status=True)
    given = pft.pft3d_mesh(*a, options={"q_per_thread": 4, "block_threads": 128}, check_status=True)
    assert torch.equal(short, given)
