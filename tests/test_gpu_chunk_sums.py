"""Short 3D launches: the chunk count that the planner takes and the finishing kernel's side-by-side sum of the
chunks, against one chunk a call.  Both add the same FP32 tile sums, across tiles in compensated FP32 pairs (48
bits) or in FP64, so they differ by less than 2^-40 of the tile sums, which stay below |Q|^2 F(0)."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("level,n_q", [(5, 1500), (5, 2049), (5, 4095), (6, 1001), (6, 515), (7, 129)])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_default_chunks_match_one_chunk(level, n_q, precision):
    import paper_2104_08309_gb300 as pft
    from paper_2104_08309_gb300 import synth
    if precision == "fp64" and level > 5:
        pytest.skip("the FP64 path is planned apart; one size pair suffices")
    v, f = (torch.from_numpy(x).cuda() for x in synth.icosphere(level))
    g = torch.Generator().manual_seed(n_q)
    q = torch.empty(n_q, 3, dtype=torch.float64).uniform_(-25, 25, generator=g)
    q[0] = 0.0
    q[1:40] *= 0.004        # the small-|Q| pass (more than its direct points)
    q = q.cuda()
    out = pft.pft3d_mesh(v, f, q, options={"precision": precision}, check_status=True)
    one = pft.pft3d_mesh(v, f, q, options={"precision": precision, "k_splits": 1}, check_status=True)
    assert torch.isfinite(out).all()
    assert (out - one).abs().max().item() < 2.0 ** -40 * 4.2
