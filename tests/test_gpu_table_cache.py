"""The table cache past its limit: a call can still be captured after its
warm-up, and a graph captured earlier still finds its tables when the cache has
been emptied."""
import pytest
import torch

from gpu_util import random_state, to_patch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def capi():
    from paper_1112_1710_gb300 import _build, capi as C
    _build.build()
    C.load()
    return C


def test_captured_calls_keep_their_tables(capi):
    from paper_1112_1710_gb300.patch import periodic_copies
    n, g = (4, 5, 6), 2
    ctx = capi.mhd_ctx_create()
    s = torch.cuda.Stream()
    sp = s.cuda_stream
    try:
        p = to_patch(random_state(n, g, seed=3), n, g, (0.1,) * 3)
        q = to_patch(random_state(n, g, seed=3), n, g, (0.1,) * 3)
        one, copies = [p.desc()], periodic_copies(n, g)
        # half a million patches in one call: about 300 MB of tables
        many = [(capi.mhd_patch_desc * k).from_buffer_copy(bytes(q.desc()) * k) for k in (500000, 499999)]
        sums = torch.zeros(8, dtype=torch.float64, device="cuda")
        dt = torch.zeros(1, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()

        def small():
            capi.mhd_ghost_fill(ctx, one, copies, sp)
            capi.mhd_conservation_sums(ctx, one, sums.data_ptr(), sp)

        def big():
            capi.mhd_cfl_dt(ctx, many[0], dt.data_ptr(), sp)

        graphs = []
        for call in (small, big):
            call()
            torch.cuda.synchronize()
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=s):
                call()
            graphs.append(graph)
        want = sums.clone(), dt.clone()
        capi.mhd_cfl_dt(ctx, many[1], dt.data_ptr(), sp)  # past the limit again, not captured
        capi.mhd_cfl_dt(ctx, one, dt.data_ptr(), sp)      # drops what no graph reads
        other = torch.full((1 << 27,), -1, dtype=torch.int32, device="cuda")  # (over what was freed)
        sums.zero_()
        dt.zero_()
        p.state[:, :g] = 0.0  # ghost planes
        r = to_patch(p.state.cpu().numpy(), n, g, (0.1,) * 3)
        fresh = capi.mhd_ctx_create()
        capi.mhd_ghost_fill(fresh, [r.desc()], copies)
        torch.cuda.synchronize()
        capi.mhd_ctx_destroy(fresh)
        for graph in graphs:
            graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(sums, want[0]) and torch.equal(dt, want[1]) and torch.equal(p.state, r.state)
        assert int(other[0]) == -1
    finally:
        capi.mhd_ctx_destroy(ctx)
