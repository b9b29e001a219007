"""A request whose workspace fits the server's budget only in the shorter default segments (sqrt(nt) steps) is admitted
and run in them: bit for bit the operator on a context of its own with that segment length."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
import paper_2206_02362_gb300 as fw  # noqa: E402
from paper_2206_02362_gb300 import serve  # noqa: E402

pytestmark = pytest.mark.gpu


def request(nt):
    """The gradient request of the serving mix with the longest record, its record cut or repeated to nt steps"""
    reqs = [serve.from_synth(r) for r in synth.serving_mix(nreq=12, rate=400.0, seed=synth.SEED0 + 377, nz_range=(40, 60),
                                                           nx_range=(100, 160), nt_range=(240, 260), nh_choices=(5,))]
    r = next(q for q in reqs if q.kind == "gradient")
    r.w = synth.ricker(nt, r.dt, 10.0).astype(np.float32)
    r.dobs = np.random.default_rng(synth.SEED0).standard_normal((nt, len(r.rec_iz))).astype(np.float32)
    r.nt = nt
    return r


@pytest.mark.parametrize("nt", [300, 1000])
def test_request_between_the_two_segment_lengths(nt):
    r = request(nt)
    least, most = serve.request_bytes(r, least=True), serve.request_bytes(r)
    assert least < most
    K = int(round(np.sqrt(nt - 1)))
    grid = fw.Grid(nz=r.nz, nx=r.nx, sponge=r.sponge, nt=nt, dt=r.dt, dx=r.dx, nh=r.nh)
    geom = fw.Geometry(np.array([r.src[0]]), np.array([r.src[1]]), r.rec_iz, r.rec_ix)
    cu = lambda a: torch.from_numpy(np.ascontiguousarray(a, np.float32)).cuda()  # noqa: E731
    g = torch.zeros((r.nz, r.nx), device="cuda")
    with fw.Context(grid, geom, segment=K, shots_per_batch=1) as ctx:
        J = ctx.gradient(cu(r.v), cu(r.w[None]), cu(r.pt), cu(r.dobs[None]), g, eps=r.eps)
    for budget in (least, (least + most) // 2):
        srv = serve.Server(memory_budget=budget)
        try:
            res = srv.serve([r], realtime=False)[0]
        finally:
            srv.close()
        np.testing.assert_array_equal(res.grad, g.cpu().numpy())
        assert res.objective == J
    srv = serve.Server(memory_budget=least - 1)
    try:
        with pytest.raises(ValueError):
            srv.serve([r], realtime=False)
    finally:
        srv.close()
