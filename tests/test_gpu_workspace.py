"""The two further fields of two-step launches are reserved only for calls that use them: the workspace of T and of the
objective with time lags and of a grouped forward grows by the same bytes per shot below and above the line (13 M
points) from which batches run two steps per launch; that of a plain forward call by two fields more."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
import paper_2206_02362_gb300 as fw  # noqa: E402

pytestmark = pytest.mark.gpu
NZ, NX, W, NT, NH = 1270, 2028, 5, 6, 3
POINTS = (NZ + 18) * (NX + 20)          # 2.6 M points of a padded field (rows of 2046, rounded up to 2048)


def workspace(kind, nshot):
    v = torch.full((NZ, NX), 2000.0, device="cuda")
    dv, pt = torch.zeros_like(v), torch.zeros((NH, NZ, NX), device="cuda")
    w = torch.from_numpy(np.stack([synth.ricker(NT, 1e-3, 25.0)] * nshot).astype(np.float32)).cuda()
    geom = fw.Geometry(np.full(nshot, 2), np.arange(nshot), np.array([3]), np.array([4]))
    d = torch.zeros((nshot, NT, 1), device="cuda")
    grid = fw.Grid(nz=NZ, nx=NX, sponge=W, nt=NT, dt=1e-3, dx=10.0, nh=NH)
    with fw.Context(grid, geom, time_lag=1 if kind.endswith("lag") else 0) as ctx:
        if kind == "tomo_lag":
            ctx.tomo(v, w, pt, dv, d)
        elif kind == "objective_lag":
            ctx.objective(v, w, pt, d)
        elif kind == "group":
            fw.forward_group([ctx], [v], [w], [d])
        else:
            ctx.forward(v, w, d)
        return ctx.get_option("workspace")


@pytest.mark.parametrize("kind,more", [("tomo_lag", 0), ("objective_lag", 0), ("group", 0), ("forward", 2)])
def test_further_fields_only_where_they_are_used(kind, more):
    size = {s: workspace(kind, s) for s in (2, 4, 6)}
    field = 4 * POINTS
    assert 4 * POINTS < 13e6 <= 6 * POINTS
    assert (size[6] - size[4]) - (size[4] - size[2]) == more * 6 * field
