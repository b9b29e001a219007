"""FWIME_OPT_LAUNCHES and the profile count kernels: the extension kernels run one launch per segment up to 47 offsets
and three at 101, in chunks of at most 48 offsets."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
import paper_2206_02362_gb300 as fw  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("op,family", [("born_ext", "scatter"), ("born_ext_adj", "image")])
def test_launches_of_many_offsets(op, family):
    nz, nx, nt, K = 5, 61, 49, 8
    geom = fw.Geometry(np.array([1]), np.array([20]), np.full(nx, 1), np.arange(nx))
    v = torch.full((nz, nx), 2000.0, device="cuda")
    w = torch.from_numpy(synth.ricker(nt, 1e-3, 25.0)[None].astype(np.float32)).cuda()
    total = {}
    for nh in (47, 101):
        grid = fw.Grid(nz=nz, nx=nx, sponge=3, nt=nt, dt=1e-3, dx=10.0, nh=nh)
        pt, d = torch.zeros((nh, nz, nx), device="cuda"), torch.zeros((1, nt, nx), device="cuda")
        for profile in (0, 1):
            with fw.Context(grid, geom, segment=K, profile=profile) as ctx:
                if op == "born_ext":
                    ctx.born_ext(v, w, pt, d)
                else:
                    ctx.born_ext_adj(v, w, d, pt)
                if profile:
                    count = ctx.profile_read()
                    assert count[family]["launches"] == (nt - 1) // K * (3 if nh == 101 else 1)
                    assert sum(c["launches"] for c in count.values()) == ctx.launches == total[nh]
                else:
                    total[nh] = ctx.launches
    assert total[101] - total[47] == (nt - 1) // K * 2
