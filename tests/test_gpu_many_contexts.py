"""Contexts beside one another on one card: a kept history takes a third of the card at most and half of what is free,
so that the next context, and the caller, still have room."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
import paper_2206_02362_gb300 as fw  # noqa: E402

pytestmark = pytest.mark.gpu


def test_every_context_leaves_room_for_the_next():
    """B* of 10 shots on 7 M points, 299 steps: a history of 84 GB; checkpoints take 21 GB for all shots, 2 for one"""
    nz, nx, nt, nshot = 1188, 5868, 300, 10
    grid = fw.Grid(nz=nz, nx=nx, sponge=2, nt=nt, dt=1e-3, dx=10.0, nh=1)
    src = 500 * np.arange(nshot) + 200
    geom = fw.Geometry(np.full(nshot, 1), src, np.full(600, 1), 9 * np.arange(600))
    gen = torch.Generator(device="cuda").manual_seed(synth.SEED0)
    v = torch.full((nz, nx), 2000.0, device="cuda")
    w = torch.from_numpy(np.stack([synth.ricker(nt, 1e-3, 25.0)] * nshot).astype(np.float32)).cuda()
    d = torch.randn((nshot, nt, 600), generator=gen, device="cuda")
    first, out = torch.zeros_like(v), torch.zeros_like(v)
    contexts = []
    try:
        for k in range(6):
            ctx = fw.Context(grid, geom)
            contexts.append(ctx)
            ctx.born_adj(v, w, d, first if k == 0 else out)
            if k:
                diff = torch.linalg.vector_norm((out - first).double()) / torch.linalg.vector_norm(first.double())
                assert float(diff) <= 2e-6      # the same sums over other batches of shots
            assert torch.cuda.mem_get_info()[0] > 4 << 30
        before = contexts[0].get_option("workspace")
        contexts[0].born_adj(v, w, d, out)      # what a context holds it keeps
        assert contexts[0].get_option("workspace") == before and torch.equal(out, first)
    finally:
        for ctx in contexts:
            ctx.close()
