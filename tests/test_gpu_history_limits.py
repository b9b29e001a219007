"""Caps around the size at which the source side's history just fits the workspace: every one is accepted, since the
checkpoints take less, and gives the same results (FP32 reorderings only: relative L2 <= 2e-6, the bound of
test_gpu_history)."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
import paper_2206_02362_gb300 as fw  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,op,fields", [("born_adj", fw.OP_BORN_ADJ, 1), ("gradient", fw.OP_GRADIENT, 2)])
def test_caps_around_the_history(name, op, fields):
    nz, nx, sponge, nt = 20, 90, 6, 301
    field = 4 * (nz + 20) * 128
    grid = fw.Grid(nz=nz, nx=nx, sponge=sponge, nt=nt, dt=1e-3, dx=10.0, nh=1)
    geom = fw.Geometry(np.array([1]), np.array([40]), np.full(30, 1), 3 * np.arange(30))
    rng = np.random.default_rng(synth.SEED0 + 1301)
    cu = lambda a: torch.from_numpy(np.ascontiguousarray(a, np.float32)).cuda()  # noqa: E731
    v = cu(1800.0 + 25.0 * np.arange(nz)[:, None] + 60.0 * np.sin(np.arange(nx)[None, :] / 11.0))
    w, d, pt = cu(synth.ricker(nt, 1e-3, 22.0)[None]), cu(rng.standard_normal((1, nt, 30))), cu(rng.standard_normal((1, nz, nx)))

    def run(ctx):
        out = torch.zeros_like(v)
        if op == fw.OP_GRADIENT:
            ctx.gradient(v, w, pt, d, out, eps=1e-3)
        else:
            ctx.born_adj(v, w, d, out)
        return out.double(), ctx.launches

    K = min(64, nt - 1)                                   # the default segment of one shot; 5 segments
    states = (4 if fields == 2 else 2) * -(-(nt - 1) // K)
    least = fw.workspace_bytes(grid, geom, op, 1)         # with checkpoints at K
    fits = least + (fields * (nt - 1 - K) - states) * field
    with fw.Context(grid, geom, segment=17) as ctx:
        want, many = run(ctx)
    kept = 0
    for cap in range(fits - 8 * 1024, fits + 8 * 1024, 512):
        with fw.Context(grid, geom, max_workspace_bytes=cap) as ctx:
            got, few = run(ctx)
            kept += few < many - (nt - 1 - K)
            assert ctx.get_option("workspace") <= cap
        assert float(torch.linalg.vector_norm(got - want)) <= 2e-6 * float(torch.linalg.vector_norm(want))
    assert 0 < kept < 32                                  # the caps lie on both sides
