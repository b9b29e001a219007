"""A tuned schedule keeps the source side's history as the automatic one does: the adjoints recompute nothing after
fwime_autotune_schedule, alone and after a forward call with background reuse.  An explicit segment of the same length
recomputes, so the launch counts tell them apart; the results are those of the same sums, in other orders at most
(relative L2 <= 2e-6, the bound of test_gpu_history)."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
import paper_2206_02362_gb300 as fw  # noqa: E402

pytestmark = pytest.mark.gpu
NT, NSHOT, NH = 131, 6, 5


def inputs():
    nz, nx = 30, 100
    rng = np.random.default_rng(synth.SEED0 + 911)
    v = (1800.0 + 25.0 * np.arange(nz)[:, None] + 40.0 * rng.random((nz, nx))).astype(np.float32)
    t = dict(v=v, w=np.stack([synth.ricker(NT, 1e-3, 20.0)] * NSHOT).astype(np.float32),
             pt=rng.standard_normal((NH, nz, nx)).astype(np.float32),
             d=rng.standard_normal((NSHOT, NT, 50)).astype(np.float32))
    geom = fw.Geometry(np.full(NSHOT, 2), np.array([10, 30, 50, 70, 90, 95]), np.full(50, 1), 2 * np.arange(50))
    grid = fw.Grid(nz=nz, nx=nx, sponge=8, nt=NT, dt=1e-3, dx=10.0, nh=NH)
    return grid, geom, {k: torch.from_numpy(np.ascontiguousarray(a)).cuda() for k, a in t.items()}


def run(ctx, name, t):
    out = torch.zeros(t["pt"].shape if name == "born_ext_adj" else t["v"].shape, device="cuda")
    args = {"born_adj": (), "born_ext_adj": (), "tomo_adj": (t["pt"],), "gradient": (t["pt"],)}[name]
    getattr(ctx, name)(t["v"], t["w"], *args, t["d"], out)
    return out.double(), ctx.launches


def close(a, b):
    assert torch.isfinite(b).all() and torch.any(b)
    assert float(torch.linalg.vector_norm(a - b)) <= 2e-6 * float(torch.linalg.vector_norm(b))


@pytest.mark.parametrize("name,op,fields", [("born_adj", fw.OP_BORN_ADJ, 1), ("born_ext_adj", fw.OP_BORN_EXT_ADJ, 1),
                                            ("tomo_adj", fw.OP_TOMO_ADJ, 2), ("gradient", fw.OP_GRADIENT, 2)])
def test_tuned_adjoint_keeps_the_history(name, op, fields):
    grid, geom, t = inputs()
    with fw.Context(grid, geom) as ctx:
        s = ctx.autotune_schedule(op)
        got, few = run(ctx, name, t)
        ctx.set_option("segment", s["segment"])            # the caller's own: checkpoints
        want, many = run(ctx, name, t)
    close(got, want)
    K, batches = s["segment"], -(-NSHOT // s["shots_per_batch"])
    states = (-(-(NT - 1) // K) - 1) * K                   # steps of the checkpointing sweep
    assert many - few >= fields * states * batches


def test_tuned_pair_keeps_the_background():
    grid, geom, t = inputs()
    d = torch.zeros_like(t["d"])
    with fw.Context(grid, geom, reuse_background=1) as ctx:
        s = ctx.autotune_schedule(fw.OP_BORN_EXT_ADJ)
        counts, outs = [], []
        for _ in range(2):
            ctx.born_ext(t["v"], t["w"], t["pt"], d)
            out, n = run(ctx, "born_ext_adj", t)
            assert ctx.get_option("background_reused") == 1
            counts.append(n)
            outs.append(out)
            ctx.set_option("segment", s["segment"])
    close(outs[0], outs[1])
    assert counts[1] - counts[0] >= (NT - 1) * -(-NSHOT // s["shots_per_batch"])


def test_tuned_batches_are_not_cut_for_a_history():
    """20 Marmousi2-sized shots, a history of 7 in the cap, checkpoints of all: the tuner keeps the batch of all shots
    (or of half of them) instead of the few shots that a history leaves room for."""
    nz, nx, nt, nshot = 350, 1700, 401, 20
    field = 4 * 458 * 1824
    grid = fw.Grid(nz=nz, nx=nx, sponge=50, nt=nt, dt=8e-4, dx=10.0, nh=3)
    geom = fw.Geometry(np.full(nshot, 2), 80 * np.arange(nshot), np.full(20, 1), np.arange(20))
    # fields per shot: 424 with the history (K = 20), 84 with checkpoints (104 at K = 40)
    with fw.Context(grid, geom, max_workspace_bytes=7 * 450 * field) as ctx:
        assert ctx.autotune_schedule(fw.OP_BORN_EXT_ADJ)["shots_per_batch"] in (nshot, nshot // 2)
