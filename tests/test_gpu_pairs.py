"""Two time steps per launch (batches whose fields exceed the L2 cache) against a launch per step (smaller batches).
The wavefields have the same bits, so the modelling operators' outputs are equal; the adjoints sum the same terms per
shot in other batches: FP32 reorderings, relative L2 <= 2e-6.  The launch counts show which one ran."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
import paper_2206_02362_gb300 as fw  # noqa: E402

pytestmark = pytest.mark.gpu


def inputs(nz, nx, nt, nshot, nh):
    rng = np.random.default_rng(synth.SEED0 + 193)
    v = (1800.0 + 600.0 * np.arange(nz)[:, None] / nz + 60.0 * np.sin(np.arange(nx)[None, :] / 11.0)).astype(np.float32)
    w = np.stack([synth.ricker(nt, 1e-3, 60.0) * (1.0 + 0.1 * (s % 7)) for s in range(nshot)]).astype(np.float32)
    rec = np.arange(0, nx, 5)
    rec_iz = np.where(np.arange(len(rec)) % 3 == 0, nz - 1, 2)       # two receiver rows, ends of the grid included
    src_ix = np.linspace(0, nx - 1, nshot).astype(int)
    geom = fw.Geometry(src_iz=(np.arange(nshot) * 7) % nz, src_ix=src_ix, rec_iz=rec_iz, rec_ix=rec)
    t = dict(v=v, w=w, pt=rng.standard_normal((nh, nz, nx)).astype(np.float32),
             dv=(40.0 * np.sin(1.0 + np.arange(nz)[:, None] / 5.0 + np.arange(nx)[None, :] / 9.0)).astype(np.float32),
             d=rng.standard_normal((nshot, nt, len(rec))).astype(np.float32))
    return geom, {k: torch.from_numpy(np.ascontiguousarray(a)).cuda() for k, a in t.items()}


def call(ctx, op, t):
    if op in ("forward", "born_ext", "tomo"):
        out = torch.full(t["d"].shape, 7.0, device="cuda")
        args = {"forward": (), "born_ext": (t["pt"],), "tomo": (t["pt"], t["dv"])}[op]
        getattr(ctx, op)(t["v"], t["w"], *args, out)
    else:
        out = torch.full(t["pt"].shape if op == "born_ext_adj" else t["v"].shape, 7.0, device="cuda")
        args = {"born_adj": (), "born_ext_adj": (), "tomo_adj": (t["pt"],), "gradient": (t["pt"],)}[op]
        getattr(ctx, op)(t["v"], t["w"], *args, t["d"], out, **({"eps": 1e-3} if op == "gradient" else {}))
    return out.cpu().numpy(), ctx.launches


# shots that just exceed the line; strips of 120 columns that end with the grid, one short of it, and inside; chunks
# of odd and even numbers of rows; odd and even numbers of steps and segments
@pytest.mark.parametrize("op,nh,opts", [
    ("forward", 1, {}), ("born_ext", 5, {}), ("tomo", 5, {}), ("born_adj", 1, {}), ("born_ext_adj", 7, {}),
    ("tomo_adj", 5, {}), ("gradient", 5, {}), ("gradient", 5, {"segment": 5}), ("born_ext_adj", 5, {"segment": 6}),
    ("born_ext", 3, {"time_lag": 1}), ("born_ext_adj", 3, {"time_lag": 1}), ("gradient", 3, {"time_lag": 1})])
@pytest.mark.parametrize("nz,nx,sponge,nt", [(43, 460, 6, 24), (150, 1001, 20, 25), (401, 130, 9, 13), (3, 700, 1, 20)])
def test_pairs_of_steps(op, nh, opts, nz, nx, sponge, nt):
    pad = 2 * (sponge + 4)
    points = (nz + pad) * (-(-(nx + pad) // 32) * 32)
    nshot = -(-13000000 // points)
    geom, t = inputs(nz, nx, nt, nshot, nh)
    grid = fw.Grid(nz=nz, nx=nx, sponge=sponge, nt=nt, dt=1e-3, dx=10.0, nh=nh)
    st = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(st):
        with fw.Context(grid, geom, stream=st, shots_per_batch=nshot, **opts) as ctx:
            got, few = call(ctx, op, t)
            again, _ = call(ctx, op, t)
        with fw.Context(grid, geom, stream=st, shots_per_batch=nshot // 2 + 1, **opts) as ctx:
            want, many = call(ctx, op, t)
    assert few < many
    assert np.isfinite(want).all() and np.any(want)
    if op in ("forward", "born_ext", "tomo"):
        np.testing.assert_array_equal(got, want)
    else:
        assert np.linalg.norm((got - want).astype(np.float64)) <= 2e-6 * np.linalg.norm(want.astype(np.float64))
    np.testing.assert_array_equal(again, got)
