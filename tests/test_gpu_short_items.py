"""Items of a few rows, down to one (a context on the default stream, few shots), against items of eight rows or more
(a stream of its own): the same arithmetic per point in the same order, so every output is equal bit by bit, whatever
the rows per item, the number of steps or the options."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
import paper_2206_02362_gb300 as fw  # noqa: E402

pytestmark = pytest.mark.gpu


def inputs(nz, nx, nt, nshot, nh):
    rng = np.random.default_rng(synth.SEED0 + 191)
    v = (1800.0 + 12.0 * np.arange(nz)[:, None] + 60.0 * np.sin(np.arange(nx)[None, :] / 11.0)).astype(np.float32)
    w = np.stack([synth.ricker(nt, 1e-3, 30.0) * (1.0 + 0.1 * s) for s in range(nshot)]).astype(np.float32)
    rec = np.arange(0, nx, 3)
    geom = fw.Geometry(src_iz=np.full(nshot, 1), src_ix=np.linspace(2, nx - 3, nshot).astype(int),
                       rec_iz=np.full(len(rec), 2), rec_ix=rec)
    t = dict(v=v, w=w, pt=rng.standard_normal((nh, nz, nx)).astype(np.float32),
             dv=(40.0 * np.sin(1.0 + np.arange(nz)[:, None] / 5.0 + np.arange(nx)[None, :] / 9.0)).astype(np.float32),
             d=rng.standard_normal((nshot, nt, len(rec))).astype(np.float32))
    return geom, {k: torch.from_numpy(np.ascontiguousarray(a)).cuda() for k, a in t.items()}


def call(ctx, op, t):
    if op in ("forward", "born_ext", "tomo"):
        out = torch.full(t["d"].shape, 7.0, device="cuda")
        {"forward": lambda: ctx.forward(t["v"], t["w"], out),
         "born_ext": lambda: ctx.born_ext(t["v"], t["w"], t["pt"], out),
         "tomo": lambda: ctx.tomo(t["v"], t["w"], t["pt"], t["dv"], out)}[op]()
    else:
        out = torch.full(t["pt"].shape if op == "born_ext_adj" else t["v"].shape, 7.0, device="cuda")
        {"born_adj": lambda: ctx.born_adj(t["v"], t["w"], t["d"], out),
         "born_ext_adj": lambda: ctx.born_ext_adj(t["v"], t["w"], t["d"], out),
         "tomo_adj": lambda: ctx.tomo_adj(t["v"], t["w"], t["pt"], t["d"], out),
         "gradient": lambda: ctx.gradient(t["v"], t["w"], t["pt"], t["d"], out, eps=1e-3)}[op]()
    return out.cpu().numpy()


@pytest.mark.parametrize("op,nh,opts", [
    ("forward", 1, {}), ("forward", 1, {"free_surface": 1}), ("born_ext", 5, {}), ("tomo", 7, {}), ("born_adj", 1, {}),
    ("born_ext_adj", 11, {}), ("tomo_adj", 7, {}), ("gradient", 5, {}), ("gradient", 7, {"segment": 5})])
@pytest.mark.parametrize("nz,nx,sponge,nt,nshot", [
    (14, 30, 6, 9, 1),            # fewer rows and columns than a strip
    (37, 131, 9, 130, 3),         # ragged strips and chunks
    (150, 470, 20, 260, 1),
])
def test_short_items(op, nh, opts, nz, nx, sponge, nt, nshot):
    geom, t = inputs(nz, nx, nt, nshot, nh)
    grid = fw.Grid(nz=nz, nx=nx, sponge=sponge, nt=nt, dt=1e-3, dx=10.0, nh=nh)
    with fw.Context(grid, geom, **opts) as ctx:
        got = call(ctx, op, t)
        again = call(ctx, op, t)
    torch.cuda.synchronize()
    with fw.Context(grid, geom, stream=torch.cuda.Stream(), **opts) as ctx:
        want = call(ctx, op, t)
    assert np.isfinite(want).all() and np.any(want)
    np.testing.assert_array_equal(got, want)
    np.testing.assert_array_equal(again, want)
