"""The adjoint operators' schedules: source-side D2t kept for the whole record, recomputed from checkpoints (an
explicit segment length, a budget the history does not fit, the plain path), and kept by a preceding B or B~
(background reuse), must agree.  FP32 reorderings only: relative L2 <= 2e-6 between the schedules on records of
130 steps (their sums run over the same terms), 1e-4 against the FP64 oracle."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
import paper_2206_02362_gb300 as fw  # noqa: E402

pytestmark = pytest.mark.gpu


def setup(nh=7, nshot=5, nt=131):
    nz, nx, W, dx, dt = 14, 90, 6, 10.0, 1e-3
    rng = np.random.default_rng(synth.SEED0 + 77)
    v = (1800.0 + 25.0 * np.arange(nz)[:, None] + 60.0 * np.sin(np.arange(nx)[None, :] / 11.0)).astype(np.float32)
    w = np.stack([synth.ricker(nt, dt, 22.0) * (1.0 + 0.1 * s) for s in range(nshot)]).astype(np.float32)
    geo = dict(src_iz=np.full(nshot, 1), src_ix=np.linspace(3, nx - 4, nshot).astype(int), rec_iz=np.full(30, 1),
               rec_ix=3 * np.arange(30))
    pt = rng.standard_normal((nh, nz, nx)).astype(np.float32)
    d = rng.standard_normal((nshot, nt, 30)).astype(np.float32)
    dv = synth.gaussian_blobs(nz, nx, rng, amp=40.0, sigma_pts=4.0, ring=1).astype(np.float32)
    grid = dict(nz=nz, nx=nx, nt=nt, dt=dt, dx=dx, nh=nh)
    return grid, W, geo, v, w, pt, d, dv


def cu(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def rel(a, b):
    a, b = np.asarray(a, np.float64), np.asarray(b, np.float64)
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


def run(ctx, name, t):
    out = torch.zeros(t["pt"].shape if name == "born_ext_adj" else t["v"].shape, device="cuda")
    if name == "born_adj":
        ctx.born_adj(t["v"], t["w"], t["d"], out)
    elif name == "born_ext_adj":
        ctx.born_ext_adj(t["v"], t["w"], t["d"], out)
    elif name == "tomo_adj":
        ctx.tomo_adj(t["v"], t["w"], t["pt"], t["d"], out)
    else:
        ctx.gradient(t["v"], t["w"], t["pt"], t["d"], out, eps=1e-3)
    return out.cpu().numpy()


@pytest.mark.parametrize("name,nh", [("born_adj", 1), ("born_ext_adj", 7), ("tomo_adj", 7), ("gradient", 7)])
def test_schedules_agree(name, nh):
    grid, W, geo, v, w, pt, d, dv = setup(nh)
    t = dict(v=cu(v), w=cu(w), pt=cu(pt), d=cu(d))
    fg, fgeo = fw.Grid(sponge=W, **grid), fw.Geometry(**geo)
    op = dict(born_adj=fw.OP_BORN_ADJ, born_ext_adj=fw.OP_BORN_EXT_ADJ, tomo_adj=fw.OP_TOMO_ADJ, gradient=fw.OP_GRADIENT)[name]
    small = fw.workspace_bytes(fg, fgeo, op, 2)          # checkpoints of two shots: the history of one does not fit
    og, ogeo = oracle.Grid(W=W, **grid), oracle.Geometry(**geo)
    f64 = [a.astype(np.float64) for a in (v, w, pt, d)]
    ref = {"born_adj": lambda: oracle.born_adj(og, f64[0], ogeo, f64[1], f64[3]),
           "born_ext_adj": lambda: oracle.born_ext_adj(og, f64[0], ogeo, f64[1], f64[3]),
           "tomo_adj": lambda: oracle.tomo_adj(og, f64[0], ogeo, f64[1], f64[2], f64[3]),
           "gradient": lambda: oracle.gradient(og, f64[0], ogeo, f64[1], f64[2], f64[3], eps=1e-3)[1]}[name]()
    outs, launches = {}, {}
    for key, opts in dict(kept=dict(), batches=dict(shots_per_batch=2), segments=dict(segment=11), plain=dict(plain=1),
                          budget=dict(max_workspace_bytes=small)).items():
        with fw.Context(fg, fgeo, **opts) as ctx:
            outs[key] = run(ctx, name, t)
            launches[key] = ctx.launches
        assert rel(outs[key], ref) <= 1e-4, key
        assert rel(outs[key], outs["kept"]) <= 2e-6, key
    assert launches["kept"] < launches["segments"]       # nothing is recomputed when the history is kept


@pytest.mark.parametrize("ext", [False, True])
@pytest.mark.parametrize("opts", [dict(), dict(shots_per_batch=2), dict(graph=1), dict(segment=9)])
def test_adjoint_after_forward_reuses_the_background(ext, opts):
    grid, W, geo, v, w, pt, d, dv = setup(7 if ext else 1)
    t = dict(v=cu(v), w=cu(w), pt=cu(pt), d=cu(d))
    fg, fgeo = fw.Grid(sponge=W, **grid), fw.Geometry(**geo)
    name = "born_ext_adj" if ext else "born_adj"
    with fw.Context(fg, fgeo, segment=9) as ctx:
        ref = run(ctx, name, t)
    stream = torch.cuda.Stream() if opts.get("graph") else None
    dout, x = torch.zeros_like(t["d"]), cu(dv)
    torch.cuda.synchronize()
    with fw.Context(fg, fgeo, stream=stream, reuse_background=1, **opts) as ctx:
        for _ in range(2):
            if ext:
                ctx.born_ext(t["v"], t["w"], t["pt"], dout)
            else:
                ctx.born(t["v"], t["w"], x, dout)
            torch.cuda.synchronize()
            assert rel(run(ctx, name, t), ref) <= 2e-6
            assert ctx.get_option("background_reused") == 1
