"""Background reuse (FWIME_OPT_REUSE_BACKGROUND) where memory is short: the adjoints give the results of the
self-contained operators, directly and captured in graphs, whatever the writer could keep.  FP32 reorderings only:
relative L2 <= 2e-6 (the bound between schedules of test_gpu_history), 1e-4 against the FP64 oracle."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
import paper_2206_02362_gb300 as fw  # noqa: E402

pytestmark = pytest.mark.gpu
NZ, NX, W, DX, DT = 20, 90, 6, 10.0, 1e-3
PLANE = 4 * (NZ + 2 * (W + 4)) * (-(-(NX + 2 * (W + 4)) // 32) * 32)       # bytes of a padded field


def problem(nt, nh):
    rng = np.random.default_rng(synth.SEED0 + 1201)
    v = (1800.0 + 25.0 * np.arange(NZ)[:, None] + 60.0 * np.sin(np.arange(NX)[None, :] / 11.0)).astype(np.float32)
    w = synth.ricker(nt, DT, 22.0)[None].astype(np.float32)
    a = dict(nz=NZ, nx=NX, nt=nt, dt=DT, dx=DX, nh=nh)
    g = dict(src_iz=np.array([1]), src_ix=np.array([40]), rec_iz=np.full(30, 1), rec_ix=3 * np.arange(30))
    x = dict(v=v, w=w, pt=rng.standard_normal((nh, NZ, NX)).astype(np.float32),
             d=rng.standard_normal((1, nt, 30)).astype(np.float32),
             dv=(40.0 * np.sin(1.0 + np.arange(NZ)[:, None] / 5.0 + np.arange(NX)[None, :] / 9.0)).astype(np.float32))
    f64 = {k: q.astype(np.float64) for k, q in x.items()}
    og, ogeo = oracle.Grid(W=W, **a), oracle.Geometry(**g)
    ref = dict(born_adj=oracle.born_adj(og, f64["v"], ogeo, f64["w"], f64["d"]),
               born_ext_adj=oracle.born_ext_adj(og, f64["v"], ogeo, f64["w"], f64["d"]))
    return fw.Grid(sponge=W, **a), fw.Geometry(**g), {k: torch.from_numpy(np.ascontiguousarray(q)).cuda() for k, q in x.items()}, ref


def adjoint(ctx, name, t):
    out = torch.full(t["pt"].shape if name == "born_ext_adj" else t["v"].shape, 7.0, device="cuda")
    torch.cuda.synchronize()
    getattr(ctx, name)(t["v"], t["w"], t["d"], out)
    return out.cpu().numpy().astype(np.float64)


def write(ctx, name, t):
    getattr(ctx, name)(t["v"], t["w"], t["pt" if name == "born_ext" else "dv"], torch.zeros_like(t["d"]))


def close(a, b, tol):
    assert np.isfinite(a).all() and np.linalg.norm(a - b) <= tol * np.linalg.norm(b)


# 399 steps, 41 offsets: a segment of 64 steps takes B~ 175 fields and B* 135, one of 20 steps 87 and 47 (and states)
@pytest.mark.parametrize("graph", [0, 1])
@pytest.mark.parametrize("planes", [100, 150, 190])
@pytest.mark.parametrize("writer", ["born_ext", "born"])
@pytest.mark.parametrize("reader", ["born_adj", "born_ext_adj"])
def test_adjoint_after_a_writer_under_a_cap(graph, planes, writer, reader):
    grid, geom, t, ref = problem(400, 41)
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    with fw.Context(grid, geom, segment=20) as ctx:
        own = adjoint(ctx, reader, t)
    close(own, ref[reader], 1e-4)
    with fw.Context(grid, geom, stream=stream, max_workspace_bytes=planes * PLANE, graph=graph,
                    reuse_background=1) as ctx:
        for _ in range(2):                    # the second time replays the graphs
            write(ctx, writer, t)
            close(adjoint(ctx, reader, t), own, 2e-6)
            assert ctx.get_option("background_reused") == 1


# 130 steps: the history is 130 fields; a segment of 64 steps takes B~ and B~* 175, one of 11 steps 69
@pytest.mark.parametrize("graph", [0, 1])
@pytest.mark.parametrize("planes", [100, 135, 150, 230])
def test_adjoint_after_a_kept_history_under_a_cap(graph, planes):
    grid, geom, t, ref = problem(131, 41)
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    with fw.Context(grid, geom, stream=stream, max_workspace_bytes=planes * PLANE, graph=graph,
                    reuse_background=1) as ctx:
        for _ in range(2):
            write(ctx, "born_ext", t)
            close(adjoint(ctx, "born_ext_adj", t), ref["born_ext_adj"], 1e-4)
            assert ctx.get_option("background_reused") == 1
            ctx.forward(t["v"], t["w"], torch.zeros_like(t["d"]))    # drops what was kept
            adjoint(ctx, "born_adj", t)
            assert ctx.get_option("background_reused") == 0


@pytest.mark.parametrize("planes", [500, 600])
def test_the_cap_holds_a_kept_history_and_the_workspace(planes):
    """A history of 399 fields beside 139 fields of workspace: only the larger cap holds both (measured as the device's
    free memory; 64 MB, 15 fields, are left for the allocator's rounding)."""
    nz, nx, sponge, nt, nh = 996, 1012, 2, 400, 5
    field = 4 * (nz + 12) * (nx + 12)
    grid = fw.Grid(nz=nz, nx=nx, sponge=sponge, nt=nt, dt=DT, dx=DX, nh=nh)
    geom = fw.Geometry(np.array([1]), np.array([500]), np.full(30, 1), 455 + 3 * np.arange(30))
    gen = torch.Generator(device="cuda").manual_seed(synth.SEED0)
    v = torch.full((nz, nx), 2000.0, device="cuda")
    w = torch.from_numpy(synth.ricker(nt, DT, 22.0)[None].astype(np.float32)).cuda()
    pt = torch.randn((nh, nz, nx), generator=gen, device="cuda")
    d = torch.randn((1, nt, 30), generator=gen, device="cuda")
    dout, img, own = torch.zeros_like(d), torch.zeros_like(pt), torch.zeros_like(pt)

    def free():
        torch.cuda.synchronize()
        return torch.cuda.mem_get_info()[0]

    with fw.Context(grid, geom, segment=20) as ctx:      # (also loads the kernels)
        ctx.born_ext(v, w, pt, dout)
        ctx.born_ext_adj(v, w, d, own)
        ctx.forward(v, w, dout)
    before = free()
    with fw.Context(grid, geom, max_workspace_bytes=planes * field, reuse_background=1) as ctx:
        for _ in range(2):
            ctx.born_ext(v, w, pt, dout)
            ctx.born_ext_adj(v, w, d, img)
            assert ctx.get_option("background_reused") == 1
            assert before - free() <= planes * field + (64 << 20)
            diff = torch.linalg.vector_norm((img - own).double()) / torch.linalg.vector_norm(own.double())
            assert float(diff) <= 2e-6
            ctx.gradient(v, w, pt, d, torch.zeros_like(v))
            assert before - free() <= planes * field + (64 << 20)


@pytest.mark.parametrize("change", ["v", "w"])
@pytest.mark.parametrize("reader", ["born_adj", "born_ext_adj"])
def test_host_pointers_tell_models_and_wavelets_apart(change, reader):
    """With host I/O every model is staged at one address: the caller's pointers decide whether the background is of
    the same v and w."""
    grid, geom, t, _ = problem(131, 5)
    a = {k: q.cpu().numpy() for k, q in t.items()}
    b = dict(a)
    b[change] = (a[change] * np.float32(1.05)).copy()

    def run(ctx, x):
        out = np.full(a["pt"].shape if reader == "born_ext_adj" else a["v"].shape, 7.0, np.float32)
        getattr(ctx, reader)(x["v"], x["w"], x["d"], out)
        return out.astype(np.float64)

    with fw.Context(grid, geom, host_io=1) as ctx:
        own = [run(ctx, a), run(ctx, b)]
    with fw.Context(grid, geom, host_io=1, reuse_background=1) as ctx:
        for _ in range(2):                     # the first writer may find the staging not yet in place
            ctx.born_ext(a["v"], a["w"], a["pt"], np.zeros_like(a["d"]))
            close(run(ctx, b), own[1], 2e-6)
            assert ctx.get_option("background_reused") == 0
        ctx.born_ext(a["v"], a["w"], a["pt"], np.zeros_like(a["d"]))
        close(run(ctx, a), own[0], 2e-6)
        assert ctx.get_option("background_reused") == 1


@pytest.mark.parametrize("planes", [150, 300, 420, 600])
@pytest.mark.parametrize("writer", ["born", "born_ext"])
@pytest.mark.parametrize("reader", ["born_adj", "born_ext_adj"])
def test_staged_inputs_stay_in_place_under_a_cap(planes, writer, reader):
    """Host I/O: the adjoint's plan may move the arena, and what was kept may be given back for it; the call then runs
    on the inputs that it staged."""
    grid, geom, t, ref = problem(131, 41)
    a = {k: q.cpu().numpy() for k, q in t.items()}
    staging = 4 * (2 * 41 * NZ * NX + 4 * 131 * 30)
    with fw.Context(grid, geom, host_io=1, max_workspace_bytes=planes * PLANE + staging, reuse_background=1) as ctx:
        for _ in range(2):
            dout = np.full_like(a["d"], 7.0)
            getattr(ctx, writer)(a["v"], a["w"], a["pt" if writer == "born_ext" else "dv"], dout)
            assert np.isfinite(dout).all() and np.abs(dout).max() > 0
            out = np.full(a["pt"].shape if reader == "born_ext_adj" else a["v"].shape, 7.0, np.float32)
            getattr(ctx, reader)(a["v"], a["w"], a["d"], out)
            close(out.astype(np.float64), ref[reader], 1e-4)
