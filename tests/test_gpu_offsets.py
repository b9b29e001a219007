"""Extension kernels at every kind of offset count: sizes served by one launch, sizes cut into several chunks of
offsets, counts at the chunks' edges, rows shorter than a CTA and offsets that reach past the grid on both sides.
GPU (FP32) against the FP64 oracle, relative L2 <= 1e-4 (the bound of the parity tests)."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
import paper_2206_02362_gb300 as fw  # noqa: E402

pytestmark = pytest.mark.gpu
TOL = 1e-4

# 15 | 16, 23 | 25, 31 | 33, 47 | 49: the last count of a chunk size and the first of the next; 97 and 101: three chunks
COUNTS = [1, 3, 7, 9, 13, 15, 17, 21, 23, 25, 29, 31, 33, 41, 47, 49, 51, 97, 101]


def setup(nh, nx, W, nshot=2):
    nz, nt, dx, dt = 5, 48, 10.0, 1e-3
    rng = np.random.default_rng(synth.SEED0 + 1000 * nh + nx)
    v = (1800.0 + 30.0 * np.arange(nz)[:, None] + 90.0 * np.sin(np.arange(nx)[None, :] / 9.0)).astype(np.float32)
    w = np.stack([synth.ricker(nt, dt, 25.0) * (1.0 + 0.2 * s) for s in range(nshot)]).astype(np.float32)
    geo = dict(src_iz=np.array([1, 3])[:nshot], src_ix=np.array([2, nx - 3])[:nshot], rec_iz=np.full(nx, 1),
               rec_ix=np.arange(nx))
    pt = rng.standard_normal((nh, nz, nx)).astype(np.float32)
    d = rng.standard_normal((nshot, nt, nx)).astype(np.float32)
    og = oracle.Grid(nz=nz, nx=nx, W=W, nt=nt, dt=dt, dx=dx, nh=nh)
    fg = fw.Grid(nz=nz, nx=nx, sponge=W, nt=nt, dt=dt, dx=dx, nh=nh)
    return og, fg, geo, v, w, pt, d


def rel(a, b):
    return float(np.linalg.norm(a.cpu().numpy().astype(np.float64) - b) / np.linalg.norm(b))


def cu(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("nh", COUNTS)
@pytest.mark.parametrize("nx,W,segment", [(61, 0, 0), (61, 6, 5), (277, 3, 0)])
def test_extension_offsets(nh, nx, W, segment):
    og, fg, geo, v, w, pt, d = setup(nh, nx, W)
    ogeo, v64, w64 = oracle.Geometry(**geo), v.astype(np.float64), w.astype(np.float64)
    with fw.Context(fg, fw.Geometry(**geo), segment=segment) as ctx:
        img = torch.zeros(pt.shape, device="cuda")
        ctx.born_ext_adj(cu(v), cu(w), cu(d), img)
        dat = torch.zeros(d.shape, device="cuda")
        ctx.born_ext(cu(v), cu(w), cu(pt), dat)
        g = torch.zeros(v.shape, device="cuda")
        ctx.tomo_adj(cu(v), cu(w), cu(pt), cu(d), g)
    assert rel(img, oracle.born_ext_adj(og, v64, ogeo, w64, d.astype(np.float64))) <= TOL
    assert rel(dat, oracle.born_ext(og, v64, ogeo, w64, pt.astype(np.float64))) <= TOL
    assert rel(g, oracle.tomo_adj(og, v64, ogeo, w64, pt.astype(np.float64), d.astype(np.float64))) <= TOL


@pytest.mark.parametrize("nx", [1, 3, 64, 130])
def test_local_imaging_rows(nx):
    """B* (pointwise imaging): rows of one to a few 4-column groups, pairs not a multiple of those in flight."""
    og, fg, geo, v, w, pt, d = setup(1, max(nx, 5), 2)
    if nx < 5:
        v, d = v[:, :nx], d[:, :, :nx]
        geo = dict(src_iz=np.array([1, 3]), src_ix=np.array([0, nx - 1]), rec_iz=np.full(nx, 1), rec_ix=np.arange(nx))
        og = oracle.Grid(nz=5, nx=nx, W=2, nt=48, dt=1e-3, dx=10.0, nh=1)
        fg = fw.Grid(nz=5, nx=nx, sponge=2, nt=48, dt=1e-3, dx=10.0, nh=1)
    for opts in (dict(), dict(segment=5), dict(shots_per_batch=1, segment=7)):
        with fw.Context(fg, fw.Geometry(**geo), **opts) as ctx:
            g = torch.zeros(v.shape, device="cuda")
            ctx.born_adj(cu(v), cu(w), cu(d), g)
        assert rel(g, oracle.born_adj(og, v.astype(np.float64), oracle.Geometry(**geo), w.astype(np.float64),
                                      d.astype(np.float64))) <= TOL
