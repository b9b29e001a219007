"""Which launches advanced the wavefields, by their exact number: two steps per launch for batches beyond the line, one
per step below it, and no step recomputed where the source side's history is kept."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
import paper_2206_02362_gb300 as fw  # noqa: E402

pytestmark = pytest.mark.gpu


def segments(nt, nshot, K=0):
    """Lengths of the segments: of K steps, or of the default length"""
    if K == 0:
        K = max(min(max(round((nt - 1) ** 0.5), 8), 128), min(64, -(-256 // nshot)))
    K = min(K, nt - 1)
    return [min(K, nt - 1 - n) for n in range(0, nt - 1, K)]


def stencil_launches(op, seg, two, kept=True):
    """Of one batch: runs of n steps take n launches, or with two per launch n / 2 (an odd one first)"""
    f = lambda n: n // 2 + n % 2 if two else n  # noqa: E731
    each, sweep = sum(f(n) for n in seg), f(sum(seg))
    if op == "forward":
        return sweep
    if op == "born_ext":
        return 2 * each
    if op == "tomo":                       # the fields that c dv scatters have a source of their own kind: one per launch
        return 2 * each + 2 * sum(seg)
    states = sum(f(n) for n in seg[:-1])   # the sweep that leaves the states, where the history is not kept
    if op in ("born_adj", "born_ext_adj"):
        return sweep + each if kept else states + 2 * each
    forward = 2 * (each if op == "gradient" or kept else states)
    return forward + 2 * each + (0 if kept else 2 * each)


def count(op, grid, geom, **opts):
    nshot, nt, nrec = geom.nshot, grid.nt, geom.nrec
    v = torch.full((grid.nz, grid.nx), 2000.0, device="cuda")
    w = torch.from_numpy(np.stack([synth.ricker(nt, grid.dt, 25.0)] * nshot).astype(np.float32)).cuda()
    pt, d, m = torch.zeros((grid.nh, grid.nz, grid.nx), device="cuda"), torch.zeros((nshot, nt, nrec), device="cuda"), v.clone()
    args = {"forward": (d,), "born_ext": (pt, d), "tomo": (pt, m, d), "born_adj": (d, m), "born_ext_adj": (d, pt),
            "tomo_adj": (pt, d, m), "gradient": (pt, d, m)}[op]
    with fw.Context(grid, geom, profile=1, **opts) as ctx:
        getattr(ctx, op)(v, w, *args)
        return ctx.profile_read()["prop"]["launches"]


def geometry(nz, nx, nshot):
    return fw.Geometry(np.full(nshot, 2), np.linspace(0, nx - 1, nshot).astype(int), np.full(20, 1), np.arange(20))


OPS = ["forward", "born_ext", "tomo", "born_adj", "born_ext_adj", "tomo_adj", "gradient"]


@pytest.mark.parametrize("op", OPS)
@pytest.mark.parametrize("nt", [24, 25])
def test_two_steps_per_launch_from_the_line_on(op, nt):
    nz, nx, W = 150, 1001, 20              # 209088 points of a padded field
    nshot = -(-13000000 // 209088)
    grid = fw.Grid(nz=nz, nx=nx, sponge=W, nt=nt, dt=1e-3, dx=10.0, nh=3)
    geom = geometry(nz, nx, nshot)
    seg = segments(nt, nshot)
    assert count(op, grid, geom, shots_per_batch=nshot) == stencil_launches(op, seg, True)
    assert count(op, grid, geom, shots_per_batch=nshot - 1) == (stencil_launches(op, seg, False) * 2)


@pytest.mark.parametrize("op", OPS[3:])
def test_no_step_is_recomputed_with_a_history(op):
    nz, nx, W, nt, nshot = 14, 90, 6, 131, 5
    grid = fw.Grid(nz=nz, nx=nx, sponge=W, nt=nt, dt=1e-3, dx=10.0, nh=3)
    geom = geometry(nz, nx, nshot)
    seg = segments(nt, nshot)
    assert [len(seg), seg[0]] == [3, 52]
    assert count(op, grid, geom) == stencil_launches(op, seg, False)
    assert count(op, grid, geom, segment=52) == stencil_launches(op, seg, False, kept=False)
