"""The split gradient (fwime_gradient_forward, fwime_gradient_backward) under a workspace cap that its state fits only
with the shorter segments: the adjoint half still starts from the kept state.  The gradient's own arithmetic at that
segment length, FP32 reorderings only: relative L2 <= 2e-6 (the bound between schedules of test_gpu_history)."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
import paper_2206_02362_gb300 as fw  # noqa: E402

pytestmark = pytest.mark.gpu


# 399 steps, 5 offsets, one shot, fields of 4.1 MB: with 2 GB set aside the state and the adjoint sweep take 3.95 GB in
# segments of 64 steps, 3.07 GB in segments of 20
@pytest.mark.parametrize("cap,kept", [(3.5e9, 1), (4.5e9, 1), (2.5e9, 0)])
def test_state_is_kept_where_the_shorter_segments_fit(cap, kept):
    nz, nx, nt, nh = 996, 1012, 400, 5
    grid = fw.Grid(nz=nz, nx=nx, sponge=2, nt=nt, dt=1e-3, dx=10.0, nh=nh)
    geom = fw.Geometry(np.array([1]), np.array([500]), np.full(30, 1), 455 + 3 * np.arange(30))
    gen = torch.Generator(device="cuda").manual_seed(synth.SEED0)
    v = torch.full((nz, nx), 2000.0, device="cuda")
    w = torch.from_numpy(synth.ricker(nt, 1e-3, 22.0)[None].astype(np.float32)).cuda()
    pt = torch.randn((nh, nz, nx), generator=gen, device="cuda")
    d = torch.randn((1, nt, 30), generator=gen, device="cuda")
    own, got = torch.zeros_like(v), torch.zeros_like(v)
    with fw.Context(grid, geom, segment=20) as ctx:
        J = ctx.gradient(v, w, pt, d, own, eps=1e-3)
    assert torch.isfinite(own).all() and torch.any(own)
    with fw.Context(grid, geom, max_workspace_bytes=int(cap)) as ctx:
        Jf = ctx.gradient_forward(v, w, pt, d, eps=1e-3)
        ctx.gradient_backward(v, w, pt, d, got, eps=1e-3)
        assert ctx.get_option("background_reused") == kept
    assert abs(Jf - J) <= 2e-6 * abs(J)
    assert float(torch.linalg.vector_norm((got - own).double())) <= 2e-6 * float(torch.linalg.vector_norm(own.double()))
