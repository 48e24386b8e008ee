"""The transfer as two kernels (geometry of all saved states, one warp per ray; then the Stokes chain,
one lane per ray) against the kernel that does both on one lane, bit for bit:
- mixed form: against the staged-fetch transfer, which is a one-lane kernel;
- FP64: against the same call with the smallest caller's workspace, which has no room for the
  records and takes the one-lane kernel, a ray at a time.
Rays of 1, 31, 32, 33, 64 and 65 states (blocks of 32: a block filled, a last block that holds the
last state alone), whole rays, and points that do not emit at the far end, in between and next to the
camera (a small grid radius, a magnetization cut)."""
import dataclasses

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def rt():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__

    __graft_entry__.build()
    from paper_2302_02733_gb300 import polrt

    torch.cuda.set_device(0)
    ctx = polrt.rt_create(0, torch.cuda.current_stream().cuda_stream)
    yield polrt, ctx
    polrt.rt_destroy(ctx)


@pytest.mark.parametrize("nmax", [1, 31, 32, 33, 64, 65, 20000])
@pytest.mark.parametrize("cut", [1.0, 2e-3])
def test_two_kernels_equal_one(rt, synth, torus_grid, nmax, cut):
    polrt, ctx = rt
    prims, g = torus_grid
    g = dataclasses.replace(g, sigma_cut=cut)
    # the camera inside the grid's radius (every step near it emits), then outside
    for r_cam in (1000.0, 1200.0):
        cam = synth.Camera(incl_deg=35.0, nx=24, ny=12, r_cam=r_cam)
        polrt.rt_set_camera(ctx, cam)
        polrt.rt_set_integrator(ctx, 0.05, nmax)
        polrt.rt_load_model(ctx, polrt.grid_model(torch.from_numpy(prims).cuda(), g))
        ws = torch.empty(polrt.rt_workspace_min_bytes(), dtype=torch.uint8, device="cuda")

        def render(form):
            dt = torch.float64 if form == polrt.RT_FP64 else torch.float32
            img = torch.full((12, 24, 4), float("nan"), dtype=dt, device="cuda")
            dep = torch.full((12, 24, 2), float("nan"), dtype=dt, device="cuda")
            st = torch.zeros((12, 24), dtype=torch.uint8, device="cuda")
            polrt.rt_render_depths(ctx, form, img, dep, st)
            c = polrt.rt_last_counters(ctx)
            return img, dep, st, (c["points"], c["emitting_points"], c["steps"])

        try:
            two = render(polrt.RT_MIXED)
            polrt.rt_set_grid_fetch(ctx, polrt.RT_FETCH_STAGED)
            one = render(polrt.RT_MIXED)
            polrt.rt_set_grid_fetch(ctx, polrt.RT_FETCH_AUTO)
            two64 = render(polrt.RT_FP64)
            polrt.rt_set_workspace(ctx, ws)
            one64 = render(polrt.RT_FP64)
        finally:
            polrt.rt_set_workspace(ctx, None)
            polrt.rt_set_grid_fetch(ctx, polrt.RT_FETCH_AUTO)
            polrt.rt_set_integrator(ctx, 0.05, 20000)
        for a, b in ((two, one), (two64, one64)):
            assert torch.isfinite(a[0]).all()
            assert all(torch.equal(x, y) for x, y in zip(a[:3], b[:3])) and a[3] == b[3]
        if nmax == 20000:
            assert two[0][..., 0].max() > 0
            assert two[3][1] < two[3][0] if cut < 1.0 or r_cam > 1000.0 else two[3][1] > 0
