"""The geodesic kernel's two register budgets (launches of up to 38,912 rays, and of more): an image of
40,800 rays as one launch against the same image in chunks of fewer rays (a caller's workspace of a third
of what it needs), bit for bit in images, status codes and step counts. The arithmetic of a ray does not
depend on the launch it is in."""
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


@pytest.mark.parametrize("incl", [1.0, 70.0])
def test_few_rays_equal_many(rt, synth, incl):
    polrt, ctx = rt
    cam = synth.Camera(incl_deg=incl, nx=240, ny=170)
    polrt.rt_set_camera(ctx, cam)
    polrt.rt_set_integrator(ctx, 0.05, 20000)
    polrt.rt_load_model(ctx, polrt.adaf_model(synth.adaf_params(1)))
    res = []
    try:
        for frac in (None, 1 / 3):
            ws = torch.empty(int(frac * polrt.rt_workspace_hint(ctx)), dtype=torch.uint8, device="cuda") if frac else None
            polrt.rt_set_workspace(ctx, ws)
            img = torch.full((170, 240, 4), float("nan"), dtype=torch.float32, device="cuda")
            st = torch.zeros((170, 240), dtype=torch.uint8, device="cuda")
            polrt.rt_render(ctx, polrt.RT_MIXED, img, st)
            res.append((img, st, polrt.rt_last_counters(ctx)))
    finally:
        polrt.rt_set_workspace(ctx, None)
    (a, sa, ca), (b, sb, cb) = res
    assert ca["geodesic_launches"] == 1 and cb["geodesic_launches"] >= 2
    assert torch.isfinite(a).all() and torch.equal(a, b) and torch.equal(sa, sb) and ca["steps"] == cb["steps"]
