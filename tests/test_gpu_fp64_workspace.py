"""FP64 images in callers' workspaces: the transfer's records take only what the paths leave of the arena.
- the hinted size holds the image in one chunk at the default step;
- at 1.6 times one ray's budget (32 arena blocks) rays of up to 28 blocks fit (an ADAF over 80 M at
  eps = 0.018, counted with the oracle), on the one-lane kernel where the records do not;
- paths of 18 blocks a ray (20 M, eps = 0.03) at the hinted size: two chunks.
Images and depths equal those of the library's workspace bit for bit."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
PER_RAY = 16 + 20 * (32 * 64 + 4)  # a ray's record and its budget of arena blocks


@pytest.mark.parametrize("fov,eps,nx,ny,rays,chunks", [(40.0, 0.05, 48, 40, 0, 1), (80.0, 0.018, 6, 4, 1.6, 24),
                                                       (20.0, 0.03, 32, 24, 0, 2)])
def test_records_beside_the_paths(synth, fov, eps, nx, ny, rays, chunks):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__

    __graft_entry__.build()
    from paper_2302_02733_gb300 import polrt

    ctx = polrt.rt_create(0, torch.cuda.current_stream().cuda_stream)
    try:
        polrt.rt_set_camera(ctx, synth.Camera(incl_deg=60.0, nx=nx, ny=ny, fov_M=fov))
        polrt.rt_set_integrator(ctx, eps, 20000)
        polrt.rt_load_model(ctx, polrt.adaf_model(synth.adaf_params(1)))
        res = []
        for own in (True, False):
            img = torch.zeros((ny, nx, 4), dtype=torch.float64, device="cuda")
            dep = torch.zeros((ny, nx, 2), dtype=torch.float64, device="cuda")
            if not own:
                size = polrt.rt_workspace_min_bytes() + int((rays - 1) * PER_RAY) if rays else polrt.rt_workspace_hint(ctx)
                ws = torch.empty(size, dtype=torch.uint8, device="cuda")
                polrt.rt_set_workspace(ctx, ws)
            polrt.rt_render_depths(ctx, polrt.RT_FP64, img, dep)
            res.append((img, dep, polrt.rt_last_counters(ctx)["chunks"]))
        assert res[0][2] == 1 and res[1][2] == chunks
        assert torch.isfinite(res[0][0]).all() and res[0][0][..., 0].max() > 0
        assert torch.equal(res[0][0], res[1][0]) and torch.equal(res[0][1], res[1][1])
    finally:
        polrt.rt_destroy(ctx)
