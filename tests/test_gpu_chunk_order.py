"""A small image in chunks of a caller's workspace after a render of the same camera: the chunks are
dealt the recorded longest-first order, so none needs more than its budget of arena blocks (20 a ray)
where a chunk of neighbouring pixels across the photon ring does. An ADAF at 64 x 64 over 20 M with
eps = 0.0285 takes 18.8 blocks a ray in all and 21.1 in the worst sixteenth of its pixels (counted with
the oracle). Images are equal bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
PER_RAY = 16 + 20 * (32 * 64 + 4)  # a ray's record and its budget of arena blocks


@pytest.mark.parametrize("form", ["mixed", "unpol"])
def test_chunks_across_the_photon_ring(synth, form):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__

    __graft_entry__.build()
    from paper_2302_02733_gb300 import polrt

    ctx = polrt.rt_create(0, torch.cuda.current_stream().cuda_stream)
    try:
        cam = synth.Camera(incl_deg=60.0, nx=64, ny=64, fov_M=20.0)
        polrt.rt_set_camera(ctx, cam)
        polrt.rt_set_integrator(ctx, 0.0285, 20000)
        polrt.rt_load_model(ctx, polrt.adaf_model(synth.adaf_params(1)))
        f = polrt.RT_MIXED if form == "mixed" else polrt.RT_UNPOL
        out = [torch.zeros((64, 64, 4 if form == "mixed" else 1), dtype=torch.float32, device="cuda") for _ in range(2)]
        polrt.rt_render(ctx, f, out[0], None)
        ws = torch.empty(polrt.rt_workspace_min_bytes() + 255 * PER_RAY, dtype=torch.uint8, device="cuda")
        polrt.rt_set_workspace(ctx, ws)
        polrt.rt_render(ctx, f, out[1], None)
        assert polrt.rt_last_counters(ctx)["chunks"] == 16
        assert np.array_equal(out[0].cpu().numpy(), out[1].cpu().numpy())
    finally:
        polrt.rt_destroy(ctx)
