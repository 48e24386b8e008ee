"""The unpolarized transfer (a warp per ray, a lane per saved state) on rays of 1, 31, 32, 33, 64 and 65
states (blocks of 32: a block filled, a last block that holds the last state alone) and whole rays,
on an ADAF that the camera
is inside of (every point emits), and on one that ends nearer to the hole than the camera (points
that do not emit at both ends), against the oracle. A state dropped, doubled or out of order changes a
pixel by a part in the number of its states; the FP32 evaluation of a state is off by its rounding
times the exponent of the emissivity's tail, x^(1/3) of up to 1e2: 1e-4 of a pixel."""
import numpy as np
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
def test_unpolarized_rays_of_few_states(rt, ora, synth, nmax):
    polrt, ctx = rt
    cam = synth.Camera(incl_deg=60.0, nx=12, ny=9, r_cam=30.0)
    for r_out in (1000.0, 20.0):
        par = synth.adaf_params(1)
        par.r_out = r_out
        model, om = polrt.adaf_model(par), ora.adaf_model(par)
        polrt.rt_set_camera(ctx, cam)
        polrt.rt_set_integrator(ctx, 0.05, nmax)
        polrt.rt_load_model(ctx, model)
        out = torch.full((9, 12), float("nan"), dtype=torch.float32, device="cuda")
        st = torch.zeros((9, 12), dtype=torch.uint8, device="cuda")
        polrt.rt_render(ctx, polrt.RT_UNPOL, out, st)
        c = polrt.rt_last_counters(ctx)
        polrt.rt_set_integrator(ctx, 0.05, 20000)
        ocam = ora.camera(cam, nmax=nmax)
        ref = ora.render_unpol(ocam, om)
        _, nsteps, status, _ = ora.render_image(ocam, om)
        assert np.array_equal(st.cpu().numpy().astype(int), status.astype(int))
        assert c["points"] == int(nsteps.sum())
        scale = np.maximum(ref, max(1e-6 * ref.max(), 1e-300))
        err = np.abs(out.double().cpu().numpy() - ref) / scale
        print(f"nmax {nmax} max {err.max():.2e}")
        assert err.max() <= 1e-4 and (r_out < 30.0) == (c["emitting_points"] < c["points"])
