"""The surrogate's features pass (a warp per ray, a lane per saved state) on rays of 1, 31, 32, 33, 64
and 65 states (blocks of 32: a block filled, a last block that holds the last state alone) and whole
rays, on an ADAF that ends nearer to the hole than the camera (points that do not emit at both ends):
- the raw features are those of the emitting states, each once: sorted, their ln Theta_e is that of the
  oracle's saved states, ln(T0 k / (m c^2 r)) at r <= r_out, within FP32's rounding of a logarithm of
  about ten and of its argument (4e-6), and their number is the number of emitting points;
- the image is the same bit for bit whether the features lie by saved state or in compact rows (the
  streamed shape).
"""
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
def test_features_of_every_state(rt, ora, synth, nmax):
    polrt, ctx = rt
    cam = synth.Camera(incl_deg=60.0, nx=24, ny=12, r_cam=30.0)
    par = synth.adaf_params(1)
    par.r_out = 20.0
    polrt.rt_set_camera(ctx, cam)
    polrt.rt_set_integrator(ctx, 0.05, nmax)
    polrt.rt_load_model(ctx, polrt.adaf_model(par, kappa=4.5))
    theta = (0.05 * np.random.default_rng(5).standard_normal(polrt.RT_MLP_PARAMS)).astype(np.float32)
    polrt.rt_mlp_set_params(ctx, theta, polrt.mlp_norm([-5.0, 1e-3, -6.0, 3.2], [40.0, 1.5707963, 4.0, 8.0],
                                                       [-30.0] * 8, [0.01] * 8))
    feat = torch.full((1 << 18, 4), float("nan"), dtype=torch.float32, device="cuda")
    imgs = []
    try:
        n = polrt.rt_render_features(ctx, feat)
        for cfg in ((0, 0, 1), (1, 0, 4)):
            polrt.rt_set_render_config(ctx, *cfg)
            img = torch.full((12, 24, 4), float("nan"), dtype=torch.float32, device="cuda")
            polrt.rt_render(ctx, polrt.RT_SURROGATE, img)
            imgs.append((img, polrt.rt_last_counters(ctx)))
    finally:
        polrt.rt_set_render_config(ctx, 0, 0, 0)
        polrt.rt_set_integrator(ctx, 0.05, 20000)
    ocam = ora.camera(cam, nmax=nmax)
    r = []
    for iy in range(12):
        for ix in range(24):
            px, py = ((ix + 0.5) / 24 - 0.5) * ocam.fov_M, ((iy + 0.5) / 12 - 0.5) * ocam.fov_M * 12 / 24
            st, _ = ora.trace_geodesic(ocam, px, py)
            r.append(st[:-1, 1])
    r = np.concatenate(r)
    te = par.T0 * 1.380649e-16 / (9.1093837015e-28 * 2.99792458e10**2) / r[r <= par.r_out]
    assert n == te.size == imgs[0][1]["emitting_points"] and r.size == imgs[0][1]["points"]
    if n:
        got = np.sort(feat[:n, 2].double().cpu().numpy())
        assert np.abs(got - np.sort(np.log(te))).max() <= 4e-6
        assert torch.isfinite(feat[:n]).all() and torch.isnan(feat[n]).all()
    assert torch.isfinite(imgs[0][0]).all() and torch.equal(imgs[0][0], imgs[1][0])
