"""The FP64 transfer's tables and fixed-length series at the ends of their ranges, against the oracle
(which evaluates the Bessel functions, Shcherbakov's factors and the matrix exponential by other
means), per pixel and outside the oracle's own sensitivity mask:
ADAFs whose Theta_e runs below, across and above the table of K_0/K_2 and K_1/K_2 (2^-40 .. 2^20),
and whose X runs below, across and above that of f(X) and g(X) (2^-30 .. 2^14), with optical depths
from none to 2e4 (series of one term up to the closed form): depths to 1e-10 of the larger of the
pixel's value and a thousandth of the image's largest. A fit with 8 powers on a sixteenth of an octave
is within (1/66)^9 = 4e-17 times a few of its value and all values are rounded to 53 bits; the
oracle's images move by 5e-15 when its own rounding is perturbed, and a ray has at most some 1e3
points."""
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


def render(polrt, ctx, cam, model):
    polrt.rt_set_camera(ctx, cam)
    polrt.rt_set_integrator(ctx, 0.05, 20000)
    polrt.rt_load_model(ctx, model)
    img = torch.zeros((cam.ny, cam.nx, 4), dtype=torch.float64, device="cuda")
    dep = torch.zeros((cam.ny, cam.nx, 2), dtype=torch.float64, device="cuda")
    polrt.rt_render_depths(ctx, polrt.RT_FP64, img, dep)
    return img.cpu().numpy(), dep.cpu().numpy()


def calm(ora, ocam, om, ref, nsteps):
    """Pixels whose image and step count do not depend on the oracle's own rounding."""
    ok = np.ones(nsteps.shape, dtype=bool)
    for pert in (1, 2):
        im, ns, _, _ = ora.render_image(ocam, om, pert=pert)
        scale = np.maximum(ref[..., 0], 1e-8 * max(ref[..., 0].max(), 1e-300))
        ok &= (np.abs(im - ref).max(axis=-1) / scale <= 1e-10) & (ns == nsteps)
    assert ok.mean() > 0.95
    return ok


@pytest.mark.parametrize("T0,n0,beta", [(0.1, 1e7, 1e-10), (2e-2, 3e7, 10.0), (1e6, 1e7, 1e6), (1e5, 1e3, 1e4),
                                        (3e11, 3e7, 10.0), (1e13, 1e3, 10.0), (1e12, 3e7, 1e-8),
                                        (1e17, 1e-6, 10.0), (1e17, 1e3, 10.0)])
def test_thermal_tables(rt, ora, synth, T0, n0, beta):
    polrt, ctx = rt
    cam = synth.Camera(incl_deg=60.0, nx=12, ny=8)
    par = synth.AdafParams(T0=T0, n0=n0, beta=beta)
    img, dep = render(polrt, ctx, cam, polrt.adaf_model(par))
    ocam, om = ora.camera(cam), ora.adaf_model(par)
    ref, nsteps, _, _, dref = ora.render_image(ocam, om, depth=True)
    ok = calm(ora, ocam, om, ref, nsteps)
    scale = np.maximum(np.abs(dref), 1e-3 * np.abs(dref).max(axis=(0, 1), keepdims=True))
    err = np.where(scale > 0, np.abs(dep - dref) / np.where(scale > 0, scale, 1.0), np.abs(dep))
    print(f"depths {err[ok].max(axis=0)}")
    assert np.abs(dref[..., 1]).max() > 0 and err[ok].max() <= 1e-10
    serr = np.abs(img - ref).max(axis=-1) / np.maximum(ref[..., 0], 1e-8 * max(ref[..., 0].max(), 1e-300))
    assert serr[ok].max() <= 1e-9
