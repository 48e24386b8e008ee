"""The persistent batch's mixed form, whose roles go to pairs of SMs: from one pair in eight that integrates
to seven, in odd shares, with one and two blocks per SM and few or many steps between checks, and with
fewer rays than one block's lanes. Every image equals rt_render's within 1e-6 per pixel (the same states
and the same transfer), with the same number of steps."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("shape", [(1, 1, 2, 0), (1, 16, 1, 1), (7, 1, 2, 7), (7, 4, 1, 1), (1, 4, 2, 7), (4, 4, 2, 4), (3, 2, 2, 4)])
def test_shares_of_sm_pairs(synth, shape):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__

    __graft_entry__.build()
    from paper_2302_02733_gb300 import polrt

    geo, tile, blocks, odd = shape
    ctx = polrt.rt_create(0, torch.cuda.current_stream().cuda_stream)
    try:
        polrt.rt_load_model(ctx, polrt.adaf_model(synth.adaf_params(1)))
        polrt.rt_set_batch_config(ctx, polrt.RT_MIXED, geo, tile, blocks, polrt.RT_BATCH_PERSISTENT, odd)
        for sizes in ([8], [40, 96, 24, 64]):
            cams = [synth.Camera(incl_deg=20.0 + 35.0 * k, nx=n, ny=n) for k, n in enumerate(sizes)]
            outs = [torch.full((n, n, 4), float("nan"), dtype=torch.float32, device="cuda") for n in sizes]
            jobs = polrt.make_jobs((c, 0.0, 0.0, o, None, None) for c, o in zip(cams, outs))
            for _ in range(2):
                polrt.rt_render_batch(ctx, polrt.RT_MIXED, jobs)
            cnt, steps = polrt.rt_last_counters(ctx), 0
            assert cnt["n_overflow"] == 0 and cnt["points"] == cnt["steps"]
            for cam, o in zip(cams, outs):
                one = torch.zeros_like(o)
                polrt.rt_set_camera(ctx, cam)
                polrt.rt_render(ctx, polrt.RT_MIXED, one)
                steps += polrt.rt_last_counters(ctx)["steps"]
                scale = torch.clamp(one[..., 0], min=1e-8 * float(one[..., 0].max()))
                assert float(((o - one).abs().amax(dim=-1) / scale).max()) <= 1e-6
            assert cnt["steps"] == steps
    finally:
        polrt.rt_destroy(ctx)
