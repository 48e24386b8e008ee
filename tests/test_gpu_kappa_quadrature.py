"""rt_kappa_coeffs at the edges of its quadrature against the oracle's (whose nodes and kernels are its
own): kappa on both sides of every change of step, close to 3 and steep; cold to hot electrons; from
below to far above nu_c; field angles near 0, at and beyond pi/2; Maxwell-Juttner rows. Tolerances
from the rules' convergence: 2e-9 relative for emission and absorption (4e-10 from the nodes, and the
light-cone scaling of Q and V by a ratio of two of them), 1e-10 for the rotativities. Then rows that
give zeros."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

E, ME, C = 4.80320471257e-10, 9.1093837015e-28, 2.99792458e10


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


@pytest.mark.parametrize("kappa", [3.001, 3.2, 4.5, 9.99, 10.0, 19.9, 20.0, 39.9, 40.0, 98.0, 0.0])
def test_quadrature_edges(rt, ora, kappa):
    polrt, ctx = rt
    nu, rows = 230e9, []
    for Te in (0.1, 1.0, 20.0):
        for X in (10.0, 600.0, 740.0, 3e4):
            for th in (0.02, 0.5 * math.pi, 2.9):
                B = nu / (1.5 * X * math.sin(th)) * 2 * math.pi * ME * C / E
                rows.append((1e5, Te, B, nu, th, kappa))
    rows = np.array(rows)
    out = np.zeros((len(rows), 8))
    polrt.rt_kappa_coeffs(ctx, rows, out)
    for p, got in zip(rows, out):
        ref = ora.kappa_coeffs(*p)
        scale = np.abs(ref)
        scale[[2, 5]] = np.maximum(scale[[2, 5]], 1e-12 * scale[[0, 3]])  # V where cot theta rounds to 0
        scale[7] = max(scale[7], 1e-12 * scale[6])
        rel = np.abs(got - ref) / np.maximum(scale, 1e-300)
        assert rel[:6].max() <= 2e-9 and rel[6:].max() <= 1e-10, (p, rel)


def test_rows_outside_give_zeros(rt):
    polrt, ctx = rt
    rows = np.array([(0.0, 1.0, 10.0, 230e9, 1.0, 4.0), (1e5, 0.0, 10.0, 230e9, 1.0, 4.0), (1e5, 1.0, 0.0, 230e9, 1.0, 4.0),
                     (1e5, 1.0, 10.0, 0.0, 1.0, 4.0), (1e5, 1.0, 10.0, 230e9, 1.0, 3.0), (1e5, 1.0, 10.0, 230e9, 1.0, 2.0),
                     (np.nan, 1.0, 10.0, 230e9, 1.0, 4.0)])
    out = np.ones((len(rows), 8))
    polrt.rt_kappa_coeffs(ctx, rows, out)
    assert (out == 0.0).all()
    # along the field: no emission, rotativities stay
    one = np.array([(1e5, 1.0, 10.0, 230e9, 0.0, 4.0)])
    o = np.ones((1, 8))
    polrt.rt_kappa_coeffs(ctx, one, o)
    assert (o[0, :7] == 0.0).all() and o[0, 7] != 0.0
