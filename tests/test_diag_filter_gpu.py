"""Diagnostics and the standalone filter at the edges of their kernels' tiles
(30-column warps, 8-row and 8-plane segments; 4- and 8-element filter runs) and
on grids narrower than a stencil, against the FP64 oracle."""
import numpy as np
import pytest

from oracle import core
from paper_1907_13088_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fmx():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1907_13088_gb300 import build
    build.build()
    from paper_1907_13088_gb300 import fmx as m
    return m


def _close(a, b):
    # both sides sum FP64 terms of one sign or of the fields' size: 1e-12, as the parity tests
    return abs(a - b) <= 1e-12 * max(abs(b), 1e-300)


@pytest.mark.parametrize("f64", [True, False])
@pytest.mark.parametrize("shape", [(1, 2), (30, 8), (31, 9), (61, 65), (2, 130), (257, 70), (1, 2, 3), (30, 5, 8),
                                   (31, 1, 9), (33, 4, 66), (64, 40, 20), (50,)])
def test_diagnostics_edges(fmx, shape, f64):
    dt = np.float64 if f64 else np.float32
    E, B, _ = (a.astype(dt) for a in synth.random_fields(shape, 421))
    kw = dict(courant=0.7, m=3, d=(1.0, 0.8, 1.2)[:len(shape)])
    g = fmx.Grid(shape, precision=1 if f64 else 0, with_current=False, **kw)
    g.set_fields(E, B)
    d = g.diagnostics()
    p = core.Params(shape=shape, coef_f32=not f64, courant=0.7, m=3, d=(1.0, 0.8, 1.2))
    E, B = E.astype(np.float64), B.astype(np.float64)
    ws, wp = core.energy(p, E, B)
    db, ge = core.div_b(p, B), core.gauss_e(p, E)
    assert _close(d["w_scheme"], ws) and _close(d["w_plain"], wp)
    assert _close(d["divb_max"], np.max(np.abs(db))) and _close(d["divb_l2"], np.linalg.norm(db))
    assert _close(d["gauss_max"], np.max(np.abs(ge))) and _close(d["gauss_l2"], np.linalg.norm(ge))


@pytest.mark.parametrize("f64,engine", [(True, 1), (True, 2), (False, 2), (False, 0)])
@pytest.mark.parametrize("shape", [(5,), (70,), (2, 3), (33, 35), (130, 65), (7, 33, 9), (2, 1, 5)])
def test_filter_edges(fmx, shape, f64, engine):
    if engine == 2 and len(shape) != 2:
        pytest.skip("the fused engine is 2D")
    dt = np.float64 if f64 else np.float32
    E, B, J = (a.astype(dt) for a in synth.random_fields(shape, 431))
    p = core.Params(shape=shape)
    for passes in (1, 2, 3, 4):
        g = fmx.Grid(shape, precision=1 if f64 else 0, engine=engine)
        g.set_fields(E, B)
        g.set_current(J)
        g.filter(fmx.FMX_E | fmx.FMX_BX | fmx.FMX_BZ | fmx.FMX_J, passes)
        Eg, Bg, Jg = g.get_fields(fmx.FMX_E | fmx.FMX_B | fmx.FMX_J)
        assert np.array_equal(Bg[1], B[1]), "a component outside the mask is left alone"
        for got, src in [(Eg[c], E[c]) for c in range(3)] + [(Bg[0], B[0]), (Bg[2], B[2])] + [(Jg[c], J[c]) for c in range(3)]:
            ref = core.filter(p, src.astype(np.float64), passes)
            err = np.linalg.norm(got.astype(np.float64) - ref) / np.linalg.norm(src)
            assert err <= (1e-14 if f64 else 1e-6), (passes, err)
