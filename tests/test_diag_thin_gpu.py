"""Diagnostics of 3D grids of one plane, whose strips of 30 columns are more than
the 32-column blocks that the partial sums' buffer is sized by, and of grids whose
segments go down to one row or plane, against the FP64 oracle."""
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
    # both sides sum FP64 terms of one sign or of the fields' size
    return abs(a - b) <= 1e-12 * max(abs(b), 1e-300)


@pytest.mark.parametrize("f64", [True, False])
@pytest.mark.parametrize("shape", [(31, 1, 1), (31, 5, 1), (32, 16, 1), (61, 43, 1), (64, 64, 1), (31, 7, 2)])
def test_diagnostics_of_one_plane(fmx, shape, f64):
    dt = np.float64 if f64 else np.float32
    E, B, _ = (a.astype(dt) for a in synth.random_fields(shape, 461))
    kw = dict(courant=0.7, m=3, d=(1.0, 0.8, 1.2)[:len(shape)])
    g = fmx.Grid(shape, precision=1 if f64 else 0, with_current=False, **kw)
    g.set_fields(E, B)
    d = g.diagnostics()
    p = core.Params(shape=shape, coef_f32=not f64, **kw)
    E, B = E.astype(np.float64), B.astype(np.float64)
    ws, wp = core.energy(p, E, B)
    db, ge = core.div_b(p, B), core.gauss_e(p, E)
    assert _close(d["w_scheme"], ws) and _close(d["w_plain"], wp)
    assert _close(d["divb_max"], np.max(np.abs(db))) and _close(d["divb_l2"], np.linalg.norm(db))
    assert _close(d["gauss_max"], np.max(np.abs(ge))) and _close(d["gauss_l2"], np.linalg.norm(ge))


@pytest.mark.parametrize("f64", [True, False])
@pytest.mark.parametrize("shape", [(64, 64), (3000, 5), (33, 2), (29, 1), (1, 1), (100, 3, 2), (20, 30, 7)])
def test_diagnostics_of_few_rows(fmx, shape, f64):
    test_diagnostics_of_one_plane(fmx, shape, f64)
