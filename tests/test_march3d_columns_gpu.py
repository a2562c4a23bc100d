"""The one-column 3D z-march kernels (FP64, and FP32 with odd n_x) at the edges
of their tiles (32 columns, 16 rows, four rows per thread) and segments,
against the FP64 oracle at the library's parity tolerances: every sweep count,
with and without the one-pass current filter and a current."""
import numpy as np
import pytest

from oracle import core
from paper_1907_13088_gb300 import synth
from tests.helpers import assert_parity

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


@pytest.mark.parametrize("f64,shape,m,passes", [
    (True, (1, 1, 5), 2, 1), (True, (9, 8, 1), 3, 1), (True, (32, 16, 4), 4, 1), (True, (33, 17, 9), 1, 0),
    (True, (31, 15, 67), 4, None), (True, (66, 35, 130), 3, 1), (True, (40, 19, 8), 0, 1),
    (False, (1, 3, 6), 2, 1), (False, (31, 17, 5), 4, 1), (False, (33, 15, 70), 3, 0), (False, (65, 34, 12), 1, None),
    (False, (95, 48, 33), 4, 1)])
def test_one_column_kernels_match_oracle(fmx, f64, shape, m, passes):
    dt = np.float64 if f64 else np.float32
    E, B, J = (a.astype(dt) for a in synth.random_fields(shape, 411))
    kw = dict(m=m, filter_passes=passes or 0, courant=0.6, d=(1.0, 0.8, 1.2))
    g = fmx.Grid(shape, with_current=passes is not None, precision=1 if f64 else 0, **kw)
    g.set_fields(E, B)
    if passes is not None:
        g.set_current(J)
    g.step(3)
    Eg, Bg, _ = g.get_fields()
    Jo = J.astype(np.float64) if passes is not None else None
    Eo, Bo, rc, _ = core.step(core.Params(shape=shape, coef_f32=not f64, **kw), E.astype(np.float64),
                              B.astype(np.float64), Jo, 3)
    assert rc == core.OK
    assert_parity(np.asarray(Eg, np.float64), np.asarray(Bg, np.float64), Eo, Bo, 1e-12 if f64 else 1e-5,
                  f"3d columns {shape} m={m} passes={passes}")
