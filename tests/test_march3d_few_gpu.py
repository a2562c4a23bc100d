"""The one-column 3D kernels on grids of few planes or few cells (one row per
thread, segments down to one plane), on either side of the rule that picks them,
and with one to three rows left over for a thread's four: against the FP64
oracle."""
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


# 152 SMs: 4 x 19 tiles of 32 x 8 on one plane are the last on one row per thread
@pytest.mark.parametrize("f64,shape,m,passes", [
    (True, (1, 1, 1), 2, 1), (True, (12, 2, 2), 3, None), (True, (128, 127, 1), 4, 1), (True, (128, 152, 1), 2, 0),
    (True, (128, 153, 1), 2, 1), (True, (33, 9, 3), 3, 1), (True, (24, 24, 24), 2, None), (True, (24, 24, 26), 2, 1),
    (True, (40, 41, 30), 2, 1), (True, (40, 42, 30), 3, 0), (True, (40, 43, 30), 1, None), (True, (113, 101, 2), 1, 0),
    (False, (1, 2, 3), 3, 1), (False, (113, 101, 2), 4, 1), (False, (97, 75, 2), 2, None), (False, (33, 42, 40), 2, 1),
    (False, (64, 64, 2), 3, 1), (False, (64, 30, 3), 2, None)])
def test_few_planes_or_cells_match_oracle(fmx, f64, shape, m, passes):
    dt = np.float64 if f64 else np.float32
    E, B, J = (a.astype(dt) for a in synth.random_fields(shape, 511))
    kw = dict(m=m, filter_passes=passes or 0, courant=0.6, d=(1.0, 0.8, 1.2))
    g = fmx.Grid(shape, with_current=passes is not None, precision=1 if f64 else 0, engine=fmx.FMX_ENGINE_STAGED, **kw)
    g.set_fields(E, B)
    if passes is not None:
        g.set_current(J)
    g.step(2)
    Eg, Bg, _ = g.get_fields()
    Jo = J.astype(np.float64) if passes is not None else None
    Eo, Bo, rc, _ = core.step(core.Params(shape=shape, coef_f32=not f64, **kw), E.astype(np.float64),
                              B.astype(np.float64), Jo, 2)
    assert rc == core.OK
    assert_parity(np.asarray(Eg, np.float64), np.asarray(Bg, np.float64), Eo, Bo, 1e-12 if f64 else 1e-5,
                  f"3d few {shape} m={m} passes={passes}")
