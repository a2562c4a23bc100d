"""The FP64 2D fused step on grids whose segments go down to one row, and where
the last segment is shorter than the others, against the FP64 oracle."""
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


@pytest.mark.parametrize("m,passes", [(0, 1), (1, None), (2, 0), (3, 2), (4, 3), (4, None)])
@pytest.mark.parametrize("shape", [(1, 1), (4, 11), (47, 49), (36, 91), (130, 152), (207, 10), (100, 307), (500, 33)])
def test_short_segments_match_oracle(fmx, shape, m, passes):
    E, B, J = synth.random_fields(shape, 501)
    kw = dict(m=m, filter_passes=passes or 0, courant=0.6, d=(1.0, 0.8))
    g = fmx.Grid(shape, with_current=passes is not None, precision=1, engine=fmx.FMX_ENGINE_FUSED, **kw)
    g.set_fields(E, B)
    if passes is not None:
        g.set_current(J)
    g.step(3)
    Eg, Bg, _ = g.get_fields()
    Eo, Bo, rc, _ = core.step(core.Params(shape=shape, **kw), E, B, J if passes is not None else None, 3)
    assert rc == core.OK
    assert_parity(Eg, Bg, Eo, Bo, 1e-12, f"f64 rows {shape} m={m} passes={passes}")
