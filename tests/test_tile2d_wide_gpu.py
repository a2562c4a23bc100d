"""Wide FP32 2D grids of few rows, where the step and its adjoint go back to the
row pipeline: which path the sizes on either side of the rule take (told by the
launches of a step), and that the fields do not depend on it."""
import numpy as np
import pytest

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


def _run(fmx, shape, m, passes, current, rows):
    E, B, J = synth.random_fields(shape, 1907041, dtype=np.float32)
    g = fmx.Grid(shape, m=m, filter_passes=passes, courant=0.6, with_current=current, engine=fmx.FMX_ENGINE_FUSED)
    g.set_option(fmx.FMX_OPT_SEGMENT_ROWS, rows)  # > 0: the row pipeline
    g.set_fields(E, B)
    if current:
        g.set_current(J)
    g.step(1)
    before = g.launches
    g.step(2)
    launches = (g.launches - before) // 2
    Eg, Bg, _ = g.get_fields()
    g.close()
    return np.array(Eg), np.array(Bg), launches


@pytest.mark.parametrize("wide,ny,m,passes,current", [(0, 1, 4, 3, True), (0, 6, 4, 0, False), (1, 5, 1, 0, True),
                                                      (-1, 6, 4, 3, True), (-2, 4, 0, 1, True)])
def test_wide_grids_of_few_rows(fmx, wide, ny, m, passes, current):
    import torch
    nx = 48 * 4 * torch.cuda.get_device_properties(0).multi_processor_count + wide
    got = _run(fmx, (nx, ny), m, passes, current, 0)
    rows = _run(fmx, (nx, ny), m, passes, current, 26)
    # up to 196608 cells the tiles take one launch, the row pipeline two
    assert nx * ny <= 196608 and got[2] == (2 if wide >= 0 else 1) and rows[2] == 2
    assert np.array_equal(got[0], rows[0]) and np.array_equal(got[1], rows[1])
