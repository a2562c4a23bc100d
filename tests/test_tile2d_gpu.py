"""The FP32 2D step on register tiles (tile2d.cu) against the row pipeline:
every cell's arithmetic is the same, operation by operation, so the fields
agree to the bit wherever a tile, a warp's rows or the periodic seam end; and
the tiles match the FP64 oracle."""
import numpy as np
import pytest

from oracle import core
from paper_1907_13088_gb300 import synth
from tests.helpers import assert_parity

pytestmark = pytest.mark.gpu

# grids smaller than a tile, one tile and one cell more, odd row lengths, the
# one-launch sizes and the first sizes beyond them
SHAPES = [(1, 1), (2, 3), (5, 7), (63, 50), (64, 49), (65, 48), (47, 200), (130, 99), (501, 388), (520, 401)]


@pytest.fixture(scope="module")
def fmx():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1907_13088_gb300 import build
    build.build()
    from paper_1907_13088_gb300 import fmx as m
    return m


def _run(fmx, shape, m, passes, current, rows, nsteps=3):
    E, B, J = synth.random_fields(shape, 1907040, dtype=np.float32)
    g = fmx.Grid(shape, m=m, filter_passes=passes, courant=0.6, with_current=current, engine=fmx.FMX_ENGINE_FUSED)
    g.set_option(fmx.FMX_OPT_SEGMENT_ROWS, rows)  # > 0: the row pipeline
    g.set_fields(E, B)
    if current:
        g.set_current(J)
    g.step(nsteps)
    Eg, Bg, _ = g.get_fields()
    g.close()
    return np.array(Eg), np.array(Bg)


@pytest.mark.parametrize("m,passes,current", [(0, 0, False), (1, 0, True), (2, 1, True), (3, 2, True), (4, 3, True),
                                              (4, 0, False), (3, 3, True)])
@pytest.mark.parametrize("shape", SHAPES)
def test_tiles_give_the_row_pipelines_bits(fmx, shape, m, passes, current):
    tiles = _run(fmx, shape, m, passes, current, 0)
    rows = _run(fmx, shape, m, passes, current, 40)
    assert np.array_equal(tiles[0], rows[0]) and np.array_equal(tiles[1], rows[1])


@pytest.mark.parametrize("shape", [(97, 51), (600, 343)])
def test_tiles_match_the_oracle(fmx, shape):
    Eg, Bg = _run(fmx, shape, 4, 3, True, 0, nsteps=5)
    E, B, J = synth.random_fields(shape, 1907040, dtype=np.float32)
    p = core.Params(shape=shape, courant=0.6, m=4, filter_passes=3, coef_f32=True)
    Eo, Bo, _, _ = core.step(p, E.astype(np.float64), B.astype(np.float64), J.astype(np.float64), 5)
    assert_parity(Eg.astype(np.float64), Bg.astype(np.float64), Eo, Bo, 1e-5, f"register tiles {shape}")
