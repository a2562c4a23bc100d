"""The standalone filter leaves the caller's other arrays alone: after a step of
the fused engine the set that is not current still holds the state before it, and
filtering E, B or j in place does not touch it."""
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


@pytest.mark.parametrize("passes", [1, 2, 3, 4])
@pytest.mark.parametrize("f64", [False, True])
def test_filter_keeps_the_other_state_set(fmx, f64, passes):
    import torch
    shape = (70, 131)
    dt = np.float64 if f64 else np.float32
    E, B, J = (a.astype(dt) for a in synth.random_fields(shape, 481))
    for mask in (fmx.FMX_J, fmx.FMX_E | fmx.FMX_B):
        g = fmx.Grid(shape, precision=1 if f64 else 0, engine=fmx.FMX_ENGINE_FUSED)
        g.set_fields(E, B)
        g.set_current(J)
        g.step(1)
        g.sync()
        own = {fmx.fmx_field_ptr(g.handle, c) for c in range(9) if mask >> c & 1}
        n = (g._slab.numel() // 15)
        before = g._slab.clone()
        g.filter(mask, passes)
        g.sync()
        for c in range(15):
            ptr = g._slab.data_ptr() + c * n * g._slab.element_size()
            part = slice(c * n, (c + 1) * n)
            assert (ptr in own) != torch.equal(g._slab[part], before[part]), (mask, c)


@pytest.mark.parametrize("f64,engine", [(True, 1), (True, 2), (False, 2)])
@pytest.mark.parametrize("shape", [(1, 1), (1, 70), (5, 5), (200, 3), (3, 200), (63, 65), (64, 64), (65, 128), (129, 190),
                                   (1000,), (7, 2, 40), (5, 130, 35), (3, 4, 131), (260, 9, 17)])
def test_filter_tiles_and_runs_match_oracle(fmx, shape, f64, engine):
    """Edges of the in-place tiles (64 x 64 cells, rows in groups of 16; grids
    whose halos fill the spare array before all six components are in), and of the
    16-element runs and 128-element blocks of the 1D and 3D kernels."""
    from oracle import core
    if engine == 2 and len(shape) != 2:
        pytest.skip("the fused engine is 2D")
    dt = np.float64 if f64 else np.float32
    E, B, J = (a.astype(dt) for a in synth.random_fields(shape, 482))
    p = core.Params(shape=shape)
    for passes in (1, 2, 3):
        g = fmx.Grid(shape, precision=1 if f64 else 0, engine=engine)
        g.set_fields(E, B)
        g.set_current(J)
        g.filter(fmx.FMX_E | fmx.FMX_B | fmx.FMX_JY, passes)
        Eg, Bg, Jg = g.get_fields(fmx.FMX_E | fmx.FMX_B | fmx.FMX_J)
        for got, src in [(Eg[c], E[c]) for c in range(3)] + [(Bg[c], B[c]) for c in range(3)] + [(Jg[1], J[1])]:
            ref = core.filter(p, src.astype(np.float64), passes)
            # up to 2 x 7 positive weights that sum to one: a few roundings of the input's size
            err = np.linalg.norm(got.astype(np.float64) - ref) / np.linalg.norm(src)
            assert err <= (1e-14 if f64 else 1e-6), (passes, err)
        assert np.array_equal(Jg[0], J[0]) and np.array_equal(Jg[2], J[2])
