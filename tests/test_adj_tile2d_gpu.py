"""The FP32 2D adjoint step on register tiles (adj_tile2d.cu): the bits of the
row pipeline (even n_x), and the oracle's adjoint everywhere, odd n_x (staged
kernels) among them, at tile edges and on grids smaller than a tile."""
import ctypes

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


def _adjoint(fmx, shape, m, passes, rows, Ebar, Bbar, jmask):
    import torch
    nx, ny = shape
    g = fmx.Grid(shape, m=m, filter_passes=passes, courant=0.6, engine=fmx.FMX_ENGINE_FUSED)
    g.set_option(fmx.FMX_OPT_SEGMENT_ROWS, rows)
    pitch = (nx + 3) // 4 * 4
    buf = torch.zeros((9, ny, pitch), device="cuda")
    buf[:3, :, :nx] = torch.from_numpy(Ebar[:, 0]).cuda()
    buf[3:6, :, :nx] = torch.from_numpy(Bbar[:, 0]).cuda()
    wb = fmx.fmx_adjoint_workspace_bytes(ctypes.byref(g.params))
    work = torch.zeros(wb + 256, dtype=torch.uint8, device="cuda")
    vp = lambda s, mask=7: (ctypes.c_void_p * 3)(*[buf[s + c].data_ptr() if mask >> c & 1 else None for c in range(3)])
    torch.cuda.synchronize()
    fmx.check(fmx.fmx_adjoint_step(g.handle, vp(0), vp(3), vp(6, jmask), (work.data_ptr() + 255) // 256 * 256, wb))
    torch.cuda.synchronize()
    out = buf[:, :, :nx].cpu().numpy()
    g.close()
    return out


@pytest.mark.parametrize("m,passes,jmask", [(0, 0, 7), (1, 1, 7), (2, 3, 4), (3, 2, 7), (4, 3, 7), (4, 3, 0), (4, 0, 3)])
@pytest.mark.parametrize("shape", [(1, 1), (2, 3), (5, 7), (46, 48), (47, 49), (64, 50), (97, 101), (130, 64), (300, 230)])
def test_adjoint_tiles(fmx, shape, m, passes, jmask):
    rng = np.random.default_rng(451)
    Ebar, Bbar = (rng.standard_normal((3, 1) + shape[::-1]).astype(np.float32) for _ in range(2))
    out = _adjoint(fmx, shape, m, passes, 0, Ebar, Bbar, jmask)
    if shape[0] % 2 == 0:
        ref = _adjoint(fmx, shape, m, passes, 26, Ebar, Bbar, jmask)
        assert np.array_equal(out, ref)
    p = core.Params(shape=shape, courant=0.6, m=m, filter_passes=passes, coef_f32=True)
    Eo, Bo, Jo = core.adjoint_step(p, Ebar.astype(np.float64), Bbar.astype(np.float64))
    for c in range(3):
        for got, want in ((out[c], Eo[c]), (out[3 + c], Bo[c])) + (((out[6 + c], Jo[c]),) if jmask >> c & 1 else ()):
            want = np.asarray(want).reshape(got.shape)
            assert np.linalg.norm(got - want) <= 1e-5 * max(np.linalg.norm(want), 1e-30), (c, m, passes)
