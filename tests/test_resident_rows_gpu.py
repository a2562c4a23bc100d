"""The resident engine on one cluster's shared memory (2D grids without a
filtered current): rows that divide unevenly over the cluster, CTAs without
rows, one row per CTA, narrow and wide rows, against the FP64 oracle, for fixed
sweeps and residual-controlled solves, with and without a raw current."""
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


@pytest.mark.parametrize("f64", [True, False])
@pytest.mark.parametrize("resid", [True, False])
@pytest.mark.parametrize("shape,current", [((64, 8), False), ((3, 16), True), ((1, 40), False), ((7, 15), True),
                                           ((257, 17), True), ((300, 33), False), ((20, 129), True), ((2, 3), True)])
def test_cluster_rows_match_oracle(fmx, shape, current, resid, f64):
    dt = np.float64 if f64 else np.float32
    E, B, J = (a.astype(dt) for a in synth.random_fields(shape, 441))
    kw = dict(iter_mode=1, tol=1e-12 if f64 else 1e-6, m_max=5000) if resid else dict(m=5)
    g = fmx.Grid(shape, with_current=current, precision=1 if f64 else 0, courant=0.7, engine=fmx.FMX_ENGINE_RESIDENT, **kw)
    g.set_fields(E, B)
    if current:
        g.set_current(J)
    g.step(4)
    g.step(1)
    Eg, Bg, _ = g.get_fields()
    okw = dict(residual=True, tol=kw["tol"], m_max=5000) if resid else dict(m=5)
    Eo, Bo, rc, st = core.step(core.Params(shape=shape, courant=0.7, coef_f32=not f64, **okw), E.astype(np.float64),
                               B.astype(np.float64), J.astype(np.float64) if current else None, 5)
    assert rc == core.OK
    assert_parity(np.asarray(Eg, np.float64), np.asarray(Bg, np.float64), Eo, Bo, 1e-12 if f64 else 1e-5,
                  f"cluster rows {shape}")
    if f64:
        assert g.diagnostics()["total_sweeps"] == (st["total_sweeps"] if resid else 25)
