"""How many clusters a resident launch takes, by path: 3D FP64 solves spread over
several above 4096 cells, the shared-memory engine keeps to one, and FP32 with
fixed m stays on one up to 65536 cells, so that it only enqueues and can be
captured in a CUDA graph.  The result does not depend on the clusters."""
import numpy as np
import pytest

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


RES = dict(iter_mode=1, tol=1e-10, m_max=5000)


@pytest.mark.parametrize("f64,shape,passes,kw,several", [
    (True, (16, 16, 16), None, RES, False), (True, (17, 17, 17), None, RES, True), (True, (20, 20, 20), 1, RES, True),
    (True, (90, 90), None, RES, False), (True, (90, 91), 2, RES, False), (True, (8000,), None, RES, False),
    (False, (200, 200), None, dict(RES, tol=1e-5), False), (False, (300, 200), None, dict(RES, tol=1e-5), True),
    (False, (160, 160), 2, dict(RES, tol=1e-5), True), (False, (32, 32, 32), None, dict(RES, tol=1e-5), True),
    (False, (256, 256), 2, dict(m=3), False), (False, (40, 40, 40), 0, dict(m=4), False), (False, (65536,), 0, dict(m=4), False)])
def test_clusters_by_path(fmx, f64, shape, passes, kw, several):
    dt = np.float64 if f64 else np.float32
    E, B, J = (a.astype(dt) for a in synth.random_fields(shape, 491))
    out = []
    for engine in (fmx.FMX_ENGINE_RESIDENT, fmx.FMX_ENGINE_STAGED):
        g = fmx.Grid(shape, with_current=passes is not None, precision=1 if f64 else 0, courant=0.5, engine=engine,
                     filter_passes=passes or 0, **kw)
        g.set_fields(E, B)
        if passes is not None:
            g.set_current(J)
        g.step(2)
        if engine == fmx.FMX_ENGINE_RESIDENT:
            n = g.get_option(fmx.FMX_OPT_RESIDENT_CLUSTERS)
            assert (n > 1) == several, n
        Eg, Bg, _ = g.get_fields()
        out.append((np.asarray(Eg, np.float64), np.asarray(Bg, np.float64)))
    assert_parity(*out[0], *out[1], 1e-12 if f64 else 1e-5, f"clusters {shape}")


@pytest.mark.parametrize("shape,passes", [((160, 160), 2), ((32, 32, 40), 0)])
def test_fixed_sweeps_fp32_can_be_captured(fmx, shape, passes):
    import torch
    E, B, J = (a.astype(np.float32) for a in synth.random_fields(shape, 492))
    s = torch.cuda.Stream()
    g = fmx.Grid(shape, stream=s, courant=0.5, m=4, filter_passes=passes, engine=fmx.FMX_ENGINE_RESIDENT)
    torch.cuda.synchronize()
    g.set_fields(E, B)
    g.set_current(J)
    g.step(2)
    g.step(2)
    want = g.get_fields()
    g.set_fields(E, B)
    assert g.get_option(fmx.FMX_OPT_RESIDENT_CLUSTERS) == 1
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        g.step(2)
    with torch.cuda.stream(s):
        graph.replay()
        graph.replay()
    got = g.get_fields()
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])
