"""Receivers recorded together: the values of every receiver, in a fluid cell, in a
solid cell or on the interface, are the bits of that receiver recorded alone,
whatever the number of receivers (partial blocks, both block sizes) and shots."""
import numpy as np
import pytest

import synth
from tests.libutil import ensure_built

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ensure_built()
    from paper_2505_15771_gb300 import hho, solver
    return hho, solver


def points(n, seed):
    rng = np.random.default_rng(seed)
    xy = rng.uniform(0.01, 0.99, (n, 2))
    xy[::3, 1] = 0.5   # on the interface
    return xy


@pytest.mark.parametrize("k", [1, 2, 3])
def test_receivers_together_and_alone(lib, k):
    hho, solver = lib
    md = synth.quad_grid(24, 24)
    P = solver.Problem(md, synth.layered_media(md), k)
    x = P.to_device(synth.random_state(P.layout.n_canonical, 3))
    xy = points(3000, k)
    P.set_receivers(xy)
    every = P.record(x).cpu().numpy()
    assert np.isfinite(every).all() and (np.abs(every[:, :3]).max(axis=1) > 0).all()
    for n in (1, 3, 4, 5, 33, 609, 2431, 2433):
        P.set_receivers(xy[:n])
        assert np.array_equal(P.record(x).cpu().numpy(), every[:n]), n
    for i in range(6):
        P.set_receivers(xy[i:i + 1])
        assert np.array_equal(P.record(x).cpu().numpy(), every[i:i + 1])


@pytest.mark.parametrize("precision", ["f64", "f32", "f32x2"])
def test_shots_and_graphs_record_alike(lib, precision):
    """Seismograms of 1 and of 7 shots, stepped from the stream and from replayed graphs
    (no sources, so both modes step with the same bits)."""
    hho, solver = lib
    prec = {"f64": hho.HHO_F64, "f32": hho.HHO_F32, "f32x2": hho.HHO_F32X2}[precision]
    md = synth.quad_grid(24, 24)
    P = solver.Problem(md, synth.layered_media(md), 2)
    U = synth.random_state(P.layout.n_canonical, 4)
    n, steps = 405, 9
    P.set_receivers(points(n, 1))
    out = []
    for mode in (hho.HHO_LAUNCH_STREAM, hho.HHO_LAUNCH_GRAPH):
        P.set_launch_mode(mode)
        for S in (1, 7):
            x = P.batch_to_device(np.tile(U, (S, 1)), prec)
            _, work = P.batch_buffers(3, S, prec)
            seis = torch.zeros((steps, S, n, 5), device="cuda", dtype=torch.float32 if precision == "f32" else torch.float64)
            P.batch_step(x, work, S, 3, 0.0, 1e-4, steps, precision=prec, seismogram=seis)
            s = seis.cpu().numpy()
            assert np.isfinite(s).all() and (np.abs(s).max(axis=(1, 2, 3)) > 0).all()
            out += [s[:, i] for i in (0, S - 1)]
    for s in out[1:]:
        assert np.array_equal(s, out[0])
