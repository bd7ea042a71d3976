"""hho_erk_run_host on meshes large enough to be taken in pieces (4096 warps of
cells and more): the same bits as packing on the device, stepping and unpacking."""
import numpy as np
import pytest

import synth
from tests.libutil import ensure_built

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MESHES = {
    # 2 pieces, the cell order of both domains follows the device order
    "quad": lambda: synth.quad_grid(487, 280, 0.0, 1.739, 0.0, 1.0, y_interface=0.6),
    # fluid only, 3 pieces
    "fluid": lambda: synth.quad_grid(470, 419, 0.0, 1.12, 0.0, 1.0, y_interface=-1.0),
    # squares and triangles in one cell order, two classes: every piece waits for the last cells
    "hybrid": lambda: synth.hybrid_grid(340, 340, 0.0, 1.0, 0.0, 1.0, 0.7, 0.5),
}


@pytest.fixture(scope="module")
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ensure_built()
    from paper_2505_15771_gb300 import hho, solver
    return hho, solver


@pytest.mark.parametrize("mesh,k,s,nsteps,arith", [
    ("quad", 1, 4, 1, "f64"), ("quad", 2, 2, 2, "f32x2"), ("quad", 1, 3, 3, "f64"),
    ("fluid", 1, 4, 2, "f64"), ("hybrid", 1, 4, 1, "f64"), ("hybrid", 2, 3, 2, "f32x2"),
])
def test_pieces_give_the_bits_of_the_device_path(lib, mesh, k, s, nsteps, arith):
    hho, solver = lib
    md = MESHES[mesh]()
    P = solver.Problem(md, synth.layered_media(md), k)
    assert P.layout.n_fluid_pad + P.layout.n_solid_pad >= 32 * 4096
    P.set_arithmetic(hho.HHO_F64 if arith == "f64" else hho.HHO_F32X2)
    P.set_sources([(0.37, 0.21)], [(0.6, 0.8)], 10.0)
    U = np.random.default_rng(5).standard_normal(P.layout.n_canonical)
    x = P.to_device(U)
    P.step(x, s, 0.01, 1e-4, nsteps)
    ref = P.to_canonical(x)
    assert np.isfinite(ref).all() and not np.array_equal(ref, U)
    h = torch.from_numpy(U.copy()).pin_memory()
    side = torch.cuda.Stream()
    for stream in (None, None, side):   # later calls reuse the pieces of the first
        h.copy_(torch.from_numpy(U))
        P.run_host(h.numpy(), s, 0.01, 1e-4, nsteps, stream=stream.cuda_stream if stream else None)
        assert np.array_equal(h.numpy(), ref)
