"""hho_erk_run_host in pieces (from the second call of an operator on, states of
40 MB and more): the bits of packing on the device, stepping and unpacking, at
every degree, with orders that overlap and one that does not, and with one stage
and one step, where the first stage is the last one too."""
import numpy as np
import pytest

import synth
from tests.libutil import ensure_built

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MESHES = {"quad4": lambda: synth.quad_grid(723, 363, 0.0, 2.0, 0.0, 1.0, y_interface=0.45),     # 4 pieces at k = 2
          "quad2": lambda: synth.quad_grid(512, 272, 0.0, 1.9, 0.0, 1.0, y_interface=0.5),       # 2 pieces at k = 3
          "quad8": lambda: synth.quad_grid(1024, 512, 0.0, 2.0, 0.0, 1.0, y_interface=0.5),      # 8 pieces at k = 1
          "hybrid8": lambda: synth.hybrid_grid(760, 700, 0.0, 1.0, 0.0, 1.0, 0.7, 0.5),          # 8, no early stage
          "tri2": lambda: synth.tri_grid(300, 271)}                                              # 2 pieces at k = 3


@pytest.fixture(scope="module")
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ensure_built()
    from paper_2505_15771_gb300 import hho, solver
    return hho, solver


@pytest.mark.parametrize("mesh,k,s,nsteps,arith", [
    ("quad4", 2, 4, 1, "f64"), ("quad4", 2, 1, 1, "f32x2"), ("quad2", 3, 3, 2, "f64"), ("quad2", 3, 1, 1, "f64"),
    ("quad8", 1, 2, 1, "f32x2"), ("hybrid8", 2, 1, 1, "f64"), ("tri2", 3, 4, 1, "f32x2")])
def test_pieces_give_the_bits_of_the_device_path(lib, mesh, k, s, nsteps, arith):
    hho, solver = lib
    md = MESHES[mesh]()
    P = solver.Problem(md, synth.layered_media(md), k)
    P.set_arithmetic(hho.HHO_F64 if arith == "f64" else hho.HHO_F32X2)
    P.set_sources([(0.37, 0.21)], [(0.6, 0.8)], 10.0)
    if s == 1:
        tab = hho.Tableau()
        tab.s = 1
        tab.b[0] = 1.0
    else:
        tab = hho.hho_tableau_erk(s)
    U = np.random.default_rng(5).standard_normal(P.layout.n_canonical)
    assert U.nbytes >= 40_000_000
    x = P.to_device(U)
    hho.hho_erk_step(P.ops, tab, 0.01, 1e-5, nsteps, x.data_ptr(), P.work(tab).data_ptr(),
                     torch.cuda.current_stream().cuda_stream)
    ref = P.to_canonical(x)
    assert np.isfinite(ref).all() and not np.array_equal(ref, U)
    h = torch.from_numpy(U.copy()).pin_memory()
    side = torch.cuda.Stream()
    for stream in (torch.cuda.current_stream(), torch.cuda.current_stream(), side):
        h.copy_(torch.from_numpy(U))
        hho.hho_erk_run_host(P.ops, tab, 0.01, 1e-5, nsteps, h.numpy(), stream.cuda_stream)
        assert np.array_equal(h.numpy(), ref)
    P.close()
