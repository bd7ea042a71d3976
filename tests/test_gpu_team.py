"""The two forms of the stage kernels, one thread a cell and one team of warps a
group of 32 cells, give the same bits: a single shot on a small mesh takes the
team form, many copies of it together the thread form (the choice goes by
groups of cells times shots).  The parity tests pin both to the oracle."""
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


def skewed(nx, ny):
    """Quadrilaterals with no axis-aligned face inside: a class for every cell."""
    md = synth.quad_grid(nx, ny)
    rng = np.random.default_rng(1)
    inner = (md.xy > 1e-9).all(1) & (md.xy < 1 - 1e-9).all(1)
    md.xy[inner] += rng.uniform(-0.2, 0.2, (inner.sum(), 2)) / max(nx, ny)
    return md


MESHES = {"squares": lambda: synth.quad_grid(33, 33), "rectangles": lambda: synth.quad_grid(31, 17),
          "triangles": lambda: synth.tri_grid(23, 17), "hybrid": lambda: synth.hybrid_grid(19, 19, 0, 1, 0, 1, 0.6, 0.5),
          "hanging": lambda: synth.hanging_node_patch(12, 9, refine_rows=(1, 4)), "skewed": lambda: skewed(5, 5),
          "one cell": lambda: synth.quad_grid(1, 1)}


@pytest.mark.parametrize("k", [1, 2, 3])
@pytest.mark.parametrize("mesh", list(MESHES))
@pytest.mark.parametrize("precision", ["f64", "f32", "f32x2"])
def test_forms_agree_bit_for_bit(lib, mesh, k, precision):
    hho, solver = lib
    md = MESHES[mesh]()
    P = solver.Problem(md, synth.layered_media(md), k)
    prec = {"f64": hho.HHO_F64, "f32": hho.HHO_F32, "f32x2": hho.HHO_F32X2}[precision]
    groups = (P.layout.n_fluid_pad + P.layout.n_solid_pad) // 32
    many = 4200 // groups + 1
    src = (0.37, 0.21) if mesh != "one cell" else (0.4, 0.4)
    U = synth.random_state(P.layout.n_canonical, k)
    dt = 0.01 / (k * k * np.sqrt(md.n_cells))
    out = {}
    for S in (1, many):
        P.set_shot_sources([src] * S, [(0.6, 0.8)] * S, 10.0, t0=0.01)
        x = P.batch_to_device(np.tile(U, (S, 1)), prec)
        for s in (3, 4):
            _, work = P.batch_buffers(s, S, prec)
            P.batch_step(x, work, S, s, 0.0, dt, 3, precision=prec)
        out[S] = P.batch_to_canonical(x, S, prec)
    assert np.isfinite(out[1]).all() and not np.array_equal(out[1][0], U)
    assert np.array_equal(out[1][0], out[many][0]) and np.array_equal(out[1][0], out[many][-1])
