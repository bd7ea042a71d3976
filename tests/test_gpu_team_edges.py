"""The team and the thread form of the stage kernels where the dispatch's lines lie
far out (double-float on general meshes and at k = 3) and on polygons with the
most faces a cell may have, 32: the same bits in both forms, and the oracle's
values.  Which form ran is read from the list of launched kernels."""
import numpy as np
import pytest

import synth
from oracle import erk as E
from tests.libutil import ensure_built, oracle_system, rel
from tests.test_gpu_team import MESHES

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ensure_built()
    from paper_2505_15771_gb300 import hho, solver
    forms(lambda: torch.zeros(1, device="cuda"))   # the profiler's first use reports nothing
    return hho, solver


def polygon(n, cx, cy, turn):
    """A regular polygon whose faces turn and turn + n/2 are horizontal to the last bit (normals with n_x = 0)."""
    a = 2 * np.pi * (np.arange(n) - turn - 0.5) / n - np.pi / 2
    xy = np.stack([cx + 0.2 * np.cos(a), cy + 0.2 * np.sin(a)], axis=1)
    for j in (turn, (turn + n // 2) % n):
        xy[(j + 1) % n, 1] = xy[j, 1]
    return xy


def with_polygons(md):
    """Two 32-gons, a fluid and a solid one, beside a mesh that they do not touch; the last face of one is horizontal."""
    xy, ptr, vtx, dom = [md.xy], list(md.cell_ptr), list(md.cell_vtx), list(md.cell_domain)
    first = len(md.xy)
    for p, d in [(polygon(32, 3.0, 0.3, 31), synth.FLUID), (polygon(32, 3.0, 0.8, 2), synth.SOLID)]:
        xy.append(p)
        vtx += range(first, first + len(p))
        first += len(p)
        ptr.append(len(vtx))
        dom.append(d)
    return synth.MeshData(xy=np.concatenate(xy), cell_ptr=np.array(ptr, np.int64), cell_vtx=np.array(vtx, np.int64),
                          cell_domain=np.array(dom, np.uint8), vertex_rep=None)


ALL = dict(MESHES, **{"32-gons": lambda: with_polygons(synth.hybrid_grid(7, 7, 0.0, 1.0, 0.0, 1.0, 0.6, 0.5))})


def forms(run):
    """The result of run() and the kinds of stage kernels it launched."""
    from torch.profiler import ProfilerActivity, profile
    with profile(activities=[ProfilerActivity.CUDA]) as p:
        out = run()
        torch.cuda.synchronize()
    return out, {w for w in ("team_kernel", "stage_kernel") for e in p.events() if w in e.name}


@pytest.mark.parametrize("mesh,k,precision,groups_many", [
    ("squares", 3, "f32x2", 24100), ("rectangles", 3, "f32x2", 24100), ("triangles", 2, "f32x2", 12100),
    ("hanging", 2, "f32x2", 12100), ("skewed", 2, "f32x2", 12100), ("32-gons", 2, "f32x2", 12100),
    ("32-gons", 1, "f64", 4200), ("32-gons", 2, "f64", 4200), ("32-gons", 3, "f64", 4200),
    ("32-gons", 1, "f32", 4200), ("32-gons", 3, "f32", 4200)])
def test_forms_agree_bit_for_bit(lib, mesh, k, precision, groups_many):
    hho, solver = lib
    md = ALL[mesh]()
    P = solver.Problem(md, synth.layered_media(md), k)
    prec = {"f64": hho.HHO_F64, "f32": hho.HHO_F32, "f32x2": hho.HHO_F32X2}[precision]
    many = groups_many // ((P.layout.n_fluid_pad + P.layout.n_solid_pad) // 32) + 1
    U = synth.random_state(P.layout.n_canonical, k)
    out, ran = {}, {}
    for S in (1, many):
        P.set_shot_sources([(0.37, 0.21)] * S, [(0.6, 0.8)] * S, 10.0, t0=0.01)
        x = P.batch_to_device(np.tile(U, (S, 1)), prec)
        _, work = P.batch_buffers(4, S, prec)
        _, ran[S] = forms(lambda: P.batch_step(x, work, S, 4, 0.0, 1e-4, 2, precision=prec))
        got = P.batch_to_canonical(x, S, prec)
        out[S] = [got[0], got[-1]]
    if ran[1] and ran[many]:   # where the profiler reports kernels
        assert ran[1] == {"team_kernel"} and ran[many] == {"stage_kernel"}
    assert np.isfinite(out[1][0]).all() and not np.array_equal(out[1][0], U)
    for a in out[many]:
        assert np.array_equal(a, out[1][0])


@pytest.mark.parametrize("k,arith", [(1, "f64"), (2, "f64"), (3, "f64"), (1, "f32x2"), (2, "f32x2"), (3, "f32x2")])
def test_polygons_of_32_faces_match_the_oracle(lib, k, arith):
    """Relative L2 <= 1e-12 over all cell values, the bar of the parity tests, and on each polygon by itself."""
    hho, solver = lib
    md = with_polygons(synth.quad_grid(4, 4))
    media = synth.layered_media(md)
    S = oracle_system(md, k, media)
    U0 = synth.random_state(S.nT, 3)
    ref = E.Stepper(S).step(U0, 0.0, 2e-5, "erk4", 6)
    P = solver.Problem(md, media, k)
    P.set_arithmetic(hho.HHO_F64 if arith == "f64" else hho.HHO_F32X2)
    x = P.to_device(U0)
    P.step(x, 4, 0.0, 2e-5, 6)
    got = P.to_canonical(x)
    n = (k + 1) * (k + 2) // 2
    assert rel(got, ref) <= 1e-12
    assert rel(got[-8 * n:-5 * n], ref[-8 * n:-5 * n]) <= 1e-12 and rel(got[-5 * n:], ref[-5 * n:]) <= 1e-12
