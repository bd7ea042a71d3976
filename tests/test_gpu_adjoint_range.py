"""hho_adjoint_vjp_f32 holds the range of its FP32 inputs: with the state scaled
by 2^a and the cotangent by 2^b the gradients scale by 2^(a + b) (the wavelet's by
2^b), also where the products of the two leave FP32's exponents.  Scaling by a
power of two is exact in every operation but for values that become subnormal:
2^-149 absolute, 2^-79 of a state of order 2^-70, over about 2^14 operations
that amplify by less than 2^20, so well below 2^-40 of the largest gradient."""
import numpy as np
import pytest

import synth
from tests.libutil import ensure_built

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

REC = [(0.31, 0.22), (0.47, 0.5), (0.83, 0.71), (0.12, 0.9)]
SRC = [(0.41, 0.23), (0.55, 0.83)]   # one in each domain
MESHES = {"squares": lambda: synth.quad_grid(8, 8),
          "hybrid": lambda: synth.hybrid_grid(6, 6, 0.0, 1.0, 0.0, 1.0, 0.7, 0.5)}


@pytest.fixture(scope="module")
def hho():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return ensure_built()


@pytest.mark.parametrize("mesh,k", [("squares", 1), ("squares", 2), ("hybrid", 2), ("hybrid", 3)])
def test_gradients_scale_with_state_and_cotangent(hho, mesh, k):
    md = MESHES[mesh]()
    nsteps, dt, ckpt, s = 12, 0.002, 5, 4
    lm = hho.hho_mesh_create(md.xy, md.cell_ptr, md.cell_vtx, md.cell_domain)
    ops = hho.hho_operators_build(lm, k, *synth.layered_media(md))
    hho.hho_mesh_destroy(lm)
    hho.hho_sources_set_samples(ops, SRC, [(0.6, 0.8)] * 2, 0.0, dt, np.zeros((2, nsteps, s)))
    hho.hho_receivers_set(ops, REC)
    tab = hho.hho_tableau_erk(s)
    lay = hho.hho_state_layout(ops)
    c = torch.as_tensor(synth.random_state(lay.n_canonical, 12)).cuda()
    x64 = torch.zeros(lay.n_state, dtype=torch.float64, device="cuda")
    hho.hho_state_pack(ops, c.data_ptr(), x64.data_ptr())
    G = torch.as_tensor(np.random.default_rng(13).standard_normal((nsteps, len(REC), 5))).float().cuda()
    nw = hho.hho_adjoint_work_size_f32(ops, tab, nsteps, ckpt)
    work = torch.empty(nw, dtype=torch.float32, device="cuda")

    def vjp(a, b):
        x, g = x64.float() * 2.0 ** a, G * 2.0 ** b
        cell, wav, tau = hho.hho_adjoint_vjp_f32(ops, tab, 0.0, dt, nsteps, ckpt, x.data_ptr(), g.data_ptr(),
                                                 work.data_ptr(), nw, md.n_cells, n_src=2, with_tau=True)
        return [np.ldexp(cell, -a - b), np.ldexp(wav, -b), np.ldexp(tau, -a - b)]

    base = vjp(0, 0)
    for a, b in [(-70, -70), (70, 70), (-70, 70), (60, -90)]:
        for name, one, ref in zip(("materials", "wavelet", "tau"), vjp(a, b), base):
            scale = np.abs(ref).max(axis=0) if name == "materials" else np.abs(ref).max()
            assert np.isfinite(one).all() and np.abs(ref).max() > 0
            assert (np.abs(one - ref) <= 2.0 ** -40 * scale).all(), (name, a, b)
    hho.hho_ops_destroy(ops)
