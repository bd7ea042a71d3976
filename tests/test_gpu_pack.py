"""hho_batch_pack / hho_batch_unpack: the canonical <-> device-layout kernels
and their conversions, bit for bit against NumPy's conversions."""
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


def values(n, seed):
    """Doubles of every magnitude: ties of the FP32 rounding, carries into the exponent, subnormal and
    overflowing results, signed zeros, infinities and NaN."""
    rng = np.random.default_rng(seed)
    v = rng.standard_normal(n) * 2.0 ** rng.integers(-180, 140, n)
    one = 1.0 + np.arange(64) * 2.0 ** -24
    ends = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 2.0 ** -149, 2.0 ** -126, 2.0 ** -127, 2.0 ** -70, 2.0 ** -71,
                     2.0 ** 126, 2.0 ** 127, 2.0 ** 128, 3.4028235677973366e38, 1e-320, np.nextafter(2.0, 1.0),
                     2.0 ** 53 - 1, 1.0 + 2.0 ** -52, 1.5 * 2.0 ** -70])
    special = np.concatenate([one, -one, one * 2.0 ** -69.0, ends, -ends])
    v[: len(special)] = special
    return v


@pytest.mark.parametrize("k", [1, 2, 3])
@pytest.mark.parametrize("precision", ["f64", "f32", "f32x2"])
def test_pack_is_a_permutation_with_numpys_conversions(lib, k, precision):
    hho, solver = lib
    md = synth.quad_grid(9, 5, 0.0, 9.0, 0.0, 5.0, y_interface=9.0)   # one class: slot = cell
    P = solver.Problem(md, synth.layered_media(md), k)
    n, nc, N = P.layout.n, md.n_cells, P.layout.n_solid_pad
    prec = {"f64": hho.HHO_F64, "f32": hho.HHO_F32, "f32x2": hho.HHO_F32X2}[precision]
    c = values(2 * nc * 5 * n, k).reshape(2, -1)
    st = P.batch_to_device(c, prec).cpu().numpy()
    with np.errstate(all="ignore"):
        hi = c.astype(np.float32)
        lo = (c - hi.astype(np.float64)).astype(np.float32)
    want = {"f64": lambda: c, "f32": lambda: hi, "f32x2": lambda: np.stack([hi, lo], -1)}[precision]()
    raw = st.view(np.float32).reshape(-1, 2) if precision == "f32x2" else st
    raw = raw.reshape((2, 5 * n, N) + raw.shape[1:])
    got = np.moveaxis(raw[:, :, :nc], 1, 2).reshape(want.shape)
    nan = np.isnan(want)
    assert np.array_equal(np.isnan(got), nan)
    bits = np.uint64 if precision == "f64" else np.uint32
    assert np.array_equal(np.ascontiguousarray(got).view(bits)[~nan], np.ascontiguousarray(want).view(bits)[~nan])
    assert not np.any(raw[:, :, nc:])                                  # padding slots are zero
    back = P.batch_to_canonical(torch.as_tensor(st).cuda(), 2, prec)
    with np.errstate(all="ignore"):
        ref = {"f64": lambda: c, "f32": lambda: hi.astype(np.float64),
               "f32x2": lambda: hi.astype(np.float64) + lo.astype(np.float64)}[precision]()
    assert np.array_equal(back, ref, equal_nan=True)


@pytest.mark.parametrize("k", [1, 2, 3])
def test_unpack_inverts_pack_on_mixed_classes(lib, k):
    """Interleaved classes, both domains, hanging nodes, odd counts."""
    hho, solver = lib
    for md in (synth.tri_grid(7, 5), synth.hanging_node_patch(5, 4, refine_rows=(1,)), synth.quad_grid(1, 2)):
        P = solver.Problem(md, synth.layered_media(md), k)
        c = synth.random_state(3 * P.layout.n_canonical, k).reshape(3, -1)
        assert np.array_equal(P.batch_to_canonical(P.batch_to_device(c, hho.HHO_F64), 3, hho.HHO_F64), c)
        got = P.batch_to_canonical(P.batch_to_device(c, hho.HHO_F32), 3, hho.HHO_F32)
        assert np.array_equal(got, c.astype(np.float32).astype(np.float64))
