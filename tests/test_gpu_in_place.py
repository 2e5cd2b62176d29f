"""Gradient and Hessian-vector product written over their own argument.  The
result is the one written elsewhere, to the rounding of one transform there and
back of the regulariser's term (tolerances of the parity tests)."""
import numpy as np
import pytest

from paper_1807_04638_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1807_04638_gb300 as p
    p.lib()
    return p


@pytest.mark.parametrize("space", ["V", "L2"])
@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("n", [(16, 12, 10), (27, 25, 45), (32, 32, 32)])
def test_in_place_equals_out_of_place(pkg, n, prec, space):
    I0, vt = synth.blob_pair_inputs(n, 61, kmax=1, max_disp_vox=1.5)
    I0 = synth.spectral_gaussian_smooth(I0, 1.0)
    I1 = np.roll(I0, 1, axis=2)
    d = synth.band_limited_field(n, synth.rng_for(62), 2.0, 3)
    dt, cd = (torch.float64, pkg.LDDMM_F64) if prec == "f64" else (torch.float32, pkg.LDDMM_F32)
    T = lambda a: torch.tensor(np.ascontiguousarray(a), dtype=dt, device="cuda")
    # a weight that makes the regulariser's term a large part of the result
    prm = pkg.default_params(alpha=0.01, weight=0.1, nt=2, compute_dtype=cd, state_dtype=cd,
                             space=pkg.LDDMM_SPACE_L2 if space == "L2" else pkg.LDDMM_SPACE_V)
    rel = lambda a, b: float(torch.linalg.vector_norm(a.double() - b.double()) / torch.linalg.vector_norm(b.double()))
    tol = 1e-10 if prec == "f64" else 1e-5
    with pkg.Handle(n, prm) as h:
        grad, hv = h.new_vec(), h.new_vec()
        h.lddmm_gradient(T(0.5 * vt), T(I0), T(I1), grad)
        h.lddmm_hessvec(T(d), hv)
        v, x = T(0.5 * vt), T(d)
        h.lddmm_gradient(v, T(I0), T(I1), v)
        h.lddmm_hessvec(x, x)
        h.lddmm_synchronize()
        assert rel(v, grad) < tol, rel(v, grad)
        assert rel(x, hv) < tol, rel(x, hv)
