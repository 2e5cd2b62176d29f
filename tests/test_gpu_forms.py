"""Which kernels a handle's sweeps run, by the launch counts of the profiler, and
their results where no other test reaches them: the shortest lengths that have a
plan for the band form, FP32 last axes beyond the compiled lengths, lengths without
a plan, and the fused stages of bfloat16 states at each of their last axes.

Tolerance against the 24-field form in FP64 (LDDMM_GENERIC_FFT=1): 1e-10 in FP64.
In FP32 the rounding of a field is raised by L, at most 6e-8 max L over the band,
on top of the 1e-5 of the parity tests."""
import math

import numpy as np
import pytest

import test_gpu_band
import test_gpu_fused
from paper_1807_04638_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
NT, ALPHA = 2, 0.01


@pytest.fixture(scope="module")
def pkg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1807_04638_gb300 as p
    p.lib()
    return p


def product(pkg, n, prec):
    """Hessian-vector product and adjoint sweep, and the launches of their classes."""
    I0, vt = synth.blob_pair_inputs(n, 61, kmax=2, max_disp_vox=1.5)
    I0 = synth.spectral_gaussian_smooth(I0, 1.0)
    r = synth.rng_for(62)
    d, be, bx = (synth.band_limited_field(n, r, 4.0, 3) for _ in range(3))
    dt, cd = (torch.float64, pkg.LDDMM_F64) if prec == "f64" else (torch.float32, pkg.LDDMM_F32)
    T = lambda a: torch.tensor(np.ascontiguousarray(a), dtype=dt, device="cuda")
    with pkg.Handle(n, pkg.default_params(alpha=ALPHA, nt=NT, compute_dtype=cd, state_dtype=cd)) as h:
        grad, hv, adj = h.new_vec(), h.new_vec(), h.new_vec()
        h.lddmm_gradient(T(0.5 * vt), T(I0), T(np.roll(I0, 1, axis=2)), grad)
        h.lddmm_profile(True)
        h.lddmm_hessvec(T(d), hv)
        h.lddmm_jacobi_adjoint(T(be), T(bx), adj)
        h.lddmm_synchronize()
        prof = h.lddmm_profile_read()
        h.lddmm_profile(False)
    return {"grad": grad, "hv": hv, "adj": adj}, {k: v[2] for k, v in prof.items()}


@pytest.mark.parametrize("n,band64,band32", [
    ((8, 10, 12), True, True),     # the smallest lengths, two stages of the smallest radices
    ((12, 8, 15), True, True),     # odd last axis, none of the lengths compiled
    ((15, 10, 8), True, True),     # the shortest last axis, odd axis 0
    ((8, 10, 9), False, False),    # 9 has no plan
    ((10, 12, 360), True, True),   # FP32 last axes with run-time radices: 3 stages each
    ((10, 12, 400), True, True),
    ((12, 10, 405), True, True),   # odd
    ((9 * 5, 9, 16), False, False),
    ((10, 8, 450), True, True),
    ((8, 15, 486), True, True),
    ((15, 9 * 3, 500), True, True),  # odd row count
    ((10, 12, 375), True, False),  # no plan of the FP32 stages
    ((8, 10, 512), True, False),
])
def test_form_and_result(pkg, n, band64, band32, monkeypatch):
    monkeypatch.setenv("LDDMM_POISON_WORKSPACE", "1")
    monkeypatch.setenv("LDDMM_GENERIC_FFT", "1")
    want, runs = product(pkg, n, "f64")
    assert runs.get("spectral_step", 0) == 0 and runs.get("adjoint_pointwise", 0) == 4 * NT
    monkeypatch.delenv("LDDMM_GENERIC_FFT")
    Lmax = (1 + ALPHA * sum(((m - 1) // 3) ** 2 for m in n)) ** 2
    for prec, band, tol, stage in (("f64", band64, 1e-10, "adjoint_stage_fp64"),
                                   ("f32", band32, 1e-5 + 6e-8 * Lmax, "adjoint_stage_fused")):
        got, runs = product(pkg, n, prec)
        # one tangent sweep and two adjoint ones, two stages a step
        assert runs.get("spectral_step", 0) == (6 * NT if band else 0), (prec, runs)
        assert runs.get(stage, 0) == (4 * NT if band else 0), (prec, runs)
        assert runs.get("adjoint_pointwise", 0) == (0 if band else 4 * NT), (prec, runs)
        for k, w in want.items():
            e = float(torch.linalg.vector_norm(got[k].double() - w) / torch.linalg.vector_norm(w))
            assert math.isfinite(e) and e < tol, (prec, k, e, tol)


@pytest.mark.parametrize("n,nt", [((32, 32, 32), 3), ((64, 36, 64), 2), ((64, 32, 128), 2), ((20, 24, 256), 2)])
def test_fused_stages_of_bfloat16_states(pkg, n, nt, monkeypatch):
    """Every last axis of k_fused_stage, also beside axes without a register-blocked
    plan: the same inputs and criterion as on 64^3."""
    test_gpu_fused.test_fused_stages_equal_separate_passes(pkg, n, "bf16", nt, monkeypatch)


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("n", [(8, 10, 16), (12, 8, 9), (15, 500, 8), (486, 8, 10)])
def test_run_time_radices_of_the_shortest_and_longest_lengths(pkg, prec, n):
    """Axes 0 and 1 of k_gen_c2c: inputs and tolerances of its other lengths."""
    test_gpu_band.test_c2c_passes_with_run_time_radices(pkg, prec, n)
