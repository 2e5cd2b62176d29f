"""Bytes of a handle's workspace, by which a server admits requests, against the
sum of the buffers that the 24-field form of the path needs: packed copies, pitches
and alignment of other forms find their room within it."""
import itertools

import pytest

import paper_1807_04638_gb300 as pkg


def field_bytes(n, p, t):
    """121 half spectra, 89 real fields and the stored states, with the maps and
    cotangents of the discrete gradient and the velocities at checkpoints."""
    N, spec = n[0] * n[1] * n[2], n[0] * n[1] * (n[2] // 2 + 1)
    every = min(p.checkpoint_every, p.nt)
    half, real = 121, 89
    if p.gradient_mode == pkg.LDDMM_GRAD_DISCRETE:
        real += 6 * (p.nt + 1) + 6
    if every <= 1 or every == p.nt:
        every = p.nt
    else:
        half += 3 * -(-p.nt // every)
    states = 2 * every * 24 * N * (2 if p.state_dtype == pkg.LDDMM_BF16 else t)
    return 2 * t * half * spec + t * real * N + states


@pytest.mark.parametrize("n", [(12, 15, 16), (27, 25, 45), (32, 32, 32), (75, 90, 81), (128, 128, 128), (256, 300, 256)])
def test_no_more_than_the_fields_of_the_24_field_form(n):
    forms = [(pkg.LDDMM_F32, pkg.LDDMM_F32), (pkg.LDDMM_F64, pkg.LDDMM_F64), (pkg.LDDMM_F32, pkg.LDDMM_BF16)]
    for (cd, sd), every, mode, dealias in itertools.product(forms, (1, 3), (0, 1), (0, 1)):
        p = pkg.default_params(nt=10, compute_dtype=cd, state_dtype=sd, checkpoint_every=every,
                               gradient_mode=mode, dealias=dealias)
        got = pkg.workspace_bytes(n, p)
        if mode == pkg.LDDMM_GRAD_DISCRETE and (every > 1 or sd == pkg.LDDMM_BF16):
            assert got == 0
            continue
        assert 0 < got <= field_bytes(n, p, 8 if cd == pkg.LDDMM_F64 else 4), (cd, sd, every, mode)
