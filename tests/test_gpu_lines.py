"""The line-resident plane kernels (plane variant 8) against the generic mixed-radix kernel
(variant 3) of the same library, on every grid they are compiled for.

Both compute the same double-float transforms (about 48 significant bits, 3e-15 of the largest
value per transform), so A_v x may differ by a few 1e-15 of the largest component; the bar is
5e-14. chi0bar at cg_tol 1e-10 differs by the solves' own errors (each within 1e-10 of its
right-hand side, amplified by at most the condition of the occupied gap): bar 1e-8, and the FP32
inner iterations have to take the same number of steps to within 3%.

Vector counts are odd (a phantom partner in the last pair) and small against a block's plane
group, so the last blocks are ragged; the band edge |n1| = N / 4 and one column more (which the
kernels refuse) are covered by denser spheres.
"""

import dataclasses
import math
import os

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

wdf = pytest.importorskip("paper_2607_14025_gb300.wdf")


def rel(a, b):
    return float(np.abs(np.asarray(a) - np.asarray(b)).max() / np.abs(np.asarray(b)).max())


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2607_14025_gb300 import build

    build.build()


def pinned(variant, s, psi, eps, precision="mixed_df"):
    old = os.environ.get("WDF_PLANE_VARIANT")
    os.environ["WDF_PLANE_VARIANT"] = str(variant)
    try:
        return wdf.Context(s, psi=psi, eps=eps, precision=precision, cg_tol=1e-10)
    finally:
        if old is None:
            del os.environ["WDF_PLANE_VARIANT"]
        else:
            os.environ["WDF_PLANE_VARIANT"] = old


def probe(n, xmax=None):
    sp = synth.grid_probe(n)
    if xmax is not None:  # the cutoff between the columns xmax and xmax + 1
        sp = dataclasses.replace(sp, ecut=((xmax + 0.5) * 2.0 * math.pi / sp.L) ** 2)
    return synth.make_system(sp)


@pytest.mark.parametrize("n", synth.GRID_SIZES)
@pytest.mark.parametrize("nvec", [1, 7])
def test_operator_and_response_match_the_generic_kernel(n, nvec):
    s = probe(n)
    with wdf.Context(s, precision="mixed_df", gs_tol=1e-8) as c0:
        eps, psi = c0.orbitals()
    x = synth.make_guess(s, nvec, 3)
    v = (np.arange(nvec) % s.nocc).astype(np.int32)
    phi = synth.make_perturbations(s, 3 if nvec > 1 else 1, 5)
    got = {}
    for variant in (8, 3):
        with pinned(variant, s, psi, eps) as c:
            assert c.plane_variant(32) == variant and c.plane_variant(48) == variant
            out, drho, st = c.apply_chi0(phi, want_drho=True)
            got[variant] = (c.apply_sternheimer_operator(v, x), out, drho, st.cg_iters)
    a, b = got[8], got[3]
    assert rel(a[0], b[0]) < 5e-14
    assert rel(a[1], b[1]) < 1e-8 and rel(a[2], b[2]) < 1e-8
    assert abs(a[3] - b[3]) <= max(2, 0.03 * b[3])


@pytest.mark.parametrize("n", synth.GRID_SIZES)
def test_fp64_form_matches_the_generic_kernel(n):
    """FP64: both within a few ulp (1e-16 of the largest value per transform); bar 1e-14."""
    s = probe(n)
    psi = synth.make_guess(s, s.nocc, 1)
    eps = np.linspace(-7.0, -3.0, s.nocc)
    x = synth.make_guess(s, 7, 3)
    v = np.arange(7) % s.nocc
    y = {}
    for variant in (8, 3):
        with pinned(variant, s, psi, eps, "fp64") as c:
            assert c.plane_variant(64) == variant
            y[variant] = (c.apply_sternheimer_operator(v, x), c.apply_hamiltonian(x[:5]))
    assert rel(y[8][0], y[3][0]) < 1e-14 and rel(y[8][1], y[3][1]) < 1e-14
    with pinned(8, s, psi, eps) as c:  # H x of a double-float context is FP64 too
        assert rel(c.apply_hamiltonian(x[:5]), y[3][1]) < 1e-14


@pytest.mark.parametrize("n", [24, 45, 64, 96])
def test_band_edge(n):
    s = probe(n, n // 4)
    psi = synth.make_guess(s, s.nocc, 1)
    eps = np.linspace(-7.0, -3.0, s.nocc)
    x = synth.make_guess(s, 5, 2)
    v = np.arange(5) % s.nocc
    y = {}
    for variant in (8, 3):
        with pinned(variant, s, psi, eps) as c:
            assert c.plane_variant(48) == variant
            y[variant] = c.apply_sternheimer_operator(v, x)
    assert rel(y[8], y[3]) < 5e-14


def test_wider_band_is_left_to_the_other_kernels():
    s = probe(24, 7)
    psi = synth.make_guess(s, s.nocc, 1)
    with pinned(8, s, psi, np.linspace(-7.0, -3.0, s.nocc)) as c:
        assert c.plane_variant(32) != 8 and c.plane_variant(48) != 8
        assert np.isfinite(c.apply_sternheimer_operator([0], synth.make_guess(s, 1, 2))).all()
