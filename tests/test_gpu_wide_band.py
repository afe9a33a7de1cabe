"""The 64 x 64 double-float kernel with a task per thread, on bands that the line-resident kernel refuses.

Plane variant 6 is the line-resident kernel while the occupied columns lie in |n| <= 16. On a sphere
one column wider it is k_plane_df: its V_loc product, right-hand-side product and orbital sum in place
against the generic kernel's (variant 3), with the bars of the line-resident kernels' tests.
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
    return float(np.abs(a - b).max() / np.abs(b).max())


@pytest.mark.parametrize("npert", [1, 3])
def test_task_per_thread_kernel_matches_the_generic_one(npert):
    sp = synth.grid_probe(64)
    s = synth.make_system(dataclasses.replace(sp, ecut=(17.5 * 2.0 * math.pi / sp.L) ** 2))
    with wdf.Context(s, precision="mixed_df", gs_tol=1e-8) as c0:
        eps, psi = c0.orbitals()
    x, v = synth.make_guess(s, 5, 3), (np.arange(5) % s.nocc).astype(np.int32)
    phi = synth.make_perturbations(s, npert, 5)
    got = {}
    old = os.environ.get("WDF_PLANE_VARIANT")
    try:
        for variant in (6, 3):
            os.environ["WDF_PLANE_VARIANT"] = str(variant)
            with wdf.Context(s, psi=psi, eps=eps, precision="mixed_df", cg_tol=1e-10) as c:
                assert c.plane_variant(48) == variant
                c.profile_kernel("plane_accum:48")
                out, drho, _ = c.apply_chi0(phi, want_drho=True)
                assert c.profile_read()[0] == 1  # the sum ran in place
                c.profile_kernel(None)
                got[variant] = (c.apply_sternheimer_operator(v, x), out, drho)
    finally:
        if old is None:
            os.environ.pop("WDF_PLANE_VARIANT", None)
        else:
            os.environ["WDF_PLANE_VARIANT"] = old
    assert rel(got[6][0], got[3][0]) < 5e-14
    assert rel(got[6][1], got[3][1]) < 1e-8 and rel(got[6][2], got[3][2]) < 1e-8
