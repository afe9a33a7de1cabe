"""Calls that ran under a limit on the library's device memory go on running under it.

Each limit (wdf_set_device_limit, bytes) was found by bisection, to within 1 KB, with kernels that need
no workspace of their own: the smallest under which a fresh context could be made and make the call. A kernel that
trades memory for time has to stay within it, or to give way to one that does. A context with
orbitals given needs most during its setup, where the plane kernels are timed on 128 pairs.
"""

import dataclasses
import gc
import os

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

wdf = pytest.importorskip("paper_2607_14025_gb300.wdf")

# system (gN: two-atom system on an N^3 grid), occupied orbitals (None: its own), form, call and vectors, limit
CALLS = [
    ("tiny", None, "mixed", "create", 0, 5941160),
    ("tiny", None, "mixed", "hamiltonian", 48, 5941087),
    ("ragged", None, "mixed_df", "solve", 40, 17648562),
    ("g36", 14, "fp64", "solve", 20, 33333937),
    ("g48", 20, "mixed_df", "residual", 3, 120981648),
    ("medium", None, "mixed_df", "create", 0, 853695569),
    ("medium", None, "fp64", "hamiltonian", 48, 585086396),
    ("g64", 4, "mixed", "create", 0, 123983511),
    ("g75", 20, "fp64", "create", 0, 356239620),
    ("g96", 8, "mixed_df", "residual", 40, 624832845),
    # the density response: the sum over orbitals in place needs no fields
    ("g36", 14, "fp64", "chi0", 1, 33334382),
    ("g36", 14, "fp64", "chi0", 4, 34647756),
    ("g45", 14, "mixed", "chi0", 4, 65270793),
    ("g48", 20, "mixed_df", "chi0", 6, 190597472),
    ("g64", 4, "mixed_df", "chi0", 16, 269822532),
    ("medium", None, "mixed_df", "chi0", 1, 1037335816),
    ("medium", None, "mixed_df", "chi0", 8, 1962374208),
    ("g75", 20, "mixed_df", "chi0", 1, 460809251),
    ("g75", 20, "fp64", "chi0", 1, 356239257),
]


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2607_14025_gb300 import build

    build.build()
    wdf.load()


def system(name, nocc):
    sp = synth.grid_probe(int(name[1:])) if name[0] == "g" else synth.spec(name)
    return synth.make_system(dataclasses.replace(sp, nocc=nocc) if nocc else sp)


@pytest.mark.parametrize("name,nocc,form,call,k,limit", CALLS, ids=[f"{c[0]}-{c[2]}-{c[3]}{c[4]}" for c in CALLS])
def test_call_is_accepted_within_its_limit(name, nocc, form, call, k, limit):
    s = system(name, nocc)
    psi, eps = synth.make_guess(s, s.nocc, 1), np.linspace(-7.0, -3.0, s.nocc)
    v = (np.arange(k) % s.nocc).astype(np.int32)
    gc.collect()
    wdf.set_device_limit(wdf.device_bytes() + limit)
    try:
        with wdf.Context(s, psi=psi, eps=eps, precision=form, cg_tol=1e-4, cg_maxiter=6) as c:
            try:
                if call == "chi0":
                    c.apply_chi0(synth.make_perturbations(s, k, 2), want_drho=True)
                elif call == "solve":
                    c.sternheimer(v, synth.make_guess(s, k, 3))
                elif call == "hamiltonian":
                    c.apply_hamiltonian(synth.make_guess(s, k, 3))
                elif call == "residual":
                    c.apply_sternheimer_operator(v, synth.make_guess(s, k, 3))
            except wdf.NotConverged:  # six iterations on made-up orbitals
                pass
    finally:
        wdf.set_device_limit(0)


def chi0(s, psi, eps, form, variant, phi, limit=0):
    """(out, drho, bytes held) of a fresh context with this plane kernel; limit: for the call alone."""
    old = os.environ.get("WDF_PLANE_VARIANT")
    os.environ["WDF_PLANE_VARIANT"] = str(variant)
    try:
        c = wdf.Context(s, psi=psi, eps=eps, precision=form, cg_tol=1e-10)
    finally:
        if old is None:
            del os.environ["WDF_PLANE_VARIANT"]
        else:
            os.environ["WDF_PLANE_VARIANT"] = old
    with c:
        assert c.plane_variant(64 if form == "fp64" else 32) == variant
        wdf.set_device_limit(limit)
        try:
            out, drho, _ = c.apply_chi0(phi, want_drho=True)
        finally:
            wdf.set_device_limit(0)
        return out, drho, wdf.device_bytes()


def rel(a, b):
    return float(np.abs(a - b).max() / np.abs(b).max())


@pytest.mark.parametrize("npert", [1, 3])
@pytest.mark.parametrize("n,natom,form", [(36, 2, "fp64"), (45, 2, "mixed"), (54, 8, "mixed_df"), (64, 12, "mixed_df")])
def test_density_response_in_groups_and_in_place(n, natom, form, npert):
    """The sum over orbitals in one or two groups, in the refinement's buffer, and in place.

    The limit is what a context with the generic plane kernel holds, which sums in place. The
    solves are the same bit for bit, the sums differ by the rounding of FP64-class transforms (a
    few 1e-15): bar 1e-12. The generic kernel's solves differ by their own errors: bar 1e-8.
    """
    s = synth.make_system(dataclasses.replace(synth.grid_probe(n), natom=natom, nocc=2 * natom))
    with wdf.Context(s, precision="fp64", gs_tol=1e-9) as c0:
        eps, psi = c0.orbitals()
    phi = synth.make_perturbations(s, npert, 5)
    gc.collect()
    generic = chi0(s, psi, eps, form, 3, phi)
    free = chi0(s, psi, eps, form, 8, phi)
    tight = chi0(s, psi, eps, form, 8, phi, generic[2])
    assert tight[2] <= generic[2]
    for a, b, g in zip(free[:2], tight[:2], generic[:2]):
        assert rel(b, a) < 1e-12 and rel(a, g) < 1e-8
