"""Calls that ran under a limit on the library's device memory go on running under it.

Each limit (wdf_set_device_limit, bytes) was found by bisection, to within 1 KB, with kernels that need
no workspace of their own: the smallest under which a fresh context could be made and make the call. A kernel that
trades memory for time has to stay within it, or to give way to one that does. A context with
orbitals given needs most during its setup, where the plane kernels are timed on 128 pairs.
"""

import dataclasses

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
    assert wdf.device_bytes() == 0
    wdf.set_device_limit(limit)
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
