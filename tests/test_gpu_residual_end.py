"""The end of a refinement in one pass: x += d, r = b - A x, its FP32 copy and <r, r> (Sec. 2.1).

The largest relative residual that a solve reports comes from that pass. The returned x goes through
the residual operator once more, b - A x is formed on the host, and the two have to agree to the
accuracy of the operator itself (1e-12 of ||b||, the bar it is held to against the oracle), for a
single short row, an odd number of rows, a row of a full chunk and a remainder, and right-hand sides
among which one is zero; an FP32 solve that overwrites its right-hand sides leaves the caller's alone.
"""

import numpy as np
import pytest

import synth
from oracle import basis

pytestmark = pytest.mark.gpu

wdf = pytest.importorskip("paper_2607_14025_gb300.wdf")

BAR = 1e-12


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2607_14025_gb300 import build

    build.build()
    wdf.load()


@pytest.mark.parametrize("prec", ["mixed", "mixed_df"])
@pytest.mark.parametrize("name,n", [("tiny", 1), ("small", 3), ("medium", 5)])
def test_reported_residual_is_that_of_the_solution(name, n, prec):
    s = synth.make_system(name)
    vidx = (np.arange(n) % s.nocc).astype(np.int32)
    with wdf.Context(s, precision="fp64") as c:
        eps, psi = c.orbitals()
    b = synth.make_guess(s, n, 11)
    full, pf = basis.expand(b), basis.expand(psi)
    pf /= np.linalg.norm(pf, axis=1, keepdims=True)
    full -= (full @ pf.conj().T) @ pf  # right-hand sides orthogonal to the orbitals
    b = basis.fold(full)
    if n > 2:
        b[1] = 0.0
    b0 = b.copy()
    with wdf.Context(s, psi=psi, eps=eps, precision=prec, cg_tol=1e-9) as c:
        x, st = c.sternheimer(vidx, b)
        Ax = c.apply_sternheimer_operator(vidx, x)
    assert np.array_equal(b, b0) and st.converged == 1
    num = np.linalg.norm(basis.expand(b - Ax), axis=1)
    den = np.linalg.norm(basis.expand(b), axis=1)
    live = den > 0
    res = (num[live] / den[live]).max()
    print(f"{name} {n} {prec}: reported {st.max_residual:.6e}, recomputed {res:.6e}")
    assert abs(res - st.max_residual) <= BAR
    assert np.all(x[~live] == 0.0)
