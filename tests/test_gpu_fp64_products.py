"""The FP64 Gram products and linear combinations behind H x, A_v x, W_p x (plain FP64) against
numpy, at the edges of their 16 x 16 output tiles, of the 1-, 2-, 4- and 8-vector groups, of the
128-element blocks and of the element splits (Gram products with 8 vectors and fewer: the narrow kernel).

W_p x = v^1/2 sum_a phibar_a lam_a / (1 - lam_a) <phibar_a, v^1/2 x> is one Gram product and one
combination; both sides sum a few thousand terms in FP64, so they agree to a few hundred ulp:
bar 1e-13 of the largest value.
"""

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

wdf = pytest.importorskip("paper_2607_14025_gb300.wdf")

_ctx = {}


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2607_14025_gb300 import build

    build.build()
    yield
    for c, _ in _ctx.values():
        c.close()
    _ctx.clear()


def context(n):
    if n not in _ctx:
        s = synth.make_system(synth.grid_probe(n))
        psi = synth.make_guess(s, s.nocc, 1)
        _ctx[n] = (wdf.Context(s, psi=psi, eps=np.linspace(-7.0, -3.0, s.nocc), precision="fp64"), s)
    return _ctx[n]


def wp_reference(s, lam, phi, x):
    g = np.sqrt(np.einsum("ij,ij->i", s.gvec, s.gvec))
    vh = np.zeros_like(g)
    vh[1:] = np.sqrt(4.0 * np.pi) / g[1:]
    w = np.full(s.npw_h, 2.0)
    w[0] = 1.0
    dot = ((np.conj(phi) * w) @ (x * vh).T).real
    return (((lam / (1.0 - lam))[:, None] * dot).T @ phi) * vh


@pytest.mark.parametrize("n", [24, 45, 64])
@pytest.mark.parametrize("neig,nvec", [(1, 9), (15, 16), (16, 17), (17, 33), (64, 47), (33, 130), (200, 12), (65, 1), (64, 2), (70, 3), (63, 8)])
def test_wp_matches_numpy(n, neig, nvec):
    c, s = context(n)
    rng = np.random.default_rng(neig * 1000 + nvec)
    phi = synth.make_perturbations(s, neig, 3)
    x = rng.standard_normal((nvec, s.npw_h)) + 1j * rng.standard_normal((nvec, s.npw_h))
    x[:, 0] = x[:, 0].real
    lam = -3.0 * rng.random(neig)
    y = c.apply_wp(lam, phi, x)
    ref = wp_reference(s, lam, phi, x)
    assert np.abs(y - ref).max() <= 1e-13 * np.abs(ref).max()


@pytest.mark.parametrize("nvec", [9, 16, 31, 64])
def test_hamiltonian_blocks_match_narrow_calls(nvec):
    c, s = context(45)
    x = synth.make_guess(s, nvec, 4)
    y = c.apply_hamiltonian(x)
    one = np.concatenate([c.apply_hamiltonian(x[i:i + 8]) for i in range(0, nvec, 8)])
    assert np.abs(y - one).max() <= 1e-13 * np.abs(one).max()
