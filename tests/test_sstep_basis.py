"""Conditioning of the complex64 GMRES(3) steps' s-step basis (CPU, the oracle's
matrices and iterates).

A step solves the normal equations of W = (w_0, w_1, w_2), w_j = scale A v_j,
v_{j+1} = (scale A - sigma) v_j, v_0 = r, scale = h_l^2 / 4, with W's columns
scaled to unit length.  Over a whole solve, the median condition of W^H W:

* fine level: 9 to 24 with sigma = 1, 600 to 1100 with sigma = 0 (the spectrum
  of scale A lies around 1, so the shift separates the vectors);
* first coarse level: 17 to 45 with sigma = 0, 2e4 to 7e4 with sigma = 1 (the
  spectrum of its Galerkin operator lies around 0.3, and the shift turns the
  powers into nearly one direction);
* below: 30 to 2400 with sigma = 0, 500 to 4e4 with sigma = 1.
"""
import numpy as np
import pytest

import synth
from oracle import cycle as ocycle
from oracle import hierarchy as ohier
from oracle import smoothers


def _conditions(n, kh, kvar, gamma, monkeypatch):
    h = 1.0 / n
    k = kh / h
    kk = synth.k_field(synth.chi_smooth(n, n, 2), 0.6 * k, k) if kvar else k
    H = ohier.build_hierarchy(n, n, h, kk, 1 / k)
    level = {H.A[q].shape[0]: q for q in range(H.nlevels)}
    cond = {}
    step = smoothers.gmres_step

    def recorded(A, x, b, *a, **kw):
        lev, r = level[A.shape[0]], b - A @ x
        scale = 0.25 * h * h * 4**lev
        for sigma in (0.0, 1.0):
            v = [r]
            for _ in range(3):
                v.append(scale * (A @ v[-1]) - sigma * v[-1])
            W = np.stack([v[j + 1] + sigma * v[j] for j in range(3)], axis=1)
            W = W / np.linalg.norm(W, axis=0)
            cond.setdefault((lev, sigma), []).append(np.linalg.cond(W.conj().T @ W))
        return step(A, x, b, *a, **kw)

    monkeypatch.setattr(smoothers, "gmres_step", recorded)
    res = ocycle.mg_solve(H, synth.point_source(n, n, h).ravel(), 1e-6, ocycle.CycleOptions(gamma, "gmres3", 2, 2, 4.5))
    assert res.converged
    return H.nlevels, {key: float(np.median(v)) for key, v in cond.items()}


@pytest.mark.parametrize("n,kh,kvar,gamma", [(64, 0.6, False, 1), (128, 0.6, False, 1), (128, 0.3, False, 1),
                                             (128, 0.6, True, 1), (64, 0.6, False, 2)])
def test_median_condition_of_the_normal_equations(n, kh, kvar, gamma, monkeypatch):
    nlev, med = _conditions(n, kh, kvar, gamma, monkeypatch)
    assert med[0, 1.0] <= 30 and med[0, 0.0] >= 500
    assert med[1, 0.0] <= 50 and med[1, 1.0] >= 1e4
    for lev in range(2, nlev - 1):
        assert med[lev, 0.0] <= 2500 and med[lev, 0.0] <= med[lev, 1.0], lev
