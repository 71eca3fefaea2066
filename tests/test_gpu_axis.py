"""Roots next to the real axis and the root 0 of the fixed-point descents
(csrc/mt_descent.cuh): a fixed-point coordinate has an absolute error however
small it is, binary64's shrinks with it, so small components are held against
the binary64 Newton step, written out in numpy."""
from __future__ import annotations

import numpy as np
import pytest

from hostpool import polish_all

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mt():
    import torch
    assert torch.cuda.is_available()
    import paper_2402_06083_gb300 as pkg
    return pkg


def _step64(kind, n, l, z):
    """One Newton step in binary64 from every point."""
    m, cap = (n, 0) if kind == "hyp" else (l + n - 1, l - 1)
    p, d = np.zeros_like(z), np.zeros_like(z)
    cp = cd = 0.0
    for k in range(1, m + 1):
        d = 2 * p * d + 1
        p = p * p + z
        if k == cap:
            cp, cd = p, d
    return z - (p + cp) / (d + cd)


def _errors(z, x4):
    return np.abs((x4[:, 0] - z.real) + x4[:, 1]), np.abs((x4[:, 2] - z.imag) + x4[:, 3])


def _rms(e):
    return float(np.sqrt(np.mean(e ** 2)))


@pytest.mark.parametrize("kind,n,l,prec", [("hyp", 13, 0, "fp64"), ("hyp", 18, 0, "fp64"), ("hyp", 20, 0, "fp64"),
                                           ("mis", 5, 8, "fp64"), ("mis", 10, 6, "fp64"), ("mis", 6, 5, "batch"),
                                           ("hyp", 23, 0, "mixed"), ("hyp", 25, 0, "mixed")])
def test_roots_as_close_as_binary64(mt, kind, n, l, prec):
    """rms errors against binary128: of all sampled roots no larger than the
    binary64 step's from the exact root; of the imaginary parts below 2^-13, and
    of those below 1e-6, no more than twice the binary64 step's (the same
    arithmetic up to fused multiply-adds); the root 0 within tol^2 = 1e-26, what
    a last step below tol = 1e-13 leaves of it."""
    if prec == "batch":
        roots, _, off, _, pairs = mt.split_misiurewicz_batch(12)
        p = pairs.index((l, n))
        z = roots[off[p]:off[p + 1]]
    elif kind == "hyp":
        z = mt.split_hyperbolic(n, prec).roots
    else:
        z = mt.split_misiurewicz(l, n, prec).roots
    z = z.cpu().numpy()
    assert np.abs(z).min() <= 1e-26
    small = np.nonzero((np.abs(z.imag) < 2.0 ** -13) & (z.imag > 0))[0][:6000]
    pick = np.unique(np.concatenate([np.linspace(0, z.size - 1, min(z.size, 6000)).astype(int), small]))
    z = z[pick]
    z = z[np.abs(z) > 0.1]  # the root 0 is held to its own bound above
    _, _, x4 = polish_all(kind, n, z, l=l)
    re, im = _errors(z, x4)
    ref = _step64(kind, n, l, x4[:, 0] + 1j * x4[:, 2])
    re64, im64 = _errors(ref, x4)
    assert _rms(np.hypot(re, im)) <= _rms(np.hypot(re64, im64))
    for hi in (2.0 ** -13, 1e-6):
        g = (np.abs(x4[:, 2]) < hi) & (x4[:, 2] != 0)
        if g.any():
            assert _rms(im[g]) <= 2 * _rms(im64[g]), (hi, int(g.sum()), _rms(im[g]), _rms(im64[g]))


@pytest.mark.parametrize("kind,n,l", [("hyp", 1, 0), ("hyp", 2, 0), ("hyp", 4, 0), ("hyp", 10, 0), ("hyp", 20, 0),
                                      ("mis", 3, 3), ("mis", 1, 2), ("mis", 6, 5)])
def test_descents_to_zero(mt, kind, n, l):
    """Starts from 1e-25 to 0.1 around the root 0, more than a block's and
    fewer than a warp's worth of them: within tol^2 of it."""
    import torch
    rng = np.random.default_rng(n)
    r = 10.0 ** rng.uniform(-25, -1, 3001) * np.exp(2j * np.pi * rng.uniform(0, 1, 3001))
    for z in (np.concatenate([r, r.real, 1j * r.imag, [0.0, 1e-300, -1e-300j]]), r[:7]):
        out, status, _ = mt.descend(kind, n, torch.tensor(z, device="cuda"), l=l)
        out, status = out.cpu().numpy(), status.cpu().numpy()
        near = (status == 0) & (np.abs(out) < 0.1)
        assert near.sum() >= 0.9 * z.size
        assert np.abs(out[near]).max() <= 1e-26
