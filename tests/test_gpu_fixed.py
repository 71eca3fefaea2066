"""The binary64 tier's fixed-point orbit (csrc/mt_fix.cuh) where it can go
wrong: levels at the edges of its ranges (12 and 200, beyond which the walk
takes fewer fraction bits or binary64), starts inside, at and outside the
range |Re|, |Im| < 4, the shortest orbits, and orbits that leave the range."""
from __future__ import annotations

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mt():
    import torch
    assert torch.cuda.is_available()
    import paper_2402_06083_gb300 as pkg
    return pkg


def _t(z):
    import torch
    return torch.tensor(np.asarray(z, dtype=np.complex128), device="cuda")


@pytest.mark.parametrize("lam", [5.0, 11.9, 12.0, 12.1, 199.0, 200.0, 201.0, 1000.0])
@pytest.mark.parametrize("kind,n,l", [("hyp", 1, 0), ("hyp", 2, 0), ("hyp", 3, 0), ("hyp", 8, 0), ("hyp", 11, 0),
                                      ("mis", 1, 2), ("mis", 4, 3), ("mis", 2, 7), ("q", 3, 3)])
def test_level_line_at_the_edges_of_the_ranges(mt, lam, kind, n, l):
    """Start s satisfies P = lambda0 i^s to the walk's tolerance (1e-2 of a
    sub-step of 1/8 turn, a quarter of it in P's relative error: 2e-3 and
    more is left to the last correction), for every range of the level."""
    if kind != "hyp" and lam < 12:
        pytest.skip("below the critical values of the family")
    g, st = mt.level_line(kind, n, l=l, lambda0=lam)
    assert st["walk_fail"] == 0
    v = mt.evaluate(kind, n, g, l=l).cpu().numpy()[:, 0] if kind != "q" else None
    if v is None:  # evaluate gives q in product form: the same value
        v = mt.evaluate("q", n, g, l=l).cpu().numpy()[:, 0]
    want = lam * (1j ** (np.arange(v.size) % 4))
    assert np.max(np.abs(v - want)) < 1e-2 * lam


@pytest.mark.parametrize("kind,n,l", [("hyp", 1, 0), ("hyp", 2, 0), ("hyp", 5, 0), ("hyp", 13, 0), ("mis", 1, 2),
                                      ("mis", 3, 2), ("mis", 2, 9), ("mis", 8, 4)])
def test_descents_from_inside_and_outside_the_range(mt, kind, n, l):
    """Starts spread over |Re|, |Im| < 6 (the range ends at 4), on the axes and
    at the edge: what converges is a root, to binary64 rounding (a binary128
    polish moves it less than 4e-16 |z| + 4e-16, two roundings of the result
    and of its last step)."""
    rng = np.random.default_rng(7 + n + 31 * l)
    z = rng.uniform(-6, 6, 1000) + 1j * rng.uniform(-6, 6, 1000)
    z = np.concatenate([z, 0.4 * z, [4.0, -4.0, 4j, np.nextafter(4.0, 0), np.nextafter(4.0, 5) * 1j, 0.3, -2.0, 1e-30,
                                     -1.75, 2.0 - 2.0j, 3.9999999 + 3.9999999j]])
    out, status, _ = mt.descend(kind, n, _t(z), l=l)
    out, status = out.cpu().numpy(), status.cpu().numpy()
    conv = out[status == 0]
    assert conv.size >= 8
    for c in conv[:: max(1, conv.size // 200)]:
        _, disp = oracle.polish(kind, n, c, steps=3, l=l)
        assert disp <= 4e-16 * abs(c) + 4e-16, (c, disp)


@pytest.mark.parametrize("kind,n,l,exps", [("hyp", 1, 0, (18, 19, 20, 38, 100, 150, 300)), ("hyp", 2, 0, (18, 20, 39, 100)),
                                           ("hyp", 3, 0, (18, 20, 39, 60)), ("hyp", 4, 0, (18, 20, 30)),
                                           ("mis", 1, 2, (18, 20, 39, 100)), ("mis", 2, 2, (18, 20, 39, 60))])
def test_descents_from_far_away(mt, kind, n, l, exps):
    """From |z0| so large that z0 alone decides (P ~ z^d), a Newton step is
    (1 - 1/d) z: 20 of them (the cap), no long jump; p_1 = z is at its root
    after one.  Relative error 20 binary64 steps of a few roundings each, and the
    next term of P, at most 2 / |z| a step and so 4 d over the last point."""
    z = np.array([s * 10.0 ** e for e in exps for s in (1, -1, 1j, 0.6 - 0.8j)])
    out, status, _ = mt.descend(kind, n, _t(z), l=l)
    out, status = out.cpu().numpy(), status.cpu().numpy()
    d = 2 ** (n - 1) if kind == "hyp" else 2 ** (l + n - 2)
    if d == 1:
        assert np.all(status == 0) and np.all(out == 0)
    else:
        assert np.all(status == 2)
        err = np.abs(out / (z * (1 - 1 / d) ** 20) - 1)
        assert np.all(err < 20 * 32 * 2.0 ** -53 + 4 * d / np.abs(out))
