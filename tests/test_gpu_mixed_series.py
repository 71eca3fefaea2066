"""The mixed tier's descents on shared anchors and the anchors' series
(csrc/mt_mixed.cu): orbit lengths on both sides of the rules (general loop
below 16, fixed lengths from 16, shared anchors, series and the fixed-point
finish from 23), starts that do not fill a
group or a queue range, and denser starts, whose groups span less of a turn."""
from __future__ import annotations

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mt():
    import torch
    assert torch.cuda.is_available()
    import paper_2402_06083_gb300 as pkg
    return pkg


@pytest.mark.parametrize("n,kw", [(1, {}), (2, {}), (3, {}), (6, {}), (7, {}), (13, {}), (15, {}), (16, {}), (17, {}),
                                  (19, {}), (20, {}), (21, {}), (22, {}), (23, {}), (24, {}), (25, {}), (23, {"M": 16, "c_L": 8}), (23, {"M": 8, "c_L": 2}),
                                  (23, {"lambda0": 5.8}), (23, {"stream_pieces": 4}), (20, {"M": 16, "c_L": 8}), (20, {"M": 8, "c_L": 2}),
                                  (20, {"lambda0": 5.8}), (18, {"stream_pieces": 4}), (21, {"stream_pieces": 2})])
def test_first_attempt_finds_every_root(mt, n, kw):
    """The first attempt alone (no binary64 repeat) is complete and certified,
    and its roots are the binary64 tier's to the Newton tolerance 1e-13 (each
    tier stops within it)."""
    few = kw.get("c_L") == 2  # half the starts: roots are missing, none is wrong
    r = mt.split_hyperbolic(n, "mixed", max_retries=-1, check_status=not few, **kw)
    st = r.stats
    assert st["n_cert_pass"] == st["n_roots"] and st["walk_fail"] == 0
    if few:
        return
    assert st["prec_used"] == 1 and st["n_roots"] == 2 ** (n - 1)
    a, b = r.roots.cpu().numpy(), mt.split_hyperbolic(n).roots.cpu().numpy()
    assert np.max(np.abs(a - b)) < 1e-13


@pytest.mark.parametrize("level", [5.935373876248844, 5.287923032490966, 5.828942694987802, 5.27979241373518,
                                   5.224064323734339, 5.820812076232031, 5.942318253715001, 5.212828084963434])
def test_close_pairs_at_the_tip_are_told_apart(mt, level):
    """Levels of p_24 whose line sends two or three starts to one root of a real
    pair at the left tip, 2e-13 to 5e-12 apart where starts lie 4e-10 to 3e-9
    apart: around an anchor of its own each start reaches its root, around a
    neighbour's one of the pair was missed."""
    st = mt.split_hyperbolic(24, "mixed", max_retries=-1, check_status=False, lambda0=level).stats
    assert st["n_roots"] == st["n_cert_pass"] == 2 ** 23
