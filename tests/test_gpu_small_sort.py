"""Lists that are sorted by one thread-block cluster and scanned by one block
(csrc/mt_dedup.cu): sizes at the edges of a warp's, a block's and the cluster's
run and one beyond, where the pass-wise sort takes over.  The certificate of a
shuffled list, with exact ties, has to be that of the same list in every order."""
from __future__ import annotations

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2, 31, 33, 1024, 1025, 8191, 8192, 8193, 16385, 32768, 32769, 40959, 40960, 40961])
def test_certificate_in_any_order(n):
    import torch
    import paper_2402_06083_gb300 as mt
    assert torch.cuda.is_available()
    roots = mt.split_hyperbolic(18, "mixed").roots
    z = roots[:n].clone()
    perm = torch.from_numpy(np.random.RandomState(n).permutation(n)).cuda()
    p = torch.from_numpy(np.random.RandomState(n).permutation(n)).cuda()
    (ok, rad, k), (ok2, rad2, k2) = mt.certify("hyp", 18, z), mt.certify("hyp", 18, z[p].contiguous())
    assert k == k2 and torch.equal(ok[p], ok2) and torch.equal(rad[p], rad2)
    # disjoint disks: no radius above half the distance to the nearest other root
    for i in range(0, min(n, 8193), 1024):
        d = (z[i:i + 1024, None] - z[None, :]).abs()
        d[torch.arange(d.shape[0]), torch.arange(i, i + d.shape[0])] = float("inf")
        assert torch.all(rad[i:i + 1024] <= d.min(1).values / 2)
