"""Batched ground states over the sizes where the kernel's paths change: more than eight sites (two
bytes of sites), one row or one column, rows longer than a CTA, both launch classes, and parameters
outside the range of the division-free eigenvalue test."""
from __future__ import annotations

import numpy as np
import pytest
import torch

from paper_1307_7542_gb300 import hub, workloads as W

pytestmark = pytest.mark.gpu

# (M, [(n_up, n_dn), ..]): sectors of at most 8192 states; 4900 and 2520 states are of the large class
JOBS = [(3, [(0, 0), (1, 0), (3, 3), (1, 2)]), (8, [(4, 4), (3, 5), (8, 1)]), (10, [(5, 1), (1, 5), (5, 0), (0, 10), (2, 2)]),
        (12, [(6, 0), (0, 6), (1, 4), (3, 1)]), (16, [(1, 2), (3, 0), (0, 4), (1, 0)])]


@pytest.mark.parametrize("scale", [1.0, 1e40])
@pytest.mark.parametrize("M,sectors", JOBS)
def test_batch_sizes(M, sectors, scale):
    bonds = W.ring_bonds(M)
    rng = np.random.default_rng(M)
    t, U, eps = (rng.normal(size=(2, n)) * scale for n in (len(bonds), M, M))
    jobs = [(a, b, p) for p in range(2) for a, b in sectors]
    nu, nd, jp = (np.array([j[k] for j in jobs], dtype=np.int32) for k in range(3))
    E, _, status = hub.hub_batch_ground(M, bonds, t, U, eps, nu, nd, jp, maxit=400, tol=1e-13 * scale)
    assert np.all(status >= 0), status
    for (a, b, p), e in zip(jobs, E):
        m = hub.Hubbard(M, a, b, bonds, t[p], U[p], eps[p])
        ref = m.ground(torch.from_numpy(W.normal(1, m.D)).cuda(), maxit=400, tol=1e-13 * scale)["E0"]
        m.close()
        # both stop at changes of 1e-13; a Lanczos value lies within a few changes of its limit and
        # the rounding of a step is 2^-52 of the operator's size (sum of |parameters| at most 60)
        assert abs(e - ref) <= 1e-10 * scale, (M, a, b, p, e, ref)
