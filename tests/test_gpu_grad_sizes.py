"""Bilinear forms a^T (dH/dtheta) b over row lengths, chunk edges and entry counts of the kernel.

H is linear in its parameters, so each form is the product of the model whose other parameters
are zero: a . (H(theta = e_k) b), one FP64 product per parameter.
"""
from __future__ import annotations

import numpy as np
import pytest
import torch

from paper_1307_7542_gb300 import hub, workloads as W

pytestmark = pytest.mark.gpu

# (M, n_up, n_dn): one state; one row; one column; rows of 255/256/257-like and 512+ lengths; hopping
# rows of more than eight entries; rows too long to stage beside the bins (48620 states)
SHAPES = [(2, 2, 0), (8, 0, 4), (8, 4, 0), (10, 5, 2), (11, 5, 1), (12, 6, 3), (12, 5, 6), (13, 6, 2), (16, 7, 2),
          (18, 9, 1)]


@pytest.mark.parametrize("M,n_up,n_dn", SHAPES)
def test_bilinear_forms(M, n_up, n_dn):
    bonds = W.square_bonds(3, 4, periodic=True) if M == 12 else W.ring_bonds(M)
    nb = len(bonds)
    rng = np.random.default_rng(M + 31 * n_up + 977 * n_dn)
    t, U, eps = rng.normal(size=nb), rng.normal(size=M), rng.normal(size=M)
    m = hub.Hubbard(M, n_up, n_dn, bonds, t, U, eps)
    b = torch.from_numpy(rng.normal(size=m.D)).cuda()
    a = torch.from_numpy(rng.normal(size=m.D)).cuda()
    _, dt, dU, de = m.vjp(a, b)
    got = np.concatenate([np.asarray(v).ravel() for v in (dt, dU, de)])
    m.close()
    z = np.zeros(nb + 2 * M)
    worst = 0.0
    for k in range(nb + 2 * M):
        e = z.copy()
        e[k] = 1.0
        u = hub.Hubbard(M, n_up, n_dn, bonds, e[:nb], e[nb:nb + M], e[nb + M:])
        y = torch.empty_like(b)
        u.apply(b, y)
        u.close()
        ref, size = float(torch.dot(a, y)), float(torch.dot(a.abs(), y.abs()))
        # both sides add up to D terms of this total size; their roundings (2^-53 each, relative to
        # partial sums no larger than it) add like a random walk: eight standard deviations, and a few
        tol = 2.0 ** -53 * (64 + 8 * np.sqrt(len(b))) * max(size, 1e-300)
        worst = max(worst, abs(got[k] - ref) / tol)
        assert abs(got[k] - ref) <= tol, (k, got[k], ref, tol)
    print(f"worst {worst:.3f} of the bound")
