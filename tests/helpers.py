"""Helpers shared by the parity tests: build both sides from one workload description."""
import numpy as np

from oracle import hub_oracle as O


def oracle_model(w):
    return O.Model(w["M"], w["bonds"], w["t"], w["U"], w.get("eps"))


def abs_bound(model, B, x, rows=None):
    """(|H| |x|)_n over rows (r0, r1): the scale of the per-entry tolerance."""
    return O.apply(model, B, x, rows=rows, absolute=True)


def assert_entrywise(y, ref, bound, rtol=1e-13):
    """|y - ref| <= rtol * (|H||x|) + 1e-300 for every entry (per-entry tolerance of the apply)."""
    err = np.abs(y - ref)
    bad = err > rtol * bound + 1e-300
    if bad.any():
        k = int(np.argmax(err / (bound + 1e-300)))
        raise AssertionError(f"{int(bad.sum())} entries exceed {rtol:g}*|H||x|; worst at {k}: "
                             f"got {y[k]!r}, want {ref[k]!r}, bound {bound[k]!r}")


def device_bound(m, x, U):
    """(|H| |x|) of every entry on the device, for vectors that the oracle would take too long for:
    the spins' CSR matrices without their signs, and a uniform U >= 0."""
    import torch
    A = []
    for spin, n in ((0, m.count_up), (1, m.count_dn)):
        rp, cols, vals = m.csr(spin)
        A.append(torch.sparse_csr_tensor(torch.from_numpy(rp.astype(np.int64)), torch.from_numpy(cols.astype(np.int64)),
                                         torch.from_numpy(np.abs(vals)), size=(n, n)).cuda())
    X = x.abs().view(m.count_dn, m.count_up)
    out = A[1] @ X
    out += (A[0] @ X.T.contiguous()).T
    bits = [torch.from_numpy(((m.basis(s).astype(np.int64)[:, None] >> np.arange(m.M)) & 1).astype(np.float64)).cuda()
            for s in (0, 1)]
    both = bits[1] @ bits[0].T
    both *= U
    out += both * X
    return out.reshape(-1)
