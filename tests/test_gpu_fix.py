"""The fixed-point product and Lanczos (csrc/hub_fix.cu): every shape (both spins gathered, both
combined, one of each; t uniform or not), and the routes a vector can take (fixed point, entries
recomputed, double-float, FP64), against the oracle's per-entry bound."""
import numpy as np
import pytest

from oracle import hub_oracle as O
from paper_1307_7542_gb300 import workloads as W

from helpers import abs_bound, assert_entrywise

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def hub(cuda_ok):
    import __graft_entry__
    __graft_entry__.build()
    from paper_1307_7542_gb300 import hub as H
    return H


# more than 2.2e7 terms each, so that hub_apply does not take the FP64 kernel: odd x odd counts
# with both spins gathered (1287 x 2002 and 1716 x 1716), long rows with one spin combined, either
# way round (48620 x 153)
SHAPES = {
    "ring13_58": (13, 5, 8, W.ring_bonds(13)),
    "ring14_95": (14, 9, 5, W.ring_bonds(14)),
    "long_up": (18, 9, 2, W.square_bonds(3, 6, True)),
    "long_dn": (18, 2, 9, W.square_bonds(3, 6, True)),
}


def _vector(kind, D):
    x = W.normal(11, D)
    if kind == "few_small":        # a few entries (and all their neighbours' sums) far below the largest
        x[D // 3: D // 3 + 3000] *= 1e-9
    elif kind == "wide":           # most entries small: the double-float kernels
        x *= 10.0 ** W.uniform(5, D, -12.0, 0.0)
    elif kind == "sparse":
        x[W.uniform(6, D) > 0.01] = 0.0
    elif kind == "one":            # every entry at the top of the grid, all ones below the leading bit
        x = np.copysign(np.full(D, np.nextafter(2.0, 1.0)), x)
    elif kind == "constant":
        x = np.full(D, 1.0 - 2.0 ** -28)
    elif kind == "outside":        # outside the double-float window: FP64
        x[7] = 1e-200
    return x


@pytest.mark.parametrize("kind", ["normal", "few_small", "wide", "sparse", "one", "constant", "outside"])
@pytest.mark.parametrize("shape", ["ring13_58", "long_up"])
def test_apply_routes(hub, shape, kind):
    M, nu, nd, b = SHAPES[shape]
    m = hub.Hubbard(M, nu, nd, b, -0.7, 3.3)
    om = O.Model(M, b, -0.7, 3.3)
    B = O.basis(M, nu, nd)
    x = _vector(kind, m.D)
    y = m.apply(torch.from_numpy(x).cuda()).cpu().numpy()
    m.close()
    assert_entrywise(y, O.apply(om, B, x), abs_bound(om, B, x))


@pytest.mark.parametrize("shape", sorted(SHAPES))
@pytest.mark.parametrize("disorder", [False, True])
def test_apply_shapes(hub, shape, disorder):
    """Uniform t, U = 4 (an integer diagonal), and per-bond t, per-site U, site energies."""
    M, nu, nd, b = SHAPES[shape]
    if disorder:
        t, U, eps = W.uniform(1, len(b), -1.3, 1.3), W.uniform(2, M, -2.0, 8.0), W.uniform(3, M, -0.5, 0.5)
    else:
        t, U, eps = np.ones(len(b)), np.full(M, 4.0), np.zeros(M)
    m = hub.Hubbard(M, nu, nd, b, t, U, eps)
    om = O.Model(M, b, t, U, eps)
    B = O.basis(M, nu, nd)
    x = W.normal(4, m.D)
    xd = torch.from_numpy(x).cuda()
    y = m.apply(xd).cpu().numpy()
    # an output vector on an odd 8-byte boundary takes the narrow stores: the same bits
    pad = torch.empty(m.D + 1, dtype=torch.float64, device="cuda")
    y2 = m.apply(xd, pad[1:]).cpu().numpy()
    m.close()
    assert np.array_equal(y, y2)
    assert_entrywise(y, O.apply(om, B, x), abs_bound(om, B, x))


@pytest.mark.parametrize("U", [0.0, -3.0, 7.25, 4000.0])
@pytest.mark.parametrize("shape", ["ring", "disordered", "long_up", "long_dn"])
def test_lanczos_against_fp64(hub, shape, U):
    """alpha, beta and the Ritz vector of 12 steps equal the FP64 driver's up to rounding."""
    if shape in ("ring", "disordered"):
        M, nu, nd, b = 9, 4, 3, W.ring_bonds(9)
    else:
        M, nu, nd, b = (18, 9, 1, W.square_bonds(3, 6, True)) if shape == "long_up" else (18, 1, 9,
                                                                                         W.square_bonds(3, 6, True))
    t = W.uniform(8, len(b), 0.2, 1.5) if shape == "disordered" else 1.25
    m = hub.Hubbard(M, nu, nd, b, t, U, W.uniform(9, M, -1.0, 1.0) if shape == "disordered" else None)
    hub.hub_set_small_dim(m.h, 0)
    x = torch.from_numpy(W.normal(2, m.D)).cuda()
    out = []
    for mode in (hub.HUB_MODE_AUTO, hub.HUB_MODE_FP64):
        hub.hub_set_mode(m.h, mode)
        r = m.ground(x, maxit=12, tol=0.0, want_psi=True)
        out.append((*hub.hub_lanczos_coeffs(m.h), r["psi"].cpu().numpy()))
    m.close()
    (a0, b0, p0), (a1, b1, p1) = out
    scale = max(np.abs(a1).max(), b1.max())
    assert np.abs(a0 - a1).max() <= 1e-12 * scale and np.abs(b0 - b1).max() <= 1e-12 * scale
    assert np.linalg.norm(p0 - p1) <= 1e-11


def test_host_buffers_in_row_chunks(hub):
    """A sector large enough for the row-chunk pipeline (3003 x 3003): within the bound of
    hub_apply's result, and several vectors in one call bit for bit equal to one call each."""
    m = hub.Hubbard(14, 6, 6, W.ring_bonds(14), 1.0, 4.0)
    om, B = O.Model(14, W.ring_bonds(14), 1.0, 4.0), O.basis(14, 6, 6)
    X = torch.from_numpy(np.stack([W.normal(s, m.D) for s in (1, 2)]))
    X[1, -5:] *= 1e6                       # the largest exponent in the last chunk
    X = X.pin_memory()
    Y = torch.empty_like(X).pin_memory()
    hub.hub_apply_host_many(m.h, 2, X, Y)
    for v in range(2):
        y1 = torch.empty(m.D, dtype=torch.float64).pin_memory()
        hub.hub_apply_host(m.h, X[v], y1)
        assert torch.equal(Y[v], y1)
        x = X[v].numpy()
        assert_entrywise(y1.numpy(), O.apply(om, B, x), abs_bound(om, B, x))
    m.close()
