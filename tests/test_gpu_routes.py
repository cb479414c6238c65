"""Products on each of the kernels that hub_apply and hub_apply_host choose between (FP64, fixed point,
double-float), the kernels asserted: sectors above the 2.2e7 terms up to which the FP64 kernel
takes every product, and above the 2^22 states from which host buffers are copied in row chunks.
Both sides of the window's edges on both routes that have a window, the parameter range, cancellation
and low parts of one sign, the row-chunk pipeline, and Lanczos runs in the shapes that only large
sectors take.  Reference: the oracle on sampled rows, and the FP64 kernel on all of them."""
import numpy as np
import pytest

from oracle import hub_oracle as O
from paper_1307_7542_gb300 import workloads as W

from helpers import abs_bound, assert_entrywise, device_bound

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def hub(cuda_ok):
    import __graft_entry__
    __graft_entry__.build()
    from paper_1307_7542_gb300 import hub as H
    return H


RING = (13, 5, 8, W.ring_bonds(13))                        # 1287 x 1287, both spins gathered
LONG = (18, 9, 2, W.square_bonds(3, 6, True))              # 48620 x 153, spin up combined
D_OF = {"ring": 1287 * 1287, "long": 48620 * 153}


def _unit(seed, n):
    """Magnitudes in [0.5, 1.5), random signs."""
    return W.uniform(seed, n, 0.5, 1.5) * np.where(W.uniform(seed + 1, n) < 0.5, -1.0, 1.0)


def _check(hub, shape, x, route, t=1.0, U=4.0, eps=None):
    """hub_apply in HUB_MODE_AUTO: the route, and every entry within the bound."""
    M, nu, nd, b = RING if shape == "ring" else LONG
    m = hub.Hubbard(M, nu, nd, b, t, U, eps)
    xd = torch.from_numpy(x).cuda()
    y = m.apply(xd)
    assert hub.hub_last_route(m.h) == route
    hub.hub_check(m.h)
    hub.hub_set_mode(m.h, hub.HUB_MODE_FP64)
    y64 = m.apply(xd)
    assert hub.hub_last_route(m.h) == hub.HUB_ROUTE_FP64
    if eps is None:
        # the FP64 product's own rounding: at most 80 operations of 2^-53 each
        assert bool(((y - y64).abs() <= 1.09e-13 * device_bound(m, xd, U) + 1e-300).all())
    m.close()
    om, B = O.Model(M, b, t, U, eps), O.basis(M, nu, nd)
    y, D = y.cpu().numpy(), len(x)
    for r0, r1 in ((0, 3000), (D // 3 - 1500, D // 3 + 1500), (D - 3000, D)):
        assert_entrywise(y[r0:r1], O.apply(om, B, x, rows=(r0, r1)), abs_bound(om, B, x, rows=(r0, r1)))


@pytest.mark.parametrize("shape", ["ring", "long"])
@pytest.mark.parametrize("kind,route", [("plain", "FIX"), ("spike 1e15", "DF"), ("spike 1e30", "FP64"),
                                        ("spike -1e200", "FP64")])
def test_spike(hub, shape, kind, route):
    """One entry far above the rest: the others are small on its grid (double-float), or further
    below it than the window reaches (FP64)."""
    x = _unit(40, D_OF[shape])
    if kind != "plain":
        x[len(x) // 3 + 5] = float(kind.split()[1])
    _check(hub, shape, x, getattr(hub, "HUB_ROUTE_" + route))


@pytest.mark.parametrize("shape", ["ring", "long"])
@pytest.mark.parametrize("log2_rel", [-60, -78, -90, -130, -1060])
@pytest.mark.parametrize("part", ["few", "most"])
def test_small_block(hub, shape, log2_rel, part):
    """A block of entries 2^log2_rel below the others, one in thirty (recomputed where their sums are
    small) or three in five (double-float); below 2^-80, and subnormals: FP64."""
    D = D_OF[shape]
    x = _unit(41, D)
    x[D // 3: D // 3 + (D // 30 if part == "few" else 3 * D // 5)] *= 2.0 ** log2_rel
    inside = hub.HUB_ROUTE_FIX if part == "few" else hub.HUB_ROUTE_DF
    _check(hub, shape, x, inside if log2_rel >= -78 else hub.HUB_ROUTE_FP64)


@pytest.mark.parametrize("shape", ["ring", "long"])
@pytest.mark.parametrize("scale_exp", [-820, 870, -830, 880])
@pytest.mark.parametrize("kind", ["even", "uneven"])
def test_vector_scale_limits(hub, shape, scale_exp, kind):
    """The largest entry just inside and just outside [2^-823, 2^877]."""
    D = D_OF[shape]
    x = _unit(42, D) if kind == "even" else _unit(42, D) * 2.0 ** np.floor(W.uniform(44, D, -60, 0))
    inside = hub.HUB_ROUTE_FIX if kind == "even" else hub.HUB_ROUTE_DF
    _check(hub, shape, np.ldexp(x, scale_exp), inside if abs(scale_exp) in (820, 870) else hub.HUB_ROUTE_FP64)


@pytest.mark.parametrize("t,U,eps,even,uneven", [
    (2.0 ** -15, 2.0 ** -13, 0.0, "FIX", "DF"), (3e4, 2.0 ** 15, 0.0, "FIX", "DF"),      # t inside [2^-16, 2^16]
    (2.0 ** -17, 2.0 ** -15, 0.0, "FIX", "FP64"), (1.0, 1e-6, 0.0, "FIX", "FP64"),       # t, U / t below it
    (1.0, 1e3, 0.0, "DF", "DF"), (1.0, 7e4, 0.0, "FP64", "FP64"),                        # too much for the grid
    (-0.7, 3.3, 0.0, "FIX", "DF"), (1.0, 0.0, 0.0, "FIX", "DF"), (1.0, 4.0, 3e-6, "FP64", "FP64")])
@pytest.mark.parametrize("kind", ["even", "uneven"])
def test_parameter_range(hub, t, U, eps, even, uneven, kind):
    D = D_OF["ring"]
    x = _unit(43, D)
    if kind == "uneven":
        x *= 2.0 ** np.floor(W.uniform(44, D, -78, 0))
    e = np.where(np.arange(13) % 3 == 0, eps, 0.0) if eps else None
    _check(hub, "ring", x, getattr(hub, "HUB_ROUTE_" + (even if kind == "even" else uneven)), t, U, e)


@pytest.mark.parametrize("shape", ["ring", "long"])
@pytest.mark.parametrize("lo_exp,route", [(-10, "DF"), (-6, "FIX")])
@pytest.mark.parametrize("kind", ["one_sign", "mixed", "zeros"])
def test_low_parts_and_cancellation(hub, shape, lo_exp, route, kind):
    """FP64 values whose FP32 low parts are nearly a unit of the high part's last place: of one sign,
    with both signs (sums that cancel), and with exact zeros (few enough not to look uneven)."""
    D = D_OF[shape]
    e = np.floor(W.uniform(50, D, lo_exp, 1)).astype(np.int64)
    x = np.ldexp(1.0 + np.floor(W.uniform(51, D) * (1 << 23)) / (1 << 23), e) + np.ldexp(0.999, e - 23)
    if kind == "mixed":
        x *= np.where(W.uniform(61, D) < 0.5, -1.0, 1.0)
    elif kind == "zeros":
        x[W.uniform(62, D) < 0.08] = 0.0
    _check(hub, shape, x, getattr(hub, "HUB_ROUTE_" + route))


def test_modes_differ(hub):
    """HUB_MODE_AUTO runs other kernels than HUB_MODE_FP64: not the same bits."""
    m = hub.Hubbard(*RING[:3], RING[3], 1.0, 4.0)
    x = torch.from_numpy(W.normal(1, m.D)).cuda()
    y = m.apply(x)
    hub.hub_set_mode(m.h, hub.HUB_MODE_FP64)
    assert not torch.equal(y, m.apply(x))
    m.close()


@pytest.mark.parametrize("shape", ["ring", "long"])
def test_captured_products(hub, shape):
    """A product captured in a CUDA graph (after a first one outside) takes each vector's own route on
    replay: bit for bit the call outside the graph."""
    M, nu, nd, b = RING if shape == "ring" else LONG
    m = hub.Hubbard(M, nu, nd, b, 1.0, 4.0)
    D = m.D
    x = torch.from_numpy(_unit(70, D)).cuda()
    y = m.apply(x)
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        m.apply(x, y, stream=side)
    kinds = [_unit(71, D), _unit(72, D) * 2.0 ** np.floor(W.uniform(73, D, -40, 0)), _unit(74, D)]
    kinds[2][5] = 1e200
    for v, route in zip(kinds, (hub.HUB_ROUTE_FIX, hub.HUB_ROUTE_DF, hub.HUB_ROUTE_FP64)):
        x.copy_(torch.from_numpy(v))
        y.zero_()
        graph.replay()
        torch.cuda.synchronize()
        out = y.clone()
        assert torch.equal(out, m.apply(x)) and hub.hub_last_route(m.h) == route
    m.close()


# ---------------------------------------------------------------------- host buffers in row chunks

@pytest.fixture(scope="module")
def big(hub):
    """14-site ring (7, 6): 3432 x 3003, an odd number of rows, 1.03e7 states."""
    m = hub.Hubbard(14, 7, 6, W.ring_bonds(14), 1.0, 4.0)
    yield m
    m.close()


def _single(hub, m, x):
    y = torch.empty_like(x).pin_memory()
    hub.hub_apply_host(m.h, x, y)
    return y


@pytest.mark.parametrize("case", ["plain", "max_in_first_chunk", "max_in_last_chunk", "outside"])
def test_row_chunks(hub, big, case):
    m = big
    x = torch.from_numpy(W.normal(17, m.D))
    if case == "max_in_first_chunk":
        x[: 2 * m.count_up] *= 64.0
    elif case == "max_in_last_chunk":
        x[-2 * m.count_up:] *= 1e6
    elif case == "outside":
        x[m.D // 3] = 1e280
    y = _single(hub, m, x.pin_memory()).cuda()
    assert hub.hub_last_route(m.h) == (hub.HUB_ROUTE_FP64 if case == "outside" else hub.HUB_ROUTE_DF)
    xd = x.cuda()
    hub.hub_set_mode(m.h, hub.HUB_MODE_FP64)
    y -= m.apply(xd)
    hub.hub_set_mode(m.h, hub.HUB_MODE_AUTO)
    assert bool((y.abs() <= 1.09e-13 * device_bound(m, xd, 4.0)).all())


def test_row_chunks_of_several_vectors(hub, big):
    """Five vectors in one call (both buffer pairs used twice and more; one whose largest exponent is
    in its last chunk, one outside the window), in place, and two after them on the same buffers:
    bit for bit one call per vector."""
    m = big
    X = torch.stack([torch.from_numpy(W.normal(30 + v, m.D)) for v in range(5)])
    X[1, -2 * m.count_up:] *= 1e6
    X[2, m.D // 3] = 1e280
    X = X.pin_memory()
    ref = torch.stack([_single(hub, m, X[v]) for v in range(5)])
    Y = torch.empty_like(X).pin_memory()
    hub.hub_apply_host_many(m.h, 5, X, Y)
    assert hub.hub_last_route(m.h) == hub.HUB_ROUTE_DF
    assert torch.equal(Y, ref)
    Z = X.clone().pin_memory()
    hub.hub_apply_host_many(m.h, 5, Z, Z)
    assert torch.equal(Z, ref)
    Y.zero_()
    hub.hub_apply_host_many(m.h, 2, X[3:], Y[3:])
    assert torch.equal(Y[3:], ref[3:]) and not bool(Y[:3].any())


# ------------------------------------------------------------- Lanczos runs of the large shapes

@pytest.mark.parametrize("U", [4.0, -3.3])
@pytest.mark.parametrize("shape", ["planes of 14400", "both combined"])
def test_lanczos_of_large_shapes(hub, shape, U):
    """Both spins gathered from the larger staged planes (3432 x 3003 states); both spins as row
    combinations (20349 x 20349, odd counts, different bases): alpha, beta and the Ritz vector equal
    the FP64 driver's up to rounding, and a product lies within the bound."""
    M, nu, nd = (14, 7, 6) if shape == "planes of 14400" else (21, 5, 16)
    steps = 8 if M == 14 else 4
    m = hub.Hubbard(M, nu, nd, W.ring_bonds(M), 1.25, U)
    g = torch.Generator(device="cuda").manual_seed(3)
    x = torch.randn(m.D, dtype=torch.float64, device="cuda", generator=g)
    out, y = [], []
    for mode in (hub.HUB_MODE_AUTO, hub.HUB_MODE_FP64):
        hub.hub_set_mode(m.h, mode)
        r = m.ground(x, maxit=steps, tol=0.0, want_psi=True)
        out.append((*hub.hub_lanczos_coeffs(m.h), r["psi"]))
        y.append(m.apply(x))
        assert hub.hub_last_route(m.h) == (hub.HUB_ROUTE_FIX if mode == hub.HUB_MODE_AUTO else hub.HUB_ROUTE_FP64)
    (a0, b0, p0), (a1, b1, p1) = out
    scale = max(np.abs(a1).max(), b1.max())
    assert np.abs(a0 - a1).max() <= 1e-13 * scale and np.abs(b0 - b1).max() <= 1e-13 * scale
    p0 -= p1
    assert float(p0.norm()) <= 1e-12
    y[0] -= y[1]
    del out, p0, p1, y[1]
    assert bool((y[0].abs() <= 1.09e-13 * device_bound(m, x, abs(U))).all())
    m.close()
