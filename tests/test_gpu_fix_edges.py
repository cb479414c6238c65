"""Edges of the fixed-point path (csrc/hub_fix.cu): more entries to recompute than its list holds; start
vectors of one sign, of zeros, and uneven ones; scratch vectors that another path allocated."""
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


def _dense(csr, n):
    rp, cols, vals = csr
    A = np.zeros((n, n))
    A[np.repeat(np.arange(n), np.diff(rp)), cols] = vals
    return A


def test_more_small_sums_than_the_list_holds(hub):
    """U = 0 and a vector in the null spaces of both spins' hopping matrices: entries of ordinary
    size, yet both hopping sums of every entry vanish, so that all of them ask to be computed
    again, far more than the list holds (1 in 64)."""
    M, nu, nd, b = 14, 4, 6, W.ring_bonds(14)
    m = hub.Hubbard(M, nu, nd, b, 1.0, 0.0)
    null = []
    for spin, n in ((0, m.count_up), (1, m.count_dn)):
        ev, v = np.linalg.eigh(_dense(m.csr(spin), n))
        null.append(v[:, np.abs(ev) < 1e-9])
    g = W.normal(21, null[0].shape[1] * null[1].shape[1]).reshape(null[1].shape[1], null[0].shape[1])
    x = (null[1] @ g @ null[0].T).ravel()
    x /= np.abs(x).max()
    y = m.apply(torch.from_numpy(x).cuda()).cpu().numpy()
    m.close()
    om, B = O.Model(M, b, 1.0, 0.0), O.basis(M, nu, nd)
    bound = abs_bound(om, B, x)
    ref = O.apply(om, B, x)
    assert (np.abs(ref) < 1e-10 * bound).mean() > 0.5 and (np.abs(x) > 2.0 ** -8).mean() > 0.9
    assert_entrywise(y, ref, bound)


@pytest.mark.parametrize("M,nu,nd", [(13, 5, 8), (14, 9, 5), (14, 7, 7)])
@pytest.mark.parametrize("top", [1.0001, 1.9999])
def test_first_coefficient_of_a_positive_vector(hub, M, nu, nd, top):
    """alpha_1 = <x, H x> / <x, x> where every entry is positive, so that errors of one sign in H x
    add up: within 5e-16 of the operator's scale of the sum in long double.  top: the largest
    entry's place between two powers of two, sixteen times the rms (a few roundings of FP64 numbers
    of at most half the scale: 3 * 1.1e-16)."""
    m = hub.Hubbard(M, nu, nd, W.ring_bonds(M), 1.0, 4.0)
    x = np.abs(W.normal(7, m.D))
    x *= 1.0 / np.sqrt((x * x).mean())
    x[m.D // 3] = 16.0
    x *= top / 16.0
    xd = torch.from_numpy(x).cuda()
    m.ground(xd, maxit=1, tol=0.0)
    alpha = hub.hub_lanczos_coeffs(m.h)[0][0]
    hub.hub_set_mode(m.h, hub.HUB_MODE_FP64)
    y = m.apply(xd).cpu().numpy()
    rows = sum(hub.hub_csr_info(m.h, s)[1] for s in (0, 1))
    m.close()
    ref = np.sum(x * y, dtype=np.longdouble) / np.sum(x * x, dtype=np.longdouble)
    assert abs(float(alpha - ref)) <= 5e-16 * (rows + 4.0 * min(nu, nd))


@pytest.mark.parametrize("driver", ["fixed", "fp64", "small"])
def test_zero_and_infinite_start_vectors(hub, driver):
    """hub_green_coeffs of c psi0 = 0 is the empty continued fraction; a ground state from zeros,
    and either from infinities, is refused."""
    m = hub.Hubbard(9, 4, 3, W.ring_bonds(9), 1.0, 4.0)
    if driver != "small":
        hub.hub_set_small_dim(m.h, 0)
    if driver == "fp64":
        hub.hub_set_mode(m.h, hub.HUB_MODE_FP64)
    x = torch.zeros(m.D, dtype=torch.float64, device="cuda")
    a, b, n2 = hub.hub_green_coeffs(m.h, x, 5)
    assert len(a) == 0 and len(b) == 0 and n2 == 0.0
    with pytest.raises(hub.HubError) as e:
        hub.hub_lanczos_ground(m.h, x, 5, 0.0)
    assert e.value.code == hub.HUB_ERR_ARG
    x[3] = float("inf")
    for call in (lambda: hub.hub_green_coeffs(m.h, x, 5), lambda: hub.hub_lanczos_ground(m.h, x, 5, 0.0)):
        with pytest.raises(hub.HubError) as e:
            call()
        assert e.value.code == hub.HUB_ERR_ARG
    m.close()


def test_scratch_vectors_of_the_double_float_path(hub):
    """17 sites (8, 7), 24310 x 19448: both spins too long to stage.  A product at strong coupling
    allocates the transposed scratch vectors for the double-float kernels; the fixed-point product
    after it takes them for vectors in the other order, whose padded rows need 311,168 bytes more."""
    m = hub.Hubbard(17, 8, 7, W.ring_bonds(17), 1.0, 4000.0)
    g = torch.Generator(device="cuda").manual_seed(5)
    x = torch.randn(m.D, dtype=torch.float64, device="cuda", generator=g)
    y = m.apply(x)
    hub.hub_set_U(m.h, [4.0])
    m.apply(x, y)
    hub.hub_set_mode(m.h, hub.HUB_MODE_FP64)
    y -= m.apply(x)
    bound = device_bound(m, x, 4.0)
    m.close()
    assert bool((y.abs() <= 1.1e-13 * bound).all())       # a tenth for the FP64 product's own rounding


def _run(hub, m, x, steps):
    r = m.ground(x, maxit=steps, tol=0.0, want_psi=True)
    return (*hub.hub_lanczos_coeffs(m.h), r["psi"])


def _same_run(one, two, tol=1e-12):
    (a0, b0, p0), (a1, b1, p1) = one, two
    scale = max(np.abs(a1).max(), b1.max())
    assert np.abs(a0 - a1).max() <= tol * scale and np.abs(b0 - b1).max() <= tol * scale
    assert float((p0 - p1).norm()) <= 10 * tol


@pytest.mark.parametrize("kind", ["single", "decades", "top", "power", "negative_top"])
def test_start_vectors_on_the_grid(hub, kind):
    """Start vectors of a single entry, of entries over nine decades, and with a largest entry just below
    and at a power of two (the ends of the range that is scaled to the top of the grid): the FP64
    driver's alpha, beta and Ritz vector."""
    m = hub.Hubbard(9, 4, 5, W.ring_bonds(9), 1.0, 4.0)
    hub.hub_set_small_dim(m.h, 0)
    x = W.normal(2, m.D)
    if kind == "single":
        x[:] = 0.0
        x[17] = -3.0
    elif kind == "decades":
        x *= 10.0 ** W.uniform(3, m.D, -9.0, -3.0)
        x[m.D // 2] = 1.0
    elif kind == "power":
        x = np.copysign(np.full(m.D, 4.0), x)
    else:
        x = np.copysign(np.full(m.D, np.nextafter(4.0, 0.0)), x if kind == "top" else np.full(m.D, -1.0))
    x = torch.from_numpy(x).cuda()
    one = _run(hub, m, x, 12)
    n2 = hub.hub_green_coeffs(m.h, x, 2)[2]
    hub.hub_set_mode(m.h, hub.HUB_MODE_FP64)
    _same_run(one, _run(hub, m, x, 12))
    m.close()
    assert abs(n2 / float(torch.dot(x, x)) - 1.0) <= 1e-14


def test_vector_that_becomes_uneven(hub):
    """U = 0, the start vector an eigenvector with one entry changed: its largest entry is 20 times
    the rms, but what the first step leaves is the changed entry's neighbourhood, 2^10 times the rms."""
    M, nu, nd = 13, 5, 8
    m = hub.Hubbard(M, nu, nd, W.ring_bonds(M), 1.0, 0.0)
    v = [np.linalg.eigh(_dense(m.csr(s), n))[1][:, 0] for s, n in ((0, m.count_up), (1, m.count_dn))]
    x = np.outer(v[1], v[0])
    x[600, 700] += 20.0 * np.sqrt((x * x).mean())
    x = torch.from_numpy(x.ravel().copy()).cuda()
    one = _run(hub, m, x, 8)
    hub.hub_set_mode(m.h, hub.HUB_MODE_FP64)
    _same_run(one, _run(hub, m, x, 8))
    m.close()


def test_short_of_memory(hub):
    """Room for three and a half more vectors: the product falls back on the FP64 kernel (room for
    one), the Lanczos run, whose fixed-point form takes four, on the FP64 driver; both come back to the
    fixed-point path once there is room."""
    m = hub.Hubbard(14, 7, 7, W.ring_bonds(14), 1.0, 4.0)
    size = 8 * m.D                                # 94 MB
    x = torch.from_numpy(W.normal(6, m.D)).cuda()
    y, psi = torch.empty_like(x), torch.empty_like(x)
    hub.hub_set_mode(m.h, hub.HUB_MODE_FP64)
    y64 = m.apply(x)
    m.close()
    m = hub.Hubbard(14, 7, 7, W.ring_bonds(14), 1.0, 4.0)
    torch.cuda.empty_cache()

    def fill(vectors):                            # leaves room for so many vectors
        room = int(vectors * size)
        return torch.empty(torch.cuda.mem_get_info()[0] - room, dtype=torch.uint8, device="cuda")

    hog = fill(1.5)
    m.apply(x, y)
    assert torch.equal(y, y64)
    del hog
    torch.cuda.empty_cache()
    m.apply(x, y)
    assert not torch.equal(y, y64)                # within the bound (other tests), but not the same bits
    hub.hub_set_mode(m.h, hub.HUB_MODE_FP64)
    E64 = hub.hub_lanczos_ground(m.h, x, 6, 0.0, psi)[0]
    m.close()
    m = hub.Hubbard(14, 7, 7, W.ring_bonds(14), 1.0, 4.0)
    torch.cuda.empty_cache()
    hog = fill(3.5)
    E = hub.hub_lanczos_ground(m.h, x, 6, 0.0, y)[0]
    assert E == E64 and torch.equal(y, psi)
    del hog
    torch.cuda.empty_cache()
    E = hub.hub_lanczos_ground(m.h, x, 6, 0.0, y)[0]
    assert abs(E - E64) <= 1e-11 and not torch.equal(y, psi)
    m.close()


@pytest.mark.parametrize("M,nu,nd", [(4, 4, 2), (6, 2, 3), (9, 4, 3), (11, 5, 2), (12, 6, 1), (16, 5, 1), (16, 8, 1),
                                     (16, 1, 8)])
@pytest.mark.parametrize("lattice", ["ring", "square"])
def test_schedules_of_all_lengths(hub, M, nu, nd, lattice):
    """Gather schedules from one position to 12,870: counts that are no multiple of a group, of a
    slice or of a warp's share of the grouping, few and many quads, a long spin beside a short one."""
    b = W.ring_bonds(M)
    if lattice == "square":                      # longer rows, uneven ones
        b = W.square_bonds(4, 4, True) if M == 16 else [(i, j) for i in range(M) for j in range(i + 1, M) if (i * j) % 3 != 1]
    m = hub.Hubbard(M, nu, nd, b, 1.0, 4.0)
    hub.hub_set_small_dim(m.h, 0)
    x = torch.from_numpy(W.normal(9, m.D)).cuda()
    steps = min(5, m.D)
    a0, b0, p0 = _run(hub, m, x, steps)
    hub.hub_set_mode(m.h, hub.HUB_MODE_FP64)
    a1, b1, p1 = _run(hub, m, x, steps)
    m.close()
    k = min(len(a0), len(a1))
    scale = max(np.abs(a1).max(), b1.max(), 1.0)
    assert np.abs(a0[:k] - a1[:k]).max() <= 1e-12 * scale and np.abs(b0[:k] - b1[:k]).max() <= 1e-12 * scale
    assert float((p0 - p1).norm()) <= 1e-10
