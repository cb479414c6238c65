"""Ground-state and Ritz vectors written over their start vector: bit for bit those of separate
buffers, in every Lanczos driver (fixed point, FP64, small sectors in both forms, momentum)."""
import pytest

from paper_1307_7542_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def hub(cuda_ok):
    import __graft_entry__
    __graft_entry__.build()
    from paper_1307_7542_gb300 import hub as H
    return H


def _model(hub, driver):
    if driver == "fixed_mixed":          # one spin gathered, one combined
        m = hub.Hubbard(18, 1, 9, W.square_bonds(3, 6, True), 1.0, 4.0)
    elif driver == "momentum":
        m = hub.Hubbard(10, 5, 5, W.ring_bonds(10), 1.0, 4.0)
        m.set_symmetry(hub.HUB_SYM_K0)
    elif driver == "cluster":
        m = hub.Hubbard(8, 4, 4, W.ring_bonds(8), 1.0, 4.0)
    else:                                # "small", "fixed", "fp64"
        m = hub.Hubbard(9, 4, 5, W.ring_bonds(9), 1.0, 4.0)
    if driver.startswith("f"):
        hub.hub_set_small_dim(m.h, 0)
    if driver == "fp64":
        hub.hub_set_mode(m.h, hub.HUB_MODE_FP64)
    return m


@pytest.mark.parametrize("driver", ["fixed", "fixed_mixed", "fp64", "small", "cluster", "momentum"])
def test_vector_over_start(hub, driver):
    m = _model(hub, driver)
    D = m.D
    x = torch.from_numpy(W.normal(3, D)).cuda()
    psi = torch.empty_like(x)
    E = hub.hub_lanczos_ground(m.h, x, 14, 0.0, psi)[0]
    assert abs(float(psi.norm()) - 1.0) < 1e-12
    z = x.clone()
    assert hub.hub_lanczos_ground(m.h, z, 14, 0.0, z)[0] == E
    assert torch.equal(z, psi)
    # partly over it: the start vector ends where the output's second half begins
    both = torch.zeros(D + D // 2, dtype=torch.float64, device="cuda")
    both[:D] = x
    assert hub.hub_lanczos_ground(m.h, both[:D], 14, 0.0, both[D // 2:])[0] == E
    assert torch.equal(both[D // 2:], psi)
    v = hub.hub_lanczos_ritz(m.h, x, 14, E + 1.0, psi)
    z = x.clone()
    assert hub.hub_lanczos_ritz(m.h, z, 14, E + 1.0, z) == v
    assert torch.equal(z, psi)
    m.close()
