"""fp64 solves whose constants are outside the fixed-point range as a whole, through
every kernel that has that form: the wide step, lanes launched per step and on a
cluster, the tiled and the resident engine.  Strong force (theta = tau c |g| >=
1/8), strong half step (c g dt / 2 = 0.1), mirrored pairs of unequal weight, and a
fluid at rest without a force; against the oracle with the tolerances of the fp64 parity tests (populations 1e-13, u 1e-12 of
its largest value; both sides round O(1) populations at 1e-16 per step)."""
import numpy as np
import pytest

import oracle
from lbm_inputs import rho_field

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SETS = [("D2V16", 3), ("D2V33", 4), ("D2V32", 3), ("D3V107xz", 3), ("D3V112xz", 2)]
KINDS = ["theta", "half_step", "weights"]


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build_library()


def _case(name, kind, Ny):
    """(e, w, c, Kn, g)"""
    import paper_1510_08886_gb300 as lbm
    e, w, c = lbm.dvm(name)
    w = np.array(w)
    tau = oracle.tau_of_kn
    if kind == "theta":
        return e, w, c, 10.0, 0.2 / (tau(10.0) * c)
    if kind == "half_step":
        return e, w, c, 0.002, 0.2 * Ny                # c g dt / 2 = g / (2 Ny)
    prod = e[:, 0] * e[:, 1]
    w = w * (1 + 1e-14 * np.sign(prod))
    assert np.any(prod > 0) and np.any(prod < 0)
    return e, w, c, 0.2, oracle.force_for_mach(0.2, 1e-2)


def _rho(Nx, Ny):
    return rho_field(Nx, Ny, seed=3, amplitude=1e-3)


def _assert_close(rho_u_v, ref):
    r_o, u_o, v_o = ref.moments()
    umax = np.max(np.abs(u_o)) + np.max(np.abs(v_o))
    r, u, v = rho_u_v
    assert np.max(np.abs(r - r_o)) < 1e-13 * max(1.0, np.max(np.abs(r_o)))
    assert np.max(np.abs(u - u_o)) < 1e-12 * umax
    assert np.max(np.abs(v - v_o)) < 1e-12 * umax


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("name,N", SETS)
# blocks with wall strips; odd rows; lanes; lanes of a channel that a large cluster
# block would hold
@pytest.mark.parametrize("Nx,Ny", [(128, 40), (67, 81), (3, 20), (1, 600)])
def test_solver(name, N, kind, Nx, Ny):
    import paper_1510_08886_gb300 as lbm
    e, w, c, Kn, g = _case(name, kind, Ny)
    steps = 2 if kind == "half_step" else 5
    s = lbm.Solver(e, w, c, N, Nx, Ny, Kn, g).init(_rho(Nx, Ny)).step(steps)
    ref = oracle.Channel(e, w, c, N, Nx, Ny, Kn, g).init(_rho(Nx, Ny)).step(steps)
    _assert_close(s.moments(), ref)
    lut = {(int(x), int(y)): i for i, (x, y) in enumerate(zip(ref.ex, ref.ey))}
    idx = [lut[(int(x), int(y))] for x, y in e]
    f_o = ref.collide(ref.f)[idx]
    assert np.max(np.abs(s.populations() - f_o)) < 1e-13 * max(1.0, np.max(np.abs(f_o)))


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("name,N", [("D2V16", 3), ("D2V33", 4), ("D3V107xz", 3)])
@pytest.mark.parametrize("Nx,Ny", [(1, 90), (3, 40), (5, 31)])
def test_engine(name, N, kind, Nx, Ny):
    import paper_1510_08886_gb300 as lbm
    e, w, c, Kn, g = _case(name, kind, Ny)
    steps = 2 if kind == "half_step" else 6
    ref = oracle.Channel(e, w, c, N, Nx, Ny, Kn, g).init(_rho(Nx, Ny)).step(steps)
    out = []
    for resident in (True, False):
        eng = lbm.Engine("fp64", max_solves=2, arena_bytes=64 << 20, chunk=steps, resident=resident)
        slot = eng.add(e, w, c, N, Nx, Ny, Kn, g, rho=_rho(Nx, Ny))
        eng.run(1)
        assert eng.paths() == ((0, 1) if resident else (1, 0))
        out.append(eng.moments(slot, Nx, Ny))
        eng.close()
        _assert_close(out[-1], ref)
    for a, b in zip(*out):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("name,N", SETS)
@pytest.mark.parametrize("Nx,Ny", [(128, 40), (3, 20), (1, 50), (1, 600)])
def test_rest_stays_at_rest(name, N, Nx, Ny):
    """rho = 1 and no force: zero deviations stay zero, in the solver and the
    engine; beside a disturbance the rest of the channel is at rest until it is
    reached."""
    import paper_1510_08886_gb300 as lbm
    e, w, c = lbm.dvm(name)
    s = lbm.Solver(e, w, c, N, Nx, Ny, 0.3, 0.0).init().step(7)
    assert np.array_equal(s.populations(), np.broadcast_to(np.asarray(w)[:, None, None], (len(w), Ny, Nx)))
    rho, ux, uy = s.moments()
    assert np.all(rho == 1) and not np.any(ux) and not np.any(uy)
    # the deviations themselves, from the saved state
    V = len(w)
    state = np.frombuffer(s.get_state(), dtype=np.uint8)
    d = state[state.size - 8 * Nx * Ny * (V + 3):state.size - 8 * Nx * Ny * 3].view(np.float64)
    assert d.size == V * Nx * Ny and not np.any(d)
    eng = lbm.Engine("fp64", max_solves=2, arena_bytes=64 << 20, chunk=6)
    slot = eng.add(e, w, c, N, Nx, Ny, 0.3, 0.0)
    eng.run(1)
    rho, ux, uy = eng.moments(slot, Nx, Ny)
    assert np.all(rho == 1) and not np.any(ux) and not np.any(uy)
    eng.close()
    far = np.ones((Ny, Nx))
    far[Ny // 2, 0] = 1.01
    s.init(far).step(1)
    ref = oracle.Channel(e, w, c, N, Nx, Ny, 0.3, 0.0).init(far).step(1)
    _assert_close(s.moments(), ref)
    reach = 2 * int(np.max(np.abs(e)))
    if Ny // 2 - reach > 0:
        assert not np.any(s.moments()[1][:Ny // 2 - reach])


# channels of more than eight warps per CTA, on 8, 16 and 32 lanes per node
LARGE = [("D2V16", 3, 1, 600), ("D2V16", 3, 1, 1500), ("D2V16", 3, 5, 290), ("D2V33", 4, 1, 400), ("D3V107xz", 3, 1, 200),
         ("D3V112xz", 3, 2, 150)]


@pytest.mark.parametrize("precision,amplitude", [("fp32", 1e-3), ("fp64", 1e-3), ("fp64", 0.3)])
@pytest.mark.parametrize("name,N,Nx,Ny", LARGE)
def test_large_cluster_blocks_bitwise_equal_launched(name, N, Nx, Ny, precision, amplitude):
    """Resident steps give the bits of launched steps; with the larger density
    amplitude nodes of one warp split between the fixed-point and the FP64 form,
    and once the host has read the status the solve goes on in launches."""
    import paper_1510_08886_gb300 as lbm
    e, w, c = lbm.dvm(name)
    rho = np.clip(rho_field(Nx, Ny, seed=5, amplitude=amplitude), 0.2, None)
    g = oracle.force_for_mach(0.2, 1e-2)
    a, b = (lbm.Solver(e, w, c, N, Nx, Ny, 0.2, g, precision=precision).set_resident(r).init(rho) for r in (True, False))
    assert a.resident_ctas() > 0 and b.resident_ctas() == 0
    for n in (33, 2, 1):
        a.step(n)
        b.step(n)
        assert np.array_equal(a.populations(), b.populations())
        for x, y in zip(a.moments(), b.moments()):
            assert np.array_equal(x, y)
    a.init(rho)
    assert a.resident_ctas() > 0
    if amplitude > 0.1:
        a.step(2)                       # density well out of range at some nodes
        assert a.status() == 0 and a.resident_ctas() == 0
        b.init(rho).step(2)
        assert a.run_to_steady(1e-16, 203, check_every=50) == b.run_to_steady(1e-16, 203, check_every=50)
        assert np.array_equal(a.populations(), b.populations())
        a.set_state(b.get_state())
        assert a.resident_ctas() > 0


def test_fixed_point_clusters_only():
    """A solve outside the range as a whole gets no block of more than eight warps
    (two FP64 lanes per SM), one inside does."""
    import paper_1510_08886_gb300 as lbm
    e, w, c, Kn, g = _case("D2V16", "theta", 1500)
    assert lbm.Solver(e, w, c, 3, 1, 1500, Kn, g).resident_ctas() == 0
    assert lbm.Solver(e, w, c, 3, 1, 64, Kn, g).resident_ctas() > 0
    assert lbm.Solver(e, w, c, 3, 1, 1500, 0.1, 1e-3).resident_ctas() > 0
