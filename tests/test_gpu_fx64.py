"""fp64 steps of the compiled velocity sets on the GPU against the oracle where
the fixed-point collision's kernels can go wrong: every set, one column, columns
narrower than the velocities, rows and blocks with remainders, strips, flows
that leave the fixed-point range (general form node by node), no force.

Tolerances: those of the fp64 parity tests (populations 1e-13, u 1e-12 of its
largest value; both sides round O(1) populations at 1e-16 per step)."""
import numpy as np
import pytest

import oracle
from lbm_inputs import rho_field

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SETS = [("D2V16", 2), ("D2V16", 3), ("D2V16", 4), ("D2V33", 3), ("D2V33", 4), ("D2V32", 3), ("D3V107xz", 3),
        ("D3V96xz", 3), ("D3V112xz", 3)]


def _compare(name, N, Nx, Ny, steps, amplitude=1e-3, mach=1e-2, Kn=0.2):
    import paper_1510_08886_gb300 as lbm
    e, w, c = lbm.dvm(name)
    g = oracle.force_for_mach(Kn, mach) if mach else 0.0
    rho = np.clip(rho_field(Nx, Ny, seed=17, amplitude=amplitude), 0.2, None)
    s = lbm.Solver(e, w, c, N, Nx, Ny, Kn, g).init(rho).step(steps)
    ref = oracle.channel(name, N, Nx, Ny, Kn, g).init(rho).step(steps)
    r_g, u_g, v_g = s.moments()
    r_o, u_o, v_o = ref.moments()
    umax = np.max(np.abs(u_o)) + np.max(np.abs(v_o))
    assert np.max(np.abs(r_g - r_o)) < 1e-13 * max(1.0, np.max(r_o))
    assert np.max(np.abs(u_g - u_o)) < 1e-12 * umax
    assert np.max(np.abs(v_g - v_o)) < 1e-12 * umax
    lut = {(int(x), int(y)): i for i, (x, y) in enumerate(zip(ref.ex, ref.ey))}
    idx = [lut[(int(x), int(y))] for x, y in e]
    assert np.max(np.abs(s.populations() - ref.collide(ref.f)[idx])) < 1e-13 * max(1.0, np.max(r_o))
    assert s.status() == 0


@pytest.mark.parametrize("name,N", SETS)
@pytest.mark.parametrize("Nx,Ny", [(1, 5001), (3, 1667), (129, 39), (128, 40)])
def test_every_set_and_shape(name, N, Nx, Ny):
    _compare(name, N, Nx, Ny, 6)


@pytest.mark.parametrize("name,N", [("D2V16", 3), ("D2V33", 4), ("D2V32", 3), ("D3V107xz", 3)])
@pytest.mark.parametrize("amplitude,mach", [(0.3, 0.1), (1e-6, 0.3), (1e-3, 0.0)])
def test_outside_the_range_and_without_force(name, N, amplitude, mach):
    _compare(name, N, 67, 81, 5, amplitude=amplitude, mach=mach)


@pytest.mark.parametrize("name,N", [("D2V16", 3), ("D2V33", 4)])
@pytest.mark.parametrize("Nx,Ny", [(1, 150), (3, 40), (2, 97)])
def test_resident_and_tiled_engine_bitwise(name, N, Nx, Ny):
    """The resident kernel reads populations where they lie, the tiled one from
    its scratch: the same bits, also where nodes leave the fixed-point range."""
    import paper_1510_08886_gb300 as lbm
    e, w, c = lbm.dvm(name)
    rho = np.clip(rho_field(Nx, Ny, seed=5, amplitude=0.2), 0.2, None)
    out = []
    for resident in (True, False):
        eng = lbm.Engine("fp64", max_solves=2, arena_bytes=64 << 20, chunk=20, resident=resident)
        slot = eng.add(e, w, c, N, Nx, Ny, 0.1, oracle.force_for_mach(0.1, 0.05), rho=rho)
        res = eng.run(2)[slot].copy()
        assert eng.paths() == ((0, 1) if resident else (1, 0))
        out.append((res, eng.moments(slot, Nx, Ny)))
        eng.close()
    assert np.array_equal(out[0][0], out[1][0])
    for a, b in zip(out[0][1], out[1][1]):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("name,N", SETS)
@pytest.mark.parametrize("Nx,Ny", [(5, 29), (1, 600)])
@pytest.mark.parametrize("amplitude,mach", [(1e-3, 1e-2), (0.3, 0.1)])
def test_small_channels_on_lanes(name, N, Nx, Ny, amplitude, mach):
    """Several lanes per node, resident on a cluster of small or large blocks;
    the second flow takes the general form on some nodes of a warp."""
    _compare(name, N, Nx, Ny, 7, amplitude=amplitude, mach=mach)


@pytest.mark.parametrize("name,N", [("D2V33", 4), ("D3V107xz", 3)])
@pytest.mark.parametrize("Nx,Ny", [(129, 60), (4, 40)])
def test_force_against_x(name, N, Nx, Ny):
    """g < 0 runs as the mirror image of g > 0."""
    _compare(name, N, Nx, Ny, 7, mach=-1e-2)
