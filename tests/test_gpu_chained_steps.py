"""Steps that follow one another on the stream (programmatic launches: a step's
blocks may start while the last step still writes the lattice they will read)
against the same steps with the stream drained after each: the same bits in
every precision, on grids just above the size from which the early trigger is
used, of odd width (wrap and wall loads on unaligned rows), with a width of
whole blocks and wall strips, below that size, and on one-column channels with
and without lanes, and for the sums of a window of averages."""
import numpy as np
import pytest

import oracle
from lbm_inputs import rho_field

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build_library()


def _solver(name, N, Nx, Ny, precision):
    import paper_1510_08886_gb300 as lbm
    e, w, c = lbm.dvm(name)
    s = lbm.Solver(e, w, c, N, Nx, Ny, 0.2, oracle.force_for_mach(0.2, 1e-2), precision=precision)
    return s.set_resident(False).init(rho_field(Nx, Ny, seed=29, amplitude=1e-3))


# (name, N, Nx, Ny): 2074 and 2080 blocks of 128 nodes, above the 1520 or 1900 from
# which fp64 and the 53-velocity set let blocks in, and 1276 below; then 40 blocks, a
# short column and a small set on lanes
SHAPES = [("D2V33", 4, 1021, 260), ("D2V33", 4, 1024, 260), ("D3V107xz", 3, 1021, 260), ("D2V33", 4, 1021, 160),
          ("D2V16", 3, 129, 39), ("D2V33", 4, 1, 5001), ("D2V16", 3, 1, 40)]


@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp16", "bf16"])
@pytest.mark.parametrize("name,N,Nx,Ny", SHAPES)
def test_chained_steps_bitwise_equal_drained(name, N, Nx, Ny, precision):
    a, b = _solver(name, N, Nx, Ny, precision), _solver(name, N, Nx, Ny, precision)
    a.step(40)
    for _ in range(40):
        b.step(1)
        torch.cuda.synchronize()
    assert np.array_equal(a.populations(), b.populations())
    for x, y in zip(a.moments(), b.moments()):
        assert np.array_equal(x, y)
    a.average(20)
    total = [0.0, 0.0, 0.0]
    for _ in range(20):
        b.step(1)
        total = [t + m for t, m in zip(total, b.moments())]
    for x, t in zip(a.moments(), total):
        assert np.array_equal(x, t * (1.0 / 20.0))
    assert np.array_equal(a.populations(), b.populations())
