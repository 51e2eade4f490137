"""The fused legs of the V-cycle (k_tile.cu) at the sides where their tiles
can go wrong: ragged open cubes (sides that are no multiple of a tile), the
smallest and largest they take, both boundaries.  The persistent batched
solve runs the one-colour passes and transfers one by one, the graph solve
and a single context the fused legs: all three must agree bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from oracle import cosmology as cz  # noqa: E402
from oracle import pm as opm  # noqa: E402
from paper_1709_04703_gb300 import ics  # noqa: E402

OM, OL = 0.3, 0.7


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1709_04703_gb300 import build
    build.build()


def _case(side, periodic):
    """(mesh, box, a) whose step solves on a cube of this side."""
    if periodic:
        return side, 4.0 * side, 0.1
    n = min(v for v in (32, 64, 128, 256) if v >= side)
    box = 8000.0
    for a in np.linspace(0.25, 0.99, 3000):
        R = cz.chi(a, OM, OL) / (box / n) + 1.0
        lo, s, per = opm.active_cube(R, n)
        if not per and s == side:
            return n, box, a
    raise AssertionError(side)


@pytest.mark.parametrize("side,periodic", [(20, False), (24, True), (28, False), (32, True),
                                           (40, False), (48, True), (56, False), (64, True),
                                           (80, False), (96, True), (112, False), (160, False),
                                           (192, True), (224, False)])
def test_fused_legs_give_the_bits_of_the_separate_passes(side, periodic):
    from paper_1709_04703_gb300.sim import Batch, Sim
    n, box, a0 = _case(side, periodic)
    m = min(n, 64)  # particles per axis: the solve is what is compared
    x, p, ids = ics.zeldovich(m, -1.5, None, 3, a0, rms_disp=0.4)
    x, p = (x * np.float32(n / m)).astype(np.float32), p * np.float32(n / m)
    x[x >= n] = 0.0
    rtol, steps = 1e-8, 400
    got = []
    for persistent in (True, False):
        b = Batch([dict(pos=x, mom=p, ids=ids, n_mesh=n, box=box)], a0, 1.0, steps, rtol=rtol,
                  store_forces=True)
        b.set_solve(persistent=persistent)
        b.step(2)
        s = b.stats(0)
        got.append((b.forces(0), *b.particles(0), s["vcycles_total"], s["resid_last"]))
        assert s["cube_side"] == side and bool(s["periodic"]) == periodic
        b.close()
    for one, two in zip(*got):
        np.testing.assert_array_equal(one, two)
    # a single context (tile shape by rule); its solve may run one V-cycle
    # more, so the forces agree to the tolerance of the solve
    sim = Sim(x, p, ids, n, box, a0, 1.0, steps, rtol=rtol, store_forces=True)
    sim.step(2)
    f = got[0][0]
    assert np.sqrt(((sim.forces() - f) ** 2).sum() / (f**2).sum()) < 1e-6
    sim.close()
