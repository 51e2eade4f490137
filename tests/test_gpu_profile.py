"""The per-class byte counts (pm_profile_read) are what the launches must
move: the counts that a rate over time is compared with the memory's."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_1709_04703_gb300 import ics  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1709_04703_gb300 import build
    build.build()


# bytes per cell of the finest level's legs (down, up): a fused leg down reads
# the right-hand side and writes the scratch grid and the coarse right-hand
# side (4 + 4 + 4/8); a fused leg up reads scratch grid, right-hand side and
# coarse values and writes the iterate (4 + 4 + 4/8 + 4); from side 192 the leg
# up is a prolongation (class transfer0: 4 + 4/8 + 4) and the two-sweep pass
# (4 + 4 + 4); the same two fused legs, or the two-sweep pass, on each coarser
# level, and the bottom (side <= 16) reads one array and writes one
@pytest.mark.parametrize("n,smooth,transfer", [(32, 21.0, 0.0), (128, 21.0, 0.0),
                                               (192, 20.5, 8.5)])
def test_vcycle_bytes(n, smooth, transfer):
    from paper_1709_04703_gb300.sim import Sim
    x, p, ids = ics.random_particles(4000, n, 3)
    sim = Sim(x, p, ids, n, 8.0 * n, 0.05, 1.0, 100, rtol=1e-6)
    sim.step(1)
    sim.profile(True)
    sim.step(2)
    prof = sim.profile_read()
    sim.close()
    vc = prof["smooth0"]["groups"] / 2  # both legs of a V-cycle are timed
    assert vc >= 2
    per = {c: prof[c]["bytes"] / vc / n**3 for c in ("smooth0", "transfer0", "coarse")}
    coarse, s = 0.0, n // 2
    while s > 16:
        coarse += 21.0 * s**3
        s //= 2
    coarse += 8.0 * s**3
    assert per["smooth0"] == pytest.approx(smooth)
    assert per["transfer0"] == pytest.approx(transfer)
    assert per["coarse"] == pytest.approx(coarse / n**3)


@pytest.mark.parametrize("n,passes", [(32, 2), (64, 3)])
def test_sort_bytes(n, passes):
    """Keys 20 B, the second pass on a histogram each (4), scatters reading
    and writing key and index (16) but for the first's index and the last's
    key (4 each), permutation and records 68."""
    from paper_1709_04703_gb300.sim import Sim
    N = 5000
    x, p, ids = ics.random_particles(N, n, 3)
    sim = Sim(x, p, ids, n, 8.0 * n, 0.05, 1.0, 100, rtol=1e-6, sort_every=1)
    sim.profile(True)
    sim.step(1)
    got = sim.profile_read()["sort"]["bytes"] / N
    sim.close()
    assert got == pytest.approx(20 + 4 * (passes - 1) + 16 * passes - 8 + 68)
