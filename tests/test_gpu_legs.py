"""The fused legs of the V-cycle (k_tile.cu) against the passes that they
stand for, bit for bit: each tile shape by itself on one level (every boundary
and operator that the solver gives it, ragged sides), and a single context's
first step, whose legs they are, against the persistent batched solve, which
runs one-colour passes and transfers on every level."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_1709_04703_gb300 import _lib as L  # noqa: E402
from paper_1709_04703_gb300 import ics  # noqa: E402
from test_gpu_tiles import _case  # noqa: E402


@pytest.fixture(scope="module")
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1709_04703_gb300 import build
    build.build()
    return L.load()


def _array(rng, s, inside=True):
    a = np.zeros((s + 2,) * 3, np.float32)
    if inside:
        a[1:-1, 1:-1, 1:-1] = rng.standard_normal((s,) * 3)
    return torch.from_numpy(a).cuda()


def _leg(lib, up, u, b, w, uc, bc, s, per, h2, gam, gam_c, d0, tile):
    code = lib.pm_mg_leg(up, *(C.c_void_p(t.data_ptr()) for t in (u, b, w, uc, bc)), s, per, h2,
                         gam, gam_c, d0, tile, None)
    assert code == L.PM_OK, lib.pm_last_error(None)


def _bits(a):
    return a.view(torch.int32).cpu().numpy()


# finest and coarse level (h2 = 4^l, ghost factors (H - 1) / (H + 1) of the
# level and the next one), and the diffusion's shifted operator
OPERATORS = [(1.0, 0.0, 1.0 / 3.0, 6.0), (16.0, 3.0 / 5.0, 7.0 / 9.0, 6.0),
             (4.0, 1.0 / 3.0, 3.0 / 5.0, 7.25)]


@pytest.mark.parametrize("s", [20, 22, 24, 28, 32, 38, 40, 48, 56, 64, 70, 80, 112, 128, 160, 192])
@pytest.mark.parametrize("per", [0, 1])
@pytest.mark.parametrize("tile", [8, 16])
def test_leg_gives_the_bits_of_the_passes(lib, s, per, tile):
    rng = np.random.default_rng(100 * s + per)
    b, w0, uc0 = _array(rng, s), _array(rng, s), _array(rng, s // 2)
    for h2, gam, gam_c, d0 in OPERATORS:
        got, ref = [], []
        for out, t in ((got, tile), (ref, 0)):
            u, w = _array(rng, s, False), _array(rng, s, False)
            uc, bc = _array(rng, s // 2, False), _array(rng, s // 2, False)
            _leg(lib, 0, u, b, w, uc, bc, s, per, h2, gam, gam_c, d0, t)
            out += [_bits(w), _bits(bc)]
            w, uc = w0.clone(), uc0.clone()
            _leg(lib, 1, u, b, w, uc, bc, s, per, h2, gam, gam_c, d0, t)
            out += [_bits(u)]
            assert torch.equal(w, w0) and torch.equal(uc, uc0)
        for name, x, y in zip(("w", "bc", "u"), got, ref):
            np.testing.assert_array_equal(x, y, err_msg=f"{name}, d0 {d0}, gam {gam}")
        assert np.any(got[2])


def test_leg_rejects_bad_arguments(lib):
    arrays = [_array(np.random.default_rng(0), 20) for _ in range(5)]
    p = [C.c_void_p(a.data_ptr()) for a in arrays]
    good = dict(up=0, s=20, per=1, h2=1.0, gam=0.0, gam_c=0.0, d0=6.0, tile=8)
    for bad in (dict(up=2), dict(s=18), dict(s=21), dict(s=2000), dict(h2=0.0), dict(d0=5.0),
                dict(tile=4)):
        g = {**good, **bad}
        assert lib.pm_mg_leg(g["up"], *p, g["s"], g["per"], g["h2"], g["gam"], g["gam_c"],
                             g["d0"], g["tile"], None) == L.PM_EINVAL
    assert lib.pm_mg_leg(0, p[0], p[1], p[0], p[3], p[4], 20, 1, 1.0, 0.0, 0.0, 6.0, 8,
                         None) == L.PM_EINVAL


@pytest.mark.parametrize("side,periodic", [(20, False), (28, False), (32, True), (40, False),
                                           (48, True), (56, False), (64, True), (80, False),
                                           (96, True), (112, False), (160, False), (192, True),
                                           (224, False)])
def test_single_context_gives_the_bits_of_the_passes(lib, side, periodic):
    """The first step: no V-cycle is run ahead of its residual there, so a
    context and a batch take the same number and their results must be equal
    bit for bit."""
    from paper_1709_04703_gb300.sim import Batch, Sim
    n, box, a0 = _case(side, periodic)
    m = min(n, 64)
    x, p, ids = ics.zeldovich(m, -1.5, None, 3, a0, rms_disp=0.4)
    x, p = (x * np.float32(n / m)).astype(np.float32), p * np.float32(n / m)
    x[x >= n] = 0.0
    batch = Batch([dict(pos=x, mom=p, ids=ids, n_mesh=n, box=box)], a0, 1.0, 400, rtol=1e-8,
                  store_forces=True)
    batch.set_solve(persistent=True)
    batch.step(1)
    sim = Sim(x, p, ids, n, box, a0, 1.0, 400, rtol=1e-8, store_forces=True)
    sim.step(1)
    a, b = sim.stats(), batch.stats(0)
    assert a["cube_side"] == side and bool(a["periodic"]) == periodic
    assert a["vcycles_last"] == b["vcycles_last"] >= 2
    np.testing.assert_array_equal(sim.forces(), batch.forces(0))
    for one, two in zip(sim.particles(), batch.particles(0)):
        np.testing.assert_array_equal(one, two)
    sim.close()
    batch.close()
