"""The binned power-spectrum pass at the sizes where its folding of mirrored
modes, its integer bins and its runs of one bin can go wrong: odd and even
meshes, rows shorter and longer than a warp, more bins than the sphere inside
the cube fills, every alias range.  Bounds as tests/test_gpu_parity.py: mode
counts exact, k to 1e-12, P to the FP32 FFT's rounding."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from oracle.pk import power_spectrum as opk  # noqa: E402
from oracle.pk import power_spectrum_jing as opkj  # noqa: E402
from paper_1709_04703_gb300 import ics  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1709_04703_gb300 import build
    build.build()


def _particles(n, N):
    from paper_1709_04703_gb300.sim import pack
    pos, mom, ids = ics.random_particles(N, n, 5)
    return pos, torch.from_numpy(pack(pos, mom, ids)[0]).cuda()


@pytest.mark.parametrize("n,n_bins,N", [(2, 1, 7), (5, 4, 300), (31, 15, 5000), (33, 40, 20000),
                                        (62, 31, 30001), (65, 56, 40000), (96, 48, 90000)])
@pytest.mark.parametrize("shot", [True, False])
def test_bins_match_oracle(n, n_bins, N, shot):
    from paper_1709_04703_gb300.sim import power_spectrum
    pos, p4 = _particles(n, N)
    k, p, m = power_spectrum(p4, 300.0, n, n_bins, subtract_shot=shot)
    ko, po, mo = opk(pos, n, 300.0, n_bins, shot_noise=shot)
    np.testing.assert_array_equal(m, mo)
    has = mo > 0
    np.testing.assert_allclose(k[has], ko[has], rtol=1e-12)
    assert np.isnan(k[~has]).all() and np.isnan(p[~has]).all()
    # Poisson points: P_obs is the shot noise's size, on which the FP32
    # transform's rounding is measured
    np.testing.assert_allclose(p[has], po[has], rtol=2e-4, atol=2e-5 * 300.0**3 / N)


@pytest.mark.parametrize("n,alias", [(5, 3), (32, 1), (33, 2), (48, 3)])
def test_alias_ranges_match_oracle(n, alias):
    from paper_1709_04703_gb300.sim import power_spectrum_jing
    pos, _, _ = ics.zeldovich(n, -2.0, None, 3, 0.5, rms_disp=0.5)
    from paper_1709_04703_gb300.sim import pack
    p4 = torch.from_numpy(pack(pos, 0 * pos)[0]).cuda()
    k, p, m, nu, _ = power_spectrum_jing(p4, 300.0, n, n // 2, subtract_shot=False,
                                         alias_range=alias, max_iter=3, tol=1e-30)
    ko, po, mo, nuo, _ = opkj(pos, n, 300.0, n // 2, shot_noise=False, m=alias,
                              max_iter=3, tol=1e-30)
    np.testing.assert_array_equal(m, mo)
    np.testing.assert_allclose(k, ko, rtol=1e-12)
    np.testing.assert_allclose(nu, nuo, rtol=0, atol=2e-3)
    np.testing.assert_allclose(p, po, rtol=3e-4, atol=3e-5 * np.abs(po).max())


def test_mean_k_is_a_64_bit_sum():
    """The mean |k| of a bin against an extended-precision sum over its modes,
    on meshes small enough that the order of the FP64 sums hides nothing.
    About 30 partial sums a bin, the wavenumber unit, a product and a quotient
    in 64 bits leave 1.4e-16 in the mean; one FP64 unit roundoff's double is
    the bound (values or sums as pairs of floats leave 3.5e-16 and more)."""
    from paper_1709_04703_gb300.sim import power_spectrum
    err = []
    for n in (8, 16, 20, 24, 32, 40):
        _, p4 = _particles(n, 500)
        x = np.arange(n // 2 + 1)
        q = np.where(np.arange(n) <= n // 2, np.arange(n), np.arange(n) - n)
        m2 = x[None, None] ** 2 + q[None, :, None] ** 2 + q[:, None, None] ** 2
        w = np.where((x == 0) | (2 * x == n), 1, 2) + 0 * m2
        root = np.sqrt(m2.astype(np.longdouble))
        b = np.floor(np.sqrt(m2) + 0.5).astype(int) - 1
        ok = (b >= 0) & (b < n // 2)
        tot = np.zeros(n // 2, np.longdouble)
        np.add.at(tot, b[ok], (w * root)[ok])
        cnt = np.bincount(b[ok], weights=w[ok], minlength=n // 2)
        for box in (100.0, 300.0, 777.0):
            k, _, m = power_spectrum(p4, box, n, n // 2)
            np.testing.assert_array_equal(m, cnt)
            ref = tot / cnt * (2 * np.longdouble("3.14159265358979323846264338327950288") / box)
            err.append(((k - ref) / ref).astype(float))
    err = np.concatenate(err)
    assert np.sqrt((err**2).mean()) < 2.0**-52
