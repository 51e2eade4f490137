"""The work space and FFT plans that the context-free calls share: more
meshes than the plan cache keeps, sizes going up and down, several streams and
threads at once, always the results of a call alone."""
import threading

import numpy as np
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


def _points(n, N, seed):
    from paper_1709_04703_gb300.sim import pack
    p4, m4 = pack(*ics.random_particles(N, n, seed))
    return torch.from_numpy(p4).cuda(), torch.from_numpy(m4).cuda()


def test_plans_and_work_space_across_sizes_streams_and_threads():
    from paper_1709_04703_gb300.sim import power_spectrum, sort_particles
    sizes = [8, 15, 32, 48, 20, 64, 33]  # more than the cache keeps
    pts = {n: _points(n, 4000 + n, n) for n in sizes}

    def one(n):
        p4, m4 = pts[n]
        spec = power_spectrum(p4, 100.0, n, n // 2)
        return spec, sort_particles(p4, m4, n)

    def same(got, ref):
        for x, y in zip(got[0], ref[0]):  # sums of doubles by atomics
            np.testing.assert_allclose(x, y, rtol=1e-12)
        for x, y in zip(got[1], ref[1]):
            assert torch.equal(x.view(torch.int32), y.view(torch.int32))

    ref = {n: one(n) for n in sizes}
    for n in sizes + sizes[::-1]:
        same(one(n), ref[n])
    bad = []

    def work(k):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for r in range(6):
                    n = sizes[(k + r) % len(sizes)]
                    same(one(n), ref[n])
        except Exception as e:  # noqa: BLE001 - reported below
            bad.append(e)
    ts = [threading.Thread(target=work, args=(k,)) for k in range(4)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not bad, bad[0]
