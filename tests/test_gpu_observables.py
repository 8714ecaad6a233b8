"""The observables kernel at the edges of its decomposition (32 x-planes a
block, eight rows at a time): per-plane sums and masses against the decoded
state on the host, summed in the kernel's population order."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    from paper_1411_2181_gb300 import build
    build.build()
    from paper_1411_2181_gb300 import lbfe
    return lbfe


@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("shape", [(1, 3, 4), (7, 5, 6), (31, 2, 9), (33, 17, 11), (65, 4, 2), (141, 75, 53),
                                   (4096, 1, 2)])
def test_sums_against_the_decoded_state(L, shape, prec):
    Lx, Ly, Lz = shape
    p = L.Params(Lx=Lx, Ly=Ly, Lz=Lz, R=2.0, Uw=0.02, eta_M=0.5, precision=prec)
    rng = np.random.default_rng(sum(shape))
    rho = rng.uniform(0.3, 0.7, (2, Lz, Ly, Lx))
    s = L.Solver(p)
    s.init(0, rho)
    s.step(1)
    o = s.observables(0)
    f = s.get_field(0, L.FIELD_F)
    d = np.zeros((2, Lz, Ly, Lx), np.float32)
    for i in range(19):
        d = d + f[:, i]
    A = d[0] > d[1]
    V = int(A.sum())
    assert o["volume"] == V and o["flags"] == 0
    assert o["Lp"] == (Lx - longest_gap(A.any((0, 1))) if V else 0)
    z, y, _ = np.nonzero(A)
    # FP64 sums of FP32 densities: exact up to the order, N 2^-53 relative
    assert np.allclose(o["mass"], d.astype(np.float64).sum((1, 2, 3)), rtol=p.N * 2.0 ** -53, atol=0)
    if V:
        # exact integer sums; the FP64 moments about the mean cancel at most N 2^16 squares
        tol = V * max(Ly, Lz) ** 2 * 2.0 ** -50
        assert abs(o["centroid"][1] - y.mean()) < 1e-9 and abs(o["centroid"][2] - z.mean()) < 1e-9
        for k, (a, b) in ((1, (y, y)), (2, (z, z)), (5, (y, z))):
            assert abs(o["M"][k] - ((a - a.mean()) * (b - b.mean())).sum()) <= tol + 1e-9
    assert s.observables(0) == o
    s.close()


def longest_gap(occupied):
    """Longest circular run of empty planes."""
    n = len(occupied)
    if occupied.all():
        return 0
    best = run = 0
    for v in np.concatenate([occupied, occupied]):
        run = 0 if v else run + 1
        best = max(best, run)
    return min(best, n)
