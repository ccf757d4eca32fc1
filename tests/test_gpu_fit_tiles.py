"""The RBF fit on ordered tiles (d = 2, 3): sizes at the edges of its tiles,
groups and clusters, and clustered points, against the oracle's fit; a fit is
bit-reproducible."""
import numpy as np
import pytest
import torch

import oracle
import paper_2108_11775_gb300 as pdmp
import workloads as wl
from gpu_util import setup_oracle_threads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    assert torch.cuda.is_available()
    setup_oracle_threads()
    yield
    assert pdmp.stream_status()[0] == 0


@pytest.mark.parametrize("d,M,n,blob", [(2, 1, 1, False), (2, 33, 65, False), (3, 31, 1000, False),
                                        (2, 1300, 4097, False), (3, 2500, 3000, False), (2, 300, 40000, False),
                                        (2, 500, 20000, True)])
def test_fit_matches_the_oracle(d, M, n, blob):
    side = 10.0 if d == 2 else 5.0
    f = wl.random_field(M + d, wl.RBF, d, M, lo=0, hi=side, gamma=8.0)
    X = wl.uniform_box(n, wl.S_POINTS, n, np.zeros(d), np.full(d, side))
    if blob:                                   # dense labels around one obstacle, a few far away
        X[: n - 50] = wl.f32(3.0 + 0.3 * wl.rng(n, 3).standard_normal((n - 50, d)))
    y = wl.inside_boxes(wl.random_boxes(n, 24, np.zeros(d), np.full(d, side), 0.3, 1.5), X)
    fld = pdmp.DeviceField.from_host(f)
    Xd, yd = torch.from_numpy(X).cuda(), torch.from_numpy(y).cuda()
    w, b, loss, alpha = pdmp.fit_occupancy(fld, Xd, yd, 1e-4, 10, 30)
    again = pdmp.fit_occupancy(fld, Xd, yd, 1e-4, 10, 30)
    assert torch.equal(w, again[0]) and (b, loss, alpha) == again[1:]
    rw, rb, rloss, ralpha = oracle.fit(f, X, y, 1e-4, 10, 30)
    # 40 sweeps each way in FP32: the sums' relative errors of about 1e-6 reach w at most 30-fold
    assert abs(alpha - ralpha) <= 1e-5 * ralpha
    assert np.linalg.norm(w.cpu().numpy() - rw) <= 3e-5 * np.linalg.norm(rw)
    assert abs(b - rb) <= 3e-5 * max(1.0, abs(rb))
    assert abs(loss - rloss) <= 1e-5 * max(rloss, 1e-2)
