"""Occupancy queries on sorted tiles (long sweeps of 2-D / 3-D RBF fields)
against the direct kernel and the oracle, on both sides of the rule that picks
them; every combination of outputs, ragged sizes, points that are not finite;
and the samples' order at the sizes where it changes its launches."""
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


def direct(fld, x):
    """pdmp_occupancy_query: the kernel without a workspace."""
    import ctypes
    N, d = x.shape
    c, s, g = torch.empty(N, device="cuda"), torch.empty(N, device="cuda"), torch.empty(N, d, device="cuda")
    f = fld.struct()
    P = lambda t: ctypes.c_void_p(t.data_ptr())
    assert pdmp.lib().pdmp_occupancy_query(ctypes.byref(f), P(x), N, P(c), P(s), P(g),
                                           ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)) == 0
    return c, s, g


@pytest.mark.parametrize("d,M,N,tiles", [(2, 2047, 1000, False), (2, 2048, 1, True), (3, 2048, 129, True),
                                         (2, 16385, 16384, True), (3, 5000, 16385, True), (2, 300, 1000003, True),
                                         (2, 2048, 1 << 21, True)])
def test_query_on_tiles(d, M, N, tiles):
    f = wl.random_field(M, wl.RBF, d, M, lo=0, hi=10, gamma=4.0, wscale=0.5, bias=0.1)
    fld = pdmp.DeviceField.from_host(f)
    assert (pdmp.lib().pdmp_occupancy_query_workspace(__import__("ctypes").byref(fld.struct()), N) > 0) == tiles
    x = torch.from_numpy(wl.uniform_box(N, 3, N, np.full(d, -0.5), np.full(d, 10.5))).cuda()
    q = pdmp.occupancy_query(fld, x)
    idx = np.unique(np.r_[0, N - 1, wl.rng(N, 9).integers(0, N, 80)])
    ev = oracle.evaluate(f, x.cpu().numpy()[idx])
    assert np.abs(q["s"].cpu().numpy()[idx] - ev["s"]).max() <= 1e-4
    assert np.abs(q["c"].cpu().numpy()[idx] - ev["c"]).max() <= 3e-5
    err = np.abs(q["grad"].cpu().numpy()[idx] - ev["grad"]).max(axis=1)
    assert np.all(err <= 1e-5 * ev["scale"] + 1e-5 * np.abs(ev["grad"]).max(axis=1) + 1e-7)
    c, s, g = direct(fld, x)
    assert float((q["s"] - s).abs().max()) <= 2e-4 and float((q["c"] - c).abs().max()) <= 5e-5
    for want in (("c",), ("grad",), ("s", "grad")):
        part = pdmp.occupancy_query(fld, x, want=want)
        for k in ("c", "s", "grad"):
            assert (part[k] is None) == (k not in want)
            assert part[k] is None or torch.equal(part[k], q[k])


def test_points_that_are_not_finite():
    f = wl.random_field(5, wl.RBF, 2, 4096, lo=0, hi=40, gamma=4.0)
    fld = pdmp.DeviceField.from_host(f)
    x = wl.uniform_box(6, 3, 5000, np.zeros(2), np.full(2, 40.0))
    x[7] = np.nan
    x[8, 0] = np.inf
    x = torch.from_numpy(x).cuda()
    q = pdmp.occupancy_query(fld, x)
    c, s, g = direct(fld, x)
    for a, b in ((q["c"], c), (q["s"], s), (q["grad"], g)):
        assert torch.equal(torch.isnan(a), torch.isnan(b))
        assert float((a - b).nan_to_num().abs().max()) <= 1e-4
