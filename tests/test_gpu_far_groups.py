"""Sorted-tile kernels on ordered centres: groups of centres whose features are
all exactly zero on a tile are not visited.  Sizes at the edges of groups (32),
order chunks (16,384), the samples' one-launch order and the cluster rules,
against the oracle, and the cases in which no group may be left out."""
import numpy as np
import pytest
import torch

import oracle
import paper_2108_11775_gb300 as pdmp
import workloads as wl
from gpu_util import max_abs, rbf_eta, setup_oracle_threads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    assert torch.cuda.is_available()
    setup_oracle_threads()
    yield
    assert pdmp.stream_status()[0] == 0


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()


def wide_field(d, M, side, seed=7):
    """Centres over a box many feature widths across, some weights zero."""
    f = wl.random_field(seed + M, wl.RBF, d, M, lo=0, hi=side, gamma=4.0, wscale=1.5, bias=-0.2)
    w = f.w.copy()
    w[3::7] = 0.0
    return f.with_weights(w, bias=-0.2)


@pytest.mark.parametrize("d,M,N", [(2, 1, 129), (2, 31, 1), (3, 33, 128), (2, 1025, 16384), (3, 700, 16385),
                                   (2, 16385, 4097), (3, 16416, 20000), (2, 4096, 150000)])
def test_morph_and_vjp_with_far_groups(d, M, N):
    side = 30.0 if d == 2 else 12.0
    f = wide_field(d, M, side)
    lo, hi = np.zeros(d), np.full(d, side)
    eta, _ = rbf_eta(f, lo, hi, cells=24 if d == 2 else 8)
    fld = pdmp.DeviceField.from_host(f)
    x0 = wl.uniform_box(N + M, 3, N, lo - 1.0, hi + 1.0)
    T, k = 4, 2
    idx = np.unique(np.r_[0, N - 1, wl.rng(N, 9).integers(0, N, 60)])
    traj, _ = pdmp.morph_trace(fld, dev(x0), T, eta)
    xT = pdmp.morph(fld, dev(x0), T, eta)
    assert torch.equal(xT, traj[-1])
    assert max_abs(xT.cpu().numpy()[idx], oracle.morph(f, x0[idx], T, eta)) <= 1e-4
    gT = wl.f32(wl.rng(N, wl.S_COTANGENT).standard_normal((N, d)))
    g0 = pdmp.morph_vjp(fld, dev(x0), T, eta, k, dev(gT)).cpu().numpy()
    r0 = oracle.morph_vjp(f, x0[idx], T, eta, gT[idx])
    assert np.linalg.norm(g0[idx] - r0) <= 1e-4 * np.linalg.norm(r0)
    ld = pdmp.logdet(fld, dev(x0), T, eta).cpu().numpy()
    assert max_abs(ld[idx], oracle.logdet(f, x0[idx], T, eta)[0]) <= 1e-4 * T


@pytest.mark.parametrize("d,tiles", [(2, 3), (3, 3), (2, 115), (3, 305), (2, 457)])
def test_weight_gradient_in_the_callers_order(d, tiles):
    """Rows are summed in the centres' own order and handed back in the caller's;
    features of zero weight have a gradient too.  Whole tiles, as many as take
    clusters of 8, 4 and 2 blocks and single ones."""
    f = wide_field(d, 1500, 20.0 if d == 2 else 8.0)
    lo, hi = np.zeros(d), np.full(d, 20.0 if d == 2 else 8.0)
    eta, _ = rbf_eta(f, lo, hi, cells=24 if d == 2 else 8)
    N, T, k = tiles * (256 if d == 2 else 192), 4, 2
    x0 = wl.uniform_box(d, 3, N, lo, hi)
    gT = wl.f32(wl.rng(d, wl.S_COTANGENT).standard_normal((N, d)))
    _, gw, gb = pdmp.morph_vjp(pdmp.DeviceField.from_host(f), dev(x0), T, eta, k, dev(gT), want_param_grad=True)
    _, rw, rb = oracle.morph_vjp(f, x0, T, eta, gT, want_gw=True)
    assert np.linalg.norm(gw.cpu().numpy() - rw) <= 1e-4 * np.linalg.norm(rw)
    assert abs(float(gb) - rb) <= 1e-4 * max(abs(rb), np.linalg.norm(rw))


def test_what_is_not_finite_reaches_everything_it_reached():
    """An infinite centre makes its coordinate NaN for every sample wherever it is,
    and a NaN sample beside far groups stays in its own row."""
    f = wide_field(2, 600, 30.0)
    x0 = wl.uniform_box(3, 3, 5000, np.zeros(2), np.full(2, 30.0))
    fld = pdmp.DeviceField.from_host(f)
    bad = x0.copy()
    bad[17, 1] = np.nan
    out = pdmp.morph(fld, dev(bad), 3, 1e-3).cpu().numpy()
    ref = pdmp.morph(fld, dev(x0), 3, 1e-3).cpu().numpy()
    good = np.arange(5000) != 17
    assert np.isnan(out[17]).any() and max_abs(out[good], ref[good]) <= 1e-5
    c = f.centres.copy()
    c[5, 0] = np.inf
    inf = pdmp.DeviceField(pdmp.RBF, c, f.w, f.gamma, None, f.bias)
    assert torch.isnan(pdmp.morph(inf, dev(x0), 1, 1e-3)[:, 0]).all()   # that coordinate of every sample
