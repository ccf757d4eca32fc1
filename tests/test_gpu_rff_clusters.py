"""Random Fourier morphs of few tiles run on clusters: sample counts that take one,
two, four and eight blocks per tile, feature counts of fewer and odd numbers of
stages, against the oracle; the trace ends in the morph bit for bit, and a morph
that writes checkpoints (one block per tile) ends within rounding of it."""
import numpy as np
import pytest
import torch

import oracle
import paper_2108_11775_gb300 as pdmp
import workloads as wl
from gpu_util import max_abs, rff_eta_sampled, setup_oracle_threads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    assert torch.cuda.is_available()
    setup_oracle_threads()
    yield
    assert pdmp.stream_status()[0] == 0


@pytest.mark.parametrize("d,M,N", [(7, 1, 5), (7, 129, 300), (5, 700, 129), (7, 1100, 3000), (3, 2100, 12001),
                                   (7, 4096, 20000), (2, 1000, 45001), (6, 900, 70000)])
def test_morph_of_few_tiles(d, M, N):
    f = wl.random_field(M + d, wl.RFF, d, M, wscale=5.0, bias=0.1)
    lo, hi = np.full(d, -np.pi), np.full(d, np.pi)
    eta, _ = rff_eta_sampled(f, lo, hi, n=400)
    fld = pdmp.DeviceField.from_host(f)
    x0 = wl.uniform_box(N, 3, N, lo, hi)
    x = torch.from_numpy(x0).cuda()
    T, k = 4, 2
    idx = np.unique(np.r_[0, N - 1, wl.rng(N, 9).integers(0, N, 60)])
    xT = pdmp.morph(fld, x, T, eta)
    traj, _ = pdmp.morph_trace(fld, x, T, eta)
    assert torch.equal(xT, traj[-1])
    y = x.clone()
    assert torch.equal(pdmp.morph(fld, y, T, eta, out=y), xT)
    ref = oracle.morph(f, x0[idx], T, eta)
    assert max_abs(xT.cpu().numpy()[idx], ref) <= 1e-4
    ck = torch.empty(T // k, N, d, device="cuda")
    xc = pdmp.morph(fld, x, T, eta, ckpt=ck, k=k)
    assert torch.equal(ck[-1], xc)
    assert float((xc - xT).abs().max()) <= 2e-5
    assert float((ck[0] - traj[k]).abs().max()) <= 2e-5


@pytest.mark.parametrize("d,M", [(7, 300), (3, 1000)])
def test_dealing_tiles_out_in_halves_keeps_the_results(d, M):
    """One launch of whole tiles and halves behind a full wave, against launches
    of halves alone: the same log-det, end points, checkpoints and gradient of
    every sample, and a weight gradient that adds up."""
    N = 128 * 3 * torch.cuda.get_device_properties(0).multi_processor_count + 700
    f = wl.random_field(M + d, wl.RFF, d, M, wscale=5.0, bias=0.1)
    lo, hi = np.full(d, -np.pi), np.full(d, np.pi)
    eta, _ = rff_eta_sampled(f, lo, hi, n=400)
    fld = pdmp.DeviceField.from_host(f)
    x0 = wl.uniform_box(N, 3, N, lo, hi)
    x = torch.from_numpy(x0).cuda()
    gT = torch.from_numpy(wl.f32(wl.rng(N, wl.S_COTANGENT).standard_normal((N, d)))).cuda()
    T, k = 4, 2

    def run(sl):
        xs, gs = x[sl].clone(), gT[sl].clone()
        ck = torch.empty(T // k, xs.shape[0], d, device="cuda")
        xT = pdmp.morph(fld, xs, T, eta, ckpt=ck, k=k)
        ld, xl = pdmp.logdet(fld, xs, T, eta, want_xT=True)
        g0, gw, gb = pdmp.morph_vjp(fld, xs, T, eta, k, gs, ckpt=ck, want_param_grad=True)
        return [xT, ck.transpose(0, 1), ld, xl, g0], gw, gb

    whole, gw, gb = run(slice(0, N))
    cuts = [0, 65, 4000, 4128, 12000, N - 700, N]
    sw = torch.zeros_like(gw)
    for a, b in zip(cuts[:-1], cuts[1:]):
        parts, pw, _ = run(slice(a, b))
        for q, r in zip(whole, parts):
            assert torch.equal(q[a:b], r)
        sw += pw
    assert float((sw - gw).norm()) <= 1e-5 * float(gw.norm())
    idx = wl.rng(N, 9).integers(0, N, 40)
    assert max_abs(whole[2].cpu().numpy()[idx], oracle.logdet(f, x0[idx], T, eta)[0]) <= 1e-4 * T
