"""The one-CTA transform where its CTAs walk more than one item of the work list:
every stamp of a large batch the same bits as alone (its transforms share nothing
with the items before), for square and oblong transforms of each length, in
evaluations and in fits whose stamps leave the loop at different times."""
import numpy as np
import pytest

import oracle
from gpu_util import assert_pix_close, noisy_image
from paper_1101_2254_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

KINDS = [synth.SERSIC, synth.SKY]
FFT_FLOOR = 2e-6  # float32 FFT round-off, relative to the peak (as in the method's other tests)


@pytest.fixture(scope="module")
def gf():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1101_2254_gb300 import build, gf as gf_
    build.build()
    return gf_


def cuda(x):
    return torch.as_tensor(np.ascontiguousarray(x, dtype=np.float32)).cuda()


# transforms of 96 x 96, 128 x 128, 160 x 160, 96 (y) x 160 (x) and 160 x 128; a launch has at
# most 4 waves of 152 SMs x 4 CTAs, fewer for the longer ones
@pytest.mark.parametrize("H,W,P,n", [(64, 64, 33, 2500), (95, 90, 33, 1900), (128, 121, 31, 700), (33, 140, 9, 1900),
                                     (130, 100, 25, 1300)])
def test_models_of_many_stamps(gf, H, W, P, n):
    rng = np.random.default_rng(H + P)
    m = 3  # distinct stamps, in turn
    p = np.array([synth.random_params(KINDS, rng, H, W) for _ in range(m)])
    psfs = [synth.random_psf(P, 5 * P + k) for k in range(m)]
    img, sig = cuda(rng.standard_normal((m, H, W))), cuda(rng.uniform(0.5, 2.0, (m, H, W)))
    d = gf.make_desc(H, W, P, KINDS, 1, 0, conv_method=gf.CONV_FFT)
    od = oracle.make_desc(H, W, P, KINDS, 1, 0)
    one = [gf.evaluate(d, p[k], img[k], sig[k], cuda(psfs[k])) for k in range(m)]
    for k in range(m):
        want = oracle.convolve_fft(oracle.model_ext(od, p[k]), psfs[k].astype(np.float64))
        assert_pix_close(one[k][1].cpu().numpy().reshape(H, W), want, floor=FFT_FLOOR, what=f"{H}x{W} P{P}")
    which = np.arange(n) % m
    at = torch.as_tensor(which).cuda()
    x2, y = gf.evaluate_batch(d, gf.make_batch([H] * n, [W] * n, psf_size=P), p[which], img[at].reshape(-1),
                              sig[at].reshape(-1), cuda(np.array(psfs))[at].reshape(-1), want_model=True)
    y = y.view(n, H, W)
    for k in range(m):
        assert bool((y[at == k] == one[k][1].view(1, H, W)).all()), k
        assert bool((x2[at == k] == one[k][0].view(-1)).all()), k


@pytest.mark.parametrize("side,P,n", [(64, 33, 450), (96, 33, 330), (128, 33, 120)])
def test_fits_of_many_stamps(gf, side, P, n):
    # eight channels a stamp in a Jacobian pass: more transforms than CTAs
    sts = synth.batch_stamps(3, seed=11 + side, smin=side, smax=side, psf_size=P)
    data = [noisy_image(st)[1:] for st in sts]
    start = [st.guess() for st in sts]
    start[1][2] *= 3.0  # (a longer way: the stamps leave the loop at different times)
    img, sig = cuda(np.array([i for i, _ in data])), cuda(np.array([s for _, s in data]))
    psf = cuda(np.array([st.psf for st in sts]))
    d = gf.make_desc(side, side, P, sts[0].kinds, 5, 8, conv_method=gf.CONV_FFT)
    opts = gf.default_opts(ladder=1)
    one = [gf.lm_fit(d, start[k], sts[k].fixed, img[k], sig[k], psf[k], opts) for k in range(3)]
    which = np.arange(n) % 3
    at = torch.as_tensor(which).cuda()
    p, r = gf.lm_fit_batch(d, gf.make_batch([side] * n, [side] * n, psf_size=P), np.array(start)[which], sts[0].fixed,
                           img[at].reshape(-1), sig[at].reshape(-1), psf[at].reshape(-1), opts)
    for k in range(3):
        assert (np.asarray(p)[which == k] == np.asarray(one[k][0])).all(), k
        assert (np.asarray(r.chi2)[which == k] == one[k][1]["chi2"]).all(), k
