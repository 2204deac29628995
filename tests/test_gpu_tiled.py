"""The tiled one-CTA transform, which batched calls take under the automatic
method for PSF sides from 23 to 39: stamps of any sizes against the oracle and
the direct sum, at the edges of its 16 x 32 blocks and of its tiles, for both
transform lengths, with rectangular and one-pixel stamps in one batch; and
batched fits against single-stamp ones, which take the direct sum."""
import numpy as np
import pytest

import oracle
from gpu_util import CHI2_REL, assert_pix_close
from paper_1101_2254_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SIZES = [(64, 64), (65, 63), (1, 1), (3, 129), (128, 65), (80, 97), (16, 32), (17, 33), (200, 40), (31, 161)] * 17  # 1887 blocks: fewer would take the direct sum
KINDS = [synth.SERSIC, synth.EXPDISK, synth.SKY]


@pytest.fixture(scope="module")
def gf():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1101_2254_gb300 import build, gf as gf_
    build.build()
    return gf_


def cuda(xs):
    return torch.as_tensor(np.concatenate([np.asarray(x, np.float32).ravel() for x in xs])).cuda()


@pytest.mark.parametrize("P", [21, 23, 33, 35, 39])
def test_tiled_models_match_the_oracle_and_the_direct_sum(gf, P):
    rng = np.random.default_rng(P)
    params = [synth.random_params(KINDS, rng, max(H, 8), max(W, 8)) for H, W in SIZES]
    psfs = [synth.random_psf(P, 7 * P + k) for k in range(len(SIZES))]
    want = []
    for (H, W), p, psf in zip(SIZES, params, psfs):
        od = oracle.make_desc(H, W, P, KINDS, 1, 0)
        want.append(oracle.convolve_direct(oracle.model_ext(od, p), psf.astype(np.float64)))
    noisy = [synth.add_noise(m, 90 + k) for k, m in enumerate(want)]
    img, sig = cuda([i for i, _ in noisy]), cuda([s for _, s in noisy])
    b = gf.make_batch([h for h, _ in SIZES], [w for _, w in SIZES], psf_size=P)
    out = {}
    for method in (gf.CONV_AUTO, gf.CONV_DIRECT):
        d = gf.make_desc(1, 1, P, KINDS, 1, 0, conv_method=method)
        x2, m = gf.evaluate_batch(d, b, np.array(params), img, sig, cuda(psfs), want_model=True)
        out[method] = m.cpu().numpy().astype(np.float64), x2.cpu().numpy()
    same = np.array_equal(out[gf.CONV_AUTO][0], out[gf.CONV_DIRECT][0])
    assert same == (P < 23)  # below the line the automatic method is the direct sum
    at = 0
    for k, (w, (i, s)) in enumerate(zip(want, noisy)):
        got = out[gf.CONV_AUTO][0][at:at + w.size].reshape(w.shape)
        assert_pix_close(got, w, what=f"P {P} stamp {w.shape}")
        xo = oracle.chi2(i, s, w)
        assert abs(out[gf.CONV_AUTO][1][k] - xo) <= CHI2_REL * xo
        at += w.size


def test_tiled_fits_match_single_stamp_fits(gf):
    P = 23
    sts = synth.batch_stamps(6, seed=5, smin=48, smax=150, psf_size=P)
    imgs, sigs = [], []
    for st in sts:
        od = oracle.make_desc(st.H, st.W, P, st.kinds, st.os_factor, 8)
        i, s = synth.add_noise(oracle.render(od, st.params, st.psf), st.noise_seed)
        imgs.append(i)
        sigs.append(s)
    p0 = np.array([st.guess() for st in sts])
    b = gf.make_batch([st.H for st in sts], [st.W for st in sts], psf_size=P)
    d = gf.make_desc(1, 1, P, sts[0].kinds, 5, 8)
    fits = [gf.lm_fit_batch(d, b, p0, sts[0].fixed, cuda(imgs), cuda(sigs), cuda([st.psf for st in sts]),
                            opts=gf.default_opts(ladder=k)) for k in (0, 1, 3)]
    for p, r in fits[1:]:  # any ladder takes the same steps
        assert np.array_equal(p, fits[0][0]) and np.array_equal(r.chi2, fits[0][1].chi2)
    for k, st in enumerate(sts):
        one = gf.make_desc(st.H, st.W, P, st.kinds, 5, 8)
        _, rs = gf.lm_fit(one, p0[k], st.fixed, cuda([imgs[k]]).view(st.H, st.W), cuda([sigs[k]]).view(st.H, st.W),
                           cuda([st.psf]).view(P, P))
        assert abs(fits[0][1].chi2[k] - rs["chi2"]) <= CHI2_REL * rs["chi2"]
