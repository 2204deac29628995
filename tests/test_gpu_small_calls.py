"""Small launches against large ones of the same work: the direct convolution's
kernel for few output blocks against the one for many (the same bits, in models,
chi^2 and a fit's trials)."""
import numpy as np
import pytest

from paper_1101_2254_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

KINDS = [synth.SERSIC, synth.EXPDISK, synth.SKY]


@pytest.fixture(scope="module")
def gf():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1101_2254_gb300 import build, gf as gf_
    build.build()
    return gf_


@pytest.mark.parametrize("P", [1, 3, 5, 7, 17, 25, 27, 33, 35])
@pytest.mark.parametrize("H,W", [(1, 1), (16, 32), (17, 33), (61, 95)])
def test_few_blocks_give_the_bits_of_many(gf, P, H, W):
    # one stamp has at most 12 output blocks of 16 x 32; 700 copies have at least
    # 700.  Every output sums its taps in the same order in both: equal bits.
    n = 700
    rng = np.random.default_rng(100 * P + H)
    p = synth.random_params(KINDS, rng, max(H, 8), max(W, 8))
    psf = torch.as_tensor(synth.random_psf(P, P).astype(np.float32).ravel()).cuda()
    img = torch.as_tensor(rng.standard_normal(H * W).astype(np.float32)).cuda()
    sig = torch.as_tensor(rng.uniform(0.5, 2.0, H * W).astype(np.float32)).cuda()
    d = gf.make_desc(1, 1, P, KINDS, 1, 0, conv_method=gf.CONV_DIRECT)
    out = []
    for k in (1, n):
        x2, m = gf.evaluate_batch(d, gf.make_batch([H] * k, [W] * k, psf_size=P), np.tile(p, (k, 1)),
                                  img.repeat(k), sig.repeat(k), psf.repeat(k), want_model=True)
        out.append((x2.cpu().numpy(), m.cpu().numpy().reshape(k, H * W)))
    assert np.isfinite(out[0][1]).all()
    assert (out[1][1] == out[0][1]).all() and (out[1][0] == out[0][0]).all()


@pytest.mark.parametrize("P,H,W", [(25, 61, 95), (7, 48, 33)])
def test_few_block_fits_take_the_steps_of_many(gf, P, H, W):
    n = 200
    rng = np.random.default_rng(P)
    p = synth.random_params(KINDS, rng, H, W)
    psf = torch.as_tensor(synth.random_psf(P, P).astype(np.float32).ravel()).cuda()
    img = torch.as_tensor(rng.standard_normal(H * W).astype(np.float32)).cuda()
    sig = torch.as_tensor(rng.uniform(0.5, 2.0, H * W).astype(np.float32)).cuda()
    sig[::7] = 0.0  # pixels that count nothing
    img[::11] = float("nan")
    d = gf.make_desc(1, 1, P, KINDS, 1, 0, conv_method=gf.CONV_DIRECT)
    fits = []
    for k in (1, n):
        b = gf.make_batch([H] * k, [W] * k, psf_size=P)
        fits.append(gf.lm_fit_batch(d, b, np.tile(p, (k, 1)), None, img.repeat(k), sig.repeat(k), psf.repeat(k)))
    (p1, r1), (pn, rn) = fits
    assert (np.asarray(pn) == np.asarray(p1)[0]).all()
    assert (np.asarray(rn.chi2) == np.asarray(r1.chi2)[0]).all()


def test_nan_amplitude_is_nan_everywhere(gf):
    # with n inside the table of b_n, above it (solved for otherwise) and below zero;
    # the stamp beside them keeps its bits
    kinds, H, W, P = [synth.SERSIC, synth.SKY], 20, 33, 5
    rng = np.random.default_rng(4)
    p = np.tile(synth.random_params(kinds, rng, H, W), (5, 1))
    p[1:, 4] = 3.0, 12.0, -1.0, 12.0
    p[1:4, 2] = np.nan
    img = torch.as_tensor(rng.standard_normal(5 * H * W).astype(np.float32)).cuda()
    psf = torch.as_tensor(np.tile(synth.random_psf(P, 1).astype(np.float32).ravel(), 5)).cuda()
    d = gf.make_desc(1, 1, P, kinds, 1, 0)

    def run(rows):
        n = H * W
        x2, m = gf.evaluate_batch(d, gf.make_batch([H] * len(rows), [W] * len(rows), psf_size=P), p[rows],
                                  torch.cat([img[r * n:(r + 1) * n] for r in rows]),
                                  torch.ones(len(rows) * n, device="cuda"), psf[:len(rows) * P * P], want_model=True)
        return x2.cpu().numpy(), m.cpu().numpy().reshape(len(rows), n)

    x2, m = run([0, 1, 2, 3, 4])
    assert np.isnan(m[1:4]).all() and np.isfinite(m[[0, 4]]).all() and np.isfinite(x2[[0, 4]]).all()
    for k in (0, 4):
        y2, my = run([k])
        assert y2[0] == x2[k] and np.array_equal(my[0], m[k])
