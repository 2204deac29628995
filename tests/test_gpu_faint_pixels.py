"""Bright compact galaxies on a faint sky under the automatic method: every pixel
of a batched evaluation to the relative tolerance of the model, with no share of
the brightest pixel's round-off, and a stamp's numbers the same bits alone, in a
small batch and in a large one."""
import numpy as np
import pytest

import oracle
from gpu_util import REL, noisy_image
from paper_1101_2254_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

KINDS = [synth.SERSIC, synth.SKY]
# (I_e, r_e, n): fluxes of about 1e5, 1e6 and 1e6
GALAXIES = [(520.0, 4.0, 1.0), (9200.0, 3.0, 1.0), (8000.0, 2.5, 0.7)]


@pytest.fixture(scope="module")
def gf():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1101_2254_gb300 import build, gf as gf_
    build.build()
    return gf_


def cuda(x):
    return torch.as_tensor(np.ascontiguousarray(x, dtype=np.float32)).cuda()


def params(H, W, galaxy):
    ie, re, n = galaxy
    return np.array([0.5 * (W - 1) + 0.3, 0.5 * (H - 1) - 0.2, ie, re, n, 0.7, 34.0, 0.0, 0.05])


@pytest.mark.parametrize("P", [23, 33, 35, 39])
@pytest.mark.parametrize("H,W", [(64, 64), (81, 65)])
def test_faint_pixels_of_batched_evaluations(gf, P, H, W):
    # REL, the tolerance of the float32 model and convolution, without the floor
    # that assert_pix_close grants to pixels far below the peak: a direct sum of
    # positive terms has an error relative to its own value.
    want = [oracle.convolve_direct(oracle.model_ext(oracle.make_desc(H, W, P, KINDS, 5, 8), params(H, W, g)),
                                   synth.moffat_psf(P, 3.0).astype(np.float64)) for g in GALAXIES]
    n = 240  # at least 8 output blocks of 16 x 32 each
    p = np.array([params(H, W, GALAXIES[k % 3]) for k in range(n)])
    psf = cuda(np.tile(synth.moffat_psf(P, 3.0).ravel(), n))
    d = gf.make_desc(1, 1, P, KINDS, 5, 8)
    ones = torch.ones(n * H * W, device="cuda")
    _, m = gf.evaluate_batch(d, gf.make_batch([H] * n, [W] * n, psf_size=P), p, ones, ones, psf, want_model=True)
    m = m.cpu().numpy().astype(np.float64).reshape(n, H, W)
    for k in range(n):
        rel = np.abs(m[k] - want[k % 3]) / want[k % 3]
        assert rel.max() <= REL, (k, rel.max(), np.unravel_index(rel.argmax(), rel.shape))


@pytest.mark.parametrize("P", [21, 23, 31, 33, 35, 37, 39])
def test_a_stamps_numbers_do_not_depend_on_its_batch(gf, P):
    H, W = 61, 95
    p = params(H, W, GALAXIES[0])
    psf = cuda(synth.moffat_psf(P, 3.0))
    one = gf.make_desc(H, W, P, KINDS, 5, 8)
    rng = np.random.default_rng(P)
    sig = cuda(rng.uniform(0.5, 2.0, (H, W)))
    img = cuda(rng.standard_normal((H, W)))
    x1, m1 = gf.evaluate(one, p, img, sig, psf)
    d = gf.make_desc(1, 1, P, KINDS, 5, 8)
    for n in (1, 40, 300):  # 12 output blocks of 16 x 32 each
        x2, m = gf.evaluate_batch(d, gf.make_batch([H] * n, [W] * n, psf_size=P), np.tile(p, (n, 1)),
                                  img.view(-1).repeat(n), sig.view(-1).repeat(n), psf.view(-1).repeat(n), want_model=True)
        assert torch.equal(m.view(n, H, W), m1.view(1, H, W).expand(n, H, W)), n
        assert torch.equal(x2, x1.view(1).expand(n)), n


@pytest.mark.parametrize("P", [23, 33, 39])
def test_a_fit_does_not_depend_on_its_batch(gf, P):
    st = synth.batch_stamps(1, seed=7, smin=81, smax=81, psf_size=P)[0]
    _, img, sig = noisy_image(st)
    img, sig, psf = cuda(img), cuda(sig), cuda(st.psf)
    p1, r1 = gf.lm_fit(gf.make_desc(st.H, st.W, P, st.kinds, st.os_factor, st.os_box), st.guess(), st.fixed, img, sig, psf)
    d = gf.make_desc(1, 1, P, st.kinds, st.os_factor, st.os_box)
    for n in (1, 60):
        p, r = gf.lm_fit_batch(d, gf.make_batch([st.H] * n, [st.W] * n, psf_size=P), np.tile(st.guess(), (n, 1)), st.fixed,
                               img.view(-1).repeat(n), sig.view(-1).repeat(n), psf.view(-1).repeat(n))
        assert (np.asarray(p) == np.asarray(p1)).all() and (np.asarray(r.chi2) == r1["chi2"]).all()
