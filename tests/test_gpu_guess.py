"""The default guess against the oracle at the sizes where its kernel's forms
change: stamps kept in shared memory or read again, more rows than are
tabulated, more aperture indices than the histogram has bins, rings of odd
length, single rows and columns.  Each size is a batch of its own, since the
largest stamp of a batch picks the form."""
import math

import numpy as np
import pytest
import oracle
from paper_1101_2254_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SIZES = [(64, 64), (33, 47), (97, 100), (98, 100), (256, 20), (257, 20), (257, 60), (300, 41), (1, 200), (150, 1),
         (2, 2), (3, 2), (1, 1)]


@pytest.fixture(scope="module")
def gf():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1101_2254_gb300 import build, gf as gf_
    build.build()
    return gf_


def stamp(H, W, seed):
    rng = np.random.default_rng(seed)
    if min(H, W) < 8:
        return rng.uniform(-0.2, 1.0, (H, W)).astype(np.float32)
    p = [W / 2 + rng.uniform(-2, 2), H / 2 + rng.uniform(-2, 2), rng.uniform(0.5, 5), rng.uniform(2, 0.2 * min(H, W) + 2),
         rng.uniform(0.7, 4), rng.uniform(0.3, 1), rng.uniform(0, 180), 0.0, -0.05]
    d = oracle.make_desc(H, W, 9, [oracle.SERSIC, oracle.SKY])
    return synth.add_noise(oracle.render(d, p, synth.moffat_psf(9, 3.0)), seed)[0]


@pytest.mark.parametrize("H,W", SIZES)
def test_default_guess_forms(gf, H, W):
    imgs = [stamp(H, W, 31 * H + W + k) for k in range(3)] + [np.full((H, W), 0.25, np.float32)]
    g = gf.default_guess(gf.make_batch([H] * 4, [W] * 4, psf_size=1),
                         torch.as_tensor(np.concatenate([im.ravel() for im in imgs])).cuda()).cpu().numpy()
    for k, im in enumerate(imgs):
        o = oracle.default_guess(im.astype(np.float64))
        assert g[k, 8] == o[8], (k, g[k], o)  # the median of the same float values
        # float64 sums of the same terms in another order
        assert np.allclose(g[k, [0, 1, 5]], o[[0, 1, 5]], rtol=1e-10, atol=1e-10), (k, g[k], o)
        assert abs((g[k, 6] - o[6] + 90.0) % 180.0 - 90.0) < 1e-7 or o[5] > 1.0 - 1e-9, (k, g[k], o)
        assert g[k, 3] == o[3] and math.isclose(g[k, 2], o[2], rel_tol=1e-10), (k, g[k], o)


def test_default_guess_of_masked_pixels(gf):
    """NaN pixels give no centre, the unit flux and r_e = 1; infinite ones no aperture."""
    im = stamp(64, 64, 5)
    im[30, 31] = np.nan
    g = gf.default_guess(gf.make_batch([64], [64], psf_size=1), torch.as_tensor(im).cuda()).cpu().numpy()[0]
    assert g[0] == g[1] == 31.5 and g[3] == 1.0 and np.isfinite(g[2])
