"""The tensor-core DFT's two forms of its contiguous contractions (16-byte loads
where the last digit of the width is even, single values where it is odd), with
several stamps in a call, so that no stamp but the first starts at the buffers'
beginning: against the oracle, and each stamp the same bits as alone."""
import numpy as np
import pytest

import oracle
from gpu_util import assert_pix_close
from paper_1101_2254_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

KINDS = [synth.SERSIC, synth.SKY]
# split-precision bf16 products: the floor of the method's other parity tests
DFT_FLOOR = 5e-5


@pytest.fixture(scope="module")
def gf():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1101_2254_gb300 import build, gf as gf_
    build.build()
    return gf_


# extended widths 63 = 1 x 63 (odd, one digit), 69 = 3 x 23, 99 = 9 x 11 (odd), 88 = 2 x 44,
# 152 = 4 x 38 (even); heights 33 = 11 x 3, 39 = 13 x 3, 84 = 12 x 7, 88 = 11 x 8, 232 = 29 x 8
@pytest.mark.parametrize("H,W,P", [(27, 57, 7), (31, 61, 9), (75, 91, 9), (64, 64, 25), (200, 120, 33)])
def test_stamps_of_one_call(gf, H, W, P):
    n = 3
    rng = np.random.default_rng(H + W)
    p = np.array([synth.random_params(KINDS, rng, H, W) for _ in range(n)])
    psfs = [synth.random_psf(P, 11 * P + k) for k in range(n)]
    psf = torch.as_tensor(np.concatenate([q.ravel() for q in psfs])).float().cuda()
    img = torch.as_tensor(rng.standard_normal(n * H * W).astype(np.float32)).cuda()
    sig = torch.as_tensor(rng.uniform(0.5, 2.0, n * H * W).astype(np.float32)).cuda()
    d = gf.make_desc(H, W, P, KINDS, 1, 0, conv_method=gf.CONV_DFT_TC)
    x2, m = gf.evaluate_batch(d, gf.make_batch([H] * n, [W] * n, psf_size=P), p, img, sig, psf, want_model=True)
    m = m.view(n, H, W)
    od = oracle.make_desc(H, W, P, KINDS, 1, 0)
    for k in range(n):
        want = oracle.convolve_fft(oracle.model_ext(od, p[k]), psfs[k].astype(np.float64))
        assert_pix_close(m[k].cpu().numpy(), want, floor=DFT_FLOOR, what=f"stamp {k} of {H}x{W} P{P}")
        at = slice(k * H * W, (k + 1) * H * W)
        y2, one = gf.evaluate(d, p[k], img[at].view(H, W), sig[at].view(H, W), psf[k * P * P:(k + 1) * P * P].view(P, P))
        assert torch.equal(one.view(H, W), m[k]) and float(y2.view(-1)[0]) == float(x2[k])
