"""The network's gradient and forward at batch sizes whose last tiles are ragged,
against the same samples repeated."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def gf():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1101_2254_gb300 import build, gf as gf_
    build.build()
    return gf_


def network(gf, nb, seed):
    g = torch.Generator().manual_seed(seed)
    x = torch.randn((nb, 64, 64), generator=g).bfloat16().float()
    t = torch.randn((nb, 8), generator=g)
    return gf.cnn_init(seed), x.cuda(), t.cuda()


@pytest.mark.parametrize("nb,copies", [(1, 64), (3, 22), (35, 3), (130, 2)])
def test_gradient_of_repeated_samples(gf, nb, copies):
    # the mean loss of a batch and of the batch repeated are the same number, and
    # all products of the gradient's sums are exact: only the order of at most
    # 260 x 1024 float32 additions and the rounding of 1 / nb differ, about
    # sqrt(2.7e5) 2^-24 = 3e-5 of a block's RMS at random signs; bound 2e-4.  A
    # pixel, tap or sample left out or counted twice is above 1e-3.
    w, x, t = network(gf, nb, 31 + nb)
    loss, g = gf.cnn_loss_grad(w, x, t)
    loss, g = float(loss.item()), g.double().clone()
    loss2, g2 = gf.cnn_loss_grad(w, x.repeat(copies, 1, 1), t.repeat(copies, 1))
    assert abs(float(loss2.item()) - loss) <= 1e-5 * loss
    ends = [0, 288, 320, 18752, 18816, 55680, 55744, 129472, 129600, 195136, 195168, 195424, 195432]
    for a, b in zip(ends, ends[1:]):
        rms = float(g[a:b].square().mean().sqrt())
        assert float((g2[a:b].double() - g[a:b]).abs().max()) <= 2e-4 * rms, (a, b)


@pytest.mark.parametrize("nb", [2047, 2048, 2051])
def test_forward_of_repeated_samples(gf, nb):
    # both sides of the batch size at which the dense layer takes four samples a
    # block: each output's sum is in the same order
    w, x, _ = network(gf, 7, 5)
    y = gf.cnn_forward(w, x)
    yn = gf.cnn_forward(w, x.repeat(nb // 7 + 1, 1, 1)[:nb])
    assert torch.equal(yn, y.repeat(nb // 7 + 1, 1)[:nb])
