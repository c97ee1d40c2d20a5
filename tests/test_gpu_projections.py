"""Projection kernels at the sizes where a launch takes another shape, against 64-bit products."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    t = pytest.importorskip("torch")
    if not t.cuda.is_available():
        pytest.skip("needs a CUDA device")
    return t


def check_linear(torch, M, N, K, ctas):
    from paper_2503_14153_b200 import spec_op_linear
    g = torch.Generator().manual_seed(M + N + K)
    x = torch.randn((M, K), generator=g).bfloat16().cuda()
    w = (torch.randn((N, K), generator=g) * 0.02).bfloat16().cuda()
    want = x.double() @ w.double().T
    y = spec_op_linear(x, w, ctas)
    # float32 sums of K products: K / 2 roundings of the running sum, each at most 2^-24 of the sum of the magnitudes
    bound = (K / 2 + 8) * 2.0 ** -24 * (x.double().abs() @ w.double().abs().T)
    assert ((y.double() - want).abs() <= bound).all()


@pytest.mark.parametrize("M,chunks", [(16, 5), (16, 6), (16, 12), (16, 13), (32, 11), (32, 12), (48, 9), (64, 4), (64, 9), (64, 10),
                                      (80, 4), (112, 7), (128, 3), (128, 8)])
def test_ring_depths(torch, M, chunks):
    """Grids of at most one CTA an SM get a stage for every K chunk of a CTA (`chunks`, here of a cluster of eight): the ring of which two fit an
    SM and one chunk more, the deepest ring full and run through again, and activation rows that fill the MMA's N only in part."""
    check_linear(torch, M, 1000, 8 * 64 * chunks, 128)
