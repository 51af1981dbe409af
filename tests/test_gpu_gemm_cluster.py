"""Products below one wave of tiles: one launch, K split over the blocks of a cluster.

Shapes at the edges of the tiles (64 / 128 columns), of K tiles and of the rows each block adds up, for
every split, with the outputs and the bias alignments that a caller may pass.  The partial sums are added in
split order, so a split product equals the sum, in that order, of the products of the K ranges bit for bit;
the ranges themselves are held to the FP32 accumulation bound against FP64."""
import numpy as np
import pytest

from paper_2503_06757_gb300 import prrtc as P

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2503_06757_gb300 import build
    build.build()


def product(a, b, splits, bias=None, relu=False, c32=True, c16=True):
    M, K = a.shape
    N = b.shape[0]
    o32 = torch.full((M + 1, N), 7.0, device="cuda") if c32 else None
    o16 = torch.full((M + 1, N), 7.0, dtype=torch.bfloat16, device="cuda") if c16 else None
    P.prrtc_gemm_bf16_splitk(a.data_ptr(), b.data_ptr(), M, N, K, bias.data_ptr() if bias is not None else 0, relu,
                             o32.data_ptr() if c32 else 0, o16.data_ptr() if c16 else 0, splits,
                             torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    assert P.prrtc_gemm_error() == 0
    for o in (o32, o16):  # nothing is written below the last row
        assert o is None or bool((o[M] == 7.0).all())
    return (o32[:M] if c32 else None), (o16[:M] if c16 else None)


SHAPES = [(1, 8, 64), (128, 64, 512), (129, 72, 520), (127, 136, 1000), (300, 1024, 4096), (512, 520, 1032),
          (1024, 2056, 512), (40, 128, 4160), (640, 1000, 640)]


@pytest.mark.parametrize("splits", [1, 2, 4, 8])
@pytest.mark.parametrize("M,N,K", SHAPES)
def test_split_product_is_the_ordered_sum_of_its_ranges(M, N, K, splits):
    g = torch.Generator(device="cpu").manual_seed(M + N + K + splits)
    a = torch.randn(M, K, generator=g).to(torch.bfloat16).cuda()
    b = torch.randn(N, K, generator=g).to(torch.bfloat16).cuda()
    got, _ = product(a, b, splits)
    tiles = -(-K // 64)
    n = min(splits, tiles)
    cuts = np.cumsum([0] + [tiles // n + (s < tiles % n) for s in range(n)]) * 64
    total = None
    for k0, k1 in zip(cuts[:-1], np.minimum(cuts[1:], K)):
        part, _ = product(a[:, k0:k1].contiguous(), b[:, k0:k1].contiguous(), 1)
        aa, bb = a[:, k0:k1].double(), b[:, k0:k1].double()
        bound = (k1 - k0) * 2.0 ** -23 * (aa.abs() @ bb.abs().T) + 1e-6
        assert bool(((part.double() - aa @ bb.T).abs() <= bound).all())
        total = part if total is None else total + part
    assert torch.equal(got, total)


@pytest.mark.parametrize("splits", [1, 2, 4, 8])
@pytest.mark.parametrize("c32,c16", [(True, True), (True, False), (False, True)])
@pytest.mark.parametrize("offset", [0, 1, 3])
def test_bias_relu_and_outputs(splits, c32, c16, offset):
    g = torch.Generator(device="cpu").manual_seed(splits)
    a = torch.randn(200, 576, generator=g).to(torch.bfloat16).cuda()
    b = torch.randn(264, 576, generator=g).to(torch.bfloat16).cuda()
    bias = torch.randn(264 + offset, generator=g).cuda()[offset:]  # any 4-byte alignment
    plain, _ = product(a, b, splits)
    want = torch.relu(plain + bias)
    o32, o16 = product(a, b, splits, bias, True, c32, c16)
    if c32:
        assert torch.equal(o32, want)
    if c16:
        assert torch.equal(o16, want.to(torch.bfloat16))
