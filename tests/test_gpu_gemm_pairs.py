"""Products whose tiles are taken by pairs of CTAs (256 x 256).

Operands of small integers: every product and sum is exact in FP32, so the outputs equal the integer product.
Shapes with a second CTA that holds no row or no column of the last tile, ragged K, several waves, K ranges
through the workspace, and the number of K tiles on both sides of the rule."""
import pytest

from paper_2503_06757_gb300 import prrtc as P

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2503_06757_gb300 import build
    build.build()


@pytest.mark.parametrize("M,N,K,splits", [
    (2305, 2320, 840, 1), (2432, 4096, 776, 1), (2432, 4096, 768, 1),  # one row, 16 columns in the last tiles
    (2560, 2184, 1032, 0), (8192, 1032, 840, 1), (300, 20000, 840, 1),
    (1, 8, 2600, 3), (257, 264, 2496, 3), (700, 1000, 4160, 5), (130, 2000, 16648, 16),
])
@pytest.mark.parametrize("relu", [False, True])
def test_integer_products_are_exact(M, N, K, splits, relu):
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    a = torch.randint(-8, 9, (M, K), generator=g, device="cuda").to(torch.bfloat16)
    b = torch.randint(-8, 9, (N, K), generator=g, device="cuda").to(torch.bfloat16)
    bias = torch.randint(-99, 100, (N,), generator=g, device="cuda").float()
    assert 64 * K + 99 < 1 << 24
    c32 = torch.full((M + 1, N), 7.0, device="cuda")
    c16 = torch.full((M + 1, N), 7.0, dtype=torch.bfloat16, device="cuda")
    P.prrtc_gemm_bf16_splitk(a.data_ptr(), b.data_ptr(), M, N, K, bias.data_ptr(), relu, c32.data_ptr(),
                             c16.data_ptr(), splits, torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    assert P.prrtc_gemm_error() == 0
    want = a.double() @ b.double().T + bias
    want = (torch.relu(want) if relu else want).float()
    assert torch.equal(c32[:M], want)
    assert torch.equal(c16[:M], want.to(torch.bfloat16))
    assert bool((c32[M] == 7.0).all()) and bool((c16[M] == 7.0).all())
