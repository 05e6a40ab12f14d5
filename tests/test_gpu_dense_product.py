"""The FP64 dense product at every row tile it runs (4 to 32 rows a CTA, one pass and two), even n by bulk
copies and odd n by 8-byte ones, and a ragged last chunk of 128.

Each entry is a sum of n FP64 products in some order: |AP - ref| <= 2 n 2^-53 (|A| |P|), for either side's order
against the other's."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mb():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2608_07327_gb300 as mb
    mb.lib()
    return mb


@pytest.mark.parametrize("n,s", [(1, 1), (3, 2), (640, 32), (1300, 4), (1301, 16), (2000, 8), (2001, 1), (2600, 32),
                                 (3500, 2), (3501, 5), (4100, 4), (4101, 32), (4700, 8), (5000, 16), (5001, 3)])
def test_dense_product(mb, n, s):
    gen = torch.Generator(device="cuda").manual_seed(n)
    A = torch.rand((n, n), generator=gen, dtype=torch.float64, device="cuda") - 0.5
    A = A + A.T
    kp = mb.mbpcg_k_padded_width(s)
    P = torch.zeros((n, kp), dtype=torch.float64, device="cuda")
    P[:, :s] = torch.rand((n, s), generator=gen, dtype=torch.float64, device="cuda") - 0.5
    AP = torch.full_like(P, float("nan"))
    assert mb.mbpcg_k_dense_product(n, A, s, P, AP, torch.cuda.current_stream().cuda_stream) == mb.MBPCG_OK
    bound = 2.0 * n * 2.0 ** -53 * (A.abs() @ P.abs())
    assert bool(((AP - A @ P).abs() <= bound).all())
