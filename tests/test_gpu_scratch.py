"""The component products write nothing past the scratch size that the library asks for."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

GUARD = 8 << 20  # more than any product here could write: (8 CTAs/SM x 152 SMs) x 564 doubles


@pytest.fixture(scope="module")
def mb():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2608_07327_gb300 as mb
    mb.lib()
    return mb


@pytest.mark.parametrize("n,s", [(300, 32), (1500, 32), (4761, 32), (4761, 17), (9800, 32), (4761, 16), (40000, 4)])
@pytest.mark.parametrize("kind", ["csr", "csr_f32", "dense"])
def test_product_stays_in_scratch(mb, kind, n, s):
    if kind == "dense" and n > 4761:
        pytest.skip("the CSR products cover this n")
    kp, nbytes = mb.mbpcg_k_padded_width(s), mb.mbpcg_k_scratch_bytes(n, s)
    scratch = torch.full((nbytes + GUARD,), 0x5A, dtype=torch.uint8, device="cuda")
    dt = torch.float32 if kind == "csr_f32" else torch.float64
    gen = torch.Generator(device="cuda").manual_seed(7)
    P = torch.zeros((n, kp), dtype=dt, device="cuda")
    P[:, :s] = torch.rand((n, s), generator=gen, dtype=dt, device="cuda")
    AP, G = torch.empty_like(P), torch.empty((s, s), dtype=torch.float64, device="cuda")
    st = torch.cuda.current_stream().cuda_stream
    if kind == "dense":
        rc = mb.mbpcg_k_dense_gram(n, 2.0 * torch.eye(n, dtype=dt, device="cuda"), s, P, AP, G, scratch, nbytes, st)
    else:
        rp = torch.arange(n + 1, dtype=torch.int32, device="cuda")
        call = mb.mbpcg_k_spmm_gram if kind == "csr" else mb.mbpcg_k_spmm_gram_f32
        rc = call(n, rp, rp[:-1], torch.full((n,), 2.0, dtype=dt, device="cuda"), s, P, AP, G, scratch, nbytes, st)
    assert rc == mb.MBPCG_OK
    assert bool((scratch[nbytes:] == 0x5A).all())
    assert torch.equal(AP, 2.0 * P)
    # same-signed terms in FP64, or in pairs of FP32 (2^-46) over the rows of one CTA: below 1e-10 relative
    assert torch.allclose(G, 2.0 * P[:, :s].double().T @ P[:, :s].double(), rtol=1e-10, atol=0)
