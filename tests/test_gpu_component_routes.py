"""Two columns in the component product of a large matrix: the Gram by tiles when its rows are long, in registers when
they are short, by whichever entry point; the row lengths are on the device only. The kernel that does the work
is read from a profile. G: sums of n <= 600,000 terms of any sign in blocks of a few hundred, off by less than
300 x 2^-53 = 3.4e-14 of the absolute terms."""
import numpy as np
import pytest

import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,factory,tiles", [
    ("stencil81", lambda: wl.stencil27(81, 2), True),
    ("poisson81", lambda: wl.poisson3d(81), False),
])
@pytest.mark.parametrize("scratch", [True, False])
def test_two_columns(name, factory, tiles, scratch):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2608_07327_gb300 as mb
    A = factory()
    n = A.n
    assert n > 1 << 19 and (A.nnz > 16 * n) is tiles
    rp, ci, av = (torch.as_tensor(a, device="cuda") for a in (A.row_ptr, A.col_idx, A.val))
    Ph = wl.initial_block(n, 2, 3)
    P = torch.as_tensor(np.ascontiguousarray(Ph), device="cuda")
    AP = torch.full_like(P, float("nan"))
    G = torch.full((2, 2), float("nan"), dtype=torch.float64, device="cuda")
    nbytes = mb.mbpcg_k_scratch_bytes(n, 2)
    buf = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    st = torch.cuda.current_stream().cuda_stream

    def call():
        if scratch:
            return mb.mbpcg_k_spmm_gram(n, rp, ci, av, 2, P, AP, G, buf, nbytes, st)
        return mb.mbpcg_k_spmm_gram_noalloc(n, rp, ci, av, 2, P, AP, G, st)

    took = {}
    for _ in range(2):  # the first profile of a process sees no kernels
        with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]) as prof:
            assert call() == 0
            torch.cuda.synchronize()
    on_device = [e for e in prof.events() if e.device_type == torch.autograd.DeviceType.CUDA]
    for e in on_device:
        if "k_spmm<2, true" in e.name:
            took["k_spmm<2, true, true" in e.name] = e.time_range.elapsed_us()
    if on_device:  # (nothing where another tool holds the profiler's interface)
        assert max(took, key=took.get) is tiles and took[tiles] > 20.0
        assert took.get(not tiles, 0.0) < 10.0
    Q = A.to_scipy() @ Ph
    assert np.allclose(AP.cpu().numpy(), Q, rtol=0, atol=1e-13 * np.abs(A.val).max())
    bound = 3.4e-14 * (np.abs(Ph).T @ np.abs(Q)).max()
    assert np.abs(G.cpu().numpy() - Ph.T @ Q).max() <= bound
