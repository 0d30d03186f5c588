"""The batched FP64 SVD of matrices of very small and very large scale. A power of two scales every operation of the
algorithm exactly, so U and V are the same bits and sigma is scaled exactly, as long as squares of the entries stay in
FP64's normal range (2^-1022 .. 2^1023) with 106 bits to spare for the columns that still count."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n,batch", [(2, 2, 1), (9, 7, 3), (64, 64, 1), (40, 130, 2), (100, 100, 2), (260, 50, 1)])
@pytest.mark.parametrize("direct", [False, True])
def test_svd_scales_exactly(m, n, batch, direct):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2201_05529_gb300 as pkg
    pkg.build()
    capi = pkg.load()
    capi.use_torch_allocator()
    rng = np.random.default_rng(m * 1021 + n)
    k = min(m, n)
    A = rng.standard_normal((batch, m, n)) + 1j * rng.standard_normal((batch, m, n))
    A[0] *= np.exp(-12.0 * np.arange(n) / n)

    def svd(X):
        S = torch.zeros((batch, k), dtype=torch.float64, device="cuda")
        U = torch.zeros((batch, m, k), dtype=torch.complex128, device="cuda")
        V = torch.zeros((batch, n, k), dtype=torch.complex128, device="cuda")
        if direct:
            capi.svd_f64_noalloc(torch.from_numpy(X).cuda(), S, U, V)
        else:
            capi.svd_f64(torch.from_numpy(X).cuda(), S, U, V,
                         torch.empty(capi.svd_scratch_bytes(m, n, batch), dtype=torch.uint8, device="cuda"))
        return [x.cpu().numpy() for x in (S, U, V)]

    S, U, V = svd(A)
    for b in range(batch):
        assert np.abs(S[b] - np.linalg.svd(A[b], compute_uv=False)).max() <= 1e-13 * max(m, n) * S[b][0]
    for e in (-400, -256, -250, 249, 256, 400):
        s, u, v = svd(A * 2.0 ** e)
        assert np.array_equal(s, S * 2.0 ** e), e
        assert np.array_equal(u, U) and np.array_equal(v, V), e
