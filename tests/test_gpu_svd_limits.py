"""The launch of the whole-GPU Jacobi behind the standalone SVD: CTAs whose matrices have converged wait for a whole sweep
of the others, which may take longer than the wait limit; the limit grows with a sweep's work. Where the device cannot
hold the launch's CTAs at once, one cluster per matrix does the work."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

PT_OK = 0


@pytest.fixture(scope="module")
def capi():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2201_05529_gb300 as pkg
    pkg.build()
    c = pkg.load()
    c.use_torch_allocator()
    return c


def _check(capi, A, **kw):
    import torch
    b, m, n = A.shape
    k = min(m, n)
    S = torch.zeros((b, k), dtype=torch.float64, device="cuda")
    U = torch.zeros((b, m, k), dtype=torch.complex128, device="cuda")
    V = torch.zeros((b, n, k), dtype=torch.complex128, device="cuda")
    scratch = torch.empty(capi.svd_scratch_bytes(m, n, b), dtype=torch.uint8, device="cuda")
    assert capi.selftest_svd(torch.from_numpy(A).cuda(), S, U, V, scratch, **kw) == PT_OK
    S, U, V = (x.cpu().numpy() for x in (S, U, V))
    for i in range(b):
        s = np.linalg.svd(A[i], compute_uv=False)
        tol = 1e-13 * max(m, n) * s[0]
        assert np.abs(S[i] - s).max() <= tol
        assert np.abs((U[i] * S[i]) @ V[i].conj().T - A[i]).max() <= tol


def test_a_sweep_may_take_longer_than_the_wait_limit(capi):
    """One matrix is diagonal, so its CTAs have nothing to do from the second sweep on; a sweep over the other takes ~1 ms,
    five times the limit."""
    rng = np.random.default_rng(1)
    A = rng.standard_normal((2, 256, 256)) + 1j * rng.standard_normal((2, 256, 256))
    A[0] = np.diag(np.arange(256, 0, -1.0))
    _check(capi, A, limit_ms=0.2)


@pytest.mark.parametrize("m,n,batch", [(1, 1, 1), (9, 7, 3), (70, 130, 2), (100, 100, 1)])
def test_a_refused_cooperative_launch_falls_back_to_clusters(capi, m, n, batch):
    """More CTAs than the device holds: the launch is refused on the host, before anything runs."""
    rng = np.random.default_rng(m + n)
    A = rng.standard_normal((batch, m, n)) + 1j * rng.standard_normal((batch, m, n))
    _check(capi, A, ctas=100000)
    _check(capi, A)
