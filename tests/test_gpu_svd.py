"""The batched FP64 one-sided Jacobi SVD (pt_svd_f64) against its definition at the sizes where the whole-GPU kernel
changes its work: single columns, odd counts, block edges (1, 2, 4 or 8 columns per block), a mix that fills
several blocks, wide matrices, columns too long for shared memory, matrices of very small and large scale, graded,
rank-deficient and repeated singular values. Bounds: |A - U S V^H| and |U^H U - I| within 1e-13 max(m, n) (rotations
unitary to rounding, at most a few thousand per column), sigma against LAPACK within 1e-13 max(m, n) of sigma_1."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n,batch,scale", [(1, 1, 1, 1.0), (5, 1, 2, 1.0), (2, 2, 3, 1.0), (3, 3, 1, 1e-60), (9, 7, 4, 1e60),
                                             (17, 16, 2, 1.0), (33, 33, 1, 1.0), (20, 50, 3, 1.0), (129, 65, 9, 1.0),
                                             (256, 130, 2, 1.0), (7200, 3, 1, 1.0)])
def test_jacobi_svd_against_definition(m, n, batch, scale):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2201_05529_gb300 as pkg
    pkg.build()
    capi = pkg.load()
    capi.use_torch_allocator()
    rng = np.random.default_rng(m * 1009 + n)
    A = rng.standard_normal((batch, m, n)) + 1j * rng.standard_normal((batch, m, n))
    A[0] *= np.exp(-12.0 * np.arange(n) / max(1, n))[None, :]            # graded
    if batch > 1 and n > 2:
        A[1][:, 2] = A[1][:, 0] - A[1][:, 1]                             # rank-deficient
    if batch > 2 and min(m, n) > 3:
        q1 = np.linalg.qr(A[2] if m >= n else A[2].T)[0]
        A[2] = (q1 if m >= n else q1.T) * 1.0                            # all singular values equal
    A = A * scale
    k = min(m, n)
    At = torch.from_numpy(A).cuda()
    S = torch.zeros((batch, k), dtype=torch.float64, device="cuda")
    U = torch.zeros((batch, m, k), dtype=torch.complex128, device="cuda")
    V = torch.zeros((batch, n, k), dtype=torch.complex128, device="cuda")
    capi.svd_f64(At, S, U, V, torch.empty(capi.svd_scratch_bytes(m, n, batch), dtype=torch.uint8, device="cuda"))
    S, U, V = S.cpu().numpy(), U.cpu().numpy(), V.cpu().numpy()
    tol = 1e-13 * max(m, n)
    for b in range(batch):
        s = np.linalg.svd(A[b], compute_uv=False)
        assert np.all(np.diff(S[b]) <= 0)
        assert np.abs(S[b] - s).max() <= tol * s[0]
        assert np.abs((U[b] * S[b]) @ V[b].conj().T - A[b]).max() <= tol * s[0]
        r = int((s > 1e-10 * s[0]).sum())                                # vectors of the null space are arbitrary in U
        assert np.abs(U[b][:, :r].conj().T @ U[b][:, :r] - np.eye(r)).max() <= 1e-13 * max(m, n)
        assert np.abs(V[b].conj().T @ V[b] - np.eye(k)).max() <= tol


@pytest.mark.parametrize("m,n,r", [(97, 130, 24), (128, 32, 8), (256, 256, 64), (64, 64, 1), (31, 31, 30)])
def test_jacobi_svd_of_low_rank(m, n, r):
    """Matrices of exact rank r: the columns of the null space shrink to rounding level over many rotations, which
    closed-form norms alone do not follow. The rest of the spectrum stays within 100 max(m, n) u of sigma_1."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2201_05529_gb300 as pkg
    pkg.build()
    capi = pkg.load()
    capi.use_torch_allocator()
    rng = np.random.default_rng(m + n + r)
    k = min(m, n)
    A = (rng.standard_normal((1, m, r)) + 1j * rng.standard_normal((1, m, r))) @ rng.standard_normal((r, n))
    S = torch.zeros((1, k), dtype=torch.float64, device="cuda")
    U = torch.zeros((1, m, k), dtype=torch.complex128, device="cuda")
    V = torch.zeros((1, n, k), dtype=torch.complex128, device="cuda")
    capi.svd_f64_noalloc(torch.from_numpy(A).cuda(), S, U, V)
    S, U, V = S.cpu().numpy()[0], U.cpu().numpy()[0], V.cpu().numpy()[0]
    s = np.linalg.svd(A[0], compute_uv=False)
    tol = 1e-13 * max(m, n)
    assert np.abs(S - s).max() <= tol * s[0]
    assert S[r:].max() <= 100 * max(m, n) * 1.2e-16 * s[0]
    assert np.abs((U * S) @ V.conj().T - A[0]).max() <= tol * s[0]


@pytest.mark.parametrize("m,n,batch,kind", [(96, 96, 1, "graded"), (97, 130, 2, "rank"), (384, 95, 2, "graded"),
                                            (128, 32, 3, "rank"), (33, 140, 1, "rows"), (100, 100, 2, "rows"),
                                            (257, 129, 2, "columns"), (160, 160, 1, "zero"), (96, 96, 2, "huge")])
def test_svd_after_two_qrs_against_the_direct_call(m, n, batch, kind):
    """The calls that go through two QR factorisations give what the direct Jacobi (the call without a workspace) gives:
    the same bounds against A, and singular values within 1e-13 max(m, n) sigma_1 of the direct call's."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2201_05529_gb300 as pkg
    pkg.build()
    capi = pkg.load()
    capi.use_torch_allocator()
    rng = np.random.default_rng(m * 1013 + n)
    k = min(m, n)
    A = rng.standard_normal((batch, m, n)) + 1j * rng.standard_normal((batch, m, n))
    if kind == "graded":
        A = A @ np.diag(np.exp(-20.0 * np.arange(n) / n)) @ (rng.standard_normal((n, n)) / np.sqrt(n))
    elif kind == "rank":
        A = A[:, :, :k // 4] @ (rng.standard_normal((k // 4, n)) + 0j)
    elif kind == "rows":
        A = A * 10.0 ** rng.uniform(-9, 0, m)[:, None]
    elif kind == "columns":
        A = A * 10.0 ** rng.uniform(-9, 0, n)
    elif kind == "zero":
        A = A * 0.0
    elif kind == "huge":
        A = A * 1e70
    At = torch.from_numpy(A).cuda()
    out = []
    for direct in (False, True):
        S = torch.zeros((batch, k), dtype=torch.float64, device="cuda")
        U = torch.zeros((batch, m, k), dtype=torch.complex128, device="cuda")
        V = torch.zeros((batch, n, k), dtype=torch.complex128, device="cuda")
        if direct:
            capi.svd_f64_noalloc(At, S, U, V)
        else:
            capi.svd_f64(At, S, U, V, torch.empty(capi.svd_scratch_bytes(m, n, batch), dtype=torch.uint8, device="cuda"))
        out.append([x.cpu().numpy() for x in (S, U, V)])
    tol = 1e-13 * max(m, n)
    (S, U, V), (S0, _, _) = out
    for b in range(batch):
        s1 = max(S0[b][0], 1e-300)
        assert np.all(np.diff(S[b]) <= 0)
        assert np.abs(S[b] - S0[b]).max() <= tol * s1
        assert np.abs((U[b] * S[b]) @ V[b].conj().T - A[b]).max() <= tol * s1
        W = (V if m >= n else U)[b]                                      # the factor that is unitary in any case
        assert np.abs(W.conj().T @ W - np.eye(k)).max() <= tol
        r = int((S0[b] > 1e-10 * s1).sum())
        X = (U if m >= n else V)[b][:, :r]
        assert r == 0 or np.abs(X.conj().T @ X - np.eye(r)).max() <= tol


@pytest.mark.parametrize("value,n", [(np.nan, 100), (np.inf, 100)])
def test_svd_of_a_non_finite_matrix_answers_as_the_direct_call(value, n):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2201_05529_gb300 as pkg
    pkg.build()
    capi = pkg.load()
    capi.use_torch_allocator()
    A = np.random.default_rng(n).standard_normal((1, n, n)) + 0j
    A[0, 3, 2] = value
    At = torch.from_numpy(A).cuda()
    said = []
    for direct in (False, True):
        S = torch.zeros((1, n), dtype=torch.float64, device="cuda")
        U, V = (torch.zeros((1, n, n), dtype=torch.complex128, device="cuda") for _ in range(2))
        try:
            if direct:
                capi.svd_f64_noalloc(At, S, U, V)
            else:
                capi.svd_f64(At, S, U, V, torch.empty(capi.svd_scratch_bytes(n, n, 1), dtype=torch.uint8, device="cuda"))
            said.append("")
        except Exception as e:
            said.append(str(e).split(":")[0])
    assert said[0] == said[1]
