"""Singular values of matrices whose columns, or rows, have very different scales, on the path with two QRs: A = B D or D B
with B well conditioned and D over twelve decades. Every singular value is then determined to a relative accuracy of
rounding times cond(B) (Demmel and Veselic), and the sorting by norms in front of the QRs is there to keep it.

Reference: a one-sided Jacobi in numpy's FP64 on the form whose columns carry the scales, which has that accuracy. Bound:
1e-13 max(m, n) cond(B), relative, for each value; cond(B) is below 10 here."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _jacobi(A):
    """Singular values by one-sided Jacobi on the columns of A (round-robin, all pairs of a round at once)."""
    A = A.copy()
    n = A.shape[1]
    if n % 2:
        A = np.concatenate([A, np.zeros((A.shape[0], 1))], axis=1)
    n2 = A.shape[1]
    order = np.arange(n2)
    for sweep in range(60):
        most = 0.0
        for _ in range(n2 - 1):
            i, j = order[:n2 // 2], order[n2 // 2:][::-1]
            x, y = A[:, i], A[:, j]
            al, be = (np.abs(x) ** 2).sum(0), (np.abs(y) ** 2).sum(0)
            g = (x.conj() * y).sum(0)
            ag = np.abs(g)
            live = (al > 0) & (be > 0) & (ag > 0)
            c = np.where(live, ag / np.sqrt(np.where(live, al * be, 1.0)), 0.0)
            most = max(most, c.max())
            z = np.where(live, (be - al) / np.where(live, 2 * ag, 1.0), 0.0)
            t = np.where(live, np.where(z >= 0, 1.0, -1.0) / (np.abs(z) + np.sqrt(1 + z * z)), 0.0)
            cs = 1 / np.sqrt(1 + t * t)
            ph = np.where(live, g / np.where(live, ag, 1.0), 1.0)
            A[:, i], A[:, j] = cs * x - cs * t * ph.conj() * y, cs * y + cs * t * ph * x
            order = np.concatenate([order[:1], order[-1:], order[1:-1]])
        if most < 4e-16 * np.sqrt(A.shape[0]):
            break
    return np.sort(np.sqrt((np.abs(A) ** 2).sum(0)))[::-1][:n]


@pytest.mark.parametrize("m,n,kind", [(96, 96, "columns"), (130, 97, "columns"), (256, 256, "columns"), (300, 33, "columns"),
                                      (96, 96, "rows"), (97, 130, "rows"), (256, 256, "rows"), (40, 200, "rows")])
def test_graded_matrices_keep_relative_accuracy(m, n, kind):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2201_05529_gb300 as pkg
    pkg.build()
    capi = pkg.load()
    capi.use_torch_allocator()
    rng = np.random.default_rng(m * 1031 + n)
    k = min(m, n)
    G = rng.standard_normal((max(m, n), k)) + 1j * rng.standard_normal((max(m, n), k))
    B = np.linalg.qr(G)[0] + 0.05 / np.sqrt(k) * (rng.standard_normal(G.shape) + 1j * rng.standard_normal(G.shape))
    cond = np.linalg.cond(B)
    assert cond < 10
    C = B * 10.0 ** rng.uniform(-12, 0, k)                # the scales on the columns
    A = C if kind == "columns" else C.conj().T            # the same values either way
    S = torch.zeros((1, k), dtype=torch.float64, device="cuda")
    U = torch.zeros((1, m, k), dtype=torch.complex128, device="cuda")
    V = torch.zeros((1, n, k), dtype=torch.complex128, device="cuda")
    At = torch.from_numpy(np.ascontiguousarray(A[None])).cuda()
    assert At.shape == (1, m, n)
    capi.svd_f64(At, S, U, V, torch.empty(capi.svd_scratch_bytes(m, n, 1), dtype=torch.uint8, device="cuda"))
    s = _jacobi(C)
    err = np.abs(S.cpu().numpy()[0] / s - 1).max()
    print(f"{m} x {n} {kind}: largest relative error {err:.1e}, cond(B) {cond:.1f}")
    assert err <= 1e-13 * max(m, n) * cond
