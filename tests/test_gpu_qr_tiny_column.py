"""The batched QR of matrices with a column so small that the square of its norm is subnormal (2^-1026): its reflector is
formed and the columns after it stay finite. Bounds: the definition as in the other QR tests, column by column; the
squares' sum carries 2 m 2^-1075 of 2^-1026, so reflectors are unitary to 2 m 2^-49 < 1e-12, with Q^H Q - I a few
hundred times that at most: 1e-10."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n", [(20, 8), (60, 30), (300, 40), (700, 70)])
@pytest.mark.parametrize("col", [0, 1, 6])
def test_tiny_column(m, n, col):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2201_05529_gb300 as pkg
    pkg.build()
    capi = pkg.load()
    capi.use_torch_allocator()
    rng = np.random.default_rng(m + n + col)
    A = rng.standard_normal((2, m, n)) + 1j * rng.standard_normal((2, m, n))
    # what is left of the column under the rows before it has the norm 2^-513
    below = np.linalg.norm(A[0, col:, col])
    A[0, :col, col] = 0.0
    A[0, :, col] *= 2.0 ** -513 / below
    if col > 0:
        A[0, col:, :col] = 0.0                            # so that the reflectors before leave it as it is
        A[0, :col, :col] += 4.0 * np.eye(col)
    At = torch.from_numpy(np.ascontiguousarray(A.transpose(0, 2, 1))).cuda()
    Rt = torch.zeros((2, n, n), dtype=torch.complex128, device="cuda")
    capi.qr_f64(At, Rt, torch.empty(capi.qr_scratch_bytes(m, n, 2), dtype=torch.uint8, device="cuda"))
    Q = At.cpu().numpy().transpose(0, 2, 1)
    R = Rt.cpu().numpy().transpose(0, 2, 1)
    assert np.isfinite(Q).all() and np.isfinite(R).all()
    for b in range(2):
        cols = np.abs(A[b]).max(axis=0)
        big = 2.0 ** 500                                  # the products of the tiny column in the normal range
        assert np.all(np.abs(Q[b] @ (R[b] * big) - A[b] * big).max(axis=0) <= 1e-10 * m * cols * big)
        assert np.abs(Q[b].conj().T @ Q[b] - np.eye(n)).max() <= 1e-10
