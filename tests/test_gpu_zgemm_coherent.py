"""The sliced complex GEMM (pt_zgemm_sliced) on operands whose slices add up coherently: constant complex entries, for
which the real part of A^H B is the sum of 2 K equal products, up to and across the 512-long chunks of K.

Error bound. Entries x (1 + i), |x| in (1/2, 1), have exponent 0. The levels 3, 4 and 5 of a chunk accumulate in one FP32
sum: at most 1024 (2 128 64 + 2 64 64) (1 + 2^-6) 2^-35 < 2^-10, so a truncation drops at most 2^-34, and a chunk of 32
K steps makes 32 x 15 x 2 = 960 of them: 2^-24.1, or 2^-33.1 per product term, 2^-31.1 relative to max|row| max|column|
>= 1/4. Dropped levels (2^-40) and the exact levels add nothing to speak of: 2^-31 K max|row| max|column|."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [320, 338, 384, 448, 512, 513, 1024])
@pytest.mark.parametrize("x", [0.5, 0.707, 0.832, 0.957, 127 / 128 + 63 * sum(2.0 ** (-7 * j) for j in range(2, 7))])
def test_constant_operands(x, k):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2201_05529_gb300 as pkg
    pkg.build()
    capi = pkg.load()
    capi.use_torch_allocator()
    m, n = 5, 3
    for sign in (1.0, -1.0):
        for conj in (1, -1):                     # Re = 2 x^2 K, or Im
            A = torch.full((1, m, k), sign * x * (1 + 1j), dtype=torch.complex128, device="cuda")
            B = torch.full((1, n, k), x * (1 + conj * 1j), dtype=torch.complex128, device="cuda")
            C = torch.zeros((1, n, m), dtype=torch.complex128, device="cuda")
            scratch = torch.empty(capi.zgemm_scratch_bytes(m, n, k, 1), dtype=torch.uint8, device="cuda")
            capi.zgemm_sliced("H", "N", A, B, C, m, n, k, scratch)
            ref = sign * 2.0 * x * x * k * (1.0 if conj > 0 else -1j)
            assert np.abs(C.cpu().numpy() - ref).max() <= 2.0 ** -31 * k * x * x
