"""The pivoted QR of the bond SVD with its columns in global memory (one CTA per matrix, the matrices beyond a CTA's
shared memory) against shared memory (sixteen CTAs per matrix): many copies of one chain against the chain alone. The
two factorisations differ by rounding, so the observables agree to the bound the FP64 path has against the oracle."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_pivoted_qr_in_global_memory_against_shared_memory():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2201_05529_gb300 as pkg
    pkg.build()
    capi = pkg.load()
    capi.use_torch_allocator()
    from oracle import problem as oprob
    from workloads import workload
    from tests.gpu_helpers import OPS, run_gpu
    K, copies = 10, 76
    w = workload("xyz5_twobaths", K=K, chi_max=128)
    cis = oprob.build_inputs(w)
    eng, obs, _ = run_gpu(w, cis, OPS, route=("cluster_smem", "grid"))
    rec, _ = eng.read_bond_log(0, K)
    largest = (rec[..., 0].astype(np.int64) * rec[..., 1]).max()
    assert 16 * largest > 227 * 1024                      # beyond one CTA's shared memory
    eng.destroy()
    eng, many, _ = run_gpu(w, cis * copies, OPS, route=("cluster_global", "cta"))
    eng.destroy()
    for c in (0, copies // 2, copies - 1):
        assert np.abs(many[:, c] - obs[:, 0]).max() < 1e-9
