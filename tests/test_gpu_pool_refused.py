"""The blocked QRs' workspace is optional: where the device has no memory left for it, the unblocked kernels do the work.
The allocator of this test refuses that one request and leaves the runtime with the error of a real failed allocation."""
import ctypes

import numpy as np
import pytest

from workloads import workload
from oracle import problem as oprob
from tests.gpu_helpers import OPS, engine_args_from_oracle

pytestmark = pytest.mark.gpu


def test_a_refused_qr_workspace_is_no_error():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2201_05529_gb300 as pkg
    pkg.build()
    capi = pkg.load()
    w = workload("random32_stress", K=2)
    w.random_state = dict(N=6, chi=24, kappa=8, K=2)
    w.kappa_max = 8
    chains, mpos = engine_args_from_oracle(oprob.build_inputs(w))
    dev = torch.cuda.current_device()
    torch.zeros(1, device="cuda")
    runtime = ctypes.CDLL(next(ln.split()[-1] for ln in open("/proc/self/maps") if "libcudart.so" in ln))
    sizes, refuse = [], [None]

    def _alloc(nbytes, ctx):
        sizes.append(int(nbytes))
        if len(sizes) - 1 == refuse[0]:
            p = ctypes.c_void_p()
            assert runtime.cudaMalloc(ctypes.byref(p), ctypes.c_size_t(1 << 50)) != 0
            return None
        return torch.cuda.caching_allocator_alloc(int(nbytes), dev, torch.cuda.current_stream(dev))

    def _free(ptr, ctx):
        if ptr:
            torch.cuda.caching_allocator_delete(ptr)

    def run():
        del sizes[:]
        eng = capi.Engine(chains, mpos, chi_max=32, eps=w.eps, max_steps=w.K, autotune=False)
        made = list(sizes)
        eng.set_observables(OPS)
        eng.step(w.K)
        obs = eng.read_history(0, w.K + 1)[0]
        kernels = eng.step_kernels()
        eng.destroy()
        return obs, kernels, made

    fa, ff = capi.ALLOC_FN(_alloc), capi.FREE_FN(_free)
    capi.lib.pt_tebd_set_allocator(fa, ff, None)
    try:
        ref, with_pool, made = run()
        # init's last requests: the workspace in one piece, then two short lists per layer
        refuse[0] = max(range(len(made) - 5, len(made)), key=lambda i: made[i])
        obs, without, _ = run()
    finally:
        capi.use_torch_allocator(dev)
    assert without < with_pool                         # fewer launches per step: the unblocked kernel
    assert np.max(np.abs(obs - ref)) < 1e-9 * np.max(np.abs(ref))
