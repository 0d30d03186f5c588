"""pt_svd_scratch_bytes depends on m, n and batch alone (no GPU here): sizes that go through two QRs include the QR's
workspace whatever the current device, or its absence, says about cluster launches."""
import os
import shutil

import pytest


@pytest.mark.parametrize("m,n,batch", [(96, 96, 1), (256, 256, 2), (64, 256, 2), (1000, 40, 2), (6400, 100, 1)])
def test_scratch_holds_the_qr_workspace_on_any_device(m, n, batch):
    if shutil.which("nvcc") is None and not os.path.exists("/usr/local/cuda/bin/nvcc"):
        pytest.skip("nvcc not available")
    import paper_2201_05529_gb300 as pkg
    pkg.build()
    capi = pkg.load()
    big, small = max(m, n), min(m, n)
    matrices = 16 * batch * (big * small + small * small)          # the Jacobi's matrix and right factor
    assert capi.svd_scratch_bytes(m, n, batch) >= matrices + capi.qr_scratch_bytes(big, small, batch)
