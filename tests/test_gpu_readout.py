"""The readout (App. A.3) of stored random augmented MPS against the oracle's, at bond dimensions around the
sizes where the kernels split their work: one CTA or a cluster per pass (24), eight columns or rows per turn, 32
lanes. Bound: the passes are N products of sums of at most 4 kappa chi terms in FP64; relative to the same
contraction of absolute values 1e-13 covers it many times over."""
import numpy as np
import pytest

from oracle import model, pttebd

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("chis,kap", [((1, 1), 3), ((1, 2, 1), 1), ((1, 4, 7, 4, 1), 2), ((1, 4, 23, 24, 25, 4, 1), 3),
                                      ((1, 16, 63, 64, 65, 16, 1), 2), ((1, 4, 130, 9, 1), 5)])
def test_readout_against_oracle(chis, kap):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2201_05529_gb300 as pkg
    pkg.build()
    capi = pkg.load()
    capi.use_torch_allocator()
    rng = np.random.default_rng(sum(chis) + kap)
    N = len(chis) - 1
    gam = [rng.standard_normal((chis[n], 4, kap, chis[n + 1])) + 1j * rng.standard_normal((chis[n], 4, kap, chis[n + 1]))
           for n in range(N)]
    lam = [np.sort(rng.uniform(0.1, 1.0, size=x))[::-1].copy() for x in chis]
    P = rng.standard_normal((kap, 4, 4, 1)) + 1j * rng.standard_normal((kap, 4, 4, 1))
    gates = np.array([np.eye(16, dtype=complex)] * max(0, N - 1))
    chain = dict(N=N, rho0=None, gates_q=gates, gates_h=gates, ptmpo_id=[0] * N, chi0=list(chis), kappa0=[kap] * N,
                 gamma0=gam, lambda0=lam)
    ops = [model.SZ, model.SX, model.SY]
    eng = capi.Engine([chain, chain], [[P]], chi_max=max(chis), eps=1e-8, autotune=False)
    out, tr = eng.observe(ops)
    eng.destroy()
    cap = pttebd.caps([P])[0]
    vecs = [np.asarray(o).T.reshape(4) for o in ops]
    ref, t = pttebd.observe(pttebd.AugmentedMPS(gam, lam, 0.0), [cap] * N, vecs)
    amps = pttebd.AugmentedMPS([np.abs(g) for g in gam], lam, 0.0)
    scale, ts = pttebd.observe(amps, [np.abs(cap)] * N, [np.abs(v) for v in vecs])
    for c in range(2):
        assert np.all(np.abs(out[c] - ref) <= 1e-13 * np.abs(scale))
        assert abs(tr[c] - t) <= 1e-13 * abs(ts)
