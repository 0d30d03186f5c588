"""What a user of this package has it do, as cases that can be timed and compared.

A user runs whole PT-TEBD simulations (an Engine from host inputs, steps, the recorded history), reads
observables out of a state, and calls the step's three building blocks on their own: the batched
Householder QR with the explicit Q, the batched sliced complex GEMM of the fast path, and the batched FP64
SVD. Sizes are those of this repository's workloads (3-, 5- and 21-site chains, the ensemble of chains of 4
to 16 sites) and of its kernel tests.

Site tensors and singular vectors are fixed only up to a phase per bond index, so a run returns the state's
gauge-independent part (observables, trace, bond weights, log-norms), and the SVD's vectors are returned with
the first entry of every right vector made real.
"""
import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_2201_05529_gb300 as pkg
from paper_2201_05529_gb300 import problem

_capi = None


def _lib():
    global _capi
    if _capi is None:
        _capi = pkg.load()
        _capi.use_torch_allocator()
    return _capi


# ------------------------------------------------------------------------------------------- the cases
def listed():
    return [
        # observables of a stored 21-site state (one call of the readout on a state that is at hand)
        dict(name="readout_21", kind="readout", N=21, chi=64, kappa=16, ops=3),
        # the smallest simulation: three spins, one bath, the whole 20-step run in FP64
        dict(name="chain3_fp64", kind="run", model="xyz", chains=1, N=3, steps=20, memory=20, dt=0.1, chi=64,
             kappa=16, eps=1e-10, precision="fp64", typical_chi=4),
        # five spins between two baths, the first steps of a long run in FP64
        dict(name="chain5_fp64", kind="run", model="xyz", chains=1, N=5, steps=8, memory=16, dt=0.05, chi=64,
             kappa=32, eps=1e-8, precision="fp64", typical_chi=16),
        # a batch of chains of uneven length in one handle, FP64
        dict(name="ensemble16_fp64", kind="run", model="ensemble", chains=16, N=16, steps=4, memory=8, dt=0.05,
             chi=64, kappa=16, eps=1e-8, precision="fp64", typical_chi=16),
        # the 21-site chain with a bath on every site on the tensor-core path: the first steps, during which
        # the bonds grow from 1 to about their largest size
        dict(name="chain21_fast", kind="run", model="xy", chains=1, N=21, steps=4, memory=10, dt=0.1, chi=128,
             kappa=16, eps=1e-6, precision="bf16_ozaki", typical_chi=48),
        # QR: blocks of a run's early steps; the fast path's sketches (chi 128 + 32 columns); the outer
        # blocks of the 21-site chain at full bond dimension
        dict(name="qr_early_blocks", kind="qr", m=61, n=24, batch=10),
        dict(name="qr_sketches", kind="qr", m=1120, n=160, batch=10),
        dict(name="qr_outer_blocks", kind="qr", m=2048, n=512, batch=20),
        # the sliced complex GEMM: ragged blocks of a small chain; D Omega of one bond layer; the site layer
        # of the 21-site chain (few columns, many rows)
        dict(name="zgemm_ragged", kind="zgemm", m=300, n=70, k=530, batch=3, opA="H", opB="N"),
        dict(name="zgemm_sketch", kind="zgemm", m=1120, n=160, k=1120, batch=10, opA="N", opB="N"),
        dict(name="zgemm_sites", kind="zgemm", m=16384, n=64, k=64, batch=21, opA="N", opB="T"),
        # the SVD of a bond layer's two-site blocks of the five-site chain
        dict(name="svd_bonds", kind="svd", m=256, n=256, batch=2),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["qr", "zgemm", "qr", "zgemm", "svd", "run", "run", "readout"])
    if kind == "readout":
        return dict(kind=kind, N=rng.randint(2, 21), chi=_log_int(rng, 4, 64), kappa=rng.randint(1, 16),
                    ops=rng.randint(1, 4))
    if kind == "qr":
        m, n = _log_int(rng, 1, 2048), _log_int(rng, 1, 512)
        return dict(kind=kind, m=max(m, n), n=min(m, n), batch=_log_int(rng, 1, 20))
    if kind == "zgemm":
        n, k = _log_int(rng, 1, 1120), _log_int(rng, 1, 1120)
        return dict(kind=kind, m=_log_int(rng, 1, 2048), n=n, k=k, batch=_log_int(rng, 1, 10),
                    opA=rng.choice("NTH"), opB=rng.choice("NTH"))
    if kind == "svd":
        return dict(kind=kind, m=_log_int(rng, 1, 320), n=_log_int(rng, 1, 256), batch=rng.randint(1, 4))
    fast = rng.random() < 0.5
    if rng.random() < 0.4:
        return dict(kind=kind, model="ensemble", chains=rng.randint(2, 12), N=rng.randint(4, 12),
                    steps=rng.randint(1, 3), memory=rng.randint(4, 10), dt=0.05, chi=rng.randint(16, 64), kappa=16,
                    eps=1e-6 if fast else 1e-8, precision="bf16_ozaki" if fast else "fp64", typical_chi=12)
    xy = rng.random() < 0.4
    N = rng.randint(3, 15 if xy else 7)
    steps = rng.randint(2, 3 if xy else 7)
    return dict(kind=kind, model="xy" if xy else "xyz", chains=1, N=N, steps=steps, memory=steps + rng.randint(2, 8),
                dt=0.1 if xy else 0.05, chi=rng.randint(24, 128 if xy else 64), kappa=16 if xy else rng.randint(8, 32),
                eps=1e-6 if fast or xy else 1e-8, precision="bf16_ozaki" if fast else "fp64",
                typical_chi=24 if xy else 12)


# -------------------------------------------------------------------------------------------- inputs
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) & 0x7FFFFFFF)
    return g


def _cgauss(gen, *shape):
    return torch.randn(*shape, dtype=torch.complex128, device="cuda", generator=gen)


def _qr_input(c, seed):
    """[batch, n, m]: columns of a matrix whose rows carry decaying bond weights (B_L = lambda Gamma), mixed as a
    sketch mixes them."""
    gen = _gen(seed)
    A = _cgauss(gen, c["batch"], c["n"], c["m"])
    w = torch.exp(-6.0 * torch.arange(c["m"], dtype=torch.float64, device="cuda") / c["m"])
    return (A * w).contiguous()


def _zgemm_input(c, seed):
    """Operands in storage order [batch, columns, rows], the rows of opA(A) and the columns of opB(B) of
    uneven scale, as a bond's blocks have them."""
    gen = _gen(seed)
    m, n, k, b = c["m"], c["n"], c["k"], c["batch"]
    ra = torch.exp(-8.0 * torch.rand(m, dtype=torch.float64, device="cuda", generator=gen))
    cb = torch.exp(-8.0 * torch.rand(n, dtype=torch.float64, device="cuda", generator=gen))
    A = _cgauss(gen, b, k, m) * ra if c["opA"] == "N" else _cgauss(gen, b, m, k) * ra[:, None]
    B = _cgauss(gen, b, n, k) * cb[:, None] if c["opB"] == "N" else _cgauss(gen, b, k, n) * cb
    return A.contiguous(), B.contiguous()


def _svd_input(c, seed):
    """[batch, m, n] with singular values that fall off over four decades, as a truncated two-site block."""
    gen = _gen(seed)
    k = min(c["m"], c["n"])
    L = torch.linalg.qr(_cgauss(gen, c["batch"], c["m"], k))[0]
    R = torch.linalg.qr(_cgauss(gen, c["batch"], c["n"], k))[0]
    s = torch.exp(-9.2 * (torch.arange(k, dtype=torch.float64, device="cuda") +
                          0.3 * torch.rand(k, dtype=torch.float64, device="cuda", generator=gen)) / k)
    return ((L * s) @ R.mH).contiguous()


PAULI = {n: problem.pauli(n) for n in "zxy"}


def _bath(alpha, omega_c, T):
    return SimpleNamespace(alpha=alpha, omega_c=omega_c, T=T, cutoff="exponential")


def _chain_inputs(c, seed):
    """(chains, PT-MPOs) on the host: couplings and baths drawn around the workloads' values."""
    rng = np.random.default_rng([int(seed), 11])
    mpos, chains = [], []

    def bath(alpha, omega_c, T):
        b = _bath(alpha, omega_c, T)
        eta = problem.eta_list(b, c["dt"], c["memory"])
        F = problem.influence_mpo(eta, c["memory"], 1e-7, c["kappa"], c["memory"])
        mpos.append(problem.pt_mpo_tensors(F))
        return len(mpos) - 1

    for i in range(c["chains"]):
        if c["model"] == "ensemble":
            N = 4 + (5 * i + c["N"]) % (c["N"] - 3)          # lengths 4 .. N, spread over the batch
            J = tuple(rng.uniform(0.5, 1.5, size=3))
            field = 0.0
            ids = [bath(rng.uniform(0.05, 0.2), 4.0, rng.uniform(0.5, 5.0))] + [-1] * (N - 2)
            ids += [bath(rng.uniform(0.05, 0.2), 4.0, rng.uniform(0.5, 5.0))]
            init = ["u" if n % 2 == 0 else "d" for n in range(N)]
        elif c["model"] == "xy":
            N = c["N"]
            j = rng.uniform(0.9, 1.1)
            J, field = (j, j, 0.0), 0.0
            ids = [bath(rng.uniform(0.04, 0.06), 3.0, rng.uniform(0.7, 0.9))] * N
            init = ["u" if n == N // 2 else "d" for n in range(N)]
        else:
            N = c["N"]
            J, field = tuple(np.array([1.3, 0.7, 1.2]) * rng.uniform(0.9, 1.1, size=3)), rng.uniform(0.4, 0.6)
            ids = [bath(rng.uniform(0.1, 0.16), 4.0, rng.uniform(1.0, 5.0))] + [-1] * (N - 1)
            if N >= 5:
                ids[-1] = bath(rng.uniform(0.1, 0.16), 4.0, rng.uniform(0.5, 1.0))
            init = ["u" if n % 2 == 0 else "d" for n in range(N)]
        spec = SimpleNamespace(N=N, eps=tuple([field] + [0.0] * (N - 1)), J=tuple([J] * (N - 1)), gksl=(), drive=None)
        gq, gh = problem.chain_gates(spec, c["dt"])
        chains.append(dict(N=N, rho0=np.array([problem.state_vec(s) for s in init]), gates_q=gq, gates_h=gh,
                           ptmpo_id=ids))
    return chains, mpos


def _readout_inputs(c, seed):
    """A stored augmented MPS of N sites: decaying bond weights, site tensors around a common positive part
    (so that its trace is of order one), and the caps of a one-step PT-MPO."""
    rng = np.random.default_rng([int(seed), 12])
    N, chi, kap = c["N"], c["chi"], c["kappa"]
    chis = [1] + [max(1, min(chi, 4 ** min(b, N - b, 6))) for b in range(1, N)] + [1]
    lam = []
    for x in chis:
        l = np.exp(-np.arange(x) / 8.0) * rng.uniform(0.9, 1.1, size=x)
        l = np.sort(l)[::-1]
        lam.append(np.ascontiguousarray(l / np.linalg.norm(l)))
    gam = []
    for n in range(N):
        a, b = chis[n], chis[n + 1]
        p = rng.uniform(0.2, 0.8)
        rho = np.array([p, 0.1 + 0.05j, 0.1 - 0.05j, 1.0 - p])
        g = rng.uniform(0.5, 1.5, size=(a, 1, kap, b)) * rho[None, :, None, None]
        g = g + 0.1 * (rng.standard_normal((a, 4, kap, b)) + 1j * rng.standard_normal((a, 4, kap, b)))
        gam.append(g / lam[n + 1].sum())
    w = rng.uniform(0.5, 1.5, size=kap)
    P = np.zeros((kap, 4, 4, 1), dtype=complex)
    for p in range(4):
        P[:, p, p, 0] = w / w.sum()
    gates = np.array([np.eye(16, dtype=complex)] * max(0, N - 1))
    chain = dict(N=N, rho0=None, gates_q=gates, gates_h=gates, ptmpo_id=[0] * N, chi0=chis, kappa0=[kap] * N,
                 gamma0=gam, lambda0=lam)
    ops = [PAULI["z"], PAULI["x"], PAULI["y"], np.eye(2, dtype=complex)][:c["ops"]]
    return chain, [[P]], ops, w / w.sum()


# ------------------------------------------------------------------------------------------- the calls
def prepare(case, seed):
    capi = _lib()
    c, dev = dict(case), "cuda"
    if c["kind"] == "qr":
        A = _qr_input(c, seed)
        return dict(c=c, A=A, Q=torch.empty_like(A),
                    R=torch.empty(c["batch"], c["n"], c["n"], dtype=torch.complex128, device=dev),
                    scratch=torch.empty(capi.qr_scratch_bytes(c["m"], c["n"], c["batch"]), dtype=torch.uint8, device=dev))
    if c["kind"] == "zgemm":
        A, B = _zgemm_input(c, seed)
        C = torch.empty(c["batch"], c["n"], c["m"], dtype=torch.complex128, device=dev)
        nb = capi.zgemm_scratch_bytes(c["m"], c["n"], c["k"], c["batch"])
        return dict(c=c, A=A, B=B, C=C, scratch=torch.empty(nb, dtype=torch.uint8, device=dev))
    if c["kind"] == "svd":
        b, m, n, k = c["batch"], c["m"], c["n"], min(c["m"], c["n"])
        return dict(c=c, A=_svd_input(c, seed), S=torch.empty(b, k, dtype=torch.float64, device=dev),
                    U=torch.empty(b, m, k, dtype=torch.complex128, device=dev),
                    V=torch.empty(b, n, k, dtype=torch.complex128, device=dev),
                    scratch=torch.empty(capi.svd_scratch_bytes(m, n, b), dtype=torch.uint8, device=dev))
    if c["kind"] == "readout":
        chain, mpos, ops, _ = _readout_inputs(c, seed)
        eng = capi.Engine([chain], mpos, chi_max=c["chi"], eps=1e-8, precision="fp64", autotune=False)
        return dict(c=c, eng=eng, ops=ops)
    chains, mpos = _chain_inputs(c, seed)
    return dict(c=c, chains=chains, mpos=mpos)


def run(state):
    capi = _lib()
    c = state["c"]
    if c["kind"] == "qr":
        state["Q"].copy_(state["A"])            # the factorisation is in place: the caller keeps A
        capi.qr_f64(state["Q"], state["R"], state["scratch"])
        return state["Q"], state["R"]
    if c["kind"] == "zgemm":
        capi.zgemm_sliced(c["opA"], c["opB"], state["A"], state["B"], state["C"], c["m"], c["n"], c["k"],
                          state["scratch"])
        return state["C"]
    if c["kind"] == "svd":
        capi.svd_f64(state["A"], state["S"], state["U"], state["V"], state["scratch"])
        ph = torch.sgn(state["V"][:, :1, :]).conj()       # first entry of every right vector real
        return state["S"], state["U"] * ph, state["V"] * ph
    if c["kind"] == "readout":
        return state["eng"].observe(state["ops"])
    eng = capi.Engine(state["chains"], state["mpos"], chi_max=c["chi"], eps=c["eps"], precision=c["precision"],
                      multiplet_tol=1e-9, max_steps=c["steps"])
    eng.set_observables([PAULI["z"], PAULI["x"]])
    eng.step(c["steps"])
    hist, trace = eng.read_history(0, c["steps"] + 1)
    lam = np.zeros((eng.n_chains, eng.n_max + 1, c["chi"]))         # bond weights, zero beyond a bond's dimension
    for i, n in enumerate(eng.N):
        for b in range(n + 1):
            l = eng.get_lambda(i, b)
            lam[i, b, :len(l)] = l
    logs = [eng.get_lognorm(i) for i in range(eng.n_chains)]
    eng.destroy()
    return dict(observables=hist, trace=trace, weights=lam, lognorm=np.array(logs))


def work(case):
    c = case
    z = 16.0                                     # bytes of a complex number
    if c["kind"] == "qr":
        m, n, b = c["m"], c["n"], c["batch"]
        return {"bytes": z * b * (2 * m * n + n * n), "flops": 16.0 * b * (m * n * n - n ** 3 / 3)}
    if c["kind"] == "zgemm":
        m, n, k, b = c["m"], c["n"], c["k"], c["batch"]
        return {"bytes": z * b * (m * k + k * n + m * n), "flops": 8.0 * b * m * n * k}
    if c["kind"] == "svd":
        m, n, b = max(c["m"], c["n"]), min(c["m"], c["n"]), c["batch"]
        return {"bytes": z * b * (2 * m * n + n * n) + 8.0 * b * n, "flops": 4.0 * b * (14.0 * m * n * n + 8.0 * n ** 3)}
    if c["kind"] == "readout":
        el = c["N"] * 4.0 * c["kappa"] * c["chi"] ** 2
        return {"bytes": z * el, "flops": 8.0 * el}
    # a run: bond dimensions come out of the run itself; the count uses the size they typically have by its
    # end (typical_chi), with the outer reductions, the two-site block, its SVD and the recovery of every bond
    # update, six layers a step over two interleaved sets of bonds
    chi, N = float(c["typical_chi"]), (0.5 * (4 + c["N"]) if c["model"] == "ensemble" else c["N"])
    baths = N if c["model"] == "xy" else 2
    r = 4.0 * chi                                # rows of a reduced block
    per_bond = 4.0 * (14.0 + 8.0) * r ** 3 + 128.0 * r * r * chi + 8.0 * r * r * chi
    state = z * (baths * c["kappa"] + (N - baths)) * 4.0 * chi * chi
    return {"bytes": c["chains"] * c["steps"] * 2.0 * state, "flops": c["chains"] * c["steps"] * 3.0 * (N - 1) * per_bond}


# -------------------------------------------------------------------- the same in plain 64-bit arithmetic
def _householder(A):
    """Q and R of [batch, m, n] with reflectors I - tau u u^H and R's diagonal -phase(alpha) ||x||."""
    A = A.clone()
    b, m, n = A.shape
    refl = []
    for j in range(n):
        x = A[:, j:, j].clone()
        nrm = torch.linalg.vector_norm(x, dim=1)
        al = x[:, 0].clone()
        ph = torch.where(al.abs() > 0, torch.sgn(al), torch.ones_like(al))
        x[:, 0] = al + ph * nrm
        u2 = (x.abs() ** 2).sum(1)
        tau = torch.where(u2 > 0, 2.0 / u2, torch.zeros_like(u2))
        w = torch.einsum("bi,bij->bj", x.conj(), A[:, j:, j:]) * tau[:, None]
        A[:, j:, j:] -= x[:, :, None] * w[:, None, :]
        refl.append((x, tau))
    R = torch.triu(A[:, :n, :])
    Q = torch.zeros_like(A)
    Q[:, torch.arange(n), torch.arange(n)] = 1.0
    for j in range(n - 1, -1, -1):
        x, tau = refl[j]
        w = torch.einsum("bi,bij->bj", x.conj(), Q[:, j:, j:]) * tau[:, None]
        Q[:, j:, j:] -= x[:, :, None] * w[:, None, :]
    return Q, R


def _keep(s, eps, cap, mtol):
    """Kept singular values: the fewest whose discarded rest is below eps s[0], at most cap, no multiplet cut."""
    n, s0 = len(s), s[0]
    tail = np.append(np.sqrt(np.cumsum((s * s)[::-1])[::-1]), 0.0)
    chi = min(int(np.argmax(tail < eps * s0)), int((s > 0).sum()))
    chi = max(1, chi)

    def cuts(x):
        return 0 < x < n and s[x - 1] - s[x] <= mtol * s0

    if chi <= cap:
        while cuts(chi) and chi < cap and s[chi] > 0:
            chi += 1
        if not cuts(chi):
            return chi
    chi = min(chi, cap)
    while chi > 1 and cuts(chi):
        chi -= 1
    return chi


def _expect(gam, lam, caps, ops, lognorm):
    """Tr(O_n rho) for every site and operator, and Tr(rho), of one augmented MPS."""
    tau = np.array([1, 0, 0, 1], dtype=complex)
    N = len(gam)
    M = [np.tensordot(g, cp, axes=(2, 0)) for g, cp in zip(gam, caps)]          # [l, p, r]
    left = [lam[0].astype(complex)]
    for n in range(N):
        left.append(np.einsum("l,lpr,p->r", left[n], M[n], tau, optimize=True) * lam[n + 1])
    right = [None] * N + [np.ones(1, dtype=complex)]
    for n in range(N - 1, -1, -1):
        right[n] = np.einsum("lpr,p,r->l", M[n], tau, lam[n + 1] * right[n + 1], optimize=True)
    out = np.array([[np.einsum("l,lpr,p,r->", left[n], M[n], o.T.reshape(4), lam[n + 1] * right[n + 1], optimize=True)
                     for o in ops] for n in range(N)])
    scale = math.exp(lognorm)
    return out * scale, complex(left[N][0]) * scale


def _bond(gam, lam, i, G, chi_max, eps, mtol):
    gl, gr = gam[i], gam[i + 1]
    a, _, ka, c = gl.shape
    _, _, kb, b = gr.shape
    BL = (gl * lam[i][:, None, None, None]).transpose(0, 2, 1, 3).reshape(a * ka, 4 * c)
    BR = (gr * lam[i + 2]).reshape(c * 4, kb * b)
    QL, RL = np.linalg.qr(BL) if a * ka > 4 * c else (None, BL)
    if kb * b > 4 * c:
        q, r = np.linalg.qr(BR.conj().T)
        QR, LR = q.conj().T, r.conj().T
    else:
        QR, LR = None, BR
    rl, rr = RL.shape[0], LR.shape[1]
    th = (RL.reshape(rl * 4, c) * lam[i + 1]) @ LR.reshape(c, 4 * rr)
    th = np.tensordot(G.reshape(4, 4, 4, 4), th.reshape(rl, 4, 4, rr), axes=([2, 3], [1, 2]))      # [P, Q, u, v]
    D = th.transpose(2, 0, 1, 3).reshape(rl * 4, 4 * rr)
    U, S, Vh = np.linalg.svd(D, full_matrices=False)
    x = _keep(S, eps, chi_max, mtol)
    nrm = float(np.linalg.norm(S[:x]))
    lam[i + 1] = S[:x] / nrm
    L = U[:, :x].reshape(rl, 4 * x)
    L = L if QL is None else QL @ L
    gam[i] = L.reshape(a, ka, 4, x).transpose(0, 2, 1, 3) / lam[i][:, None, None, None]
    R = Vh[:x].reshape(x * 4, rr)
    R = R if QR is None else R @ QR
    gam[i + 1] = R.reshape(x, 4, kb, b) / lam[i + 2]
    return math.log(nrm)


def _simulate(c, ch, mpos):
    """One chain's history, bond weights and log-norm by plain TEBD with PT-MPOs."""
    N, eps, mtol, chi = ch["N"], c["eps"], 1e-9, c["chi"]
    gam = [np.asarray(v, dtype=complex).reshape(1, 4, 1, 1) for v in ch["rho0"]]
    lam = [np.ones(1) for _ in range(N + 1)]
    caps = {}
    for m in set(ch["ptmpo_id"]) - {-1}:
        cp = [np.ones(mpos[m][-1].shape[3], dtype=complex)]
        for P in mpos[m][::-1]:
            io = P[:, [0, 0, 3, 3], [0, 3, 0, 3], :].sum(axis=1)
            cp.append(0.5 * io @ cp[-1])
        caps[m] = cp[::-1]
    one = np.ones(1, dtype=complex)
    log, hist, trace = 0.0, [], []

    def read(k):
        o, t = _expect(gam, lam, [caps[m][k] if m >= 0 else one for m in ch["ptmpo_id"]], [PAULI["z"], PAULI["x"]], log)
        hist.append(o)
        trace.append(t)

    read(0)
    for k in range(c["steps"]):
        for half in range(2):
            for gates, first in ((ch["gates_q"], 0), (ch["gates_h"], 1), (ch["gates_q"], 0)):
                for b in range(first, N - 1, 2):
                    log += _bond(gam, lam, b, gates[b], chi, eps, mtol)
            if half == 0:
                for n, m in enumerate(ch["ptmpo_id"]):
                    if m >= 0:
                        gam[n] = np.tensordot(gam[n], mpos[m][k], axes=([1, 2], [1, 0])).transpose(0, 2, 3, 1)
        read(k + 1)
    return np.array(hist), np.array(trace), lam, log


def exact(case, seed):
    c = dict(case)
    if c["kind"] == "qr":
        Q, R = _householder(_qr_input(c, seed).mT)
        return Q.mT.contiguous(), R.mT.contiguous()
    if c["kind"] == "zgemm":
        A, B = _zgemm_input(c, seed)
        op = {"N": lambda X: X.mT, "T": lambda X: X, "H": lambda X: X.conj()}     # stored [columns, rows]
        return (op[c["opA"]](A) @ op[c["opB"]](B)).mT.contiguous()
    if c["kind"] == "svd":
        U, S, Vh = torch.linalg.svd(_svd_input(c, seed).cpu(), full_matrices=False)
        V = Vh.mH
        ph = torch.sgn(V[:, :1, :]).conj()
        return S, U * ph, V * ph
    if c["kind"] == "readout":
        chain, _, ops, cap = _readout_inputs(c, seed)
        o, t = _expect(chain["gamma0"], chain["lambda0"], [cap] * c["N"], ops, 0.0)
        return o[None], np.array([t])
    chains, mpos = _chain_inputs(c, seed)
    res = [_simulate(c, ch, mpos) for ch in chains]
    n_max = max(ch["N"] for ch in chains)
    hist = np.zeros((c["steps"] + 1, len(chains), n_max, 2), dtype=complex)
    for i, r in enumerate(res):
        hist[:, i, :chains[i]["N"]] = r[0]
    weights = np.zeros((len(chains), n_max + 1, c["chi"]))
    for i, r in enumerate(res):
        for b, l in enumerate(r[2]):
            weights[i, b, :len(l)] = l
    return dict(observables=hist, trace=np.array([r[1] for r in res]).T.copy(), weights=weights,
                lognorm=np.array([r[3] for r in res]))
