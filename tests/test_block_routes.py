"""Which inputs the block form takes, what it computes for those near its limits, and what the inputs outside it
get: results of the general kernels (GF_KERNEL=direct), of the CPU oracle, or of a fresh context."""
import numpy as np
import pytest

import oracle
from paper_1111_2157_gb300 import gf, synth
from tests.test_block_form import _inputs, _rel, _run


def _context(s, **kw):
    g = gf.GreensFunction.for_systems([s], **kw)
    g.set_hamiltonian(s.H)
    g.set_projectors(s.P)
    g.set_sigma(s.sigma, s.sigma_inf)
    return g


@pytest.mark.gpu
@pytest.mark.parametrize("call", ["evaluate", "backward"])
@pytest.mark.parametrize("precision,other,size", [("fp64", "not_hermitian", (4, 20, 6, 64)),
                                                  ("mixed", "larger_norm", (150, 6, 2, 1024))])
def test_a_captured_graph_does_not_outlive_the_scratch_it_writes(precision, other, size, call):
    """N(mu) captured for one H, another H on another path (or with more FP64 frequencies) in a call that is not an
    N(mu) call and needs more partial sums, then the first H again: the replay must not use the scratch given back."""
    s = _inputs(*size, 40.0, 3)
    H2 = s.H.copy()
    if other == "not_hermitian":
        H2[0, 1, 3] += 1e-5
    else:
        H2 *= 40.0
    g = _context(s, precision=precision)
    ref = g.occupation([0.2])
    g.close()
    g = _context(s, precision=precision, graph=True)
    for _ in range(2):
        for _ in range(3):
            n, dn = g.occupation([0.2])
            assert n[0] == ref[0][0] and dn[0] == ref[1][0]
        g.set_hamiltonian(H2)
        if call == "evaluate":
            g.evaluate([0.2])
        else:
            g.backward([0.2], n_bar=[1.0])
        g.set_hamiltonian(s.H)
    g.close()


@pytest.mark.gpu
@pytest.mark.parametrize("why", ["not_hermitian", "kernel_named"])
def test_a_call_on_the_general_kernels_does_not_pay_for_the_set_up(why, monkeypatch):
    """N(mu) right after an upload against N(mu) repeated: the whole set-up of these windows (8 ms) would double the
    first, the check of H and P is 0.1 ms of it.  (Bound: a third of the pass, and 0.5 ms for what follows an
    upload.)"""
    import time
    rng = synth.rng_for(1)
    nk, nb, m, n_iw = 152, 128, 14, 40
    pole = synth.sigma_two_pole(rng, m, 4.0)
    s = synth.System(synth.hamiltonian_dense(rng, nk, nb, -8.0, 8.0, 0.3), synth.projectors(rng, nk, nb, m), pole,
                     pole.sample(40.0, n_iw), 40.0, nb / 2.0)
    if why == "kernel_named":
        monkeypatch.setenv("GF_KERNEL", "f32r")
    else:
        s.H[-1, 0, 1] += 1e-3
    g = _context(s, precision="mixed")

    def seconds():
        t = time.perf_counter()
        g.occupation([0.1])
        return time.perf_counter() - t

    seconds()  # (autotuner)
    first, again = [], []
    for _ in range(5):
        g.set_hamiltonian(s.H)
        first.append(seconds())
        again.append(seconds())
    g.close()
    assert min(first) < 1.33 * min(again) + 5e-4


def _near_dependent(s, delta, seed):
    """P of every k with singular values 1 but for one delta."""
    rng = np.random.default_rng(seed)
    nk, m, nb = s.P.shape

    def unitary(n, k):
        return np.linalg.qr(rng.standard_normal((n, k)) + 1j * rng.standard_normal((n, k)))[0]

    for k in range(nk):
        s.P[k] = (unitary(m, m) * np.r_[np.ones(m - 1), delta]) @ np.conj(unitary(nb, m).T)
    return s


@pytest.mark.gpu
@pytest.mark.parametrize("precision,delta,on_block", [
    ("fp64", 0.11, True), ("fp64", 0.09, False), ("fp64", 0.002, False), ("fp64", 0.0, False),
    ("mixed", 0.2, True), ("mixed", 0.16, False), ("mixed", 0.01, False), ("mixed", 0.002, False)])
def test_projectors_with_nearly_dependent_rows(precision, delta, on_block):
    """delta^-2 is the condition number of (P P^+)^{-1}: the limits are 32 in mixed precision and 100 in FP64.  The
    bounds are the contracts (mixed: of the G_loc, N, rho and dN/dmu tests; FP64 1e-10)."""
    s = _near_dependent(_inputs(3, 40, 14, 64, 100.0, 31), delta, 7)
    a, log = _run(s, None, precision=precision)
    b, _ = _run(s, "direct")
    assert ("mode 7: block form" in log) == on_block
    assert on_block or "P ill-conditioned" in log
    tol = {"N": 1e-7, "occ": 1e-7, "gloc": 1e-8, "loc": 1e-8, "rho": 1e-5, "dm": 1e-5, "dN_dmu": 1e-5, "docc": 1e-5,
           "n_corr": 1e-6, "dm_nc": 1e-6}
    for key in b:
        bound = tol.get(key, 1e-5 if key.startswith("mb") else 1e-8) if precision == "mixed" else 1e-10
        assert _rel(a[key], b[key]) < bound, key


@pytest.mark.gpu
@pytest.mark.parametrize("precision,scale", [("mixed", 1e-20), ("mixed", 1e-7), ("fp64", 1e-70)])
def test_projectors_of_a_scale_that_the_block_form_cannot_hold(precision, scale):
    """(P P^+)^{-1} of such rows leaves the number range of S: N and rho_k are those of H_k alone."""
    s = _inputs(2, 20, 6, 48, 40.0, 5)
    s.P *= scale
    g = _context(s, precision=precision)
    r = g.evaluate([0.1])
    assert "block form, " not in g.tuning_log()
    g.close()
    ref = oracle.get().density(s.H, s.P, s.sigma, s.sigma_inf, s.beta, 0.1)
    assert abs(r["N"][0] - ref["N"]) < (1e-7 if precision == "mixed" else 1e-10) * ref["N"]
    assert _rel(r["rho"].cpu().numpy(), ref["rho"].reshape(-1)) < (1e-5 if precision == "mixed" else 1e-10)


@pytest.mark.gpu
@pytest.mark.parametrize("split", [3e-5, 3e-6, 1e-6, 3e-7, 1e-7, 1e-9, 1e-11])
@pytest.mark.parametrize("nb,m,p", [(31, 5, 2), (60, 6, 5)])
def test_levels_that_nearly_coincide(nb, m, p, split):
    """Clusters of p levels, split of the norm apart, in the block that the set-up makes diagonal, and as eigenvalues
    of the pseudo-Hamiltonian: unitary eigenvectors to rounding.  (Bound: cond(A) ~ |H| / w_0 = 1e2 roundings, 1e2
    of their sums; vectors orthogonal to 1e-11 fail it.)"""
    from oracle import pole as pole_oracle
    s = _inputs(4, nb, m, 48, 40.0, 17)
    rng = np.random.default_rng(int(1e12 * split) + nb)
    n2 = nb - m
    for k in range(4):
        lev = np.linspace(-8.0, 8.0, n2) + 0.1 * rng.standard_normal(n2)
        hidden = np.zeros(n2, bool)
        for c in range(1, n2 - p, n2 // 3):
            lev[c:c + p] = lev[c] + 8.0 * split * np.arange(p) * (1.0 + 0.3 * rng.random(p))
            hidden[c:c + p] = k >= 2  # (k 0 and 1: coupled to the orbitals; 2 and 3: not, so levels of the whole H)
        B = 0.3 * (rng.standard_normal((m, n2)) + 1j * rng.standard_normal((m, n2)))
        B[:, hidden] = 0.0
        U = np.linalg.qr(rng.standard_normal((n2, n2)) + 1j * rng.standard_normal((n2, n2)))[0]
        H = s.H[k].copy()
        H[m:, m:] = (U * lev) @ np.conj(U.T)
        H[:m, m:] = B @ np.conj(U.T)
        H[m:, :m] = np.conj(H[:m, m:].T)
        s.H[k] = 0.5 * (H + np.conj(H.T))
        s.P[k] = np.eye(m, nb)
    a, log = _run(s, None)
    b, _ = _run(s, "direct")
    assert "mode 7: block form" in log
    for key in ("N", "rho", "n_corr", "gloc"):
        assert _rel(a[key], b[key]) < 1e-12, key
    g = gf.GreensFunction.for_systems([s])
    g.set_hamiltonian(s.H)
    g.set_projectors(s.P)
    g.set_sigma_poles([len(s.pole.p)], s.pole.p, s.pole.V.reshape(-1), s.pole.sigma_inf.reshape(-1))
    n, _ = g.pole_occupation([0.1])
    rho, _ = g.pole_density_matrix([0.1])
    g.close()
    ref = pole_oracle.density(s.H, s.P, s.sigma_inf, s.pole.p, s.pole.V, s.beta, 0.1)
    assert abs(n[0] - ref["N"]) < 1e-12 * ref["N"]
    assert _rel(rho.cpu().numpy(), np.asarray(ref["rho"]).reshape(-1)) < 1e-12


@pytest.mark.gpu
@pytest.mark.parametrize("nb,m,n_iw", [(13, 5, 300), (40, 14, 200), (60, 20, 130), (9, 1, 257)])
def test_mixed_frequency_sums_keep_more_bits_than_their_terms(nb, m, n_iw):
    """Levels that do not couple to the orbitals: rho_k there is the sum over the frequencies of 1 / (i w + mu - e),
    FP32 numbers above the FP64 limit.  Against the FP64 sum of the same FP32 numbers (bound: 1e2 roundings of FP64
    times beta; FP32 sums of a batch are off by 1e-9)."""
    beta, rng = 1.0, np.random.default_rng(nb)
    s = _inputs(2, nb, m, n_iw, beta, 1)
    e = rng.choice([-1.0, 1.0], (2, nb)) * rng.integers(40 * 64, 80 * 64, (2, nb)) / 64.0
    s.H[:] = e[:, :, None] * np.eye(nb)
    s.P[:] = np.eye(m, nb)
    g = _context(s, precision="mixed")
    rho = g.density_matrix([0.0])[0].cpu().numpy().reshape(2, nb, nb)
    log = g.tuning_log()
    g.close()
    n64 = int(log.split("block form, ")[1].split()[0])
    assert "in FP32 and FP32 pairs" in log and n64 < n_iw
    w = (2.0 * np.arange(n_iw) + 1.0) * np.pi / beta
    x, w32 = (-e[:, m:]).astype(np.float32)[:, :, None], w.astype(np.float32)
    q = np.float32(1.0) / (x.astype(np.float64) ** 2 + (w32 * w32).astype(np.float64)).astype(np.float32)
    d = np.where(np.arange(n_iw) < n64, -e[:, m:, None] / (e[:, m:, None] ** 2 + w * w), (x * q).astype(np.float64))
    tail = 2.0 / beta * np.sum((1.0 / (w * w))[::-1]) - beta / 4.0
    ref = 2.0 / beta * d.sum(2) + tail * e[:, m:] + 0.5
    got = np.diagonal(rho, axis1=1, axis2=2)[:, m:]
    assert np.max(np.abs(got - ref)) < 2e-14


@pytest.mark.gpu
def test_low_temperature_does_not_multiply_the_scratch_of_rho(monkeypatch):
    """Mixed precision at beta = 1e4, where 400 frequencies run in FP64, over many k-points: device memory of rho_k no
    more than the general kernels take, but for the tables of the set-up (U, the n2 blocks, the pairs of B with their
    moments in three widths, the rotation: 12 times H for these windows)."""
    import torch
    nk, nb, m, n_iw, beta = 6000, 12, 3, 512, 1e4
    rng = synth.rng_for(2)
    pole = synth.sigma_two_pole(rng, m, 4.0)
    s = synth.System(synth.hamiltonian_dense(rng, nk, nb, -8.0, 8.0, 0.3), synth.projectors(rng, nk, nb, m), pole,
                     pole.sample(beta, n_iw), beta, nb / 2.0)

    def taken():
        g = _context(s, precision="mixed")
        out = torch.zeros(nk * nb * nb, dtype=torch.complex128, device="cuda")
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        g.density_matrix([0.1], out=out)
        used = free - torch.cuda.mem_get_info()[0]
        log = g.tuning_log()
        g.close()
        return used, log

    block, log = taken()
    assert int(log.split("block form, ")[1].split()[0]) >= 400
    monkeypatch.setenv("GF_KERNEL", "f32r")
    general, _ = taken()
    assert block < general + 12 * 16 * nk * nb * nb


@pytest.mark.gpu
@pytest.mark.parametrize("precision,mu", [("fp64", 1e170), ("fp64", -1e155), ("fp64", 1e100), ("mixed", 1e30),
                                          ("mixed", -1e18)])
def test_a_chemical_potential_whose_square_overflows(precision, mu):
    """1 / (i w + mu - e) of every level is below the sums' last place: N and dN/dmu are the tail's, as on the general
    kernels."""
    s = _inputs(2, 40, 14, 64, 40.0, 8)
    a, log = _run(s, None, precision=precision, mu=mu)
    b, _ = _run(s, "direct", mu=mu)
    assert "mode 7: block form" in log
    for key in ("N", "occ", "dN_dmu", "docc", "rho", "n_corr"):
        assert _rel(a[key], b[key]) < (1e-10 if precision == "fp64" else 1e-6), key


@pytest.mark.gpu
@pytest.mark.parametrize("precision,lowrank,n_iw,on_block", [
    ("fp64", False, 15, False), ("fp64", False, 16, True), ("mixed", False, 39, False), ("mixed", False, 40, True),
    ("mixed", True, 16, True)])
def test_few_frequencies_do_not_pay_for_the_set_up(precision, lowrank, n_iw, on_block):
    """The first number of frequencies on the block form of each precision, and N on both sides of it."""
    s = _inputs(2, 24, 7, n_iw, 20.0, 4)
    g = _context(s, precision=precision, lowrank=lowrank)
    n, _ = g.occupation([0.1])
    assert ("block form, " in g.tuning_log()) == on_block
    g.close()
    ref = oracle.get().density(s.H, s.P, s.sigma, s.sigma_inf, s.beta, 0.1, want_rho=False)
    assert abs(n[0] - ref["N"]) < (1e-7 if precision == "mixed" else 1e-10) * ref["N"]


@pytest.mark.gpu
def test_the_log_does_not_grow_with_the_uploads():
    s = _inputs(2, 12, 4, 24, 20.0, 4)
    s.H[0, 0, 1] += 1e-3
    g = _context(s)
    g.occupation([0.1])
    log = g.tuning_log()
    assert log.count("H not Hermitian") == 1
    for _ in range(3):
        g.set_hamiltonian(s.H)
        g.occupation([0.1])
    assert g.tuning_log() == log
    g.close()


@pytest.mark.gpu
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_scratch_that_does_not_fit_beside_the_tables(precision):
    """Device memory for the block form's tables but not for its scratch beside them, and enough for the general
    kernels: the call runs on those."""
    import torch
    nk, nb, m, n_iw = 2000, 40, 24, 64
    rng = synth.rng_for(2)
    pole = synth.sigma_two_pole(rng, m, 4.0)
    s = synth.System(synth.hamiltonian_dense(rng, nk, nb, -8.0, 8.0, 0.3), synth.projectors(rng, nk, nb, m), pole,
                     pole.sample(40.0, n_iw), 40.0, nb / 2.0)
    out = torch.zeros(nk * nb * nb, dtype=torch.complex128, device="cuda")
    torch.cuda.empty_cache()

    def free():
        torch.cuda.synchronize()
        return torch.cuda.mem_get_info()[0]

    def taken(kernel):
        with pytest.MonkeyPatch.context() as mp:
            if kernel:
                mp.setenv("GF_KERNEL", kernel)
            g = _context(s, precision=precision)
            before = free()
            g.density_matrix([0.1], out=out)
            used = before - free()
            log = g.tuning_log()
            g.close()
        return used, log, out.clone()

    block, log, ref = taken(None)
    general, _, _ = taken("direct" if precision == "fp64" else "f32r")
    assert "block form, " in log and general < block - (64 << 20)
    g = _context(s, precision=precision)
    hold = torch.empty(free() - block + (24 << 20), dtype=torch.uint8, device="cuda")
    try:
        g.density_matrix([0.1], out=out)
        log = g.tuning_log()
    finally:
        del hold
        torch.cuda.empty_cache()
    assert "does not fit in device memory" in log and "mode 2: block form" not in log
    assert _rel(out.cpu().numpy(), ref.cpu().numpy()) < (1e-10 if precision == "fp64" else 1e-5)
    g.close()
