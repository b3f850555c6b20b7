"""Block form of the lattice points: P_k^+ = Q [R; 0], the rows of Q^+ A Q that hold H_k alone made
diagonal once, and every output from the m x m matrix S(z) that is left.

CPU: the algebra in numpy against the inverse of the whole window, for every form of H and P that the
rule accepts.  GPU: the kernels against the general ones (GF_KERNEL=direct) at the edges of the lane
groups, batches and chunks, the inputs that keep the general kernels, and the precisions.
"""
import os

import numpy as np
import pytest

from paper_1111_2157_gb300 import synth


def _inputs(nk, nb, m, n_iw, beta, seed, rows="orthonormal", ragged=False):
    rng = synth.rng_for(seed)
    nbs = rng.integers(m + 1, nb + 1, size=nk) if ragged else [nb] * nk
    H = [synth.hamiltonian_dense(rng, 1, int(n), -8.0, 8.0, 0.3)[0] for n in nbs]
    P = [synth.projectors(rng, 1, int(n), m)[0] for n in nbs]
    if rows == "general":
        P = [p + 0.3 * (rng.standard_normal(p.shape) + 1j * rng.standard_normal(p.shape)) for p in P]
    pole = synth.sigma_two_pole(rng, m, 4.0)
    if not ragged:
        H, P = np.array(H), np.array(P)
    return synth.System(H, P, pole, pole.sample(beta, n_iw), beta, nb / 2.0)


def _block_form(H, P):
    """(e, B, H11, O, U) of one k-point."""
    m = P.shape[0]
    Q, R = np.linalg.qr(np.conj(P.T), mode="complete")
    Ri = np.linalg.inv(R[:m])
    Hq = np.conj(Q.T) @ H @ Q
    e, V = np.linalg.eigh(Hq[m:, m:])
    U = np.concatenate([Q[:, :m] @ np.conj(Ri.T), Q[:, m:] @ V], axis=1)
    return e, Ri @ Hq[:m, m:] @ V, Ri @ Hq[:m, :m] @ np.conj(Ri.T), Ri @ np.conj(Ri.T), U


@pytest.mark.parametrize("nb,m,rows", [(9, 3, "orthonormal"), (15, 14, "orthonormal"), (40, 14, "general"),
                                       (2, 1, "general"), (24, 5, "orthonormal")])
def test_block_algebra_equals_the_whole_inverse(nb, m, rows):
    beta, n_iw, mu = 40.0, 24, 0.17
    s = _inputs(3, nb, m, n_iw, beta, 11 + nb, rows)
    wn = (2 * np.arange(n_iw) + 1) * np.pi / beta
    for H, P in zip(s.H, s.P):
        e, B, H11, O, U = _block_form(H, P)
        for n in range(n_iw):
            z = 1j * wn[n] + mu
            G = np.linalg.inv(z * np.eye(nb) - H - np.conj(P.T) @ s.sigma[n] @ P)
            d = 1.0 / (z - e)
            A = np.linalg.inv(z * O - H11 - s.sigma[n] - (B * d) @ np.conj(B.T))
            F = O + (B * d * d) @ np.conj(B.T)
            X = A @ F
            BD = B * d
            DB = d[:, None] * np.conj(B.T)
            full = U @ np.block([[A, A @ BD], [DB @ A, np.diag(d) + DB @ A @ BD]]) @ np.conj(U.T)
            # condition numbers up to ~1e3 at the lowest frequency: 1e-11 is 1e2 of their rounding
            scale = np.max(np.abs(G))
            assert np.max(np.abs(full - G)) < 1e-11 * scale
            assert np.max(np.abs(A - P @ G @ np.conj(P.T))) < 1e-11 * scale
            assert np.max(np.abs(A @ F @ A - P @ G @ G @ np.conj(P.T))) < 1e-11 * scale**2 * nb
            tr2 = np.sum(d * d) + np.trace(X @ X) + 2 * np.trace(A @ (B * d**3) @ np.conj(B.T))
            assert abs(np.sum(d) + np.trace(X) - np.trace(G)) < 1e-11 * scale * nb
            assert abs(tr2 - np.trace(G @ G)) < 1e-10 * scale**2 * nb


def _run(s, kernel, precision="fp64", lowrank=False, mu=0.1, seed=5):
    from paper_1111_2157_gb300 import gf
    prev = os.environ.pop("GF_KERNEL", None)
    if kernel:
        os.environ["GF_KERNEL"] = kernel
    try:
        g = gf.GreensFunction.for_systems([s], precision=precision, lowrank=lowrank)
        g.set_hamiltonian(s.H)
        g.set_projectors(s.P)
        g.set_sigma(s.sigma, s.sigma_inf)
        rng = np.random.default_rng(seed)
        gbar = rng.standard_normal(s.sigma.shape) + 1j * rng.standard_normal(s.sigma.shape)
        r = g.evaluate([mu])
        out = {k: (v.cpu().numpy() if hasattr(v, "cpu") else v) for k, v in r.items()}
        out["loc"] = g.local([mu]).cpu().numpy()
        out["occ"], out["docc"] = g.occupation([mu])
        out["dm"], out["dm_nc"] = (x.cpu().numpy() if hasattr(x, "cpu") else x for x in g.density_matrix([mu]))
        for name, kw in (("both", dict(gloc_bar=gbar.reshape(-1), n_bar=[0.7])), ("g", dict(gloc_bar=gbar.reshape(-1))),
                         ("n", dict(n_bar=[1.3]))):
            sb, mb = g.backward([mu], **kw)
            out["sb_" + name], out["mb_" + name] = sb.cpu().numpy(), mb
        log = g.tuning_log()
        g.close()
        return out, log
    finally:
        os.environ.pop("GF_KERNEL", None)
        if prev is not None:
            os.environ["GF_KERNEL"] = prev


def _rel(a, b):
    return float(np.max(np.abs(np.asarray(a) - b)) / np.max(np.abs(b)))


@pytest.mark.gpu
@pytest.mark.parametrize("nk,nb,m,n_iw,rows,ragged", [
    (3, 9, 8, 33, "orthonormal", False),    # one band more than orbitals, eight lanes per matrix full
    (3, 18, 9, 17, "general", False),       # the first size of sixteen lanes
    (2, 17, 16, 40, "orthonormal", False),  # sixteen lanes full
    (2, 33, 17, 19, "general", False),      # the first size of 32 lanes
    (1, 60, 32, 16, "orthonormal", False),  # 32 lanes full, one k-point
    (21, 40, 14, 130, "orthonormal", False),  # several chunks and k-groups
    (5, 70, 10, 65, "general", True),       # windows that differ from k to k
    (2, 97, 2, 30, "orthonormal", False),   # wide window, few orbitals: eigenproblem outside shared memory
])
def test_block_kernels_equal_the_general_ones(nk, nb, m, n_iw, rows, ragged):
    s = _inputs(nk, nb, m, n_iw, 40.0, nb + m, rows, ragged)
    a, log = _run(s, None)
    b, log_d = _run(s, "direct")
    assert "mode 7: block form" in log and "mode 7: block form" not in log_d
    for key in b:
        assert _rel(a[key], b[key]) < 1e-10, key
    c, _ = _run(s, None, precision="pair")
    for key in b:
        assert _rel(c[key], b[key]) < 1e-9, key
    if m < 32:  # (the low-rank path's tiles refuse the adjoint at 32 orbitals)
        d, _ = _run(s, None, lowrank=True)
        for key in b:
            assert _rel(d[key], b[key]) < 1e-10, key


@pytest.mark.gpu
@pytest.mark.parametrize("kind", ["diagonal", "degenerate", "nearly_degenerate", "scalar", "split"])
def test_levels_that_the_parallel_eigenvectors_cannot_separate(kind):
    """Degenerate, nearly degenerate and split blocks take the QR steps: same results as the general kernels, on the
    block form and (against its own oracle) on the pole path."""
    from oracle import pole as pole_oracle
    from paper_1111_2157_gb300 import gf
    s = _inputs(3, 30, 5, 40, 40.0, 21)
    rng = np.random.default_rng(4)
    for k in range(3):
        U = np.linalg.qr(rng.standard_normal((30, 30)) + 1j * rng.standard_normal((30, 30)))[0]
        lev = np.repeat(np.arange(6.0) - 2.5, 5)
        if kind == "nearly_degenerate":
            lev = lev + 1e-9 * rng.standard_normal(30)
        H = {"diagonal": np.diag(rng.uniform(-4, 4, 30)).astype(complex), "scalar": 0.7 * np.eye(30, dtype=complex),
             "split": np.kron(np.eye(3), s.H[k, :10, :10])}.get(kind, (U * lev) @ np.conj(U.T))
        s.H[k] = 0.5 * (H + np.conj(H.T))
    a, log = _run(s, None)
    b, _ = _run(s, "direct")
    assert "mode 7: block form" in log
    for key in b:
        assert _rel(a[key], b[key]) < 1e-10, key
    g = gf.GreensFunction.for_systems([s])
    g.set_hamiltonian(s.H)
    g.set_projectors(s.P)
    g.set_sigma_poles([len(s.pole.p)], s.pole.p, s.pole.V.reshape(-1), s.pole.sigma_inf.reshape(-1))
    n, dn = g.pole_occupation([0.1])
    r = pole_oracle.density(s.H, s.P, s.sigma_inf, s.pole.p, s.pole.V, s.beta, 0.1)
    assert abs(n[0] - r["N"]) < 1e-10 * r["N"]
    assert _rel(g.pole_density_matrix([0.1])[0].cpu().numpy().reshape(3, 30, 30), r["rho"]) < 1e-10
    g.close()


@pytest.mark.gpu
@pytest.mark.parametrize("nk,nb,m,n_iw", [(3, 40, 14, 200), (2, 96, 20, 70), (2, 24, 7, 300), (2, 48, 32, 40)])
def test_mixed_block_kernels_against_fp64(nk, nb, m, n_iw):
    """The mixed contract (N 1e-7, G_loc 1e-8, rho 1e-5, dN/dmu 1e-5, n_corr 1e-6) on both sides of the FP64 limit."""
    s = _inputs(nk, nb, m, n_iw, 100.0, nb)
    a, log = _run(s, None, precision="mixed")
    b, _ = _run(s, "direct")
    assert "in FP32 and FP32 pairs" in log
    tol = {"N": 1e-7, "occ": 1e-7, "gloc": 1e-8, "loc": 1e-8, "rho": 1e-5, "dm": 1e-5, "dN_dmu": 1e-5, "docc": 1e-5,
           "n_corr": 1e-6, "dm_nc": 1e-6}
    for key in b:
        assert _rel(a[key], b[key]) < tol.get(key, 1e-5 if key.startswith("mb") else 1e-8), key


@pytest.mark.gpu
@pytest.mark.parametrize("nk,nb,m,n_iw,beta,ragged", [
    (1, 3, 1, 5, 4.0, False),        # one pair, fewer frequencies than a tile
    (3, 9, 3, 200, 5.0, False),      # most frequencies by the series
    (7, 40, 14, 512, 100.0, True),   # both, windows that differ from k to k
    (2, 30, 23, 130, 20.0, False),   # two pairs per thread
    (2, 36, 32, 65, 20.0, False),    # three
    (2, 20, 5, 24, 400.0, False),    # every frequency as it stands
])
def test_pole_local_by_moments_equals_the_resolvent(nk, nb, m, n_iw, beta, ragged):
    """G_loc of the pole path, sums and Chebyshev moments, against the inverse at every frequency."""
    from oracle import pole as pole_oracle
    from paper_1111_2157_gb300 import gf
    s = _inputs(nk, nb, m, n_iw, beta, 7 * nb + m, "orthonormal", ragged)
    g = gf.GreensFunction.for_systems([s])
    g.set_hamiltonian(s.H)
    g.set_projectors(s.P)
    g.set_sigma_poles([len(s.pole.p)], s.pole.p, s.pole.V.reshape(-1), s.pole.sigma_inf.reshape(-1))
    for mu in (0.1, -30.0):  # inside and outside the levels
        ref = pole_oracle.local(s.H, s.P, s.sigma_inf, s.pole.p, s.pole.V, s.beta, mu, s.n_iw).reshape(n_iw, -1)
        gl = g.pole_local([mu]).cpu().numpy().reshape(n_iw, -1)
        assert np.max(np.abs(gl - ref) / np.max(np.abs(ref), axis=1, keepdims=True)) < 1e-11
    g.close()


@pytest.mark.gpu
@pytest.mark.parametrize("what", ["non_hermitian", "rank_deficient", "few_frequencies"])
def test_inputs_outside_the_rule_keep_the_general_kernels(what):
    s = _inputs(3, 20, 6, 8 if what == "few_frequencies" else 40, 40.0, 9)
    if what == "non_hermitian":
        s.H[1, 2, 5] += 1e-6
    if what == "rank_deficient":
        s.P[2, 3] = s.P[2, 1]
    a, log = _run(s, None)
    b, _ = _run(s, "direct")
    assert "mode 7: block form" not in log
    for key in b:
        assert np.array_equal(a[key], b[key]), key


@pytest.mark.gpu
def test_new_inputs_change_the_path_and_a_replayed_graph():
    """H replaced by one outside the rule and back: each N(mu) equals a fresh context's, also by graph replay."""
    from paper_1111_2157_gb300 import gf
    s = _inputs(4, 20, 6, 64, 40.0, 3)
    bad = s.H.copy()
    bad[0, 1, 3] += 1e-5
    ref = {}
    for name, H in (("good", s.H), ("bad", bad)):
        g = gf.GreensFunction.for_systems([s])
        g.set_hamiltonian(H)
        g.set_projectors(s.P)
        g.set_sigma(s.sigma, s.sigma_inf)
        ref[name] = g.occupation([0.2])
        g.close()
    g = gf.GreensFunction.for_systems([s], graph=True)
    g.set_projectors(s.P)
    g.set_sigma(s.sigma, s.sigma_inf)
    for name, H in (("good", s.H), ("bad", bad), ("good", s.H)):
        g.set_hamiltonian(H)
        for _ in range(3):
            n, dn = g.occupation([0.2])
            assert n[0] == ref[name][0][0] and dn[0] == ref[name][1][0]
    g.close()
