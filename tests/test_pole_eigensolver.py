"""The eigensolver of the pole path and the block form's set-up on matrices that are not generic."""
import numpy as np
import pytest

from oracle import pole as pole_oracle
from paper_1111_2157_gb300 import gf, synth
from tests.test_block_form import _rel, _run

pytestmark = pytest.mark.gpu


def _matrix(kind, n, rng):
    X = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    Q = np.linalg.qr(X)[0]
    H = {"two_levels": lambda: (Q * np.repeat([0.0, 1.0], (n + 1) // 2)[:n]) @ np.conj(Q.T),
         "three_levels": lambda: (Q * np.repeat([-1.0, 0.0, 2.0], (n + 2) // 3)[:n]) @ np.conj(Q.T),
         "ten_levels": lambda: (Q * np.repeat(rng.uniform(-8, 8, 10), (n + 9) // 10)[:n]) @ np.conj(Q.T),
         "rank_one": lambda: np.outer(X[0], np.conj(X[0])),
         "ones": lambda: np.ones((n, n), complex),
         "chain": lambda: np.diag(np.ones(n - 1), 1) + np.diag(np.ones(n - 1), -1) + 0j,
         "ring": lambda: np.roll(np.eye(n), 1, 0) + np.roll(np.eye(n), -1, 0) + 0j,
         "spin": lambda: np.kron((X + np.conj(X.T))[:n // 2, :n // 2], np.eye(2)),
         "repeated_blocks": lambda: np.kron(np.eye((n + 4) // 5), (X + np.conj(X.T))[:5, :5])[:n, :n]}[kind]()
    return 0.5 * (H + np.conj(H.T))


@pytest.mark.parametrize("n,m", [(13, 3), (70, 6), (130, 4), (200, 3)])
@pytest.mark.parametrize("kind", ["two_levels", "three_levels", "ten_levels", "rank_one", "ones", "chain", "ring", "spin",
                                  "repeated_blocks"])
def test_few_distinct_levels(kind, n, m):
    """N and rho_k of the pole path against the oracle, and of the block form against the inverse (bound: 1e2 roundings
    of the norm over w_0 and 1e1 of the sums)."""
    rng = np.random.default_rng(n)
    H = _matrix(kind, n, rng)
    n = H.shape[0]
    P = np.linalg.qr(rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n)))[0][:m]
    pole = synth.sigma_two_pole(synth.rng_for(3), m, 3.0)
    s = synth.System(H[None], P[None], pole, pole.sample(40.0, 24), 40.0, n / 2.0)
    g = gf.GreensFunction.for_systems([s])
    g.set_hamiltonian(s.H)
    g.set_projectors(s.P)
    g.set_sigma_poles([len(pole.p)], pole.p, pole.V.reshape(-1), pole.sigma_inf.reshape(-1))
    num, _ = g.pole_occupation([0.1])
    rho, _ = g.pole_density_matrix([0.1])
    g.close()
    ref = pole_oracle.density(s.H, s.P, s.sigma_inf, pole.p, pole.V, s.beta, 0.1)
    assert abs(num[0] - ref["N"]) < 1e-12 * ref["N"]
    assert _rel(rho.cpu().numpy(), np.asarray(ref["rho"]).reshape(-1)) < 1e-12
    if n <= 70:
        a, log = _run(s, None)
        b, _ = _run(s, "direct")
        assert "mode 7: block form" in log
        for key in ("N", "rho", "gloc", "n_corr"):
            assert _rel(a[key], b[key]) < 1e-12, key


@pytest.mark.parametrize("n,m,offset", [(12, 3, 100.0), (31, 5, 1000.0), (70, 6, 1e4), (31, 5, 8.0), (20, 12, 100.0)])
def test_few_electrons(n, m, offset):
    """Bands far above mu, where N is the bands' small share of the occupied pole levels: relative to N, not to the
    number of poles.  (Bound: the eigenvectors' 1e-15, over amplitudes of U / offset, on two k-points that differ.)"""
    rng = np.random.default_rng(n)
    H = np.array([synth.hamiltonian_dense(synth.rng_for(n), 1, n, -2.0, 2.0, 0.3)[0] + x * np.eye(n)
                  for x in (offset, 0.0)])
    P = np.array([np.linalg.qr(rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n)))[0][:m] for _ in range(2)])
    pole = synth.sigma_two_pole(synth.rng_for(3), m, 3.0)
    for ks in ([0], [0, 1]):
        g = gf.GreensFunction([n] * len(ks), [m], 24, [40.0])
        g.set_hamiltonian(H[ks].reshape(-1))
        g.set_projectors(P[ks].reshape(-1))
        g.set_sigma_poles([len(pole.p)], pole.p, pole.V.reshape(-1), pole.sigma_inf.reshape(-1))
        num, dn = g.pole_occupation([0.1])
        g.close()
        ref = pole_oracle.density(H[ks], P[ks], pole.sigma_inf, pole.p, pole.V, 40.0, 0.1)
        assert abs(num[0] - ref["N"]) < 1e-15 * (10.0 + offset) * 10.0 * ref["N"]
        assert abs(dn[0] - ref["dN_dmu"]) < 1e-10 * abs(ref["dN_dmu"])
