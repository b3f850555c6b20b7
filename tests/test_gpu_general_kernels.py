"""The general kernels, which take the inputs outside the block form, against the oracle: the tests of each precision
again with GF_KERNEL naming them (the block form would run otherwise), inputs outside the rule in every precision,
and the mixed block kernels over systems that differ in orbitals, windows and temperature."""
import numpy as np
import pytest

from paper_1111_2157_gb300 import synth
from tests import test_gpu_batched, test_gpu_lowrank, test_gpu_mixed, test_gpu_pair
from tests.parity import check_system_set, make_gf, oracle_all, rel, split_sys
from tests.test_block_form import _inputs

pytestmark = pytest.mark.gpu
MIXED, PAIR = test_gpu_mixed.TOL, test_gpu_pair.TOL
FP64 = {"G_loc": 1e-10, "N": 1e-10, "dN_dmu": 1e-10, "n_corr": 1e-10, "rho": 1e-10}


@pytest.mark.parametrize("precision,lowrank,kernel", [
    ("fp64", False, "direct"), ("pair", False, "direct"), ("fp64", True, "direct"), ("mixed", True, "direct"),
    ("mixed", False, "f32r"), ("mixed", False, "w32"), ("mixed", False, "direct")])
def test_a_named_kernel_keeps_the_block_form_out(precision, lowrank, kernel, monkeypatch):
    monkeypatch.setenv("GF_KERNEL", kernel)
    s = synth.ce_like(nk=3, n_iw=48).systems[0]
    g = make_gf([s], precision=precision, lowrank=lowrank)
    g.evaluate([0.1])
    g.backward([0.1], n_bar=[1.0])
    assert "block form" not in g.tuning_log()


@pytest.mark.parametrize("name", ["ce_like_small", "nio_like_small", "ragged_multi_system", "complex64_inputs",
                                  "tail_order_one", "backward", "find_mu", "ce_like_full_size_sampled"])
def test_pair_kernels(name, monkeypatch):
    monkeypatch.setenv("GF_KERNEL", "direct")
    getattr(test_gpu_pair, "test_" + name)()


@pytest.mark.parametrize("name", ["ce_like_small_all_outputs", "ragged_systems_and_edge_shapes", "find_mu_and_backward",
                                  "new_hamiltonian_refreshes_the_eigenbasis",
                                  "graph_replay_of_the_low_rank_mu_search", "mixed_precision_backward_and_mu_search",
                                  "ce_like_full_size_sampled"])
def test_low_rank_kernel(name, monkeypatch):
    monkeypatch.setenv("GF_KERNEL", "direct")
    getattr(test_gpu_lowrank, "test_" + name)()


@pytest.mark.parametrize("case", ["ce_like", "ragged"])
def test_low_rank_kernel_with_pair_band_sums(case, monkeypatch):
    monkeypatch.setenv("GF_KERNEL", "direct")
    test_gpu_lowrank.test_mixed_precision_band_sums(case)


@pytest.mark.parametrize("name", ["d_toy_full_size", "ce_like_small", "nio_like_small", "window_128",
                                  "ragged_multi_system", "complex64_inputs", "tail_order_one", "backward", "find_mu",
                                  "ce_like_full_size_sampled", "nio_like_full_size_sampled"])
def test_mixed_register_tiles(name, monkeypatch):
    monkeypatch.setenv("GF_KERNEL", "f32r")
    getattr(test_gpu_mixed, "test_" + name)()


@pytest.mark.parametrize("precision,kernel", [("fp64", "direct"), ("mixed", "f32r"), ("pair", "direct")])
def test_batched_systems(precision, kernel, monkeypatch):
    monkeypatch.setenv("GF_KERNEL", kernel)
    test_gpu_batched.test_one_launch_for_all_systems_matches_oracle(precision)


@pytest.mark.parametrize("what", ["dependent_rows", "few_frequencies", "no_rest"])
@pytest.mark.parametrize("precision,lowrank,tol", [("fp64", False, FP64), ("mixed", False, MIXED), ("pair", False, PAIR),
                                                   ("fp64", True, FP64)])
def test_inputs_outside_the_rule_against_the_oracle(what, precision, lowrank, tol):
    m = 20 if what == "no_rest" else 6  # (as many orbitals as bands)
    s = _inputs(3, 20, m, 12 if what == "few_frequencies" else 48, 40.0, 9)
    if what == "dependent_rows":
        s.P[2, 3] = s.P[2, 1]
    check_system_set([s], [0.15], tol, precision=precision, lowrank=lowrank)


def test_mixed_block_kernels_over_systems_that_differ():
    """Orbitals below the context's largest (5, 9, 14), windows that differ from k to k, projectors that are not
    orthonormal, beta 20 to 400, one context."""
    rng = synth.rng_for(99)
    systems, mus = [], [0.2, -0.4, 0.7]
    for m, nbs, beta in ((5, [9, 17, 30], 20.0), (9, [12, 33], 100.0), (14, [40, 21, 16, 64], 400.0)):
        H = [synth.hamiltonian_dense(rng, 1, n, -6.0, 6.0, 0.3)[0] for n in nbs]
        P = [synth.projectors(rng, 1, n, m)[0] for n in nbs]
        P = [p + 0.06 * (rng.standard_normal(p.shape) + 1j * rng.standard_normal(p.shape)) for p in P]
        pole = synth.sigma_two_pole(rng, m, 4.0)
        systems.append(synth.System(H, P, pole, pole.sample(beta, 130), beta, 1.0))
    g = make_gf(systems, precision="mixed")
    gl = split_sys(g.local(mus).cpu().numpy(), systems, lambda s: s.n_iw * s.m * s.m)
    n, dn = g.occupation(mus)
    rho, nc = g.density_matrix(mus)
    rho = split_sys(rho.cpu().numpy(), systems, lambda s: int(np.sum(s.nb.astype(np.int64) ** 2)))
    r = g.evaluate(mus)
    log = g.tuning_log()
    assert all(f"mode {mode}: block form" in log for mode in (1, 2, 4, 7)) and "in FP32 and FP32 pairs" in log
    assert np.max(np.abs(r["N"] - n) / n) < 1e-7
    for i, s in enumerate(systems):
        ref, glo = oracle_all(s, mus[i])
        assert rel(gl[i], glo.reshape(-1)) < MIXED["G_loc"]
        assert abs(n[i] - ref["N"]) < MIXED["N"] * ref["N"]
        assert abs(dn[i] - ref["dN_dmu"]) < MIXED["dN_dmu"] * abs(ref["dN_dmu"])
        assert abs(nc[i] - ref["n_corr"]) < MIXED["n_corr"] * abs(ref["n_corr"])
        assert rel(rho[i], np.concatenate([np.asarray(x).reshape(-1) for x in ref["rho"]])) < MIXED["rho"]
