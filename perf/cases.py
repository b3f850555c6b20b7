"""What this library is measured on: the work that LDA+DMFT programs have it do.

Inputs are seeded and synthetic, with the shapes of the d-shell toy, the Ce-like f system, the
NiO-like antiferromagnet, the ragged batch and the adjoint workload of bench.py: a Hermitian
band-window H_k (diagonal uniform in [-8, 8] eV, off-diagonal complex Gaussian), projectors with
orthonormal rows, and a causal pole-form self-energy sampled on the Matsubara grid.  k-meshes
are the symmetry-reduced or coarse ones of such runs, so that a pass stays below a second.

Everything a program has before the call (tensors on the GPU, the context with H_k and P_k) is
made by prepare; run is one pass of the program.  G_loc and Sigma_bar are kept as complex128 in
every mode.  Where a program chooses the mixed mode, what it takes from the single-precision
inverse (rho_k, N, dN/dmu, n_corr, a chemical potential and whatever depends on it) is kept in
single-precision arrays.
"""
import math

import numpy as np
import torch

from paper_1111_2157_gb300 import autograd, gf

DEV = "cuda:0"
ETA = 0.1          # Lorentzian half width of the density of states (eV)
N_EPS = 201        # energies of the density of states


def listed():
    return [
        # the smallest call: N(mu) of the d-shell toy (8 bands, diagonal H), launch bound
        dict(name="toy_occupation", kind="occupation", precision="fp64", nk=64, nb=8, m=5, n_iw=256, beta=40.0,
             U=4.0, diag=True),
        # one DMFT step in FP64 with a new Sigma: mu search, then G_loc (Ce-like f shell)
        dict(name="ce_step_fp64", kind="step", precision="fp64", nk=64, nb=40, m=14, n_iw=1024, beta=100.0, U=6.0),
        # every output of the fused pass in FP64: G_loc, rho_k, N, dN/dmu, n_corr
        dict(name="ce_evaluate_fp64", kind="evaluate", precision="fp64", nk=216, nb=40, m=14, n_iw=1024, beta=100.0,
             U=6.0),
        # the same DMFT step in mixed precision on a denser mesh
        dict(name="ce_step_mixed", kind="step", precision="mixed", nk=256, nb=40, m=14, n_iw=1024, beta=100.0, U=6.0),
        # the fused pass of a two-atom antiferromagnet: wide window, many frequencies
        dict(name="nio_evaluate_mixed", kind="evaluate", precision="mixed", nk=48, nb=96, m=20, n_iw=2048, beta=40.0,
             U=8.0, afm=True),
        # several materials in one context, windows that differ from k to k, complex128 and complex64 inputs
        dict(name="batched_evaluate_mixed", kind="evaluate", precision="mixed", nk=24, nb=128, nb_min=48, m=14, m_min=10,
             n_iw=1024, beta=40.0, U=6.0, n_sys=4, dtype="per_system"),
        # forward and backward of a loss on G_loc and N through torch.autograd, FP64
        dict(name="adjoint_fp64", kind="autograd", precision="fp64", nk=32, nb=64, m=14, n_iw=1024, beta=100.0, U=6.0),
        # the vector-Jacobian product alone in mixed precision, complex64 inputs
        dict(name="adjoint_mixed", kind="backward", precision="mixed", nk=128, nb=64, m=14, n_iw=512, beta=100.0, U=6.0,
             dtype="c64"),
        # charge self-consistency: new H_k, P_k and Sigma on every pass, odd sizes, mu search and rho_k
        dict(name="charge_step_fp64", kind="charge", precision="fp64", nk=75, nb=37, m=10, n_iw=333, beta=60.0, U=4.5),
        # the low-rank option: the fused pass in the eigenbasis of H_k
        dict(name="lowrank_evaluate_fp64", kind="evaluate", precision="fp64", nk=216, nb=40, m=14, n_iw=1024, beta=100.0,
             U=6.0, lowrank=True),
        # Sigma in pole form: mu search, rho_k, G_loc and the density of states from the pseudo-Hamiltonian
        dict(name="pole_step", kind="pole", precision="fp64", nk=125, nb=40, m=14, n_iw=512, beta=100.0, U=6.0),
        # around the lattice sums, full 10x10x10 mesh: projectors from raw projections, levels, hybridization
        dict(name="dmft_update", kind="dmft", precision="fp64", nk=1000, nb=40, m=14, n_iw=1024, beta=100.0, U=6.0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["occupation", "step", "evaluate", "evaluate", "batched", "backward", "autograd", "charge", "pole",
                       "dmft"])
    c = dict(kind=kind, precision="fp64", beta=round(rng.uniform(20.0, 100.0), 2), U=round(rng.uniform(4.0, 8.0), 2))
    nb = _log_int(rng, 8, 64 if kind in ("pole", "dmft", "charge") else 128)
    m = rng.randint(2, max(2, min(20, (3 * nb) // 5)))
    n_iw = _log_int(rng, 128, 2048)
    if kind in ("step", "evaluate", "backward"):
        c["precision"] = rng.choice(["fp64", "mixed", "mixed"])
    if kind == "evaluate" and rng.random() < 0.3:
        c["precision"], c["lowrank"] = "fp64", True
    if kind in ("evaluate", "backward", "charge"):
        c["dtype"] = rng.choice(["c128", "c128", "c64"])
    if kind == "step" and rng.random() < 0.3:
        c["graph"] = True
    if kind == "occupation":
        nb, m, c["diag"] = rng.randint(8, 24), rng.randint(3, 7), rng.random() < 0.5
    if kind == "batched":
        c["kind"], c["precision"], c["dtype"], c["n_sys"] = "evaluate", "mixed", "per_system", rng.randint(2, 5)
        nb, m, n_iw = max(nb, 32), rng.randint(5, 14), min(n_iw, 1024)
        c["nb_min"], c["m_min"] = rng.randint(16, nb), rng.randint(3, m)
    # points of a pass, so that it costs no more than the largest listed one of its kind and precision
    mixed = c["precision"] == "mixed"
    cost = {"step": (4e9, 1.5e10), "evaluate": (1.2e10, 6e10), "batched": (0, 6e10), "backward": (4e9, 1.5e10),
            "autograd": (8e9, 0), "charge": (1.2e9, 0), "occupation": (1e9, 0)}.get(kind, (1e9, 0))[mixed]
    points = cost / float(max(nb, 24)) ** 3
    most = max(4, min(512, int(points) // (n_iw * c.get("n_sys", 1))))
    if kind == "dmft":
        most = 1000
    if kind == "pole":
        most = max(4, min(125, int(125 * (68.0 / (nb + 2 * m)) ** 3)))
    c.update(nb=nb, m=m, n_iw=n_iw, nk=_log_int(rng, max(2, most // 6), most))
    return c


# ------------------------------------------------------------------------------------------- inputs
def _systems(case, seed):
    """The inputs of every system, complex128 on the GPU: lists over k of H and P, and Sigma in pole form."""
    gen = torch.Generator(device=DEV).manual_seed(int(seed))
    host = np.random.Generator(np.random.PCG64(int(seed)))

    def normal(*shape):
        return torch.complex(torch.randn(*shape, generator=gen, device=DEV, dtype=torch.float64),
                             torch.randn(*shape, generator=gen, device=DEV, dtype=torch.float64))

    out = []
    shape = np.random.Generator(np.random.PCG64(1111))  # windows and orbitals: the case's, not the seed's
    for s in range(case.get("n_sys", 1)):
        nk, m = case["nk"], int(shape.integers(case.get("m_min", case["m"]), case["m"] + 1))
        nb_max = case["nb"]
        nb = (shape.integers(max(case["nb_min"], m), nb_max + 1, size=nk) if "nb_min" in case else np.full(nk, nb_max))
        diag = 16.0 * torch.rand(nk, nb_max, generator=gen, device=DEV, dtype=torch.float64) - 8.0
        if case.get("diag"):
            H = torch.diag_embed(diag).to(torch.complex128)
        else:
            X = torch.triu(normal(nk, nb_max, nb_max) * (0.3 / math.sqrt(2.0)), 1)
            H = X + X.mH + torch.diag_embed(diag)
        Z = normal(nk, nb_max, m)
        # two poles per orbital near +-U/2 with weight U^2/8 each, rotated by a unitary matrix
        # (antiferromagnet: block-diagonal over atoms and spins of five orbitals, poles shifted by -+1 eV)
        U = case["U"]
        rot = np.zeros((m, m), np.complex128)
        step = 5 if case.get("afm") else m
        for a in range(0, m, step):
            w = min(step, m - a)
            rot[a:a + w, a:a + w] = np.linalg.qr(host.standard_normal((w, w)) + 1j * host.standard_normal((w, w)))[0]
        shift = [(-1.0) ** (a // step + a // (2 * step) + 1) if case.get("afm") else 0.0 for a in range(m)]
        p = np.array([sg * U / 2 + shift[a] + 0.1 * host.standard_normal() for a in range(m) for sg in (1, -1)])
        V = np.array([math.sqrt(U * U / 8) * np.conj(rot[:, a]) for a in range(m) for _ in (1, -1)])
        p, V = torch.tensor(p, device=DEV), torch.tensor(V, device=DEV)
        sinf = (U / 2) * torch.eye(m, dtype=torch.complex128, device=DEV)
        wn = _wn(case)
        f = 1.0 / (1j * wn[:, None] - p[None, :])
        sig = torch.einsum("ia,ni,ib->nab", V.conj(), f, V) + sinf
        # projectors: orthonormal rows, or raw projections with unit rows that are not orthogonal
        Hk, Pk = [], []
        for k in range(nk if "nb_min" in case else 0):
            n = int(nb[k])
            Hk.append(H[k, :n, :n].contiguous())
            Pk.append(torch.linalg.qr(Z[k, :n])[0].mH.resolve_conj().contiguous())
        if "nb_min" not in case:
            Hk = H.contiguous()
            Pk = (Z / torch.linalg.vector_norm(Z, dim=1, keepdim=True) if case["kind"] == "dmft"
                  else torch.linalg.qr(Z)[0]).mH.resolve_conj().contiguous()
        dtype = case.get("dtype", "c128")
        if dtype == "per_system":
            dtype = ("c128", "c64")[s % 2]
        if dtype == "c64":  # what the program holds: values rounded to single precision
            def low(x):
                return x.to(torch.complex64).to(torch.complex128)
            Hk = low(Hk) if torch.is_tensor(Hk) else [low(h) for h in Hk]
            Pk = low(Pk) if torch.is_tensor(Pk) else [low(h) for h in Pk]
            sig, sinf = low(sig), low(sinf)
        out.append(dict(nb=[int(n) for n in nb], m=m, H=Hk, P=Pk, p=p, V=V, sinf=sinf, sig=sig, dtype=dtype,
                        target=float(np.mean(nb)) / 2, mu=0.1 + 0.05 * s + 0.1 * float(host.random())))
    return out


def _wn(case):
    return (2.0 * torch.arange(case["n_iw"], device=DEV, dtype=torch.float64) + 1.0) * (math.pi / case["beta"])


def _flat(xs):
    return xs.reshape(-1) if torch.is_tensor(xs) else torch.cat([x.reshape(-1) for x in xs])


def _tol(case, sys):
    """Tolerance of the mu search: 1e-10 electrons in FP64, 1e-8 of the filling in mixed precision."""
    return 1e-10 if case["precision"] == "fp64" else 1e-8 * sys[0]["target"]


def prepare(case, seed):
    sys = _systems(case, seed)
    nb = np.concatenate([s["nb"] for s in sys])
    dts = [s["dtype"] for s in sys]
    cdt = {"c128": torch.complex128, "c64": torch.complex64}
    several = len(sys) > 1
    g = gf.GreensFunction(nb, [s["m"] for s in sys], case["n_iw"], [case["beta"]] * len(sys),
                          k_system=np.repeat(np.arange(len(sys)), [len(s["nb"]) for s in sys]) if several else None,
                          precision=case["precision"], input_dtype=dts if several else dts[0],
                          graph=case.get("graph", False), lowrank=case.get("lowrank", False))

    def held(key):
        parts = [_flat(s[key]).to(cdt[s["dtype"]]) for s in sys]
        return parts if several else parts[0]

    st = dict(case=case, g=g, mu=[s["mu"] for s in sys], target=[s["target"] for s in sys], tol=_tol(case, sys),
              H=held("H"), P=held("P"), sig=held("sig"), sinf=held("sinf"))
    if case.get("diag"):
        st["H"] = torch.diagonal(sys[0]["H"], dim1=1, dim2=2).contiguous().reshape(-1)
    gen = torch.Generator(device=DEV).manual_seed(int(seed) + 1)
    n_sig = sum(case["n_iw"] * s["m"] ** 2 for s in sys)
    # the gradient of a loss that is a mean over the frequencies
    st["gbar"] = torch.complex(torch.randn(n_sig, generator=gen, device=DEV, dtype=torch.float64),
                               torch.randn(n_sig, generator=gen, device=DEV, dtype=torch.float64)) / case["n_iw"]
    if case["kind"] == "charge":
        return st
    g.set_hamiltonian(st["H"], diagonal=bool(case.get("diag")))
    if case["kind"] == "dmft":
        wn, m = _wn(case), sys[0]["m"]
        e = torch.linspace(-2.0, 2.0, m, device=DEV, dtype=torch.float64)
        gl = torch.diag_embed(1.0 / (1j * wn[:, None] + st["mu"][0] - e[None, :]))
        st["gloc"] = (gl + 0.1 * case["n_iw"] * gl @ st["gbar"].view(-1, m, m) @ gl).reshape(-1)
        st["vdc"] = [case["U"] * 0.5]
    else:
        g.set_projectors(st["P"])
    if case["kind"] == "pole":
        st["poles"] = (len(sys[0]["p"]), sys[0]["p"], sys[0]["V"].reshape(-1), sys[0]["sinf"].reshape(-1))
        st["eps"] = np.linspace(-10.0, 10.0, N_EPS)
    else:
        g.set_sigma(st["sig"], st["sinf"])
    if case["kind"] == "autograd":
        m = sys[0]["m"]
        st["leaf"] = st["sig"].view(case["n_iw"], m, m)
        st["mu_t"] = torch.tensor(st["mu"], dtype=torch.float64)
    return st


# ------------------------------------------------------------------------------------------- one pass
def run(st):
    case, g, mu = st["case"], st["g"], st["mu"]
    kind, single = case["kind"], case["precision"] == "mixed"
    if kind == "occupation":
        n, dn = g.occupation(mu)
        return {"N": n, "dN": dn}
    if kind == "step":
        g.set_sigma(st["sig"], st["sinf"])
        mu, _ = g.find_mu(st["target"], mu0=0.0, tol=st["tol"])
        gl = g.local(mu)
        return {"mu": np.float32(mu), "gloc": gl.to(torch.complex64)} if single else {"mu": mu, "gloc": gl}
    if kind == "evaluate":
        r = g.evaluate(mu)
        if single:
            r = {"gloc": r["gloc"], "rho": r["rho"].to(torch.complex64), "N": np.float32(r["N"]),
                 "dN_dmu": np.float32(r["dN_dmu"]), "n_corr": np.float32(r["n_corr"])}
        return r
    if kind == "autograd":
        sig = st["leaf"].detach().requires_grad_(True)
        mu_t = st["mu_t"].detach().requires_grad_(True)
        gl, n = autograd.lattice_green(g, sig, mu_t, st["sinf"])
        loss = torch.sum((gl.reshape(-1) * st["gbar"].conj()).real).cpu() + 3.0 * n.sum()
        loss.backward()
        return {"loss": loss.detach(), "gloc": gl.detach(), "N": n.detach(), "sigma_bar": sig.grad, "mu_bar": mu_t.grad}
    if kind == "backward":
        sb, mb = g.backward(mu, gloc_bar=st["gbar"], n_bar=[1.5] * len(mu))
        return {"sigma_bar": sb, "mu_bar": np.float32(mb) if single else mb}
    if kind == "charge":
        g.set_hamiltonian(st["H"])
        g.set_projectors(st["P"])
        g.set_sigma(st["sig"], st["sinf"])
        mu, _ = g.find_mu(st["target"], mu0=0.0, tol=st["tol"])
        rho, nc = g.density_matrix(mu)
        return {"mu": mu, "rho": rho, "n_corr": nc}
    if kind == "pole":
        g.set_sigma_poles(*st["poles"])
        mu, _ = g.pole_find_mu(st["target"], mu0=0.0, tol=st["tol"])
        rho, nc = g.pole_density_matrix(mu)
        gl = g.pole_local(mu)
        dos, pdos = g.pole_spectral(mu, st["eps"], ETA)
        return {"mu": mu, "rho": rho, "n_corr": nc, "gloc": gl, "dos": dos, "pdos": pdos[0]}
    # dmft: projectors from raw projections, impurity levels, hybridization function
    P = g.set_projectors_lowdin(st["P"])
    e_imp = g.impurity_levels(st["vdc"])
    delta = g.hybridization(mu, st["gloc"], st["vdc"])
    return {"P": P, "e_imp": e_imp, "delta": delta}


# ------------------------------------------------------------------------------------------- its work
def work(case):
    """Inputs and outputs once, and the complex multiply-adds (8 flops) of the outputs that are asked for: an
    m x m block of the inverse and traces of it need the (N_b - m) m^2 products that couple the block to the
    rest of the window and m^3 for its own inverse, not the whole window's; rho_k needs m N_b^2 more per
    frequency; an eigenproblem is counted as 10 n^3."""
    ns, nk, niw = case.get("n_sys", 1), case["nk"], case["n_iw"]
    nb = 0.5 * (case.get("nb_min", case["nb"]) + case["nb"])
    m = 0.5 * (case.get("m_min", case["m"]) + case["m"])
    size = 8.0 if case.get("dtype") == "c64" else 16.0
    pts, kind = float(ns * nk * niw), case["kind"]
    hk, pk, sg = ns * nk * nb * nb, ns * nk * nb * m, ns * niw * m * m
    block = (nb - m) * m * m + m ** 3
    inputs = size * ((ns * nk * nb if case.get("diag") else hk) + pk + sg)
    if kind == "occupation":
        return {"bytes": inputs, "flops": 8 * pts * (3 * block)}
    if kind == "step":
        return {"bytes": inputs + 16 * sg, "flops": 8 * pts * (4 * 3 * block + block)}
    if kind in ("evaluate", "charge"):
        n_mu = 4 if kind == "charge" else 1
        return {"bytes": inputs + 16 * (hk + (sg if kind == "evaluate" else 0)),
                "flops": 8 * pts * (n_mu * 3 * block + m * nb * nb)}
    if kind == "backward":
        return {"bytes": inputs + 32 * sg, "flops": 8 * pts * (2 * block + 4 * m ** 3)}
    if kind == "autograd":
        return {"bytes": inputs + 64 * sg, "flops": 8 * pts * (5 * block + 4 * m ** 3)}
    if kind == "pole":
        n = nb + 2 * m
        return {"bytes": inputs + 16 * (hk + sg),
                "flops": 8 * nk * (4 * 10 * n ** 3 + n * nb * nb + niw * n * m * m / 2 + N_EPS * n * m / 4)}
    return {"bytes": 16 * (hk + 2 * pk + 3 * sg), "flops": 8.0 * (nk * (m * nb * nb + 2 * m * m * nb + 10 * m ** 3) + niw * m ** 3)}


# ------------------------------------------------------------------------------------------- in 64 bits
class _Sums:
    """The lattice sums of one system, by the definition: A = (i w + mu) - H - P^+ Sigma P inverted in
    complex128 for every k and frequency."""

    def __init__(self, case, s):
        self.case, self.s, self.wn = case, s, _wn(case)
        self.nk, self.beta = len(s["nb"]), case["beta"]
        w = self.wn
        # (2/beta) sum 1/w^2 over the grid minus its exact sum beta/4
        self.tail = float(2.0 / self.beta * torch.sum(1.0 / (w * w).flip(0)) - self.beta / 4)

    def blocks(self):
        """(k range, H, P) in groups of equal windows."""
        s = self.s
        if torch.is_tensor(s["H"]):
            n = max(1, int(3.0e4 * (40.0 / s["nb"][0]) ** 2) // self.case["n_iw"])
            for k in range(0, self.nk, n):
                yield k, s["H"][k:k + n], s["P"][k:k + n]
        else:
            for k in range(self.nk):
                yield k, s["H"][k][None], s["P"][k][None]

    def green(self, H, P, mu):
        n = H.shape[-1]
        A = (-H[:, None] - P.mH[:, None] @ self.s["sig"][None] @ P[:, None])
        z = mu + 1j * self.wn
        A.diagonal(dim1=-2, dim2=-1).add_(z[None, :, None].expand(H.shape[0], -1, n))
        return torch.linalg.inv(A)

    def all(self, mu, gloc=False, rho=False, bar=None):
        s, beta = self.s, self.beta
        out = dict(N=0.0, dN=0.0, n_corr=0.0, mu_bar=0.0, rho=[], gloc=0.0, sigma_bar=0.0)
        for _, H, P in self.blocks():
            G = self.green(H, P, mu)
            n = H.shape[-1]
            eye = torch.eye(n, dtype=torch.complex128, device=DEV)
            M2 = H + P.mH @ s["sinf"] @ P - mu * eye
            S = G.sum(1)
            r = (S + S.mH) / beta + self.tail * M2 + 0.5 * eye
            out["N"] += float(torch.einsum("kii->", r).real) / self.nk
            g2 = torch.einsum("knij,knji->", G, G).real
            out["dN"] += float(-2.0 / beta * g2 - H.shape[0] * n * self.tail) / self.nk
            if rho:
                out["rho"].append(r.reshape(-1))
                out["n_corr"] += float(torch.einsum("kai,kij,kaj->", P, r, P.conj()).real) / self.nk
            if gloc or bar is not None:
                Y = G @ P.mH[:, None]
                A = P[:, None] @ Y
                if gloc:
                    out["gloc"] = out["gloc"] + A.sum(0) / self.nk
                if bar is not None:
                    B = (P[:, None] @ G) @ Y
                    gb, nbar = bar
                    out["sigma_bar"] = out["sigma_bar"] + (A.mH @ gb[None] @ A.mH + nbar * (2 / beta) * B.mH).sum(0) / self.nk
                    out["mu_bar"] -= float((gb.conj()[None] * B).real.sum()) / self.nk
            del G
        if bar is not None:
            out["mu_bar"] += bar[1] * out["dN"]
        return out


def _newton(f, target, tol=1e-12):
    mu, lo, hi = 0.0, -math.inf, math.inf
    for _ in range(40):
        n, dn = f(mu)
        if abs(n - target) <= tol:
            break
        lo, hi = (max(lo, mu), hi) if n < target else (lo, min(hi, mu))
        new = mu + max(-4.0, min(4.0, (target - n) / max(dn, 1e-300)))
        if not lo < new < hi:
            new = 0.5 * (lo + hi)
        if new == mu or abs(new - mu) < 1e-15 * max(1.0, abs(mu)):
            break
        mu = new
    return mu


def _exact_pole(case, s):
    beta, wn, nk, m = case["beta"], _wn(case), len(s["nb"]), s["m"]
    H, P, p, V = s["H"], s["P"], s["p"], s["V"]
    nb, n_p = H.shape[-1], len(p)
    Hp = torch.zeros(nk, nb + n_p, nb + n_p, dtype=torch.complex128, device=DEV)
    Hp[:, :nb, :nb] = H + P.mH @ s["sinf"] @ P
    W = V[None] @ P
    Hp[:, nb:, :nb], Hp[:, :nb, nb:] = W, W.mH
    i = torch.arange(n_p, device=DEV) + nb

    def eig(mu):
        A = Hp.clone()
        A[:, i, i] = (p + mu).to(torch.complex128)
        return torch.linalg.eigh(A)

    def occ(mu):
        E, X = eig(mu)
        x = E - mu
        f = 0.5 * (1 - torch.tanh(0.5 * beta * x))
        B = X[:, :nb]
        n = float((B.abs().square().sum(1) * f).sum()) / nk
        O = (B.mH @ B).abs().square()
        u = 0.5 * beta * (x[:, :, None] - x[:, None, :])
        sh = torch.where(u.abs() < 1e-4, 1 + u * u / 6, torch.sinh(u.clamp(-1, 1)) / torch.where(u == 0, 1.0, u.clamp(-1, 1)))
        ch = torch.cosh((0.5 * beta * x).clamp(-300, 300))
        near = -0.25 * beta * sh / (ch[:, :, None] * ch[:, None, :])
        dd = torch.where(u.abs() > 1, (f[:, :, None] - f[:, None, :]) / torch.where(u.abs() > 1, x[:, :, None] - x[:, None, :], 1.0), near)
        return n, float(-(O * dd).sum()) / nk

    mu = _newton(occ, s["target"])
    E, X = eig(mu)
    f = 0.5 * (1 - torch.tanh(0.5 * beta * (E - mu)))
    B = X[:, :nb]
    rho = (B * f[:, None, :]) @ B.mH
    phi = P @ B
    gl = torch.zeros(case["n_iw"], m, m, dtype=torch.complex128, device=DEV)
    e = torch.linspace(-10.0, 10.0, N_EPS, device=DEV, dtype=torch.float64)
    eps = torch.tensor(np.linspace(-10.0, 10.0, N_EPS), device=DEV)
    dos, pdos = torch.zeros_like(e), torch.zeros(N_EPS, m, device=DEV, dtype=torch.float64)
    for k in range(nk):
        d = 1.0 / (1j * wn[:, None] + mu - E[k][None])
        gl += (phi[k][None] * d[:, None, :]) @ phi[k].mH / nk
        lor = (ETA / math.pi) / ((eps[:, None] + mu - E[k][None]) ** 2 + ETA * ETA)
        dos += lor @ B[k].abs().square().sum(0) / nk
        pdos += lor @ phi[k].abs().square().T / nk
    nc = float((phi.abs().square() * f[:, None, :]).sum()) / nk
    return {"mu": np.array([mu]), "rho": rho.reshape(-1), "n_corr": np.array([nc]), "gloc": gl.reshape(-1),
            "dos": dos[None], "pdos": pdos}


def _exact_dmft(case, s, st):
    W, H, m, nk = s["P"], s["H"], s["m"], len(s["nb"])
    lam, V = torch.linalg.eigh(W @ W.mH)
    P = (V * lam.rsqrt()[:, None, :]) @ V.mH @ W
    eye = torch.eye(m, dtype=torch.complex128, device=DEV)
    e_imp = (P @ H @ P.mH).mean(0) - st["vdc"][0] * eye
    gl = st["gloc"].view(-1, m, m)
    z = (st["mu"][0] + 1j * _wn(case))[:, None, None] * eye
    delta = z - e_imp - s["sig"] - torch.linalg.inv(gl)
    return {"P": P.reshape(-1), "e_imp": e_imp.reshape(-1), "delta": delta.reshape(-1)}


def exact(case, seed):
    kind = case["kind"]
    sys = _systems(case, seed)
    if kind == "pole":
        return _exact_pole(case, sys[0])
    if kind == "dmft":
        return _exact_dmft(case, sys[0], prepare(case, seed))
    sums = [_Sums(case, s) for s in sys]
    mu = [s["mu"] for s in sys]
    if kind in ("step", "charge"):
        mu = []
        for q, s in zip(sums, sys):
            def f(x, q=q):
                r = q.all(x)
                return r["N"], r["dN"]
            mu.append(_newton(f, s["target"], 1e-11))
    gen = torch.Generator(device=DEV).manual_seed(int(seed) + 1)
    n_sig = sum(case["n_iw"] * s["m"] ** 2 for s in sys)
    gbar = torch.complex(torch.randn(n_sig, generator=gen, device=DEV, dtype=torch.float64),
                         torch.randn(n_sig, generator=gen, device=DEV, dtype=torch.float64)) / case["n_iw"]
    bars, at = [], 0
    for s in sys:
        n = case["n_iw"] * s["m"] ** 2
        bars.append(gbar[at:at + n].view(case["n_iw"], s["m"], s["m"]))
        at += n
    nbar = {"autograd": 3.0, "backward": 1.5}.get(kind)
    rs = [q.all(x, gloc=kind in ("step", "evaluate", "autograd"), rho=kind in ("evaluate", "charge"),
                bar=(b, nbar) if nbar is not None else None) for q, x, b in zip(sums, mu, bars)]

    def arr(key):
        return np.array([r[key] for r in rs])

    def cat(key):
        return torch.cat([_flat(r[key]) for r in rs])

    if kind == "occupation":
        return {"N": arr("N"), "dN": arr("dN")}
    if kind == "step":
        return {"mu": np.array(mu), "gloc": cat("gloc")}
    if kind == "evaluate":
        return {"gloc": cat("gloc"), "rho": cat("rho"), "N": arr("N"), "dN_dmu": arr("dN"), "n_corr": arr("n_corr")}
    if kind == "charge":
        return {"mu": np.array(mu), "rho": cat("rho"), "n_corr": arr("n_corr")}
    if kind == "backward":
        return {"sigma_bar": cat("sigma_bar"), "mu_bar": arr("mu_bar")}
    r = rs[0]
    loss = torch.sum((r["gloc"].reshape(-1) * gbar.conj()).real).cpu() + 3.0 * r["N"]
    return {"loss": loss, "gloc": r["gloc"], "N": arr("N"), "sigma_bar": r["sigma_bar"], "mu_bar": arr("mu_bar")}
