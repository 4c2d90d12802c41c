"""The work that users of this library have it do, as measurable cases.

Kinds of case
  rrsvd   one batch of given matrices truncated by a plan on device buffers (rrsvd_execute);
  host    the same from and to page-locked host buffers (rrsvd_execute_host), singular values only;
  check   the fixed-precision truncation (accuracy check, basis grown on the device);
  quench  one XXZ chain evolved from a product state and measured (tebd handle, graphs);
  chains  many uneven XXZ chains in one handle, one second-order Trotter step and its measurements;
  boson   a spin-boson chain at its bond caps, one second-order Trotter step and its measurements;
  grad    forward pass and gradient of an Ising observable through the autograd function.

Outputs are what such programs keep, in forms that do not depend on the arbitrary phases of singular vectors: the
singular values, the kept weight 1 - w and the two centre-site factors U s and s V^H with the sum of each left vector
made real and positive; for chains, the Schmidt values of every bond, a local observable of every site and the
accumulated fidelity prod(1 - w).  A mixed form states its results to single precision, and its factors and chain
measurements are kept in single precision here, as its users keep them.
"""
import numpy as np
import torch

from paper_1504_00992_gb300 import binding as B
from paper_1504_00992_gb300 import inputs as I
from paper_1504_00992_gb300.autograd import tfim_observable

FORMS = {"fp64": B.TEBD_PREC_FP64, "tf32": B.TEBD_PREC_TF32, "bf16": B.TEBD_PREC_BF16}


def listed():
    return [
        # the smallest call: one small matrix truncated in place of a dense SVD, where latency is everything
        {"name": "one_small_fp64", "kind": "rrsvd", "form": "fp64", "m": 96, "n": 80, "k": 12, "p": 6, "q": 2,
         "batch": 1},
        # the thetas of all bonds of a set of small chains (chi 32, d 2), truncated for a TEBD code of the user's own
        {"name": "small_batch_fp64", "kind": "rrsvd", "form": "fp64", "m": 64, "n": 64, "k": 32, "p": 10, "q": 2,
         "batch": 256},
        # large bonds (d 20, chi 100) in the plain form, the one a user takes when FP64 accuracy is asked for
        {"name": "stress_fp64", "kind": "rrsvd", "form": "fp64", "m": 2000, "n": 2000, "k": 100, "p": 20, "q": 2,
         "batch": 16},
        # ragged middle sizes in the mixed form: d 11 x chi 97 against d 9 x chi 71, one power iteration
        {"name": "ragged_tf32", "kind": "rrsvd", "form": "tf32", "m": 1067, "n": 639, "k": 71, "p": 15, "q": 1,
         "batch": 48},
        # the benchmark's batch of large bonds, mixed form with BF16 sketches
        {"name": "stress_bf16", "kind": "rrsvd", "form": "bf16", "m": 2000, "n": 2000, "k": 100, "p": 20, "q": 2,
         "batch": 152},
        # matrices that live in host memory: the whole call with its copies, entanglement spectra only
        {"name": "host_tf32", "kind": "host", "form": "tf32", "m": 2000, "n": 2000, "k": 100, "p": 20, "q": 2,
         "batch": 32},
        # a prescribed accuracy instead of a prescribed rank
        {"name": "check_fp64", "kind": "check", "m": 2000, "n": 2000, "k": 40, "p": 10, "q": 2, "batch": 8, "r": 10,
         "eps": 1e-3, "lmax": 200},
        # the plain configuration: XXZ N=20, chi 32, quench to t = 1
        {"name": "quench_fp64", "kind": "quench", "N": 20, "chi": 32, "p": 10, "q": 2, "dt": 0.05, "steps": 20},
        # a sample of the many-chain batch (uneven N, d and chi), mixed form as in its configuration
        {"name": "chains_tf32", "kind": "chains", "form": "tf32", "count": 12, "nmin": 16, "nmax": 64, "p": 10, "q": 1},
        # the same sample in the plain form
        {"name": "chains_fp64", "kind": "chains", "form": "fp64", "count": 12, "nmin": 16, "nmax": 64, "p": 10, "q": 1},
        # star-to-chain model with local dimensions 32 -> 4 and bond caps 256 -> 64
        {"name": "boson_tf32", "kind": "boson", "form": "tf32", "bosons": 16, "d0": 32, "d1": 4, "chi0": 256,
         "chi1": 64, "p": 10, "q": 2},
        # sensitivity of an observable to every coupling
        {"name": "ising_grad", "kind": "grad", "N": 40, "chi": 64, "p": 10, "q": 2, "dt": 0.02, "steps": 12},
    ]


def _between(rng, lo, hi):
    """A whole number in [lo, hi], even over its logarithm."""
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    kind = rng.choice(["rrsvd", "rrsvd", "rrsvd", "rrsvd", "host", "check", "quench", "chains", "boson", "grad"])
    if kind in ("rrsvd", "host"):
        form = rng.choice(["fp64", "tf32", "bf16"])
        m = _between(rng, 60 if kind == "rrsvd" else 500, 2000)
        n = max(48, min(2000, _between(rng, max(48, m // 3), m * 2)))
        k = _between(rng, 8, max(9, min(120, min(m, n) // 3)))
        # as many instances as the largest listed case of the form has elements, at most
        most = {"fp64": 60e6, "tf32": 300e6, "bf16": 500e6}[form] if kind == "rrsvd" else 120e6
        batch = _between(rng, 1, max(1, min(256, int(most / (m * n)))))
        return {"kind": kind, "form": form, "m": m, "n": n, "k": k, "p": rng.randint(8, 20), "q": rng.randint(1, 2),
                "batch": batch}
    if kind == "check":
        m, n = _between(rng, 400, 2000), _between(rng, 400, 2000)
        return {"kind": kind, "m": m, "n": n, "k": rng.randint(20, 40), "p": 10, "q": rng.randint(1, 2),
                "batch": rng.randint(1, 6), "r": 10, "eps": 1e-3, "lmax": 200}
    if kind == "quench":
        return {"kind": kind, "N": rng.randint(8, 20), "chi": rng.choice([16, 24, 32, 48]), "p": 10,
                "q": rng.randint(1, 2), "dt": 0.05, "steps": rng.randint(4, 16)}
    if kind == "chains":
        return {"kind": kind, "form": rng.choice(["fp64", "tf32", "bf16"]), "count": rng.randint(2, 10), "nmin": 16,
                "nmax": rng.randint(24, 64), "p": 10, "q": rng.randint(1, 2)}
    if kind == "boson":
        return {"kind": kind, "form": rng.choice(["tf32", "bf16"]), "bosons": rng.randint(6, 14),
                "d0": rng.randint(8, 32), "d1": rng.randint(3, 5), "chi0": rng.randint(70, 256),
                "chi1": rng.randint(24, 64), "p": 10, "q": rng.randint(1, 2)}
    return {"kind": "grad", "N": rng.randint(8, 40), "chi": rng.choice([16, 32, 64]), "p": 10, "q": 2, "dt": 0.02,
            "steps": rng.randint(3, 10)}


# ------------------------------------------------------------------ matrices
def _spectrum(case):
    """Decaying as exp(-j / s): s = 15 for k = 100, in proportion otherwise (15 for the prescribed accuracy)."""
    s = 15.0 if case["kind"] == "check" else max(2.0, 0.15 * case["k"])
    j = torch.arange(min(case["m"], case["n"]), dtype=torch.float64, device="cuda")
    return torch.exp(-j / s)


def _reflectors(case, seed):
    """Four complex Gaussian reflector vectors per side and instance (unit norm)."""
    g = torch.Generator(device="cuda").manual_seed(1000003 * seed + 17)
    out = []
    for size in (case["m"], case["n"]):
        v = torch.view_as_complex(torch.randn((4, case["batch"], size, 2), dtype=torch.float64, device="cuda",
                                              generator=g))
        out.append(v / torch.linalg.vector_norm(v, dim=-1, keepdim=True))
    return out


def _reflect(X, v):
    """X <- (I - 2 v v^H) X per instance, in place."""
    w = torch.bmm(v.conj().unsqueeze(1), X)
    X.baddbmm_(v.unsqueeze(2), w, alpha=-2.0)


def _theta(case, seed):
    """theta = U diag(s) V^H with U and V products of four reflectors (exactly unitary)."""
    s = _spectrum(case)
    u, v = _reflectors(case, seed)
    r = len(s)
    X = torch.zeros((case["batch"], case["m"], case["n"]), dtype=torch.complex128, device="cuda")
    X[:, torch.arange(r), torch.arange(r)] = s.to(torch.complex128)
    for i in range(4):
        _reflect(X, u[i])
    for i in range(4):  # from the right: X <- X (I - 2 v v^H)
        w = torch.bmm(X, v[i].unsqueeze(2))
        X.baddbmm_(w, v[i].conj().unsqueeze(1), alpha=-2.0)
    return X


def _centre_factors(sigma, U, Vh, dtype):
    """U s and s V^H with the sum of each left vector real and positive."""
    t = U.sum(dim=1)
    a = t.abs()
    ph = torch.where(a > 0, t / torch.where(a > 0, a, torch.ones_like(a)), torch.ones_like(t))
    s = sigma.to(torch.complex128)
    return (U * (s * ph.conj()).unsqueeze(1)).to(dtype), (Vh * (s * ph).unsqueeze(2)).to(dtype)


class _Plan:
    """A truncation plan and its workspace, kept by the program between calls."""

    def __init__(self, case, seed):
        self.case = case
        c = case
        if c["kind"] == "check":
            self.plan = B.rrsvd_plan_create_ex(c["m"], c["n"], c["k"], c["p"], c["q"], c["batch"], B.TEBD_PREC_FP64,
                                               seed, c["r"], c["eps"], c["lmax"])
        else:
            self.plan = B.rrsvd_plan_create(c["m"], c["n"], c["k"], c["p"], c["q"], c["batch"], FORMS[c["form"]],
                                            seed)
        self.k, _ = B.rrsvd_plan_dims(self.plan)
        self.bytes = B.rrsvd_workspace_size(self.plan)
        self.ws = None if c["kind"] == "host" else torch.empty(self.bytes, dtype=torch.uint8, device="cuda")

    def __del__(self):
        torch.cuda.synchronize()
        B.rrsvd_plan_destroy(self.plan)


def _pinned(shape, dtype):
    return torch.empty(shape, dtype=dtype, pin_memory=True)


def _prepare_matrices(case, seed):
    st = _Plan(case, seed)
    theta = _theta(case, seed)
    if case["kind"] == "host":
        st.theta = _pinned(theta.shape, theta.dtype)
        st.theta.copy_(theta)
        b = case["batch"]
        st.sigma = _pinned((b, st.k), torch.float64)
        st.w, st.rank = _pinned((b,), torch.float64), _pinned((b,), torch.int32)
    else:
        st.theta = theta
    torch.cuda.synchronize()
    return st


def _run_matrices(st):
    c, b, k, dev = st.case, st.case["batch"], st.k, "cuda"
    if c["kind"] == "host":
        B.rrsvd_execute_host(st.plan, st.theta.numpy(), 0, st.sigma.numpy(), None, None, st.w.numpy(),
                             st.rank.numpy(), torch.cuda.current_stream().cuda_stream)
        return {"sigma": st.sigma, "kept": 1.0 - st.w, "rank": st.rank}
    sigma = torch.empty((b, k), dtype=torch.float64, device=dev)
    U = torch.empty((b, c["m"], k), dtype=torch.complex128, device=dev)
    Vh = torch.empty((b, k, c["n"]), dtype=torch.complex128, device=dev)
    w = torch.empty((b,), dtype=torch.float64, device=dev)
    rank = torch.empty((b,), dtype=torch.int32, device=dev)
    B.rrsvd_execute(st.plan, st.theta.data_ptr(), 0, sigma.data_ptr(), U.data_ptr(), Vh.data_ptr(), w.data_ptr(),
                    rank.data_ptr(), st.ws.data_ptr(), st.bytes, torch.cuda.current_stream().cuda_stream)
    dtype = torch.complex128 if c["kind"] == "check" or c["form"] == "fp64" else torch.complex64
    left, right = _centre_factors(sigma, U, Vh, dtype)
    return {"sigma": sigma, "left": left, "right": right, "kept": 1.0 - w, "rank": rank}


def _exact_matrices(case, seed):
    s = _spectrum(case)
    b = case["batch"]
    if case["kind"] == "check":  # the kept rank follows the grown basis: no closed form
        return None
    k = min(case["k"], case["m"], case["n"])
    total = float((s ** 2).sum())
    out = {"sigma": s[:k].expand(b, k).contiguous(), "kept": torch.full((b,), float((s[:k] ** 2).sum()) / total,
                                                                        dtype=torch.float64),
           "rank": torch.full((b,), k, dtype=torch.int32)}
    if case["kind"] == "host":
        return {name: x.cpu() for name, x in out.items()}
    u, v = _reflectors(case, seed)
    sides = []
    for vecs, size in ((u, case["m"]), (v, case["n"])):
        E = torch.eye(size, k, dtype=torch.complex128, device="cuda").expand(b, size, k).contiguous()
        for i in range(4):
            _reflect(E, vecs[i])
        sides.append(E)
    out["left"], out["right"] = _centre_factors(out["sigma"], sides[0], sides[1].mH, torch.complex128)
    return out


# ------------------------------------------------------------------ chains
def _spinors(N, d, seed):
    """Seeded product state: random amplitudes, each site near one of its extreme levels by turns."""
    rng = np.random.default_rng(seed)
    out = []
    for s in range(N):
        v = 0.35 * (rng.standard_normal(d) + 1j * rng.standard_normal(d))
        v[0 if s % 2 == 0 else d - 1] += 1.0
        out.append(v / np.linalg.norm(v))
    return out


def _padded(rows, width):
    out = np.zeros((len(rows), width))
    for i, r in enumerate(rows):
        out[i, :len(r)] = r
    return out


def _quench_terms(case, seed):
    return I.xxz_bond_terms(case["N"], 2, 1.0, 0.3 + 0.4 * np.random.default_rng(seed).random())


class _Quench:
    def __init__(self, case, seed):
        c = self.case = case
        N = c["N"]
        hs = _quench_terms(c, seed)
        self.psi = _spinors(N, 2, seed)
        self.sim = B.Tebd(N, 2, c["chi"], c["p"], c["q"], seed % 1000, use_graph=1)
        self.sim.set_gates(0, I.trotter_gates(hs, c["dt"] / 2))
        self.sim.set_gates(1, I.trotter_gates(hs, c["dt"]))

    def __del__(self):
        self.sim.close()


def _run_quench(st):
    sim, c = st.sim, st.case
    sim.set_product_state(st.psi)
    for _ in range(c["steps"]):
        sim.step_even()
        sim.step_odd()
        sim.step_even()
    sz = I.spin_ops(2)[2]
    lam = _padded([sim.get_lambda(b) for b in range(c["N"] - 1)], c["chi"])
    return {"lambda": lam, "sz": np.array([sim.expect(s, sz).real for s in range(c["N"])]),
            "kept": sim.discarded_weight()[1]}


def _exact_quench(case, seed):
    """Gate by gate on the full state vector; the Schmidt values by dense SVDs (what the cap drops is far below the
    sketch's own accuracy at these times)."""
    N, chi = case["N"], case["chi"]
    hs = _quench_terms(case, seed)
    half, full = I.trotter_gates(hs, case["dt"] / 2), I.trotter_gates(hs, case["dt"])
    psi = torch.ones(1, dtype=torch.complex128, device="cuda")
    for v in _spinors(N, 2, seed):
        psi = torch.kron(psi, torch.from_numpy(v).to("cuda"))
    gates = [torch.from_numpy(half[b] if b % 2 == 0 else full[b]).to("cuda") for b in range(N - 1)]
    for _ in range(case["steps"]):
        for par in (0, 1, 0):
            for b in range(par, N - 1, 2):
                x = psi.reshape(2 ** b, 4, 2 ** (N - b - 2))
                psi = torch.einsum("ij,ajb->aib", gates[b], x).reshape(-1)
    lam = np.zeros((N - 1, chi))
    for b in range(N - 1):
        s = np.linalg.svd(psi.reshape(2 ** (b + 1), -1).cpu().numpy(), compute_uv=False)[:chi]
        lam[b, :len(s)] = s / np.linalg.norm(s)
    sz = []
    for s in range(N):
        p = psi.reshape(2 ** s, 2, -1).abs().square().sum(dim=(0, 2)).cpu().numpy()
        sz.append(0.5 * (p[0] - p[1]) / (p[0] + p[1]))
    return {"lambda": lam, "sz": np.array(sz), "kept": None}


def _specs(case):
    """Uneven chains like those of the many-chain batch, sizes fixed by the case."""
    rng = np.random.default_rng(0)
    out = []
    for _ in range(case["count"]):
        out.append((int(rng.integers(case["nmin"], case["nmax"] + 1)), int(rng.choice([2, 3, 4])),
                    int(rng.choice([32, 64, 128]))))
    return out


class _Chains:
    """Chains brought to their bond caps by a few coarse sweeps, then evolved at the working time step."""

    def __init__(self, case, seed):
        c = self.case = case
        self.specs = _specs(c)
        rng = np.random.default_rng(seed)
        self.sim = B.MultiTebd([(N, [d] * N, [chi] * (N - 1)) for N, d, chi in self.specs], c["p"], c["q"],
                               seed % 1000, use_graph=1, workspace_budget=16 << 30, precision=FORMS[c["form"]])
        deltas = rng.random(len(self.specs))
        for step, (even, odd) in enumerate(((0.3, 0.3), (0.005, 0.01))):
            for i, (N, d, _) in enumerate(self.specs):
                h = I.xxz_bond_terms(2, d, 1.0, deltas[i])[0]
                if step == 0:
                    self.sim.set_product_state(i, _spinors(N, d, seed + 31 * i))
                self.sim.set_gates(i, 0, [I.unitary_from_hermitian(h, even)] * (N - 1))
                self.sim.set_gates(i, 1, [I.unitary_from_hermitian(h, odd)] * (N - 1))
            if step == 0:
                for _ in range(3):
                    self.sim.step_even()
                    self.sim.step_odd()

    def __del__(self):
        self.sim.close()


def _run_chains(st):
    sim = st.sim
    sim.step_even()
    sim.step_odd()
    sim.step_even()
    lam, obs, kept = [], [], []
    for i, (N, d, chi) in enumerate(st.specs):
        lam.append(_padded([sim.get_lambda(i, b) for b in range(N - 1)], chi).ravel())
        sz = I.spin_ops(d)[2]
        obs.append(np.array([sim.expect(i, s, sz).real for s in range(N)]))
        kept.append(sim.discarded_weight(i)[1])
    dtype = np.float64 if st.case["form"] == "fp64" else np.float32
    return {"lambda": np.concatenate(lam).astype(dtype), "sz": np.concatenate(obs).astype(dtype),
            "kept": np.array(kept).astype(dtype)}


class _Boson:
    """Spin-boson chain at its bond caps: seeded Gaussian tensors, Schmidt weights falling by e^-8 over a bond."""

    def __init__(self, case, seed):
        c = self.case = case
        self.dims, caps = I.spin_boson_sizes(c["bosons"], c["d0"], c["d1"], c["chi0"], c["chi1"])
        N = len(self.dims)
        self.sim = B.Tebd(N, 2, 0, c["p"], c["q"], seed % 1000, d_site=self.dims, chi_bond=caps,
                          precision=FORMS[c["form"]], use_graph=1, workspace_budget=40 << 30)
        g = torch.Generator(device="cuda").manual_seed(seed)
        chi = [1] + self.sim.caps + [1]
        gam, lam = [], []
        for s in range(N):
            shape = (self.dims[s], chi[s], chi[s + 1], 2)
            x = torch.view_as_complex(torch.randn(shape, dtype=torch.float64, device="cuda", generator=g))
            gam.append((x / np.sqrt(2.0 * self.dims[s] * chi[s])).cpu().numpy())
        for b in range(N - 1):
            x = np.exp(-np.arange(chi[b + 1]) / max(1.0, chi[b + 1] / 8.0))
            lam.append(x / np.linalg.norm(x))
        self.sim.set_mps(gam, lam)
        hs = I.spin_boson_bond_terms(self.dims)
        self.sim.set_gates(0, _gates(hs, 0.025))
        self.sim.set_gates(1, _gates(hs, 0.05))

    def __del__(self):
        self.sim.close()


def _gates(hs, tau):
    """exp(-i h tau) of real symmetric bond terms of up to 1024 x 1024, on the device."""
    out = []
    for h in hs:
        e, V = torch.linalg.eigh(torch.from_numpy(np.ascontiguousarray(h.real)).to("cuda"))
        V = V.to(torch.complex128)
        out.append(((V * torch.exp(-1j * tau * e)) @ V.mH).cpu().numpy())
    return out


def _run_boson(st):
    sim = st.sim
    sim.step_even()
    sim.step_odd()
    sim.step_even()
    lam = np.concatenate([np.pad(x, (0, sim.caps[b] - len(x)))
                          for b, x in enumerate(sim.get_lambda(b) for b in range(sim.N - 1))])
    occ = np.array([sim.expect(s, I.boson_ops(d)[2]).real for s, d in enumerate(st.dims)])
    return {"lambda": lam.astype(np.float32), "occupation": occ.astype(np.float32),
            "kept": np.array(sim.discarded_weight()[1], dtype=np.float32)}


# ------------------------------------------------------------------ the interface
def prepare(case, seed):
    kind = case["kind"]
    if kind in ("rrsvd", "host", "check"):
        return _prepare_matrices(case, seed)
    if kind == "quench":
        return _Quench(case, seed)
    if kind == "chains":
        return _Chains(case, seed)
    if kind == "boson":
        return _Boson(case, seed)
    return case, torch.from_numpy(np.random.default_rng(seed).uniform(0.5, 1.5, case["N"] - 1))


def run(state):
    if isinstance(state, _Plan):
        return _run_matrices(state)
    if isinstance(state, _Quench):
        return _run_quench(state)
    if isinstance(state, _Chains):
        return _run_chains(state)
    if isinstance(state, _Boson):
        return _run_boson(state)
    c, J = state
    J = J.clone().requires_grad_(True)
    L = tfim_observable(J, c["N"], 1.0, c["dt"], c["steps"], c["chi"], c["p"], c["q"], 0, c["N"] // 2 - 1)
    L.backward()
    return {"value": L.detach(), "grad": J.grad}


def exact(case, seed):
    if case["kind"] in ("rrsvd", "host", "check"):
        return _exact_matrices(case, seed)
    if case["kind"] == "quench":
        return _exact_quench(case, seed)
    return None


def _update_work(m, n, k, l, q, real=8.0):
    """Real operations of one truncation: 2q + 2 products with theta, 2q + 2 QRs with their Q, the factors."""
    prod = real * m * n * l
    qrs = (q + 1) * 2 * real * m * l * l + (q + 1) * 2 * real * n * l * l
    return (2 * q + 2) * prod + qrs + real * (m + n) * l * k


def _chain_work(dims, chis, q, p, sweeps):
    """Bytes and operations of sweeps (per parity) over a chain at its caps."""
    N = len(dims)
    cap = [1]
    left = 1.0
    for b in range(N - 1):
        left = min(left * dims[b], 1e9)
        right = 1.0
        for s in range(b + 1, N):
            right = min(right * dims[s], 1e9)
        cap.append(int(min(chis[b], left, right)))
    cap.append(1)
    by = fl = 0.0
    for b in range(N - 1):
        m, n, x = dims[b] * cap[b], dims[b + 1] * cap[b + 2], cap[b + 1]
        k = min(x, m, n)
        dd = dims[b] * dims[b + 1]
        t = sweeps[b % 2]
        by += t * 2 * 16.0 * (m + n) * x
        fl += t * (8.0 * m * n * x + 8.0 * m * n * dd + _update_work(m, n, k, min(k + p, m, n), q))
    return by, fl


def work(case):
    kind = case["kind"]
    if kind in ("rrsvd", "host", "check"):
        m, n, b = case["m"], case["n"], case["batch"]
        k = min(case["k"], m, n)
        if kind == "check":  # the basis at least once, the rounds' growth at the accuracy asked for
            l = min(case["lmax"], m, n)
            return {"bytes": 16.0 * b * (m * n + (m + n) * (l - case["p"])),
                    "flops": b * _update_work(m, n, l - case["p"], l, case["q"])}
        l = min(k + case["p"], m, n)
        out = 0 if kind == "host" else (m + n) * k
        return {"bytes": 16.0 * b * (m * n + out) + 8.0 * b * k, "flops": b * _update_work(m, n, k, l, case["q"])}
    if kind == "quench":
        by, fl = _chain_work([2] * case["N"], [case["chi"]] * (case["N"] - 1), case["q"], case["p"],
                             (2 * case["steps"], case["steps"]))
        return {"bytes": by, "flops": fl}
    if kind == "chains":
        each = [_chain_work([d] * N, [chi] * (N - 1), case["q"], case["p"], (2, 1)) for N, d, chi in _specs(case)]
        return {"bytes": sum(x[0] for x in each), "flops": sum(x[1] for x in each)}
    if kind == "boson":
        dims, caps = I.spin_boson_sizes(case["bosons"], case["d0"], case["d1"], case["chi0"], case["chi1"])
        by, fl = _chain_work(dims, caps, case["q"], case["p"], (2, 1))
        return {"bytes": by, "flops": fl}
    by, fl = _chain_work([2] * case["N"], [case["chi"]] * (case["N"] - 1), case["q"], case["p"],
                         (2 * case["steps"], case["steps"]))
    return {"bytes": 3 * by, "flops": 3 * fl}
