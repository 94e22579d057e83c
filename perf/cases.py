"""Performance cases of the QR-CTMRG framework: what its users have it do, through its public entry points.

Kinds
  step     ctm_step on one real instance, then the environment read back (C, T, Q): the framework's inner loop
  zstep    ctm_complex_step on one complex (E-irrep) instance, then the environment
  batch    ctm_batch_step on a ragged parameter sweep, then every instance's corner and edge
  solve    a new site tensor swapped in, ctm_converge from a fresh environment, ctm_energy (an evaluation at fixed A)
  grad     a new site tensor swapped in, ctm_grad (energy and adjoint gradient, one evaluation of the optimiser)
  gemm     ctm_gemm, the contraction engine on its own

Site tensors are the repository's seeded stand-ins (inputs.py): uniform random tensors for everything that is
compared along a trajectory, the near-product states that converge for `solve`.
"""
import math

import numpy as np
import torch

from paper_2509_05090_gb300 import binding, inputs

PHI = 0.3 * math.pi
PRODUCT = np.array([0.8, 0.6])


def listed():
    return [
        # oracle-sized Heisenberg instance in the default precision: a step-by-step loop that reads delta,
        # where launches and latency count
        dict(name="step_d2_chi8_fp64", kind="step", d=2, D=2, chi=8, precision="fp64", nsteps=1),
        # a mid-sized Kitaev instance between convergence checks
        dict(name="step_d4_chi32_split", kind="step", d=2, D=4, chi=32, precision="split_bf16", nsteps=4),
        # the benchmark's flagship size, in the mixed precision and in the default one
        dict(name="step_d6_chi72_split", kind="step", d=2, D=6, chi=72, precision="split_bf16", nsteps=4),
        dict(name="step_d6_chi72_fp64", kind="step", d=2, D=6, chi=72, precision="fp64", nsteps=2),
        # the large-bond-dimension instance that final evaluations run in the default precision
        dict(name="step_d8_chi128_fp64", kind="step", d=2, D=8, chi=128, precision="fp64", nsteps=1),
        # the top of the runtime-versus-chi sweep
        dict(name="step_d5_chi480_split", kind="step", d=2, D=5, chi=480, precision="split_bf16", nsteps=1),
        # complex tensors of the Kitaev model's representation
        dict(name="zstep_d6_chi72_split", kind="zstep", d=2, D=6, chi=72, precision="split_bf16", nsteps=1),
        dict(name="zstep_d4_chi32_fp64", kind="zstep", d=2, D=4, chi=32, precision="fp64", nsteps=2),
        # a sweep over the Kitaev-Heisenberg angle, instances of mixed sizes
        dict(name="batch24_split", kind="batch", count=24, Dmin=3, Dmax=6, chimin=24, chimax=72,
             precision="split_bf16", nsteps=2),
        # energy of one state: environment converged from scratch, then the bonds
        dict(name="solve_d6_chi72_split", kind="solve", D=6, chi=72, eps=0.002, precision="split_bf16"),
        # one evaluation of the variational loop at its usual size (chi = 3 D^2)
        dict(name="grad_d3_chi27_fp64", kind="grad", D=3, chi=27, precision="fp64", warmup=4, k=6),
        # a ragged product through the engine alone
        dict(name="gemm_2592x1300x1000_split", kind="gemm", M=2592, N=1300, K=1000, precision="split_bf16", n_split=4),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("step", "step", "step", "zstep", "batch", "solve", "grad", "gemm"))
    prec = rng.choice(("fp64", "split_bf16"))
    if kind == "step":
        D = rng.randint(2, 8)
        # n = chi D^2 up to 8192 in FP64 and 12000 in the mixed precision, chi up to 480
        top = min(480, (8192 if prec == "fp64" else 12000) // (D * D))
        return dict(kind=kind, d=rng.choice((2, 2, 3)) if D <= 5 else 2, D=D,
                    chi=min(_log(rng, 2 * D, top), 128 if prec == "fp64" else top), precision=prec,
                    nsteps=rng.randint(1, 4))
    if kind == "zstep":
        D = rng.randint(2, 6)
        return dict(kind=kind, d=2, D=D, chi=_log(rng, 2 * D, 72), precision=prec, nsteps=rng.randint(1, 3))
    if kind == "batch":
        Dmin, chimin = rng.randint(2, 4), rng.randint(12, 32)
        return dict(kind=kind, count=rng.randint(4, 24), Dmin=Dmin, Dmax=rng.randint(Dmin, 6 if prec != "fp64" else 5),
                    chimin=chimin, chimax=rng.randint(chimin, 72 if prec != "fp64" else 48), precision=prec,
                    nsteps=rng.randint(1, 3))
    if kind == "solve":
        return dict(kind=kind, D=rng.randint(3, 6), chi=_log(rng, 16, 72), eps=rng.choice((0.002, 0.005)),
                    precision=prec)
    if kind == "grad":
        D = rng.randint(2, 4)
        return dict(kind=kind, D=D, chi=rng.randint(2 * D, 3 * D * D), precision="fp64", warmup=rng.randint(2, 5),
                    k=rng.randint(2, 6))
    M, N, K = (_log(rng, 32, 3000) for _ in range(3))
    return dict(kind=kind, M=M, N=N, K=K, precision=prec, n_split=rng.randint(3, 5))


# ---------------------------------------------------------------- inputs
def _seed(seed, i=0):
    return (int(seed) * 7919 + 104729 * i + 17) % (1 << 31)


def _batch_instances(case, seed):
    """(A, chi) of every instance: sizes by the case alone (a sweep has them fixed), tensors by the seed."""
    rng = np.random.default_rng(case["count"] * 1000 + case["chimax"])
    Ds = rng.integers(case["Dmin"], case["Dmax"] + 1, size=case["count"])
    chis = rng.integers(case["chimin"], case["chimax"] + 1, size=case["count"])
    chis = np.where(np.arange(case["count"]) % 4 == 3, chis, np.maximum(case["chimin"], chis // 8 * 8))
    return [(inputs.random_site_tensor(2, int(D), _seed(seed, i)), int(chi))
            for i, (D, chi) in enumerate(zip(Ds, chis))]


def _site(case, seed):
    if case["kind"] == "zstep":
        return inputs.random_complex_site_tensor(case["d"], case["D"], _seed(seed))
    if case["kind"] == "solve":
        return inputs.perturbed_product_site_tensor(PRODUCT, case["D"], case["eps"], _seed(seed))
    return inputs.random_site_tensor(case.get("d", 2), case["D"], _seed(seed))


def _hamiltonians(case):
    if case["kind"] == "grad":
        return inputs.bond_hamiltonians(0.0, 1.0, rotate_b=True)
    return inputs.bond_hamiltonians(math.cos(PHI), math.sin(PHI))


def _gemm_inputs(case, seed):
    g = torch.Generator(device="cuda").manual_seed(_seed(seed))
    M, N, K = case["M"], case["N"], case["K"]
    return (torch.randn((M, K), generator=g, dtype=torch.float64, device="cuda"),
            torch.randn((K, N), generator=g, dtype=torch.float64, device="cuda"))


def prepare(case, seed):
    kind, s = case["kind"], {"case": case}
    if kind == "gemm":
        s["A"], s["B"] = _gemm_inputs(case, seed)
    elif kind == "batch":
        inst = _batch_instances(case, seed)
        s["ctm"] = binding.CTMBatch([A for A, _ in inst], [chi for _, chi in inst], precision=case["precision"],
                                    n_split=5)
    elif kind == "zstep":
        s["ctm"] = binding.CTMComplex(_site(case, seed), case["chi"], irrep="E", precision=case["precision"], n_split=5)
    else:
        s["A"] = torch.from_numpy(_site(case, seed)).cuda()
        s["ctm"] = binding.CTM(s["A"], case["chi"], precision=case["precision"], n_split=5)
        if kind in ("solve", "grad"):
            s["h"] = torch.from_numpy(_hamiltonians(case)).cuda()
    return s


def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind == "gemm":
        return {"C": binding.ctm_gemm(state["A"], state["B"], precision=case["precision"], n_split=case["n_split"])}
    ctm = state["ctm"]
    if kind == "step":
        delta = ctm.ctm_step(case["nsteps"])
        C, T, Q = ctm.ctm_get_env()
        return {"delta": delta, "C": C, "T": T, "Q": Q}
    if kind == "zstep":
        delta = ctm.ctm_complex_step(case["nsteps"])
        C, T, Q = ctm.ctm_complex_get_env()
        return {"delta": delta, "C": C, "T": T, "Q": Q}
    if kind == "batch":
        ctm.ctm_batch_step(case["nsteps"])
        env = [ctm.instance(i).ctm_get_env() for i in range(case["count"])]
        return {"C": [e[0] for e in env], "T": [e[1] for e in env]}
    ctm.ctm_set_site(state["A"], reset_env=True)
    if kind == "solve":
        ctm.ctm_converge(max_steps=40, tol=1e-10)
        e, E, rho = ctm.ctm_energy(state["h"])
        return {"e": e, "E": E, "rho": rho, "s": ctm.ctm_get_intermediate("s")}
    E, dA = ctm.ctm_grad(state["h"], warmup=case["warmup"], k_tracked=case["k"])
    return {"E": E, "dA": dA}


# ---------------------------------------------------------------- work
def _step_flops(D, chi):
    """One step's contractions (M Q counted once) and its QR with Q formed: 2 x multiply-adds."""
    D2, n = D * D, chi * D * D
    gemm = 2.0 * (n * chi * chi + 2.0 * n * n * chi + 4.0 * chi * chi * D2 ** 3 + 2.0 * n * n * chi + n * chi * chi
                  + n * n * chi)
    return gemm + 4.0 * n * chi * chi


def _env_bytes(D, chi):
    """C, T, Q and the double layer read, C, T, Q written."""
    D2, n = D * D, chi * D * D
    return 8.0 * (2 * (chi * chi + 2 * n * chi) + D2 ** 3)


def work(case):
    kind = case["kind"]
    if kind == "gemm":
        M, N, K = case["M"], case["N"], case["K"]
        return {"bytes": 8.0 * (M * K + K * N + M * N), "flops": 2.0 * M * N * K}
    if kind == "batch":
        inst = _batch_instances(case, 0)
        sizes = [(A.shape[1], chi) for A, chi in inst]
        return {"bytes": sum(_env_bytes(D, chi) for D, chi in sizes),
                "flops": case["nsteps"] * sum(_step_flops(D, chi) for D, chi in sizes)}
    D, chi = case["D"], case["chi"]
    if kind == "zstep":
        return {"bytes": 2.0 * _env_bytes(D, chi), "flops": 4.0 * case["nsteps"] * _step_flops(D, chi)}
    if kind == "step":
        return {"bytes": _env_bytes(D, chi), "flops": case["nsteps"] * _step_flops(D, chi)}
    if kind == "solve":
        # about five steps and the energy's extra step, its two open-layer contractions among it
        return {"bytes": _env_bytes(D, chi), "flops": 6.0 * _step_flops(D, chi) + 16.0 * chi * chi * D ** 6}
    # the tracked steps forward and twice that backward
    return {"bytes": _env_bytes(D, chi), "flops": (case["warmup"] + 3.0 * (case["k"] + 1)) * _step_flops(D, chi)}


# ---------------------------------------------------------------- plain torch in 64 bits
def _dev():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _project(A):
    P = sum(A.permute(0, *p) for p in ((1, 2, 3), (1, 3, 2), (2, 1, 3), (2, 3, 1), (3, 1, 2), (3, 2, 1))) / 6.0
    return P / torch.linalg.norm(P)


def _z_project(A):
    """The average over the six elements generated by the three-fold spin rotation about (1,1,1) with the leg
    cycle and the anti-unitary reflection with the exchange of the first two legs (spin 1/2)."""
    Sx = torch.tensor([[0, 0.5], [0.5, 0]], dtype=torch.complex128)
    Sy = torch.tensor([[0, -0.5j], [0.5j, 0]], dtype=torch.complex128)
    Sz = torch.tensor([[0.5, 0], [0, -0.5]], dtype=torch.complex128)
    U = -torch.linalg.matrix_exp(2j * math.pi / 3.0 * (Sx + Sy + Sz) / math.sqrt(3.0)) * np.exp(2j * math.pi / 3.0)
    Kh = torch.tensor([[0, 1], [-1, 0]], dtype=torch.complex128)
    P = Kh @ torch.linalg.matrix_exp(1j * math.pi * (Sx - Sy) / math.sqrt(2.0)).conj()
    U, P = U.to(A.device), P.to(A.device)
    rot = lambda X: torch.einsum("st,tijk->sijk", U, X.permute(0, 2, 3, 1))  # noqa: E731
    ref = lambda X: torch.einsum("st,tijk->sijk", P, X.conj().permute(0, 2, 1, 3))  # noqa: E731
    R1, R2 = rot(A), rot(rot(A))
    S = (A + R1 + R2 + ref(A) + ref(R1) + ref(R2)) / 6.0
    return S / torch.linalg.norm(S)


def _layer(K, B):
    D = K.shape[1]
    return torch.einsum("sijk,slmn->iljmkn", K, B.conj()).reshape(D * D, D * D, D * D)


class _Env:
    """The step, written out in plain torch: sector wiring, warm start and gauge as the library documents them."""

    def __init__(self, A, chi):
        self.A, self.chi = A, chi
        self.aB = _layer(A, A)
        Az = A.permute(0, 3, 1, 2) if A.is_complex() else A   # the apex site's z leg first
        self.aA = _layer(Az, Az)
        D = A.shape[1]
        self.D2 = D * D
        dg = torch.arange(D, device=A.device) * (D + 1)
        t = self.aB[:, dg][:, :, dg].sum(dim=(1, 2))
        eye = torch.eye(chi, dtype=A.dtype, device=A.device)
        self.C, self.T = eye, eye[:, None, :] * t[None, :, None]
        self.Q = torch.eye(chi * self.D2, chi, dtype=A.dtype, device=A.device)
        self.s = torch.full((chi,), 1.0 / math.sqrt(chi), dtype=torch.float64, device=A.device)

    def _x(self):
        chi, D2 = self.chi, self.D2
        W = (self.T.reshape(-1, chi) @ self.C)
        X = W @ self.T.conj().reshape(-1, chi).T                                # (a u), (b l)
        return X.reshape(chi, D2, chi, D2).permute(0, 2, 1, 3).reshape(chi * chi, D2 * D2)

    def _corner(self):
        chi, D2 = self.chi, self.D2
        Y1 = self._x() @ self.aB.reshape(D2 * D2, D2)                            # (a b), z
        M = Y1 @ self.aA.reshape(D2, D2 * D2)                                    # (a b), (x y)
        return M.reshape(chi, chi, D2, D2).permute(0, 3, 1, 2).reshape(chi * D2, chi * D2)

    def _projector(self, M):
        S = torch.where(torch.diagonal(self.C).real < 0, -1.0, 1.0).to(M.dtype)
        Q, R = torch.linalg.qr(M @ (self.Q * S[None, :]), mode="reduced")
        r = torch.diagonal(R)
        ph = torch.where(r.abs() > 0, r / r.abs().clamp_min(1e-300), torch.ones_like(r))
        return Q * ph[None, :]

    def _new_corner(self, M, Q):
        Cr = Q.mH @ (M @ Q)
        Cn = 0.5 * (Cr + Cr.mH)
        return Cn / torch.linalg.norm(Cn)

    def step(self, spectrum=True):
        chi, D2 = self.chi, self.D2
        M = self._corner()
        Q = self._projector(M)
        Cn = self._new_corner(M, Q)
        del M
        Q3 = Q.reshape(chi, D2, chi)
        H = self.T.reshape(chi * D2, chi) @ Q3.reshape(chi, D2 * chi)            # (a u), (w j)
        H = H.reshape(chi, D2, D2, chi).permute(0, 3, 1, 2).reshape(chi * chi, D2 * D2)
        H = (H @ self.aB.reshape(D2 * D2, D2)) @ self.aA.reshape(D2, D2 * D2)    # (a j), (x y)
        H = H.reshape(chi, chi, D2, D2).permute(0, 3, 2, 1).reshape(chi * D2, D2 * chi)   # (a y), (x j)
        Tn = (Q.mH @ H).reshape(chi, D2, chi)
        self.C, self.T, self.Q = Cn, Tn / torch.linalg.norm(Tn), Q
        if not spectrum:
            return None
        s = torch.linalg.eigvalsh(Cn.detach()).abs().sort(descending=True)[0]
        s = s / torch.linalg.norm(s)
        delta, self.s = float(torch.linalg.norm(s - self.s)), s
        return delta

    def energy(self, h):
        chi, D2, A, d = self.chi, self.D2, self.A, self.A.shape[0]
        M = self._corner()
        Q = self._projector(M)
        Ch = self._new_corner(M, Q)
        E = (Q @ torch.linalg.matrix_power(Ch, 5)) @ Q.T
        E = E.reshape(chi, D2, chi, D2).permute(0, 2, 1, 3).reshape(chi * chi, D2 * D2)   # (a b), (y x)
        X = self._x()
        Yb, Gb = [], []
        for s in range(d):
            for t in range(d):
                b = _layer(A[s:s + 1], A[t:t + 1])
                Yb.append(X @ b.reshape(D2 * D2, D2))
                Gb.append(E @ b.permute(2, 1, 0).reshape(D2 * D2, D2))                  # rows (y, x), columns z
        raw = torch.stack([torch.stack([(y * g).sum() for g in Gb]) for y in Yb])       # [pB][pA]
        r4 = raw.reshape(d, d, d, d)                                                     # sB tB sA tA
        rho = r4.permute(2, 0, 3, 1).reshape(d * d, d * d)
        rho = rho / torch.diagonal(rho).sum()
        e = torch.stack([(rho * h[k].T).sum() for k in range(3)])
        return e, 0.5 * e.sum(), rho


def _exact_env(A, chi, nsteps):
    env, delta = _Env(A, chi), None
    for _ in range(nsteps):
        delta = env.step()
    return env, delta


def exact(case, seed):
    kind = case["kind"]
    if kind == "gemm":
        A, B = _gemm_inputs(case, seed)
        return {"C": A @ B}
    if kind == "batch":
        envs = [_exact_env(_project(torch.from_numpy(A).to(_dev())), chi, case["nsteps"])[0]
                for A, chi in _batch_instances(case, seed)]
        return {"C": [e.C for e in envs], "T": [e.T for e in envs]}
    A = torch.from_numpy(_site(case, seed)).to(_dev())
    if kind in ("step", "zstep"):
        env, delta = _exact_env(_project(A) if kind == "step" else _z_project(A), case["chi"], case["nsteps"])
        return {"delta": delta, "C": env.C, "T": env.T, "Q": env.Q}
    h = torch.from_numpy(_hamiltonians(case)).to(_dev())
    if kind == "solve":
        env = _Env(_project(A), case["chi"])
        for _ in range(40):
            if env.step() < 1e-10:
                break
        e, E, rho = env.energy(h)
        return {"e": e.cpu().numpy(), "E": float(E), "rho": rho.cpu().numpy(), "s": env.s}
    A.requires_grad_(True)
    env = _Env(_project(A), case["chi"])
    with torch.no_grad():
        for _ in range(case["warmup"]):
            env.step(False)
    # the environment entering the tracked steps is a constant
    env.C, env.T, env.Q = (x.detach() for x in (env.C, env.T, env.Q))
    for _ in range(case["k"]):
        env.step(False)
    E = env.energy(h)[1]
    (g,) = torch.autograd.grad(E, A)
    return {"E": float(E.detach()), "dA": g}
