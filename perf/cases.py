"""What a user of this framework has it do, as cases that can be timed and compared.

Four kinds of work, each through the public Python entry points:

  flips    one call of ``afqmc_apply_flips`` (or its no-allocation form) on a caller's G;
  hubbard  one full sweep of Hubbard walkers: slices 1..M forward, M..1 backward, the FP64
           recompute at every multiple of the recompute period, then the energy;
  soc      the same for the spin-coupled engine (spin-y or spin-z decoupling), with the pairing
           observables at the middle slice where a production run takes them;
  cpqmc    projection steps of a constrained-path ensemble, then population control,
           re-orthonormalisation and the mixed energy.

A sweep is short (M of 5 to 40 slices instead of 80 to 920) so that a pass stays under a second;
lattice, precision, update scheme, walkers and recompute period are those of real runs.  Results of
an FP32 bulk G leave the library as doubles; ``run`` hands them on in FP32, the precision they have.

``exact`` computes the same passes in plain FP64 torch: the same Markov chain (numpy's Philox
uniforms, one rank-1 or rank-2 update per site, dense propagation), so the fields can be compared too.
"""
import ctypes
import functools
import math

import numpy as np
import torch

from paper_2506_09611_gb300 import afqmc, soc

T_HOP, DTAU = 1.0, 0.05


# ---------------------------------------------------------------- the cases

def listed():
    return [
        # A single-site move on a small FP64 G held by a host program: the smallest call, all latency.
        {"name": "flips-8x8-fp64-m4", "kind": "flips", "precision": "fp64", "N": 64, "pad": 0, "m": 4, "alloc": True},
        # A 64-site collective move on an odd lattice without padding (41 x 41, odd leading dimension),
        # FP32, under a fixed memory budget (no allocation).
        {"name": "flips-41x41-fp32-m64", "kind": "flips", "precision": "fp32", "N": 1681, "pad": 0, "m": 64,
         "alloc": False},
        # The 4 x 4 parity workload as an ensemble of independent chains in FP64: launch latency.
        {"name": "hubbard-4x4-fp64-k16-32w", "kind": "hubbard", "sizes": "4", "walkers": 32, "precision": "fp64",
         "U": 4.0, "filling": 0.875, "M": 40, "stab": 10, "mode": "delayed", "k": 16, "nb": 1, "graphs": False},
        # The 16 x 16 workload, one FP32 walker, delayed update.
        {"name": "hubbard-16x16-fp32-k32", "kind": "hubbard", "sizes": "16", "walkers": 1, "precision": "fp32",
         "U": 4.0, "filling": 0.875, "M": 20, "stab": 10, "mode": "delayed", "k": 32, "nb": 1, "graphs": False},
        # An odd lattice (N = 441) in FP64 throughout, attractive model in the charge channel, two chains.
        {"name": "hubbard-21x21-fp64-k32-2w", "kind": "hubbard", "sizes": "21", "walkers": 2, "precision": "fp64",
         "U": -4.0, "filling": 0.625, "M": 10, "stab": 5, "mode": "delayed", "k": 32, "nb": 1, "graphs": False},
        # The headline: 40 x 40, U = 6, FP32 bulk, delayed k = 64, recompute every 5 slices, graph replay.
        {"name": "hubbard-40x40-fp32-k64", "kind": "hubbard", "sizes": "40", "walkers": 1, "precision": "fp32",
         "U": 6.0, "filling": 0.875, "M": 10, "stab": 5, "mode": "delayed", "k": 64, "nb": 1, "graphs": True},
        # The same walker with the block force-bias update, and with the conventional local update.
        {"name": "hubbard-40x40-fp32-fb16", "kind": "hubbard", "sizes": "40", "walkers": 1, "precision": "fp32",
         "U": 6.0, "filling": 0.875, "M": 5, "stab": 5, "mode": "blockfb", "k": 1, "nb": 16, "graphs": False},
        {"name": "hubbard-40x40-fp32-local", "kind": "hubbard", "sizes": "40", "walkers": 1, "precision": "fp32",
         "U": 6.0, "filling": 0.875, "M": 2, "stab": 2, "mode": "local", "k": 1, "nb": 1, "graphs": False},
        # The mixed-size walker population of a production node: groups on concurrent streams, graph replay.
        {"name": "population-8to24-fp32-k64-64w", "kind": "hubbard", "sizes": "8,12,16,24", "walkers": 64,
         "precision": "fp32", "U": 4.0, "filling": 0.875, "M": 3, "stab": 3, "mode": "delayed", "k": 64, "nb": 1,
         "graphs": True},
        # The spin-orbit workload: 24 x 24 Rashba-Hubbard, complex64 G of 1152 orbitals, block force bias.
        {"name": "soc-24x24-fp32-fb16", "kind": "soc", "L": 24, "walkers": 1, "precision": "fp32", "hs": "sy",
         "lam": 0.5, "U": -4.0, "filling": 1.0, "M": 5, "stab": 5, "mode": "blockfb", "k": 1, "nb": 16,
         "pairing": False},
        # The pairing runs of the attractive model: 20 x 20, spin-z channel, several chains, observables.
        {"name": "pairing-20x20-fp32-k32-8w", "kind": "soc", "L": 20, "walkers": 8, "precision": "fp32", "hs": "sz",
         "lam": 0.0, "U": -4.0, "filling": 1.0, "M": 10, "stab": 5, "mode": "delayed", "k": 32, "nb": 1,
         "pairing": True},
        # Constrained-path AFQMC, 16 x 16, 32 walkers, five steps between population controls.
        {"name": "cpqmc-16x16-k32-32w", "kind": "cpqmc", "L": 16, "walkers": 32, "U": 4.0, "filling": 0.875,
         "steps": 5, "mode": "delayed", "k": 32, "nb": 1},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["flips", "hubbard", "hubbard", "hubbard", "hubbard", "soc", "cpqmc"])
    if kind == "flips":
        prec = rng.choice(["fp32", "fp64"])
        N = _log_int(rng, 32, 2304 if prec == "fp32" else 1600)
        m = _log_int(rng, 1, min(N // 2, 128 if prec == "fp32" else 64))
        return {"kind": "flips", "precision": prec, "N": N, "pad": rng.choice([0, 0, 1, 4, 13]), "m": m,
                "alloc": rng.random() < 0.5}
    if kind == "hubbard":
        prec = rng.choice(["fp32", "fp32", "fp64"])
        charge = rng.random() < 0.25
        U = (-1.0 if charge else 1.0) * round(rng.uniform(1.0, 6.0), 2)
        L = _log_int(rng, 4, 40 if prec == "fp32" else 22)
        mode = rng.choice(["delayed", "delayed", "blockfb", "local"])
        if mode == "local":
            walkers = rng.choice([1, 2])
        else:
            walkers = max(1, min(32, _log_int(rng, 1, 1600 // (L * L) + 1)))
        stab = rng.choice([2, 4, 5]) if L <= 16 else 2
        periods = 1 if L > 12 else rng.choice([1, 2])
        return {"kind": "hubbard", "sizes": str(L), "walkers": walkers, "precision": prec, "U": U,
                "filling": round(rng.uniform(0.5, 1.0), 3), "M": stab * periods, "stab": stab, "mode": mode,
                "k": rng.randint(8, min(L * L, 128 if prec == "fp32" else 64)), "nb": rng.randint(2, min(L * L, 32)),
                "graphs": rng.random() < 0.3}
    if kind == "soc":
        prec = rng.choice(["fp32", "fp32", "fp64"])
        hs = rng.choice(["sy", "sz"])
        L = _log_int(rng, 4, 24 if prec == "fp32" else 10)
        return {"kind": "soc", "L": L, "walkers": rng.choice([1, 2, 4]) if L <= 12 else 1, "precision": prec,
                "hs": hs, "lam": round(rng.uniform(0.1, 0.7), 2) if hs == "sy" else 0.0,
                "U": -round(rng.uniform(1.0, 4.0), 2), "filling": round(rng.uniform(0.5, 1.0), 3), "M": 4, "stab": 2,
                "mode": rng.choice(["delayed", "blockfb"]), "k": rng.randint(4, min(L * L, 32)),
                "nb": rng.randint(2, min(L * L, 20)), "pairing": hs == "sz" and rng.random() < 0.5}
    L = rng.randint(4, 15)
    return {"kind": "cpqmc", "L": L, "walkers": rng.randint(4, 24), "U": round(rng.uniform(1.0, 6.0), 2),
            "filling": round(rng.uniform(0.5, 0.9), 3), "steps": rng.randint(1, 3),
            "mode": rng.choice(["delayed", "delayed", "blockfb"]), "k": rng.randint(8, min(L * L, 48)),
            "nb": rng.randint(2, min(L * L, 16))}


# ---------------------------------------------------------------- inputs

def _n_sigma(L, filling):
    return max(1, min(L * L - 1, int(round(filling * L * L / 2))))


def _ring(L):
    """Periodic nearest-neighbour hopping of a chain (both bonds coincide at L = 2)."""
    K = np.zeros((L, L))
    for x in range(L):
        K[x, (x + 1) % L] -= T_HOP
        K[x, (x - 1) % L] -= T_HOP
    return K


def _hopping(L):
    I1 = np.eye(L)
    return np.kron(I1, _ring(L)) + np.kron(_ring(L), I1)


def _soc_h0(L, lam):
    """Rashba-coupled hopping on the 2N orbitals: (dn, r) <- (up, r') amplitude -i lam for r' = r + y,
    +i lam for r' = r - y, -lam for r' = r + x, +lam for r' = r - x."""
    N = L * L
    s = np.zeros((L, L))
    for x in range(L):
        s[x, (x + 1) % L] = 1.0
    sx, sy = np.kron(np.eye(L), s), np.kron(s, np.eye(L))
    V = -1j * lam * (sy - sy.T) - lam * (sx - sx.T)
    H = np.zeros((2 * N, 2 * N), np.complex128)
    H[:N, :N] = H[N:, N:] = _hopping(L)
    H[N:, :N] = V
    H[:N, N:] = V.conj().T
    return H


@functools.lru_cache(maxsize=None)
def _trial(L, ns):
    """The lowest ns hopping orbitals, the open shell split by a fixed small symmetric perturbation."""
    S = np.random.default_rng(12345).standard_normal((L * L, L * L))
    return np.ascontiguousarray(np.linalg.eigh(_hopping(L) + 5e-7 * (S + S.T))[1][:, :ns])


@functools.lru_cache(maxsize=None)
def _soc_trial(L, n_e, lam, hs):
    """spin-y: the lowest n_e orbitals of H0 with a time-reversal-invariant perturbation; spin-z: the
    same real orbitals in both spin blocks (the condition under which the walk is sign-free)."""
    N = L * L
    if hs == "sz":
        P = np.zeros((2 * N, n_e), np.complex128)
        P[:N, :n_e // 2] = P[N:, n_e // 2:] = _trial(L, n_e // 2)
        return P
    rng = np.random.default_rng(54321)
    A = rng.standard_normal((N, N)) + 1j * rng.standard_normal((N, N))
    B = rng.standard_normal((N, N)) + 1j * rng.standard_normal((N, N))
    A, B = 0.5 * (A + A.conj().T), 0.5 * (B - B.T)
    S = np.block([[A, B], [-B.conj(), A.conj()]])
    return np.ascontiguousarray(np.linalg.eigh(_soc_h0(L, lam) + 1e-6 * S)[1][:, :n_e])


def _lattices(case):
    sizes = [int(s) for s in case["sizes"].split(",")]
    if len(sizes) == 1:
        return sizes * case["walkers"]
    return [sizes[i] for i in np.random.default_rng(5).integers(0, len(sizes), case["walkers"])]


def _fields(seed, walker, M, N):
    return np.where(np.random.default_rng([seed, walker]).random((M, N)) < 0.5, 1, -1).astype(np.int8)


def _hs(U):
    """(kind, coupling lam, (c_up, c_dn)) of the real decouplings."""
    lam = math.acosh(math.exp(DTAU * abs(U) / 2.0))
    return (afqmc.HS_SZ_REAL, lam, (lam, -lam)) if U >= 0 else (afqmc.HS_CHARGE_REAL, lam, (lam, lam))


def _flips_inputs(case, seed):
    """G = 1 - Q Q^T of a random half-filled state for both spins, padded rows, and the flipped sites."""
    N, m = case["N"], case["m"]
    dt = torch.float64 if case["precision"] == "fp64" else torch.float32
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    g = torch.Generator(device="cpu").manual_seed(seed)
    G = torch.zeros(2, N, N + case["pad"], dtype=dt, device=dev)
    for s in range(2):
        Q = torch.linalg.qr(torch.randn(N, (N + 1) // 2, generator=g, dtype=torch.float32).to(dev).double())[0]
        G[s, :, :N] = (torch.eye(N, dtype=torch.float64, device=dev) - Q @ Q.T).to(dt)
    rng = np.random.default_rng(seed)
    sites = rng.permutation(N)[:m].astype(np.int32)
    x = np.where(rng.random(m) < 0.5, 1.0, -1.0)
    c = _hs(4.0)[2]
    delta = np.concatenate([np.exp(-2.0 * c[0] * x) - 1.0, np.exp(-2.0 * c[1] * x) - 1.0])
    return G, torch.from_numpy(sites).to(dev), torch.from_numpy(delta).to(dev)


def prepare(case, seed):
    kind = case["kind"]
    st = torch.cuda.current_stream()
    if kind == "flips":
        G, sites, delta = _flips_inputs(case, seed)
        return {"case": case, "G0": G, "G": torch.empty_like(G), "sites": sites, "delta": delta}
    if kind == "hubbard":
        Ls = _lattices(case)
        ns = [_n_sigma(L, case["filling"]) for L in Ls]
        P = np.concatenate([np.tile(_trial(L, n).ravel(), 2) for L, n in zip(Ls, ns)])
        X = np.concatenate([_fields(seed, w, case["M"], L * L).ravel() for w, L in enumerate(Ls)])
        ctx = afqmc.Context(case["M"], dtau=DTAU, U=case["U"], t=T_HOP, precision=case["precision"],
                            hs=_hs(case["U"])[0], stab_every=case["stab"], seed=seed)
        ctx.init_walkers(Ls, ns, ns, P, X, stream=st)
        ctx.set_graphs(case["graphs"])
        return {"case": case, "ctx": ctx}
    if kind == "soc":
        L, M = case["L"], case["M"]
        n_e = 2 * _n_sigma(L, case["filling"])
        X = np.concatenate([_fields(seed, w, M, L * L).ravel() for w in range(case["walkers"])])
        ctx = soc.SocContext(L, M, n_e, case["walkers"], case["precision"], "tc3", case["stab"], T_HOP, case["lam"],
                             case["U"], DTAU, seed, hs=case["hs"])
        ctx.init(_soc_trial(L, n_e, case["lam"], case["hs"]), X, stream=st)
        return {"case": case, "ctx": ctx}
    ns = _n_sigma(case["L"], case["filling"])
    P, phi0, u0 = _cp_inputs(case, seed)
    cp = afqmc.CPContext(case["L"], ns, case["walkers"], P, phi0=phi0, dtau=DTAU, U=case["U"], t=T_HOP,
                         hs=_hs(case["U"])[0], seed=seed, stream=st)
    return {"case": case, "ctx": cp, "u0": u0}


def _cp_inputs(case, seed):
    """Trial determinant, walkers started near it, the comb's offset."""
    L = case["L"]
    P = _trial(L, _n_sigma(L, case["filling"]))
    rng = np.random.default_rng(seed)
    phi0 = P + 0.01 * rng.standard_normal((case["walkers"], 2) + P.shape) / L
    return P, phi0, float(rng.random())


# ---------------------------------------------------------------- one pass

def _order(M):
    return [(l, +1) for l in range(1, M + 1)] + [(l, -1) for l in range(M, 0, -1)]


def run(state):
    case = state["case"]
    return {"flips": _run_flips, "hubbard": _run_hubbard, "soc": _run_soc, "cpqmc": _run_cpqmc}[case["kind"]](
        case, state, torch.cuda.current_stream())


def _run_flips(case, s, st):
    """A trial move on a copy: the caller's G is kept until the move is taken."""
    G = s["G"]
    G.copy_(s["G0"])
    fn = afqmc.afqmc_apply_flips if case["alloc"] else afqmc.afqmc_apply_flips_noalloc
    fn(case["precision"], case["N"], G.stride(1), G[0].data_ptr(), G[1].data_ptr(), s["sites"].data_ptr(),
       s["delta"].data_ptr(), case["m"], stream=st)
    return G


def _run_hubbard(case, s, st):
    ctx = s["ctx"]
    for ell, d in _order(case["M"]):
        ctx.sweep_slice(ell, d, case["mode"], k=case["k"], nb=case["nb"], stream=st)
        if (ell if d > 0 else ell - 1) % case["stab"] == 0:
            afqmc.afqmc_recompute_G(ctx.h, None, st)
    e, sign = ctx.measure_energy(stream=st)
    out = {"energy": e, "sign": sign, "fields": [ctx.fields(w) for w in range(case["walkers"])]}
    if case["walkers"] <= 2:  # a single chain's G, for the caller's own correlation functions
        out["G"] = [ctx.G(w, sp) for w in range(case["walkers"]) for sp in range(2)]
    else:
        out["fields"] = np.concatenate([f.ravel() for f in out["fields"]])
    return _as_bulk(case, out)


def _run_soc(case, s, st):
    ctx, got = s["ctx"], []
    for ell, d in _order(case["M"]):
        ctx.sweep_slice(ell, d, case["mode"], k=case["k"], nb=case["nb"], stream=st)
        pos = ell if d > 0 else ell - 1
        if pos % case["stab"] == 0:
            soc.afqmc_soc_recompute_G(ctx.h, None, st)
        if case["pairing"] and pos == case["M"] // 2 // case["stab"] * case["stab"]:
            got.append(ctx.measure_pairing(stream=st))
    out = {"energy": ctx.measure_energy(stream=st), "fields": [ctx.fields(w) for w in range(case["walkers"])]}
    if case["pairing"]:
        out["pairing"] = got
    else:
        out["G"] = [ctx.G(w) for w in range(case["walkers"])]
    return _as_bulk(case, out)


def _run_cpqmc(case, s, st):
    cp = s["ctx"]
    out = {"logw": [cp.step(case["mode"], case["k"], case["nb"], stream=st) for _ in range(case["steps"])]}
    out["fields"] = np.stack([cp.fields(j) for j in range(case["walkers"])])
    out["idx"] = cp.comb(s["u0"], stream=st)
    cp.reorth(stream=st)
    out["e_local"], out["e_mean"] = cp.energy(stream=st)
    out["phi"] = np.stack([cp.walker(j)[0] for j in range(case["walkers"])])
    return out


def _as_bulk(case, v):
    """FP32-bulk results in FP32 (the library's accessors widen them)."""
    if case["precision"] == "fp64":
        return v
    if isinstance(v, dict):
        return {k: _as_bulk(case, x) for k, x in v.items()}
    if isinstance(v, list):
        return [_as_bulk(case, x) for x in v]
    return v.astype({"f": np.float32, "c": np.complex64}.get(v.dtype.kind, v.dtype))


# ---------------------------------------------------------------- what a pass cannot do without

def work(case):
    if case["kind"] == "flips":
        N, m, es = case["N"], case["m"], 8 if case["precision"] == "fp64" else 4
        return {"bytes": 2 * 2 * N * N * es, "flops": 2 * 2 * N * N * m}
    if case["kind"] == "cpqmc":
        N, ns = case["L"] ** 2, _n_sigma(case["L"], case["filling"])
        # per walker, spin and step: propagation, U_L U_R, its inverse, one rank-1 update of T per site
        f = 4 * case["L"] * N * ns + 2 * N * ns * ns + 2 * ns ** 3 + N * 2 * ns * ns
        return {"bytes": case["walkers"] * 2 * N * ns * 8 * 2, "flops": case["walkers"] * 2 * case["steps"] * f}
    M, es = case["M"], 8 if case["precision"] == "fp64" else 4
    b = f = 0
    if case["kind"] == "hubbard":
        for L in _lattices(case):
            N, ns = L * L, _n_sigma(L, case["filling"])
            per_slice = 8 * L * N * N + 0.7 * N * 2 * N * N + 4 * L * N * ns  # wrap, updates, propagation
            rec = 2 * N * ns * ns + 2 * ns ** 3 + 2 * ns * ns * N + 2 * N * N * ns
            f += 2 * (2 * M * per_slice + 2 * (M // case["stab"]) * rec)
            b += 2 * 2 * N * N * es + 2 * M * N + 2 * N * ns * 8
        return {"bytes": b, "flops": f}
    L = case["L"]
    N, n_e = L * L, 2 * _n_sigma(L, case["filling"])
    n2 = 2 * N
    per_slice = 2 * 8 * n2 ** 3 + 0.7 * N * 2 * 8 * n2 * n2
    rec = 8 * (n2 * n_e * n_e + n_e ** 3 + n_e * n_e * n2 + n2 * n2 * n_e)
    f = case["walkers"] * (2 * M * per_slice + 2 * (M // case["stab"]) * rec)
    b = case["walkers"] * (2 * n2 * n2 * 2 * es + 2 * M * N)
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------- the same passes in plain FP64

def exact(case, seed):
    with torch.no_grad():
        return {"flips": _exact_flips, "hubbard": _exact_hubbard, "soc": _exact_soc, "cpqmc": _exact_cpqmc}[
            case["kind"]](case, seed)


def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _t(a, dtype=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(a)).to(_dev(), dtype)


def _uniforms(seed, walker, visit, count):
    raw = np.random.Philox(key=np.array([seed, walker], np.uint64),
                           counter=np.array([0, visit, 0, 0], np.uint64)).random_raw(4 * count)[0::4]
    return (raw >> np.uint64(11)).astype(np.float64) * 2.0 ** -53


def _exact_flips(case, seed):
    G0, sites, delta = _flips_inputs(case, seed)
    N, m = case["N"], case["m"]
    out = G0.double()
    I = sites.long()
    for s in range(2):
        G, D = G0[s, :, :N].double(), torch.diag(delta[s * m:(s + 1) * m])
        eye = torch.eye(N, dtype=torch.float64, device=G.device)[I]
        W = D @ torch.linalg.inv(torch.eye(m, dtype=torch.float64, device=G.device)
                                 + (torch.eye(m, dtype=torch.float64, device=G.device) - G[I][:, I]) @ D)
        out[s, :, :N] = G - G[:, I] @ (W @ (eye - G[I]))
    return out


def _exp_k(L, tau):
    w, v = np.linalg.eigh(_ring(L))
    e = (v * np.exp(-tau * w)) @ v.T
    return _t(np.kron(e, e))


def _qr_cols(U):
    """Orthonormal basis of the columns and the sign of the triangular factor's determinant."""
    Q, R = torch.linalg.qr(U)
    return Q, torch.sign(torch.diagonal(R, dim1=-2, dim2=-1)).prod(-1) if not R.is_complex() else None


def _scratch_g(E, P, d, M):
    """G at slice 0 and the sign of det(P^T B_M .. B_1 P) for batched slice diagonals d[l]: [..., N]."""
    Lt = P.clone()  # U_L^T
    sign = torch.ones(P.shape[:-2], dtype=torch.float64, device=P.device)
    for l in range(M - 1, -1, -1):
        Lt, s = _qr_cols(E.T @ (d[l].unsqueeze(-1) * Lt))
        sign = sign * s
    Lf = Lt.transpose(-1, -2)
    O = Lf @ P
    G = torch.eye(P.shape[-2], dtype=P.dtype, device=P.device) - P @ torch.linalg.solve(O, Lf)
    return G, sign * torch.linalg.slogdet(O)[0]


def _rank1(G, i, f):
    """G <- G - f G[:, i] (e_i^T - G[i, :]) for every matrix of the batch (f: one factor each)."""
    row = -G[..., i, :].clone()
    row[..., i] += 1.0
    col = G[..., :, i] * f.unsqueeze(-1)
    n = G.shape[-1]
    torch.baddbmm(G.view(-1, n, n), col.reshape(-1, n, 1), row.reshape(-1, 1, n), alpha=-1.0, out=G.view(-1, n, n))


def _exact_hubbard(case, seed):
    M, k_hs = case["M"], _hs(case["U"])
    _, lam, cc = k_hs
    charge = case["U"] < 0
    Ls = _lattices(case)
    walkers = len(Ls)
    energy, sign = np.zeros(walkers), np.zeros(walkers)
    fields, greens = [None] * walkers, [None] * walkers
    for L in sorted(set(Ls)):
        ids = [w for w in range(walkers) if Ls[w] == L]
        N, ns = L * L, _n_sigma(L, case["filling"])
        W, dev = len(ids), _dev()
        E, Ei = _exp_k(L, DTAU), _exp_k(L, -DTAU)
        P = _t(_trial(L, ns)).expand(W, 2, N, ns).contiguous()
        x = _t(np.stack([_fields(seed, w, M, N) for w in ids]))  # W x M x N
        c = torch.tensor(cc, dtype=torch.float64, device=dev)
        diag = lambda l: torch.exp(c[None, :, None] * x[:, l, None, :])  # noqa: E731  W x 2 x N
        G, sg = _scratch_g(E, P, [diag(l) for l in range(M)], M)
        sg = sg.prod(-1)
        for visit, (ell, d) in enumerate(_order(M)):
            u = _t(np.stack([_uniforms(seed, w, visit, 2 * N) for w in ids]))
            if d > 0:
                D = diag(ell - 1)
                G = D.unsqueeze(-1) * (E @ G @ Ei) / D.unsqueeze(-2)
            G = G.contiguous()
            xl = x[:, ell - 1]
            if case["mode"] == "blockfb":
                sg = _exact_blocks(G, xl, u, c, lam, charge, case["nb"], sg)
            else:
                for i in range(N):
                    dl = torch.exp(-2.0 * c[None, :] * xl[:, i, None]) - 1.0
                    r = 1.0 + dl * (1.0 - G[:, :, i, i])
                    R = r.prod(-1) * (torch.exp(2.0 * lam * xl[:, i]) if charge else 1.0)
                    acc = (u[:, i] < R.abs()).double()
                    _rank1(G, i, dl / r * acc[:, None])
                    xl[:, i] *= 1.0 - 2.0 * acc
                    sg = torch.where((acc > 0) & (R < 0), -sg, sg)
            if d < 0:
                D = diag(ell - 1)
                G = Ei @ (G * D.unsqueeze(-2) / D.unsqueeze(-1)) @ E
        G, _ = _scratch_g(E, P, [diag(l) for l in range(M)], M)
        A = torch.eye(N, dtype=torch.float64, device=dev) - G
        n = torch.diagonal(A, dim1=-2, dim2=-1)
        K = _t(_hopping(L))
        e = (K * A.transpose(-1, -2)).sum((-1, -2)).sum(-1) + case["U"] * (
            n[:, 0] * n[:, 1] - 0.5 * (n[:, 0] + n[:, 1])).sum(-1)
        for j, w in enumerate(ids):
            energy[w], sign[w] = float(e[j]), float(sg[j])
            fields[w] = x[j].cpu().numpy().astype(np.int8)
            if walkers <= 2:
                greens[w] = [G[j, 0].cpu().numpy(), G[j, 1].cpu().numpy()]
    out = {"energy": energy, "sign": sign}
    if walkers <= 2:
        out["fields"] = fields
        out["G"] = [g for pair in greens for g in pair]
    else:
        out["fields"] = np.concatenate([f.ravel() for f in fields])
    return out


def _exact_blocks(G, xl, u, c, lam, charge, nb, sg):
    """Block force bias on one slice (in place): stripped densities, joint proposal, determinant ratio."""
    N = G.shape[-1]
    for b, p in enumerate(range(0, N, nb)):
        q = min(N, p + nb)
        I = torch.eye(q - p, dtype=torch.float64, device=G.device)
        A = I - G[:, :, p:q, p:q]
        x = xl[:, p:q].clone()
        ds = torch.exp(-c[None, :, None] * x[:, None, :]) - 1.0
        bar = (1.0 + ds).unsqueeze(-1) * torch.linalg.solve(I + A * ds.unsqueeze(-2), A)
        h = (c[None, :, None] * torch.diagonal(bar, dim1=-2, dim2=-1)).sum(1)
        if charge:
            h = h - lam
        xp = torch.where(u[:, p:q] < 1.0 / (1.0 + torch.exp(-2.0 * h)), 1.0, -1.0).to(torch.float64)
        ls = -lam if charge else 0.0
        logq = (ls * (xp - x) + (x - xp) * h).sum(-1)
        df = torch.exp(c[None, :, None] * (xp - x)[:, None, :]) - 1.0
        R = torch.exp(logq) * torch.linalg.det(I + A * df.unsqueeze(-2)).prod(-1)
        acc = u[:, N + b] < R.abs()
        df = df * acc[:, None, None]
        W = df.unsqueeze(-1) * torch.linalg.inv(I + A * df.unsqueeze(-2))
        rows = -G[:, :, p:q, :].clone()
        rows[:, :, :, p:q] += I
        G -= G[:, :, :, p:q] @ (W @ rows)
        xl[:, p:q] = torch.where(acc[:, None], xp, x)
        sg = torch.where(acc & (R < 0), -sg, sg)
    return sg


def _site_matrix(hs, t):
    """The field's 2 x 2 matrix as its four entries (uu, ud, du, dd), for angles t of any shape."""
    if hs == "sz":
        z = torch.zeros_like(t, dtype=torch.complex128)
        return torch.exp(1j * t), z, z, torch.exp(-1j * t)
    co, si = torch.cos(t).to(torch.complex128), torch.sin(t).to(torch.complex128)
    return co, si, -si, co


def _apply_left(m, X):
    """D X for the pair-wise site matrices m (entries: [..., N]) and X: [..., 2N, C]."""
    N = X.shape[-2] // 2
    a, b, c, d = (v.unsqueeze(-1) for v in m)
    return torch.cat([a * X[..., :N, :] + b * X[..., N:, :], c * X[..., :N, :] + d * X[..., N:, :]], dim=-2)


def _pair_delta(hs, t):
    """A(t) - 1 on a block of sites as a matrix on (their up, their down) orbitals; t: [W, n]."""
    a, b, c, d = _site_matrix(hs, t)
    z = torch.diag_embed
    return torch.cat([torch.cat([z(a - 1.0), z(b)], -1), torch.cat([z(c), z(d - 1.0)], -1)], -2)


def _exact_soc(case, seed):
    L, M, W, hs, dev = case["L"], case["M"], case["walkers"], case["hs"], _dev()
    N, n_e = L * L, 2 * _n_sigma(case["L"], case["filling"])
    gamma = math.acos(math.exp(DTAU * case["U"] / 2.0))
    H = _soc_h0(L, case["lam"])
    w, v = np.linalg.eigh(H)
    cplx = torch.complex128
    E, Ei = (_t((v * np.exp(-s * DTAU * w)) @ v.conj().T, cplx) for s in (1.0, -1.0))
    P = _t(_soc_trial(L, n_e, case["lam"], hs), cplx).expand(W, 2 * N, n_e)
    x = _t(np.stack([_fields(seed, j, M, N) for j in range(W)]))
    eye = torch.eye(2 * N, dtype=cplx, device=dev)

    def scratch(pos):
        R, Lt = P, P
        for l in range(pos):
            R = torch.linalg.qr(_apply_left(_site_matrix(hs, gamma * x[:, l]), E @ R))[0]
        for l in range(M - 1, pos - 1, -1):  # U_L^+ <- B_l^+ U_L^+ = E (D_l^+ U_L^+)
            a, b, c, d = (z.conj() for z in _site_matrix(hs, gamma * x[:, l]))
            Lt = torch.linalg.qr(E @ _apply_left((a, c, b, d), Lt))[0]
        Lf = Lt.mH
        return eye - R @ torch.linalg.solve(Lf @ R, Lf)

    def wrap(G, xl, d):
        fw, bw = _site_matrix(hs, gamma * xl), _site_matrix(hs, -gamma * xl)
        right = lambda X, m: _apply_left((m[0], m[2], m[1], m[3]), X.mT).mT  # noqa: E731  X D
        if d > 0:
            return right(_apply_left(fw, E @ G @ Ei), bw)
        return Ei @ right(_apply_left(bw, G), fw) @ E

    G, got = scratch(0), []
    for visit, (ell, d) in enumerate(_order(M)):
        u = _t(np.stack([_uniforms(seed, j, visit, 2 * N) for j in range(W)]))
        xl = x[:, ell - 1]
        if d > 0:
            G = wrap(G, xl, +1)
        step = case["nb"] if case["mode"] == "blockfb" else 1
        for b, p in enumerate(range(0, N, step)):
            q = min(N, p + step)
            S = torch.cat([torch.arange(p, q), torch.arange(N + p, N + q)]).to(dev)
            I = torch.eye(2 * (q - p), dtype=cplx, device=dev)
            rows = G[:, S]
            A = I - rows[:, :, S]
            xo = xl[:, p:q].clone()
            if case["mode"] == "blockfb":
                ds = _pair_delta(hs, -gamma * xo)
                bar = (I + ds) @ torch.linalg.solve(I + A @ ds, A)
                n = q - p
                dg = lambda r, s: torch.diagonal(bar[:, r * n:(r + 1) * n, s * n:(s + 1) * n], dim1=-2, dim2=-1)  # noqa: E731
                ob = 1j * (dg(0, 0) - dg(1, 1)) if hs == "sz" else dg(1, 0) - dg(0, 1)
                h = gamma * ob.real
                xp = torch.where(u[:, p:q] < 1.0 / (1.0 + torch.exp(-2.0 * h)), 1.0, -1.0).to(torch.float64)
                logq, ua = ((xo - xp) * h).sum(-1), u[:, N + b]
            else:
                xp, logq, ua = -xo, 0.0, u[:, p]
            dl = _pair_delta(hs, gamma * (xp - xo))
            R = torch.linalg.det(I + dl @ A).abs() * (torch.exp(logq) if case["mode"] == "blockfb" else 1.0)
            acc = ua < R
            dl = dl * acc[:, None, None]
            Wm = dl @ torch.linalg.inv(I + A @ dl)
            Y = -rows
            Y[:, :, S] += I
            G = torch.baddbmm(G, G[:, :, S], Wm @ Y, alpha=-1.0)
            xl[:, p:q] = torch.where(acc[:, None], xp, xo)
        if d < 0:
            G = wrap(G, xl, -1)
        pos = ell if d > 0 else ell - 1
        if case["pairing"] and pos == M // 2 // case["stab"] * case["stab"]:
            got.append(_exact_pairing(scratch(pos), L))
    G = scratch(0)
    A = eye - G
    up, dn = torch.arange(N, device=dev), torch.arange(N, 2 * N, device=dev)
    n, m = A[:, up, up], A[:, dn, dn]
    e = (_t(H, cplx) * A.mT).sum((-1, -2)) + case["U"] * (n * m - A[:, dn, up] * A[:, up, dn] - 0.5 * (n + m)).sum(-1)
    out = {"energy": e.cpu().numpy(), "fields": [x[j].cpu().numpy().astype(np.int8) for j in range(W)]}
    if case["pairing"]:
        out["pairing"] = got
    else:
        out["G"] = [G[j].cpu().numpy() for j in range(W)]
    return out


def _exact_pairing(G, L):
    N, dev = L * L, G.device
    A = torch.eye(2 * N, dtype=G.dtype, device=dev) - G
    uu, dd, ud, du = A[:, :N, :N], A[:, N:, N:], A[:, :N, N:], A[:, N:, :N]
    dg = lambda X: torch.diagonal(X, dim1=-2, dim2=-1)  # noqa: E731
    D = (dg(uu) * dg(dd) - dg(du) * dg(ud)).mean(-1)
    # <D+_i D_j> = A_{ju,iu} A_{jd,id} - A_{jd,iu} A_{ju,id};  <D_i D+_j> the same with G_{i,j}
    g = lambda a, b: G[:, a * N:(a + 1) * N, b * N:(b + 1) * N]  # noqa: E731
    tot = (uu * dd - du * ud).sum((-1, -2)) + (g(0, 0) * g(1, 1) - g(1, 0) * g(0, 1)).sum((-1, -2))
    delta2 = tot / (4.0 * N * N)
    f1 = np.exp(-2j * np.pi * np.outer(np.arange(L), np.arange(L)) / L) / math.sqrt(L)
    F = _t(np.kron(f1, f1), G.dtype)
    At = [[F @ X @ F.mH for X in row] for row in ((uu, ud), (du, dd))]
    nk = torch.cat([dg(At[0][0]), dg(At[1][1])], -1)
    minus = torch.tensor([(L - k % L) % L + L * ((L - k // L) % L) for k in range(N)], device=dev)
    # Mk[k][k'] = At_{k'u,ku} At_{-k'd,-kd} - At_{-k'd,ku} At_{k'u,-kd}
    Mk = At[0][0].mT * At[1][1][:, minus][:, :, minus].mT - At[1][0][:, minus].mT * At[0][1][:, :, minus].mT
    return {"D": D.cpu().numpy(), "Delta2": delta2.cpu().numpy(), "nk": nk.cpu().numpy(), "Mk": Mk.cpu().numpy()}


def _exact_cpqmc(case, seed):
    L, W, dev = case["L"], case["walkers"], _dev()
    N, ns = L * L, _n_sigma(L, case["filling"])
    _, lam, cc = _hs(case["U"])
    charge = case["U"] < 0
    P0, phi0, u0 = _cp_inputs(case, seed)
    E, UL = _exp_k(L, DTAU), _t(P0).T
    phi = _t(phi0)
    c = torch.tensor(cc, dtype=torch.float64, device=dev)
    eye = torch.eye(N, dtype=torch.float64, device=dev)
    logdet = lambda p: torch.linalg.slogdet(UL @ p)[1].sum(-1)  # noqa: E731
    sx = lambda xv: torch.exp(-lam * xv) if charge else torch.ones_like(xv)  # noqa: E731
    logw, total = [], torch.zeros(W, dtype=torch.float64, device=dev)
    for step in range(case["steps"]):
        u = _t(np.stack([_uniforms(seed, j, step, 2 * N) for j in range(W)]))
        old = logdet(phi)
        phi = E @ phi
        lw = logdet(phi) - old
        G = (eye - phi @ torch.linalg.solve(UL @ phi, UL.expand(W, 2, ns, N))).contiguous()
        x = torch.zeros(W, N, dtype=torch.float64, device=dev)
        one = torch.ones(W, dtype=torch.float64, device=dev)
        if case["mode"] == "blockfb":
            for p in range(0, N, case["nb"]):
                q = min(N, p + case["nb"])
                I = torch.eye(q - p, dtype=torch.float64, device=dev)
                A = I - G[:, :, p:q, p:q]
                n = torch.diagonal(A, dim1=-2, dim2=-1)
                F = lam * (n[:, 0] + n[:, 1] - 1.0) if charge else c[0] * n[:, 0] + c[1] * n[:, 1]
                xs = torch.where(u[:, p:q] < 1.0 / (1.0 + torch.exp(-2.0 * F)), 1.0, -1.0).to(torch.float64)
                df = torch.exp(c[None, :, None] * xs[:, None, :]) - 1.0
                lw = lw + (torch.log(sx(xs) * torch.cosh(F)) - xs * F).sum(-1) + torch.log(
                    torch.linalg.det(I + A * df.unsqueeze(-2)).prod(-1))
                Wm = df.unsqueeze(-1) * torch.linalg.inv(I + A * df.unsqueeze(-2))
                rows = -G[:, :, p:q, :].clone()
                rows[:, :, :, p:q] += I
                G -= G[:, :, :, p:q] @ (Wm @ rows)
                x[:, p:q] = xs
        else:
            for i in range(N):
                a = 1.0 - G[:, :, i, i]
                rp, rm = (1.0 + (torch.exp(c * s) - 1.0) * a for s in (1.0, -1.0))
                lp, lm = ((0.5 * sx(s * one) * r.prod(-1)).clamp(min=0.0) for s, r in ((1.0, rp), (-1.0, rm)))
                xi = torch.where(u[:, i] < lp / (lp + lm), 1.0, -1.0).to(torch.float64)
                lw = lw + torch.log(lp + lm)
                _rank1(G, i, (torch.exp(c[None] * xi[:, None]) - 1.0) / torch.where(xi[:, None] > 0, rp, rm))
                x[:, i] = xi
        phi = phi * torch.exp(c[None, :, None] * x[:, None, :]).unsqueeze(-1)
        logw.append(lw.cpu().numpy())
        total = total + lw
    tw = total.cpu().numpy()
    if not np.all(np.isfinite(tw)):
        return None
    cum = np.cumsum(np.exp(tw - tw.max()))
    idx = np.minimum(np.searchsorted(cum, (np.arange(W) + u0) * cum[-1] / W, side="right"), W - 1)
    phi = phi[torch.from_numpy(idx).to(dev)]
    Pm, Lm, _ = torch.linalg.lu(phi)
    phi = Pm @ Lm
    A = phi @ torch.linalg.solve(UL @ phi, UL.expand(W, 2, ns, N))
    n = torch.diagonal(A, dim1=-2, dim2=-1)
    e = (_t(_hopping(L)) * A.mT).sum((-1, -2)).sum(-1) + case["U"] * (
        n[:, 0] * n[:, 1] - 0.5 * (n[:, 0] + n[:, 1])).sum(-1)
    e = e.cpu().numpy()
    return {"logw": logw, "fields": x.cpu().numpy().astype(np.int8), "idx": idx.astype(np.int32), "e_local": e,
            "e_mean": float(e.mean()), "phi": phi.cpu().numpy()}
