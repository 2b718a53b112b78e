"""What is timed: the work a user of this library has it do, through its public entry points.

Every case is a dict of plain values; ``kind`` picks the entry point.  Sizes are the repository's own
configurations (the plain L=8 case, the medium, benchmark and large streamed configurations, the ragged batch,
the projection, triplet and eigensolver benchmarks) or generic ones around them.  Inputs are made on the GPU from
the seed alone: orthonormal complex Gaussian vectors, as LapH eigenvectors are, and smoothed SU(3) links.
"""
import math

import numpy as np
import torch

from paper_2510_26313_gb300 import binding as laph
from paper_2510_26313_gb300 import synth


def listed():
    return [
        # a script that wants a few packed baryon blocks at once and their dense tensor: temporary plan and all
        {"name": "one-shot", "kind": "oneshot", "L": 8, "T": 1, "N": 16, "P": 3, "mode": "f16x3"},
        # the plain L=8 configuration through a kept plan: latency and launches are all there is
        {"name": "blocks-plain", "kind": "blocks", "L": 8, "T": 1, "N": 16, "P": 3, "mode": "f16x3", "out": "c128"},
        # a workflow that streams its configuration one timeslice at a time
        {"name": "blocks-one-slice", "kind": "blocks", "L": 24, "T": 1, "N": 32, "P": 7, "mode": "f16x3", "out": "c128"},
        # the medium configuration
        {"name": "blocks-medium", "kind": "blocks", "L": 24, "T": 48, "N": 32, "P": 7, "mode": "f16x3", "out": "c128"},
        # the benchmark configuration
        {"name": "blocks-benchmark", "kind": "blocks", "L": 32, "T": 64, "N": 64, "P": 19, "mode": "f16x3", "out": "c128"},
        # one timeslice of the large streamed configuration
        {"name": "blocks-large", "kind": "blocks", "L": 48, "T": 1, "N": 128, "P": 33, "mode": "f16x3", "out": "c128"},
        # many small problems of different sizes in one plan
        {"name": "blocks-ragged", "kind": "ragged", "count": 24, "Lmin": 16, "Lmax": 24, "Nmin": 24, "Nmax": 64,
         "Pmax": 19, "Tmax": 4, "pick": 5, "mode": "f16x3"},
        # smeared quark sinks, three different fields, dense N^3
        {"name": "triplets", "kind": "triplets", "L": 32, "T": 2, "N": 64, "P": 19, "mode": "f16x3", "out": "c128"},
        # mesons alone (no baryon rows), in the other split type with half-size outputs
        {"name": "mesons", "kind": "mesons", "L": 32, "T": 16, "N": 64, "P": 19, "mode": "bf16x3", "out": "c64"},
        # solution vectors projected onto the eigenvectors: inner products, n = 0
        {"name": "projection", "kind": "projection", "L": 32, "T": 16, "N": 128, "Nc": 512, "P": 1, "mode": "f16x3",
         "out": "c128"},
        # the plain FP32 path at the medium configuration
        {"name": "blocks-fp32", "kind": "blocks", "L": 24, "T": 48, "N": 32, "P": 7, "mode": "fp32", "out": "c128"},
        # the LapH eigenvectors themselves, then the check every user makes: -Delta applied to all of them
        {"name": "eigenvectors", "kind": "lanczos", "L": 32, "T": 8, "n_ev": 64, "m": 128, "degree": 48, "lo": 0.95},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["oneshot", "blocks", "blocks", "blocks", "blocks", "ragged", "triplets", "mesons", "projection",
                       "fp32", "lanczos"])
    split = rng.choice(["f16x3", "f16x3", "bf16x3"])
    out = rng.choice(["c128", "c128", "c64"])
    P = rng.choice([1, 3, 7, 19, 33])
    if kind == "oneshot":
        return {"kind": kind, "L": rng.randint(6, 20), "T": rng.randint(1, 3), "N": _log_int(rng, 8, 40), "P": P,
                "mode": split}
    if kind == "ragged":
        return {"kind": kind, "count": rng.randint(2, 24), "Lmin": rng.randint(6, 16), "Lmax": rng.randint(17, 24),
                "Nmin": rng.randint(8, 24), "Nmax": rng.randint(32, 64), "Pmax": rng.choice([7, 19]),
                "Tmax": rng.randint(1, 4), "pick": rng.randint(0, 1 << 20), "mode": split}
    if kind == "lanczos":
        # as many eigenpairs per site as the listed case has, so that the same filter bound lies above them
        L = rng.choice([12, 15, 16, 20, 21, 24, 28, 32])
        n_ev = max(3, 64 * L ** 3 // 32 ** 3)
        return {"kind": kind, "L": L, "T": _log_int(rng, 1, 8), "n_ev": n_ev, "m": max(24, 2 * n_ev),
                "degree": rng.choice([40, 47, 48]), "lo": 0.95}
    if kind == "projection":
        return {"kind": kind, "L": rng.randint(12, 32), "T": _log_int(rng, 1, 16), "N": _log_int(rng, 16, 160),
                "Nc": _log_int(rng, 32, 512), "P": rng.choice([1, 1, 7]), "mode": split, "out": out}
    # the rest: lattice and vectors over their range, timeslices up to the listed cases' work
    L = rng.randint(6, 32)
    N = _log_int(rng, 8, 96)
    cost = 8 * 3 * L ** 3 * P
    if kind == "triplets":
        N = _log_int(rng, 6, 64)
        T = max(1, min(_log_int(rng, 1, 8), int(8e12 / (cost * N ** 3))))
    elif kind == "mesons":
        T = max(1, min(_log_int(rng, 1, 32), int(2e12 / (cost * N * N))))
    elif kind == "fp32":
        kind, split, out = "blocks", "fp32", "c128"
        N = _log_int(rng, 8, 48)
        T = max(1, min(_log_int(rng, 1, 48), int(6e11 / (cost * (math.comb(N, 3) + N * N)))))
    else:
        T = max(1, min(_log_int(rng, 1, 64), int(1.5e13 / (cost * (math.comb(N, 3) + N * N)))))
    return {"kind": kind, "L": L, "T": T, "N": N, "P": P, "mode": split, "out": out}


# ---------------------------------------------------------------- inputs

def _momenta(P):
    """The first P momenta of the full shells; the plain configuration's three are 0 and two unit vectors."""
    if P == 3:
        return np.array([[0, 0, 0], [1, 0, 0], [0, 1, 0]], dtype=np.int32)
    return synth.momenta_for_count(P)


def _generator(seed, field=0):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1000003 + 7919 * field) % (1 << 62))
    return g


def _vectors(L, T, N, seed, field=0):
    """complex64 [T][N][L^3][3]: complex Gaussian vectors, orthonormal over (site, colour) on every timeslice."""
    K = 3 * L ** 3
    g = _generator(seed, field)
    out = torch.empty((T, N, K), dtype=torch.complex64, device="cuda")
    for t in range(T):
        z = torch.view_as_complex(torch.randn((N, K, 2), generator=g, device="cuda"))
        if N <= K:
            gram = (z.conj() @ z.T).to(torch.complex128)
            c = torch.linalg.cholesky(gram.T.contiguous())
            z = torch.linalg.inv(c).to(torch.complex64) @ z
        out[t] = z
    return out.reshape(T, N, L ** 3, 3)


def _ragged(case):
    insts = synth.ragged_instances(case["count"], seed=case["pick"], Ls=tuple(range(case["Lmin"], case["Lmax"] + 1)),
                                   Nrange=(case["Nmin"], case["Nmax"]),
                                   Pset=tuple(p for p in (1, 7, 19) if p <= case["Pmax"]), Trange=(1, case["Tmax"]))
    return [(i.L, i.T, i.N, i.momenta) for i in insts]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "lanczos":
        L, T = case["L"], case["T"]
        U = synth.random_links_device(L, T, 0.6, seed=int(seed))
        need = laph.lanczos_workspace_size(L, T, case["n_ev"], case["m"], case["degree"], case["lo"])
        return {"case": case, "U": U, "ws": torch.empty(need, dtype=torch.uint8, device="cuda")}
    if kind == "ragged":
        specs = _ragged(case)
        plan = laph.Plan(specs, mode=case["mode"])
        phis = [_vectors(L, T, N, seed, n) for n, (L, T, N, _) in enumerate(specs)]
        return {"case": case, "plan": plan, "phis": phis, "out": plan.alloc_outputs(), "ws": plan.alloc_workspace()}
    L, T, N, mom = case["L"], case["T"], case["N"], _momenta(case["P"])
    if kind == "oneshot":
        return {"case": case, "phi": _vectors(L, T, N, seed), "mom": mom}
    flags = laph.PLAN_OUT_C64 if case["out"] == "c64" else 0
    if kind == "triplets":
        fields = [_vectors(L, T, N, seed, f) for f in range(3)]
        plan = laph.Plan([(L, T, N, mom)], mode=case["mode"], flags=flags | laph.PLAN_FIELDS | laph.PLAN_SKIP_M)
    elif kind == "projection":
        fields = [_vectors(L, T, N, seed), _vectors(L, T, case["Nc"], seed, 1)]
        plan = laph.Plan([(L, T, N, mom, case["Nc"])], mode=case["mode"],
                         flags=flags | laph.PLAN_FIELDS | laph.PLAN_SKIP_B)
    else:
        fields = [_vectors(L, T, N, seed)]
        plan = laph.Plan([(L, T, N, mom)], mode=case["mode"],
                         flags=flags | (laph.PLAN_SKIP_B if kind == "mesons" else 0))
    return {"case": case, "plan": plan, "fields": fields, "out": plan.alloc_outputs(), "ws": plan.alloc_workspace()}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "oneshot":
        B = laph.baryon_blocks(state["phi"], case["L"], state["mom"], mode=case["mode"])
        return {"B": B, "dense": laph.baryon_dense(B, case["N"])}
    if kind == "lanczos":
        # the residual norms (FP32 rounding noise of a converged solve) follow from what is returned
        vecs, ev, _ = laph.lanczos(state["U"], case["L"], case["n_ev"], case["m"], cheb_degree=case["degree"],
                                   cheb_lo=case["lo"], workspace=state["ws"])
        return {"evals": ev, "vecs": vecs, "lap": laph.laplacian(state["U"], vecs, case["L"])}
    plan, (Bs, Ms) = state["plan"], state["out"]
    if kind == "ragged":
        plan.execute(state["phis"], Bs, Ms, state["ws"])
        return {"B": Bs, "M": Ms}
    if kind == "triplets":
        plan.execute_fields([state["fields"]], Bs, state["ws"])
        return {"B": Bs[0]}
    if kind == "projection":
        plan.execute_fields([state["fields"]], Ms, state["ws"])
        return {"M": Ms[0]}
    plan.execute(state["fields"], Bs, Ms, state["ws"])
    return {"M": Ms[0]} if kind == "mesons" else {"B": Bs[0], "M": Ms[0]}


# ---------------------------------------------------------------- work and exact results

def _blocks_work(L, T, N, P, entry):
    """Baryon and meson blocks of one instance: 8 real flops per complex multiply-add, i < j < k only."""
    n = math.comb(N, 3) + N * N
    return {"flops": 8.0 * 3 * L ** 3 * n * P * T, "bytes": T * (8.0 * N * 3 * L ** 3 + entry * n * P)}


def work(case):
    kind = case["kind"]
    if kind == "ragged":
        w = [_blocks_work(L, T, N, len(m), 16) for L, T, N, m in _ragged(case)]
        return {k: sum(x[k] for x in w) for k in ("bytes", "flops")}
    L, T = case["L"], case["T"]
    K = 3 * L ** 3
    if kind == "lanczos":
        # the filter's stencil (three links of a site, vector in, previous and out) and four passes over the basis per
        # step for the two Gram-Schmidt passes; Ritz vectors; -Delta on them twice
        m, d, nr = case["m"], case["degree"], case["n_ev"]
        site = 3 * (2 * 66 + 2 * 9)
        flops = T * (m * d * L ** 3 * site + 32.0 * K * m * (m + 1) / 2 + 4.0 * K * m * nr + 2.0 * nr * L ** 3 * site)
        return {"flops": flops, "bytes": T * (L ** 3 * 216.0 + 8.0 * K * (m + 2 * nr))}
    N, P = case["N"], case["P"]
    entry = 8 if case.get("out") == "c64" else 16
    if kind == "triplets":
        n = N ** 3
        return {"flops": 8.0 * K * n * P * T, "bytes": T * (8.0 * 3 * N * K + entry * n * P)}
    if kind == "mesons":
        return {"flops": 8.0 * K * N * N * P * T, "bytes": T * (8.0 * N * K + entry * N * N * P)}
    if kind == "projection":
        Nc = case["Nc"]
        return {"flops": 8.0 * K * N * Nc * P * T, "bytes": T * (8.0 * (N + Nc) * K + entry * N * Nc * P)}
    if kind == "oneshot":
        n = math.comb(N, 3)
        return {"flops": 8.0 * K * n * P * T, "bytes": T * (8.0 * N * K + 16.0 * n * P + 16.0 * N ** 3 * P)}
    return _blocks_work(L, T, N, P, entry)


def _phases(L, mom):
    x = torch.arange(L ** 3, device="cuda", dtype=torch.int64)
    xc = torch.stack([x % L, (x // L) % L, x // (L * L)])
    r = (torch.from_numpy(np.asarray(mom, dtype=np.int64)).cuda().unsqueeze(2) * xc.unsqueeze(0)).sum(1) % L
    return torch.polar(torch.ones(r.shape, dtype=torch.float64, device="cuda"), -2.0 * math.pi * r.double() / L)


def _exact_mesons(a, b, ph):
    """sum_x ph_p conj(a_i) . b_j: complex128 [P][Na][Nb]; a, b complex128 [N][V][3]."""
    ac = a.conj().reshape(a.shape[0], -1)
    return torch.stack([ac @ (b * p[None, :, None]).reshape(b.shape[0], -1).T for p in ph])


def _exact_baryons(f, ph):
    """Packed blocks of one timeslice, complex128 [P][C(N,3)]: f complex128 [N][V][3]."""
    N, P = f.shape[0], ph.shape[0]
    out = torch.empty((P, math.comb(N, 3)), dtype=torch.complex128, device=f.device)
    d = torch.empty((math.comb(N, 2), f.shape[1] * 3), dtype=torch.complex128, device=f.device)
    for k in range(1, N):
        if k >= 2:
            q = math.comb(k, 2)
            out[:, math.comb(k, 3):math.comb(k + 1, 3)] = (ph[:, :, None] * f[k]).reshape(P, -1) @ d[:q].T
        d[math.comb(k, 2):math.comb(k + 1, 2)] = torch.linalg.cross(f[:k], f[k:k + 1].expand(k, -1, -1)).reshape(k, -1)
    return out


def _exact_triplets(u, v, w, ph):
    """Dense three-field blocks of one timeslice, complex128 [P][N][N][N]."""
    N, P = u.shape[0], ph.shape[0]
    out = torch.empty((P, N, N, N), dtype=torch.complex128, device=u.device)
    psi = (ph[:, None, :, None] * w[None]).reshape(P * N, -1)
    for i in range(N):
        d = torch.linalg.cross(u[i:i + 1].expand(N, -1, -1), v).reshape(N, -1)
        out[:, i] = (d @ psi.T).reshape(N, P, N).permute(1, 0, 2)
    return out


def _exact_dense(packed, N):
    """Dense [T][P][N][N][N] from packed [T][P][C(N,3)]: sign of the sorting permutation."""
    dense = torch.zeros(packed.shape[:2] + (N, N, N), dtype=packed.dtype, device=packed.device)
    n = torch.arange(N, device=packed.device)
    i, j, k = torch.combinations(n, 3).unbind(1)
    idx = k * (k - 1) * (k - 2) // 6 + j * (j - 1) // 2 + i
    for perm, s in (((i, j, k), 1), ((j, k, i), 1), ((k, i, j), 1), ((j, i, k), -1), ((i, k, j), -1), ((k, j, i), -1)):
        dense[:, :, perm[0], perm[1], perm[2]] = s * packed[:, :, idx]
    return dense


def exact(case, seed):
    kind = case["kind"]
    if kind == "lanczos":
        return None   # eigenvectors of a filtered Krylov space: no closed form within seconds
    # baryon blocks of the largest problems take minutes in 64 bits: their mesons stand for them
    long = kind != "ragged" and work(case)["flops"] > 1.2e13
    if kind == "ragged":
        long = work(case)["flops"] > 1.2e13
        Bs, Ms = [], []
        for n, (L, T, N, mom) in enumerate(_ragged(case)):
            ph, f = _phases(L, mom), _vectors(L, T, N, seed, n).to(torch.complex128)
            Bs.append(None if long else torch.stack([_exact_baryons(f[t], ph) for t in range(T)]))
            Ms.append(torch.stack([_exact_mesons(f[t], f[t], ph) for t in range(T)]))
        return {"B": Bs, "M": Ms}
    L, T, N = case["L"], case["T"], case["N"]
    ph = _phases(L, _momenta(case["P"]))
    u = _vectors(L, T, N, seed)
    if kind == "triplets":
        if long:
            return None
        v, w = _vectors(L, T, N, seed, 1), _vectors(L, T, N, seed, 2)
        return {"B": torch.stack([_exact_triplets(*(x[t].to(torch.complex128) for x in (u, v, w)), ph)
                                  for t in range(T)])}
    if kind in ("mesons", "projection"):
        w = _vectors(L, T, case["Nc"], seed, 1) if kind == "projection" else u
        return {"M": torch.stack([_exact_mesons(u[t].to(torch.complex128), w[t].to(torch.complex128), ph)
                                  for t in range(T)])}
    B = None if long else torch.stack([_exact_baryons(u[t].to(torch.complex128), ph) for t in range(T)])
    if kind == "oneshot":
        return {"B": B, "dense": _exact_dense(B, N)}
    return {"B": B, "M": torch.stack([_exact_mesons(*(u[t].to(torch.complex128),) * 2, ph) for t in range(T)])}
