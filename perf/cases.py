"""The calls that a user of this library makes, over the sizes it is used at.

Systems: an active space with its exact singlet ground state (the ones of the
named configurations: 4e/4o "tiny", 8e/8o "medium", and 6e/6o between them)
and virtual orbitals drawn from the seed, with the one-electron and Cholesky
distributions of the repository's generator.  The virtual levels are raised a
little with their number so that H0 - E0 stays positive for every draw, as it
is for the configurations' own seeds.

Layers: the density-matrix eigensolvers, the local operators of one bond, the
third-order energy of a given first-order MPS, the block preconditioner's
network.  Whole calls: the Hylleraas sweep, the partitioned sweep, and the
ground-state DMRG that makes a reference.  The sweeps run a set number of
sweeps (no early stop) and return the energies; their MPSs are defined up to
a choice of basis on every bond, so the state is returned through E3 where
the full-Hamiltonian operator is small.
"""
import functools
import math

import numpy as np
import torch

import synthetic
from paper_1408_5092_gb300 import _lib as L

QSITE = ((0, 0), (1, 1), (1, -1), (2, 0))      # (N, 2Sz) of |0>, |a>, |b>, |ab>


def listed():
    return [
        # a handful of small symmetry sectors, from a host that has reserved
        # the device memory: the smallest call, launch and latency bound
        {"name": "eigh_small_noalloc", "kind": "eigh", "entry": "noalloc", "batch": 12, "n0": 13, "ragged": False},
        # the sectors of one truncation at M = 128, float64 throughout
        {"name": "eigh_sectors_M128_fp64", "kind": "eigh", "entry": "fp64", "batch": 7, "n0": 90, "ragged": True},
        # the sectors of one truncation at M = 256 (largest about 173), with the
        # truncation step's own solver
        {"name": "eigh_sectors_M256", "kind": "eigh", "entry": "mixed", "batch": 10, "n0": 173, "ragged": True},
        # sigma at the active/virtual border of the medium chain, M = 256, Dyall
        {"name": "sigma_medium_M256", "kind": "local", "op": "sigma", "k_act": 8, "k_virt": 24, "h0": "dyall",
         "M": 256, "bond": 7},
        # the right-hand side inside the virtual space, an odd M, Fock
        {"name": "rhs_medium_M101", "kind": "local", "op": "rhs", "k_act": 8, "k_virt": 24, "h0": "fock", "M": 101,
         "bond": 19},
        # E3 of a given first-order state (6e/6o + 13 virtual orbitals)
        {"name": "e3_6o13v_M60", "kind": "e3", "k_act": 6, "k_virt": 13, "h0": "dyall", "M": 60},
        # backward pass of the block preconditioner on one sweep's harvest
        {"name": "mlp_gradient_4099", "kind": "mlp", "pass": "gradient", "batch": 4099},
        # the small system to a few sweeps, with its E3
        {"name": "sweep_tiny_fock_M16_fp64", "kind": "sweep", "k_act": 4, "k_virt": 8, "h0": "fock", "M": 16,
         "prec": "fp64", "sweeps": 2, "tuned": False, "e3": True},
        # the medium system at a working M, float64 throughout
        {"name": "sweep_medium_dyall_M64_fp64", "kind": "sweep", "k_act": 8, "k_virt": 24, "h0": "dyall", "M": 64,
         "prec": "fp64", "sweeps": 1, "tuned": False, "e3": False},
        # the benchmark's configuration: M = 256, split-bf16 inner operator, tuned tiles
        {"name": "sweep_medium_dyall_M256_mixed", "kind": "sweep", "k_act": 8, "k_virt": 24, "h0": "dyall", "M": 256,
         "prec": "mixed", "sweeps": 1, "tuned": True, "e3": False},
        # virtual-pair partitions on concurrent lanes, graphs and tuned tiles as the README runs them
        {"name": "partitions_medium_12", "kind": "partitions", "k_act": 8, "k_virt": 24, "h0": "fock", "parts": 12,
         "M": 48, "prec": "fp64", "sweeps": 2},
        # the reference itself: ground-state DMRG of the 8e/8o active space
        {"name": "dmrg_8o_M48", "kind": "dmrg", "k_act": 8, "M": 48, "sweeps": 2},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["eigh", "eigh", "local", "e3", "mlp", "sweep", "sweep", "partitions", "dmrg"])
    h0 = rng.choice(["fock", "dyall"])
    k_act = rng.choice([4, 6, 8])
    k_virt = rng.randint(5, 24)
    if kind == "eigh":
        entry = rng.choice(["noalloc", "batched", "fp64", "mixed"])
        n0 = _log_int(rng, 5, 90 if entry in ("noalloc", "batched") else 190)
        return {"kind": kind, "entry": entry, "batch": rng.randint(1, 16), "n0": n0, "ragged": rng.random() < 0.6}
    if kind == "local":
        return {"kind": kind, "op": rng.choice(["sigma", "rhs", "diag"]), "k_act": k_act, "k_virt": k_virt, "h0": h0,
                "M": _log_int(rng, 12, 256), "bond": rng.randint(0, k_act + k_virt - 2)}
    if kind == "e3":
        return {"kind": kind, "k_act": rng.choice([4, 6]), "k_virt": rng.randint(5, 13), "h0": h0,
                "M": _log_int(rng, 8, 90)}
    if kind == "mlp":
        return {"kind": kind, "pass": rng.choice(["forward", "gradient"]), "batch": _log_int(rng, 17, 20000)}
    if kind == "partitions":
        return {"kind": kind, "k_act": k_act, "k_virt": k_virt, "h0": h0, "parts": rng.randint(2, 12),
                "M": _log_int(rng, 8, 48), "prec": rng.choice(["fp64", "mixed"]), "sweeps": 2}
    if kind == "dmrg":
        return {"kind": kind, "k_act": rng.choice([6, 8]), "M": _log_int(rng, 8, 64), "sweeps": rng.randint(1, 2)}
    M = _log_int(rng, 8, 256)
    return {"kind": "sweep", "k_act": k_act, "k_virt": k_virt, "h0": h0, "M": M,
            "prec": rng.choice(["fp64", "mixed", "mixed_fp16"] if M < 160 else ["mixed", "mixed_fp16"]),
            "sweeps": rng.randint(1, 2) if k_act * M < 400 else 1, "tuned": rng.random() < 0.5,
            "e3": k_act == 4 and k_virt <= 10}


# ---------------------------------------------------------------- systems
@functools.lru_cache(maxsize=None)
def _active(k_act):
    """Active block (h, L) and its singlet ground state, as the named configurations have it."""
    if k_act == 8:
        h, Lc, _, ci = synthetic.config_reference("medium")
    else:
        h, Lc = synthetic.integrals(synthetic.EVAL_SEED, k_act, 2 * k_act, 5 * k_act)
        ci, _ = synthetic.fci_reference(h, Lc, k_act, k_act)
    return h[:k_act, :k_act], Lc[:, :k_act, :k_act], ci


def _system(k_act, k_virt, seed):
    """(h, L, ci): the active block and virtual orbitals drawn from the seed."""
    ha, La, ci = _active(k_act)
    h, Lc = synthetic.integrals(seed, k_act, k_virt, La.shape[0])
    h[:k_act, :k_act] = ha
    Lc[:, :k_act, :k_act] = La
    v = np.arange(k_act, k_act + k_virt)
    h[v, v] += 0.25 * math.sqrt(k_virt)
    return h, Lc, ci


def _context(case, seed, k_virt, **opts):
    o = L.mpspt_default_options()
    for k, v in opts.items():
        setattr(o, k, v)
    h, Lc, ci = _system(case["k_act"], k_virt, seed)
    if case["kind"] == "dmrg":      # another geometry of the active space
        a = case["k_act"]
        d = np.random.default_rng(seed).normal(size=(a, a)) * 0.01
        h[:a, :a] += 0.5 * (d + d.T)
    ctx = L.mpspt_create(o)
    L.mpspt_set_integrals(ctx, case["k_act"], k_virt, case["k_act"], h, Lc)
    return ctx, ci


class _Handle:
    """A context (and an MPS) that is given back with the state."""

    def __init__(self, ctx, psi=None):
        self.ctx, self.psi = ctx, psi

    def __del__(self):
        if self.psi is not None:
            L.mpspt_mps_free(self.psi)
        L.mpspt_destroy(self.ctx)


def _sectors(k_act, k_virt, n_elec, M):
    """Per cut {(N, 2Sz): dimension} of a first-order MPS (of the reference, without virtual
    orbitals) of bond dimension about M."""
    k = k_act + k_virt

    def passes(cut, q):
        return cut != k_act or k_virt == 0 or q[0] in (n_elec - 1, n_elec - 2)

    left = [{(0, 0): 1}]
    for c in range(k):
        nxt = {}
        for q, d in left[c].items():
            for s in QSITE:
                r = (q[0] + s[0], q[1] + s[1])
                if passes(c + 1, r):
                    nxt[r] = min(1 << 40, nxt.get(r, 0) + d)
        left.append(nxt)
    right = [None] * k + [{(n_elec, 0): 1}]
    for c in range(k - 1, -1, -1):
        nxt = {}
        for q, d in right[c + 1].items():
            for s in QSITE:
                r = (q[0] - s[0], q[1] - s[1])
                if passes(c, r):
                    nxt[r] = min(1 << 40, nxt.get(r, 0) + d)
        right[c] = nxt
    out = []
    for c in range(k + 1):
        w = {q: min(d, right[c][q], M) for q, d in sorted(left[c].items()) if q in right[c]}
        tot = sum(w.values())
        out.append({q: d if tot <= M else min(d, max(1, M * d // tot)) for q, d in w.items()})
    return out


def _random_mps(k_act, k_virt, n_elec, M, rng, centre):
    """A random first-order MPS, left-orthonormal before site `centre` and right-orthonormal after it."""
    secs = _sectors(k_act, k_virt, n_elec, M)
    tensors, labels = [], []
    for s in secs:
        labels.append(np.array([q for q, d in s.items() for _ in range(d)], dtype=np.int32).reshape(-1, 2))
    for c in range(k_act + k_virt):
        ql, qr = labels[c], labels[c + 1]
        mask = np.stack([np.all(ql[:, None, :] + np.array(q) == qr[None, :, :], axis=2) for q in QSITE], axis=1)
        A = rng.normal(size=mask.shape) * mask
        side = qr if c < centre else ql
        X = A.reshape(-1, A.shape[2]) if c < centre else A.reshape(A.shape[0], -1).T
        Q = np.zeros_like(X)
        for q in {tuple(v) for v in side}:
            cols = np.flatnonzero(np.all(side == q, axis=1))
            rows = np.flatnonzero(np.any(X[:, cols] != 0, axis=1))
            if rows.size >= cols.size:
                Q[np.ix_(rows, cols)] = np.linalg.qr(X[np.ix_(rows, cols)])[0]
            elif rows.size:      # more states than directions: a bounded frame
                Q[np.ix_(rows, cols)] = np.linalg.qr(X[np.ix_(rows, cols)].T)[0].T
        tensors.append(Q.reshape(A.shape) if c < centre else np.ascontiguousarray(Q.T).reshape(A.shape))
    return tensors, labels


# --------------------------------------------------------- density matrices
def _sizes(case):
    if not case["ragged"]:
        return [case["n0"]] * case["batch"]
    return [max(1, int(round(case["n0"] * 0.8 ** i))) for i in range(case["batch"])]


def _density_matrices(case, seed):
    """Density matrices of a truncation: eigenvalues spread over four decades."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    out = []
    for n in _sizes(case):
        j = torch.arange(n, device="cuda", dtype=torch.float64)
        u = torch.rand(n, device="cuda", dtype=torch.float64, generator=g)
        lam = 10.0 ** (-4.0 * (j + 0.25 + 0.5 * u) / n)
        Q = torch.linalg.qr(torch.randn(n, n, device="cuda", dtype=torch.float64, generator=g))[0]
        A = (Q * (lam / lam.sum())) @ Q.T
        out.append(0.5 * (A + A.T))
    return out


def _in_order(w, V):
    """Eigenpairs as a caller takes them: largest first, each vector's largest component positive."""
    w, order = torch.sort(w, dim=-1, descending=True)
    V = torch.gather(V, -1, order.unsqueeze(-2).expand_as(V))
    top = torch.gather(V, -2, V.abs().argmax(dim=-2, keepdim=True))
    return w, V * top.sign()


# ------------------------------------------------------------------- cases
def prepare(case, seed):
    kind = case["kind"]
    rng = np.random.default_rng(seed)
    st = {"case": case}
    if kind == "eigh":
        mats = _density_matrices(case, seed)
        st["n"] = [m.shape[0] for m in mats]
        st["A"] = torch.cat([m.reshape(-1) for m in mats])
        st["V"] = torch.empty_like(st["A"])
        st["w"] = torch.empty(sum(st["n"]), device="cuda", dtype=torch.float64)
        return st
    if kind == "mlp":
        st["p"] = {"W1": (256, L.MLP_NF), "b1": 256, "W2": (256, 256), "b2": 256, "W3": (2, 256), "b3": 2}
        for k, shape in st["p"].items():
            scale = 0.05 if k[0] == "b" else math.sqrt(2.0 / shape[1])
            st["p"][k] = (rng.normal(size=shape) * scale).astype(np.float32)
        st["net"] = _Net(st["p"])
        st["x"] = rng.normal(size=(case["batch"], L.MLP_NF)).astype(np.float32)
        st["t"] = rng.normal(size=(case["batch"], 2)).astype(np.float32)
        return st
    if kind == "dmrg":
        st["h"] = _Handle(_context(case, seed, 6, max_sweeps=case["sweeps"], e_tol=1e-14)[0])
        return st
    if kind in ("local", "e3"):
        ctx, ci = _context(case, seed, case["k_virt"])
        L.mpspt_set_reference_ci(ctx, ci)
        i = case.get("bond", 0)
        tensors, labels = _random_mps(case["k_act"], case["k_virt"], case["k_act"], case["M"], rng, i)
        st["h"] = _Handle(ctx, L.mpspt_mps_import(ctx, tensors, labels))
        if kind == "local":
            st["shape"] = (len(labels[i]), 4, 4, len(labels[i + 2]))
            st["x"] = rng.normal(size=st["shape"])
        return st
    opts = {"prec": L.PREC[case["prec"]], "max_sweeps": case["sweeps"], "e_tol": 1e-14}
    if kind == "partitions" or case["tuned"]:
        opts["autotune"] = 1
    if kind == "partitions":
        opts["cuda_graphs"] = 1
    ctx, ci = _context(case, seed, case["k_virt"], **opts)
    L.mpspt_set_reference_ci(ctx, ci)
    st["h"] = _Handle(ctx)
    if kind == "partitions":
        kv = case["k_virt"]
        pairs = [(a, b) for a in range(kv) for b in range(a, kv)]
        at = rng.choice(len(pairs), size=min(case["parts"], len(pairs)), replace=False)
        st["pairs"] = [pairs[p] for p in sorted(at)]
        st["M"] = [max(4, int(case["M"] * (1.0 - 0.06 * q))) for q in range(len(st["pairs"]))]   # uneven
    return st


class _Net:
    def __init__(self, params):
        self.h = L.mpspt_mlp_create()
        L.mpspt_mlp_set_params(self.h, params)

    def __del__(self):
        L.mpspt_mlp_free(self.h)


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "eigh":
        call = {"noalloc": L.mpspt_eigh_batched_noalloc, "batched": L.mpspt_eigh_batched,
                "fp64": L.mpspt_eigh_batched_ex, "mixed": L.mpspt_eigh_batched_ex}[case["entry"]]
        extra = {"fp64": (0,), "mixed": (1,)}.get(case["entry"], ())
        n = st["n"]
        call(0, torch.cuda.current_stream().cuda_stream, n, st["A"].data_ptr(), st["V"].data_ptr(),
             st["w"].data_ptr(), *extra)
        if not case["ragged"]:
            return _in_order(st["w"].view(len(n), n[0]), st["V"].view(len(n), n[0], n[0]))
        return [_in_order(w, V.view(m, m)) for m, w, V in
                zip(n, torch.split(st["w"], n), torch.split(st["V"], [m * m for m in n]))]
    if kind == "mlp":
        if case["pass"] == "forward":
            return L.mpspt_mlp_forward(st["net"].h, st["x"])
        return L.mpspt_mlp_gradient(st["net"].h, st["x"], st["t"])
    ctx = st["h"].ctx
    if kind == "local":
        op = {"sigma": L.MPSPT_LOCAL_SIGMA, "rhs": L.MPSPT_LOCAL_RHS, "diag": L.MPSPT_LOCAL_DIAG}[case["op"]]
        return L.mpspt_local_apply(ctx, case["h0"], st["h"].psi, case["bond"], op,
                                   st["x"] if case["op"] == "sigma" else None, st["shape"])
    if kind == "e3":
        return L.mpspt_third_order(ctx, case["h0"], st["h"].psi)
    if kind == "partitions":
        total, each, _ = L.mpspt_minimize_partitioned(ctx, case["h0"], st["pairs"], st["M"])
        return total, each
    if kind == "dmrg":
        e_ref, _, rep = L.mpspt_ground_state(ctx, case["M"], 1.0)
        return e_ref, np.array(rep.e2_per_sweep[: rep.n_sweeps])
    e2, psi, rep = L.mpspt_minimize_hylleraas(ctx, case["h0"], case["M"])
    out = [e2, np.array(rep.e2_per_sweep[: rep.n_sweeps])]
    if case["e3"]:
        out.append(L.mpspt_third_order(ctx, case["h0"], psi))
    L.mpspt_mps_free(psi)
    return out


def _mps_values(secs):
    """(entries of all site tensors, flops of one two-site operator application per bond, summed)."""
    vals = two = 0
    for c in range(len(secs) - 1):
        for q, d in secs[c].items():
            for s in QSITE:
                vals += d * secs[c + 1].get((q[0] + s[0], q[1] + s[1]), 0)
    for c in range(len(secs) - 2):
        for q, d in secs[c].items():
            for s in QSITE:
                for t in QSITE:
                    e = secs[c + 2].get((q[0] + s[0] + t[0], q[1] + s[1] + t[1]), 0)
                    two += 2 * d * e * (d + e)      # one left and one right operator block at the least
    return vals, two


def work(case):
    kind = case["kind"]
    if kind == "eigh":
        n = _sizes(case)
        return {"bytes": 8 * sum(2 * m * m + m for m in n), "flops": 9 * sum(m ** 3 for m in n)}
    if kind == "mlp":
        b, w = case["batch"], 256
        mac = b * (16 * w + w * w + 2 * w)
        params = 16 * w + w * w + 2 * w + 2 * w + 2
        if case["pass"] == "forward":
            return {"bytes": 4 * b * 18 + 2 * params, "flops": 2 * mac}
        return {"bytes": 4 * b * 18 + 6 * params, "flops": 2 * (mac * 3 - b * 16 * w)}
    ne, ka = case["k_act"], case["k_act"]
    kv = 0 if kind == "dmrg" else case["k_virt"]
    nq = _active(ka)[1].shape[0]
    ints = 8 * (ka + kv) ** 2 * (1 + nq)
    if kind == "dmrg":
        secs = _sectors(ka, 0, ne, case["M"])
        vals, two = _mps_values(secs)
        return {"bytes": ints + 8 * vals, "flops": 2 * case["sweeps"] * two}
    if kind == "partitions":
        vals = two = 0
        for q in range(min(case["parts"], kv * (kv + 1) // 2)):
            v, t = _mps_values(_sectors(ka, 2, ne, max(4, int(case["M"] * (1.0 - 0.06 * q)))))
            vals, two = vals + v, two + t
        return {"bytes": ints + 8 * vals, "flops": 2 * case["sweeps"] * two}
    secs = _sectors(ka, kv, ne, case["M"])
    vals, two = _mps_values(secs)
    if kind == "local":
        i = case["bond"]
        n = 16 * sum(secs[i].values()) * sum(secs[i + 2].values())
        return {"bytes": 8 * (vals + (2 if case["op"] == "sigma" else 1) * n), "flops": two}
    if kind == "e3":
        return {"bytes": 8 * vals, "flops": 3 * two}
    return {"bytes": ints + 8 * vals, "flops": 2 * case["sweeps"] * two}


# ------------------------------------------------- in 64 bits, by plain torch
def exact(case, seed):
    """Eigenpairs and the network's passes in 64 bits; the sweeps' energies
    after a set number of sweeps depend on the sweep itself, and the local
    operators and E3 would need a second implementation of the operators:
    those have none here."""
    if case["kind"] == "eigh":
        mats = _density_matrices(case, seed)
        if not case["ragged"]:
            return _in_order(*torch.linalg.eigh(torch.stack(mats).cpu()))
        return [_in_order(*torch.linalg.eigh(m.cpu())) for m in mats]
    if case["kind"] == "mlp":
        st = prepare(case, seed)
        p = st["p"]
        x, t = torch.from_numpy(st["x"]).double(), torch.from_numpy(st["t"]).double()
        W = [torch.from_numpy(p[k]).bfloat16().double() for k in ("W1", "W2", "W3")]
        b = [torch.from_numpy(p[k]).double() for k in ("b1", "b2", "b3")]
        h1 = torch.relu(x @ W[0].T + b[0])
        h2 = torch.relu(h1 @ W[1].T + b[1])
        y = h2 @ W[2].T + b[2]
        if case["pass"] == "forward":
            return y
        B = x.shape[0]
        dy = (y - t) / B
        d2 = (dy @ W[2]) * (h2 > 0)
        d1 = (d2 @ W[1]) * (h1 > 0)
        g = {"W1": d1.T @ x, "b1": d1.sum(0), "W2": d2.T @ h1, "b2": d2.sum(0), "W3": dy.T @ h2, "b3": dy.sum(0)}
        return float(0.5 * ((y - t) ** 2).sum() / B), g
    return None
