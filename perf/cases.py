"""The work that a user has this package do, as cases that can be timed.

Every case goes through the package's public entry points (``Propagator``,
``BatchPropagator``, ``autograd.thermal_coefficients``).  The Hamiltonians are the
transverse-field Ising chains and lattices of the paper, built here from numpy
arrays; the seed draws their fields (and, for disordered ones, every field and
coupling), so another seed is another problem of the same size.

Sizes: the smallest chain is a whole thermal run of some thousand terms, where every
gate is a handful of microseconds of kernels; the largest holds 2^25 terms (0.8 GB of
state, several times the L2 cache).
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2601_14400_gb300 as itpp
from paper_2601_14400_gb300.autograd import thermal_coefficients


def listed():
    return [
        # A thermal run of a small chain to beta = 1 with the coefficient threshold
        # alone (the bound is never met).  About 12 thousand terms: launches and
        # latency.
        dict(name="chain_n8", kind="chain", n=8, periodic=False, dtau=0.05, layers=20,
             delta=1e-8, cap=1 << 16, policy=0, field=1.0, disorder=0.0, order=1,
             max_weight=0, out="correlators", term_gates=2.54e6),
        # One point of a fixed-K scan (K-truncation proper: no threshold, the K
        # largest coefficients after every gate): 12 layers, beta = 0.24; the
        # state read out whole.
        dict(name="ktrunc_n24_2e13", kind="chain", n=24, periodic=False, dtau=0.02,
             layers=12, delta=0.0, cap=1 << 13, policy=1, field=0.5, disorder=0.0,
             order=1, max_weight=0, out="state", term_gates=4.52e6),
        # A production-style run at a bound that fits the L2 cache: the uniform
        # critical chain, whose symmetries make many exactly equal coefficients
        # (the bound's tie rule works for its living); all <X_i>, <Z_i Z_j>.
        dict(name="chain_n64_2e18", kind="chain", n=64, periodic=True, dtau=0.01,
             layers=14, delta=1e-6, cap=1 << 18, policy=1, field=1.0, disorder=0.0,
             order=1, max_weight=0, out="correlators", term_gates=4.23e8),
        # The symmetric product formula with a Pauli weight cutoff on a
        # disordered chain, a bound in between.
        dict(name="strang_n48_2e20", kind="chain", n=48, periodic=False, dtau=0.04,
             layers=4, delta=1e-6, cap=1 << 20, policy=1, field=1.0, disorder=0.2,
             order=2, max_weight=9, out="correlators", term_gates=6.43e8),
        # The benchmark chain at half its bound: growth from the identity, then
        # layers at the bound, far beyond the caches.
        dict(name="chain_n64_2e25", kind="chain", n=64, periodic=True, dtau=0.01,
             layers=13, delta=1e-6, cap=1 << 25, policy=1, field=1.0, disorder=0.0,
             order=1, max_weight=0, out="correlators", term_gates=1.81e10),
        # The 11 x 11 lattice (two mask words) at a smaller bound.
        dict(name="lattice_11x11_2e22", kind="lattice", L=11, dtau=0.02, layers=3,
             delta=1e-5, cap=1 << 22, policy=1, field=3.04, disorder=0.0,
             out="correlators", term_gates=3.15e9),
        # A field sweep: 64 open chains of 16 to 64 sites advanced together, a
        # handle made, run and read for each sweep.
        dict(name="batch_64_2e16", kind="batch", B=64, n_min=16, n_max=64, dtau=0.02,
             layers=6, delta=1e-7, cap=1 << 16, policy=1),
        # A parameter sweep of a few small chains, where a gate of the whole
        # batch is a few thousand terms.
        dict(name="batch_12_2e12", kind="batch", B=12, n_min=9, n_max=20, dtau=0.05,
             layers=10, delta=1e-6, cap=1 << 12, policy=1),
        # Forward and backward of an energy through autograd: 63 parameters of a
        # disordered chain.
        dict(name="gradient_n32_2e18", kind="gradient", n=32, dtau=0.02, layers=10,
             delta=1e-7, cap=1 << 18, policy=1, disorder=0.2),
        # The energy of the squared (positive) state, read from a state at hand.
        dict(name="psd_n32_2e18", kind="psd", n=32, dtau=0.02, layers=8, delta=1e-7,
             cap=1 << 18),
        # Coefficients of a list of strings read from a large state at hand.
        dict(name="read_n64_2e22", kind="read", n=64, terms=1 << 22, m=2080),
        # A state taken from the host (a checkpoint, another program), one
        # Trotter layer of a two-word chain on it, and the state back in the
        # canonical order.
        dict(name="resume_n121_2e16", kind="resume", n=121, terms=1 << 16, dtau=0.02,
             delta=1e-6, cap=1 << 16),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["small", "ktrunc", "chain", "chain", "strang", "lattice", "batch",
                       "batch", "gradient", "psd", "read", "resume"])
    if kind == "small":
        n = rng.randint(6, 9)
        return dict(kind="chain", n=n, periodic=rng.random() < 0.5, dtau=0.05,
                    layers=rng.randint(8, 30), delta=10.0 ** rng.uniform(-9, -6),
                    cap=1 << 16, policy=0, field=rng.uniform(0.5, 1.5),
                    disorder=rng.choice([0.0, 0.2]), order=1, max_weight=0, out="correlators")
    if kind == "ktrunc":
        return dict(kind="chain", n=rng.randint(12, 48), periodic=False, dtau=0.02,
                    layers=rng.randint(4, 12), delta=0.0, cap=_log_int(rng, 1 << 9, 1 << 16),
                    policy=1, field=0.5, disorder=0.0, order=1, max_weight=0, out="state")
    if kind == "chain":
        cap = _log_int(rng, 1 << 12, 1 << 24)
        return dict(kind="chain", n=rng.randint(20, 64), periodic=rng.random() < 0.7,
                    dtau=rng.choice([0.01, 0.02]), layers=rng.randint(8, 13),
                    delta=10.0 ** rng.uniform(-7, -5.5), cap=cap, policy=1,
                    field=rng.uniform(0.6, 1.4), disorder=rng.choice([0.0, 0.2]), order=1,
                    max_weight=0, out="correlators")
    if kind == "strang":
        return dict(kind="chain", n=rng.randint(24, 64), periodic=False, dtau=0.04,
                    layers=rng.randint(2, 4), delta=10.0 ** rng.uniform(-7, -5),
                    cap=_log_int(rng, 1 << 14, 1 << 21), policy=1,
                    field=rng.uniform(0.6, 1.4), disorder=rng.choice([0.0, 0.2]), order=2,
                    max_weight=rng.choice([0, rng.randint(6, 12)]), out="correlators")
    if kind == "lattice":
        return dict(kind="lattice", L=rng.randint(5, 11), dtau=0.02, layers=rng.randint(2, 3),
                    delta=1e-5, cap=_log_int(rng, 1 << 14, 1 << 22), policy=1,
                    field=rng.uniform(2.0, 4.0), disorder=0.0, out="correlators")
    if kind == "batch":
        lo = rng.randint(9, 30)
        return dict(kind="batch", B=_log_int(rng, 4, 64), n_min=lo, n_max=rng.randint(lo, 64),
                    dtau=0.02, layers=rng.randint(3, 6), delta=1e-7,
                    cap=_log_int(rng, 1 << 11, 1 << 16), policy=1)
    if kind == "gradient":
        return dict(kind="gradient", n=rng.randint(12, 40), dtau=0.02,
                    layers=rng.randint(4, 10), delta=1e-7, cap=_log_int(rng, 1 << 12, 1 << 18),
                    policy=1, disorder=0.2)
    if kind == "psd":
        return dict(kind="psd", n=rng.randint(16, 64), dtau=0.02, layers=rng.randint(4, 8),
                    delta=1e-7, cap=_log_int(rng, 1 << 12, 1 << 18))
    if kind == "read":
        return dict(kind="read", n=rng.choice([48, 64, 100, 128]),
                    terms=_log_int(rng, 1 << 12, 1 << 22), m=_log_int(rng, 1, 4096))
    return dict(kind="resume", n=rng.choice([40, 64, 90, 121]),
                terms=(t := _log_int(rng, 1 << 10, 1 << 17)), dtau=0.02, delta=1e-6, cap=t)


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
class _Strings:
    """Pauli strings as (x, z) rows of 64-bit words, with weights."""

    def __init__(self, n, letters, w):
        W = (n + 63) // 64
        self.n = n
        self.x = np.zeros((len(letters), W), dtype=np.uint64)
        self.z = np.zeros((len(letters), W), dtype=np.uint64)
        self.w = np.asarray(w, dtype=np.float64)
        for j, string in enumerate(letters):
            for site, letter in string:
                bit = np.uint64(1 << (site % 64))
                if letter in "XY":
                    self.x[j, site // 64] |= bit
                if letter in "ZY":
                    self.z[j, site // 64] |= bit


class _Ham:
    """A Hamiltonian as the package takes it: gates in Trotter order."""

    def __init__(self, n, bonds, J, h):
        s = _Strings(n, [((a, "Z"), (b, "Z")) for a, b in bonds] + [((i, "X"),) for i in range(n)],
                     np.concatenate([-J, -h]))
        self.n, self.gate_x, self.gate_z, self.alpha = n, s.x, s.z, s.w
        self.n_gates = len(s.w)
        self.energy = s


def _fields(rng, case, n_bonds, n):
    """Couplings and fields: uniform ones (the field moved a little by the
    seed), or every one of them drawn."""
    d = case.get("disorder", 0.0)
    f = case.get("field", 1.0)
    if d:
        return rng.uniform(1 - d, 1 + d, n_bonds), f * rng.uniform(1 - d, 1 + d, n)
    return np.ones(n_bonds), np.full(n, f * (1.0 + 0.02 * rng.uniform(-1, 1)))


def _hamiltonian(case, seed):
    rng = np.random.default_rng([seed, 5])
    if case["kind"] == "lattice":
        L = case["L"]
        n = L * L
        bonds = [(r * L + c, r * L + c + 1) for r in range(L) for c in range(L - 1)]
        bonds += [(r * L + c, (r + 1) * L + c) for r in range(L - 1) for c in range(L)]
    else:
        n = case["n"]
        bonds = [(i, i + 1) for i in range(n - 1)]
        if case.get("periodic"):
            bonds.append((n - 1, 0))
    J, h = _fields(rng, case, len(bonds), n)
    return _Ham(n, bonds, J, h)


def _sizes(case):
    """Sites of the instances of a batch, spread evenly over its range."""
    B, lo, hi = case["B"], case["n_min"], case["n_max"]
    return [lo + (hi - lo) * b // max(1, B - 1) for b in range(B)]


def _batch_hamiltonians(case, seed):
    rng = np.random.default_rng([seed, 6])
    hams = []
    for n in _sizes(case):
        hams.append(_Ham(n, [(i, i + 1) for i in range(n - 1)], np.ones(n - 1),
                         np.full(n, rng.uniform(0.5, 2.0))))
    return hams


def _correlators(n):
    """All <X_i> and <Z_i Z_j>."""
    return _Strings(n, [((i, "X"),) for i in range(n)] +
                    [((i, "Z"), (j, "Z")) for i in range(n) for j in range(i + 1, n)],
                    np.ones(n + n * (n - 1) // 2))


def _random_terms(n, count, seed):
    """`count` distinct random strings, the identity first; log-uniform
    magnitudes down to 1e-6."""
    rng = np.random.default_rng([seed, 7])
    W = (n + 63) // 64
    top = np.full(W, ~np.uint64(0))
    if n % 64:
        top[-1] = np.uint64((1 << (n % 64)) - 1)
    x = rng.integers(0, 1 << 64, (count, W), dtype=np.uint64) & top
    z = rng.integers(0, 1 << 64, (count, W), dtype=np.uint64) & top
    # the row number in the low bits of x: no string twice
    x[:, 0] = (x[:, 0] & ~np.uint64((1 << 23) - 1)) | np.arange(count, dtype=np.uint64)
    x[0], z[0] = 0, 0
    c = np.exp(rng.uniform(math.log(1e-6), 0.0, count)) * rng.choice([-1.0, 1.0], count)
    c[0] = 1.0
    return x, z, c


def _new_propagator(case, H, stream, cap=None):
    return itpp.Propagator(H.n, H.gate_x, H.gate_z, H.alpha, case.get("dtau", 0.02),
                           case.get("delta", 0.0), cap or case["cap"], case.get("policy", 1),
                           stream=stream, max_weight=case.get("max_weight", 0),
                           trotter_order=case.get("order", 1))


def prepare(case, seed):
    stream = torch.cuda.Stream()
    s = dict(case=case, stream=stream)
    kind = case["kind"]
    if kind == "batch":
        # a batch handle has no reset: a sweep makes its own (see run)
        s["hams"] = _batch_hamiltonians(case, seed)
        s["obs"] = [H.energy for H in s["hams"]]
        return s
    if kind == "read":
        H = _Ham(case["n"], [], np.zeros(0), np.ones(case["n"]))
        s["prop"] = _new_propagator(case, H, stream, cap=case["terms"])
        x, z, c = _random_terms(case["n"], case["terms"], seed)
        s["prop"].set_terms(x, z, c)
        # half of the strings asked for are there, half are not
        rng = np.random.default_rng([seed, 8])
        at = rng.integers(0, case["terms"], case["m"])
        s["ox"], s["oz"] = x[at].copy(), z[at].copy()
        s["oz"][::2, 0] ^= np.uint64(2)
        return s
    H = _hamiltonian(case, seed)
    s["prop"] = _new_propagator(case, H, stream)
    if kind == "resume":
        s["terms"] = _random_terms(case["n"], case["terms"], seed)
    elif kind == "gradient":
        s["alpha"] = torch.tensor(H.alpha, dtype=torch.float64, requires_grad=True)
        s["ham"] = H
    elif kind == "psd":
        s["prop"].apply_trotter_layer(case["layers"])
        s["energy"] = H.energy
    elif case["out"] == "correlators":
        s["obs"] = _correlators(H.n)
    return s


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------
def run(s):
    case, kind = s["case"], s["case"]["kind"]
    if kind == "batch":
        with torch.cuda.stream(s["stream"]):
            bp = itpp.BatchPropagator(s["hams"], case["dtau"], case["delta"], case["cap"],
                                      case["policy"])
            bp.apply_trotter_layer(case["layers"])
            counts, status = bp.counts()
            energies = [bp.expect(b, o) for b, o in enumerate(s["obs"])]
            bp.close()
        return {"counts": counts, "status": status, "energies": np.array(energies)}
    p = s["prop"]
    if kind == "read":
        return p.coeffs(s["ox"], s["oz"])
    if kind == "psd":
        return np.array(p.expect_psd(s["energy"]))
    if kind == "gradient":
        a, H = s["alpha"], s["ham"]
        a.grad = None
        c = thermal_coefficients(a, p, case["layers"], H.gate_x, H.gate_z)
        energy = (a * c).sum()
        energy.backward()
        return {"energy": energy.detach(), "coefficients": c.detach(), "gradient": a.grad}
    if kind == "resume":
        p.set_terms(*s["terms"])
        p.apply_trotter_layer(1)
        x, z, c = p.sorted_terms()
        return {"x": x.view(np.int64), "z": z.view(np.int64), "c": c}
    p.reset()
    p.apply_trotter_layer(case["layers"])
    if case["out"] == "state":
        x, z, c = p.sorted_terms()
        return {"x": x.view(np.int64), "z": z.view(np.int64), "c": c}
    return {"count": p.count(), "correlators": p.coeffs(s["obs"].x, s["obs"].z)}


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------
def _term_gates(case, n, gates):
    """Terms that the gates of a run from the identity read, summed: counted
    for the listed runs (the default field); otherwise the support reaches
    about 2 n^2 strings in the first layer, grows about eightfold per layer
    until it meets the bound, and stays there."""
    if "term_gates" in case:
        return case["term_gates"]
    most = min(float(case["cap"]), float(math.comb(2 * n, n)))
    size, total = 1.0, 0.0
    for layer in range(case["layers"]):
        end = min(most, 2.0 * n * n if layer == 0 else size * 8.0)
        total += gates * 0.5 * (size + end)
        size = end
    return total


def work(case):
    kind = case["kind"]
    if kind == "read":
        b = 16 * ((case["n"] + 63) // 64)
        return {"bytes": case["terms"] * b + case["m"] * (2 * b + 16), "flops": 0}
    if kind == "psd":
        W = (case["n"] + 63) // 64
        t = min(case["cap"], math.comb(2 * case["n"], case["n"]))
        g = 2 * case["n"] - 1
        return {"bytes": t * (16 * W + 8), "flops": 3.0 * t * g}
    if kind == "batch":
        tg = sum(_term_gates(case, n, 2 * n - 1) for n in _sizes(case))
        return {"bytes": 2 * tg * 24, "flops": 3.0 * tg}
    if kind == "lattice":
        n = case["L"] ** 2
        gates = 2 * case["L"] * (case["L"] - 1) + n
    else:
        n = case["n"]
        gates = (2 * n if case.get("periodic") else 2 * n - 1)
        if case.get("order", 1) == 2:
            gates = 2 * gates - 1
    term = 16 * ((n + 63) // 64) + 8
    if kind == "resume":
        tg = gates * case["terms"]
        return {"bytes": 2 * tg * term + 4 * case["terms"] * term, "flops": 3.0 * tg}
    tg = _term_gates(case, n, gates)
    if kind == "gradient":
        # forward, and the backward sweep through every gate
        return {"bytes": 4 * tg * term, "flops": 9.0 * tg}
    return {"bytes": 2 * tg * term, "flops": 3.0 * tg}


# ---------------------------------------------------------------------------
# The same results in plain torch, 64 bits
# ---------------------------------------------------------------------------
_TOP = -(1 << 63)


def _i64(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.uint64).view(np.int64))


def _lex_order(keys):
    """Ascending order of the rows, columns compared as unsigned words."""
    idx = torch.arange(keys.shape[0], device=keys.device)
    for j in reversed(range(keys.shape[1])):
        idx = idx[torch.argsort(keys[idx, j] ^ _TOP, stable=True)]
    return idx


def _parity(v):
    for sh in (32, 16, 8, 4, 2, 1):
        v = v ^ (v >> sh)
    return (v & 1).bool()


def _weight(v):
    total = torch.zeros_like(v)
    for i in range(64):
        total += (v >> i) & 1
    return total


def _commute_and_sign(K, q, W):
    """Whether each row commutes with q, and the sign s of q P = s R."""
    par = torch.zeros(K.shape[0], dtype=torch.bool, device=K.device)
    e = torch.zeros(K.shape[0], dtype=torch.int64, device=K.device)
    for w in range(W):
        qx, qz = int(q[w]), int(q[W + w])
        par ^= _parity((K[:, w] & qz) ^ (K[:, W + w] & qx))
        for i in range(64):
            bx, bz = (qx >> i) & 1, (qz >> i) & 1
            if bx | bz:
                px, pz = (K[:, w] >> i) & 1, (K[:, W + w] >> i) & 1
                e += bx * bz + px * pz - (px ^ bx) * (pz ^ bz) + 2 * bz * px
    return ~par, torch.where((e & 3) == 2, -1.0, 1.0).to(torch.float64)


def _rows_equal(a, b):
    return (a == b).all(dim=1)


def _propagate(K, c, gates, theta, delta, cap, max_weight):
    """The gates on the state (rows K ascending, the identity first)."""
    W = K.shape[1] // 2
    for q, th in zip(gates, theta):
        comm, sign = _commute_and_sign(K, q.tolist(), W)
        ch, sh = (torch.cosh(th), torch.sinh(th)) if torch.is_tensor(th) else \
            (math.cosh(th), math.sinh(th))
        at = comm.nonzero().squeeze(1)
        keys = torch.cat([K, K[at] ^ q])
        vals = torch.cat([torch.where(comm, c * ch, c), c[at] * (sign[at] * -sh)])
        idx = _lex_order(keys)
        keys = keys[idx]
        new = torch.ones(keys.shape[0], dtype=torch.bool, device=K.device)
        new[1:] = ~_rows_equal(keys[1:], keys[:-1])
        group = torch.cumsum(new, 0) - 1
        keys = keys[new]
        out = torch.zeros(keys.shape[0], dtype=torch.float64, device=K.device)
        out = out.index_add(0, group, vals[idx])
        mag = out.detach().abs()
        keep = mag > delta
        if max_weight:
            wt = sum(_weight(keys[:, w] | keys[:, W + w]) for w in range(W))
            keep &= wt <= max_weight
        keep = keep.nonzero().squeeze(1)
        if keep.shape[0] > cap:
            # the largest, equal ones by ascending key
            order = torch.argsort(mag[keep], descending=True, stable=True)
            keep = keep[order[:cap].sort().values]
        K, out = keys[keep], out[keep]
        c = torch.cat([torch.ones(1, dtype=torch.float64, device=K.device),
                       out[1:] * (1.0 / out[0])])
    return K, c


def _schedule(H, case, device, alpha=None):
    G = H.n_gates
    if case.get("order", 1) == 2 and G > 1:
        at = list(range(G)) + list(range(G - 2, -1, -1))
        scale = [0.5] * (G - 1) + [1.0] + [0.5] * (G - 1)
    else:
        at, scale = list(range(G)), [1.0] * G
    q = torch.cat([_i64(H.gate_x), _i64(H.gate_z)], dim=1).to(device)
    a = H.alpha if alpha is None else alpha
    return [q[k] for k in at], [a[k] * f * case["dtau"] for k, f in zip(at, scale)]


def _thermal(H, case, device, layers, alpha=None):
    W = H.gate_x.shape[1]
    gates, theta = _schedule(H, case, device, alpha)
    if alpha is None:
        theta = [float(t) for t in theta]
    K = torch.zeros((1, 2 * W), dtype=torch.int64, device=device)
    c = torch.ones(1, dtype=torch.float64, device=device)
    # a run without a bound that acts (policy 0) never meets it
    for _ in range(layers):
        K, c = _propagate(K, c, gates, theta, case["delta"], case["cap"],
                          case.get("max_weight", 0))
    return K, c


def _lookup(K, c, ox, oz):
    """c of the strings asked for, zero where absent."""
    want = torch.cat([_i64(ox), _i64(oz)], dim=1).to(K.device)
    m = want.shape[0]
    keys = torch.cat([K, want])
    idx = _lex_order(keys)
    keys = keys[idx]
    new = torch.ones(keys.shape[0], dtype=torch.bool, device=K.device)
    new[1:] = ~_rows_equal(keys[1:], keys[:-1])
    group = torch.empty_like(idx)
    group[idx] = torch.cumsum(new, 0) - 1
    vals = torch.zeros(int(new.sum()), dtype=torch.float64, device=K.device)
    vals = vals.index_add(0, group[: K.shape[0]], c)
    return vals[group[K.shape[0]:][:m]]


def _state_arrays(K, c):
    W = K.shape[1] // 2
    K = K.cpu().numpy()
    return {"x": np.ascontiguousarray(K[:, :W]), "z": np.ascontiguousarray(K[:, W:]),
            "c": c.cpu().numpy()}


def exact(case, seed):
    device = "cuda" if torch.cuda.is_available() else "cpu"
    kind = case["kind"]
    if kind == "read":
        x, z, c = _random_terms(case["n"], case["terms"], seed)
        rng = np.random.default_rng([seed, 8])
        at = rng.integers(0, case["terms"], case["m"])
        ox, oz = x[at].copy(), z[at].copy()
        oz[::2, 0] ^= np.uint64(2)
        K = torch.cat([_i64(x), _i64(z)], dim=1).to(device)
        return _lookup(K, torch.from_numpy(c).to(device), ox, oz).cpu().numpy()
    # propagations whose sorted merges would take too long
    per_gate = 2e-3 + 3e-8 * case["cap"]
    if kind == "batch":
        gates = sum(2 * n - 1 for n in _sizes(case)) * case["layers"]
        if gates * per_gate > 18:
            return None
        energies, counts = [], []
        for H in _batch_hamiltonians(case, seed):
            K, c = _thermal(H, case, device, case["layers"])
            o = H.energy
            w = torch.from_numpy(o.w).to(device)
            energies.append(float((w * _lookup(K, c, o.x, o.z)).sum()))
            counts.append(K.shape[0])
        return {"counts": np.array(counts), "status": np.zeros(case["B"], dtype=np.int32),
                "energies": np.array(energies)}
    H = _hamiltonian(case, seed)
    gates = H.n_gates * case.get("order", 1)
    if gates * case.get("layers", 1) * per_gate > 18:
        return None
    if kind == "resume":
        x, z, c = _random_terms(case["n"], case["terms"], seed)
        K = torch.cat([_i64(x), _i64(z)], dim=1).to(device)
        order = _lex_order(K)
        g, theta = _schedule(H, case, device)
        K, c = _propagate(K[order], torch.from_numpy(c).to(device)[order], g,
                          [float(t) for t in theta], case["delta"], case["cap"], 0)
        return _state_arrays(K, c)
    if kind == "gradient":
        a = torch.tensor(H.alpha, dtype=torch.float64, device=device, requires_grad=True)
        K, c = _thermal(H, case, device, case["layers"], alpha=a)
        co = _lookup(K, c, H.gate_x, H.gate_z)
        energy = (a * co).sum()
        energy.backward()
        return {"energy": energy.detach().cpu(), "coefficients": co.detach().cpu(),
                "gradient": a.grad.cpu()}
    K, c = _thermal(H, case, device, case["layers"])
    if kind == "psd":
        W = K.shape[1] // 2
        purity = float((c * c).sum())
        total = 0.0
        q = torch.cat([_i64(H.gate_x), _i64(H.gate_z)], dim=1).to(device)
        for j in range(H.n_gates):
            comm, sign = _commute_and_sign(K, q[j].tolist(), W)
            at = comm.nonzero().squeeze(1)
            R = (K[at] ^ q[j]).cpu().numpy().view(np.uint64)
            other = _lookup(K, c, R[:, :W], R[:, W:])
            total += float(H.alpha[j]) * float((sign[at] * c[at] * other).sum())
        return np.array([total / purity, total, purity])
    if case["out"] == "state":
        return _state_arrays(K, c)
    o = _correlators(H.n)
    return {"count": K.shape[0], "correlators": _lookup(K, c, o.x, o.z).cpu().numpy()}
