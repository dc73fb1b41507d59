"""The kernels behind one gate, at the sizes where they change their way.

A bound up to 2^20 terms runs a layer in one launch (teams of CTAs, in-place
merge, candidates selected by one CTA); with per-kernel timing on, or above
that bound, every gate is a chain of separate launches.  Both must give the
oracle's state bit for bit: strings, coefficients and the kept set at the
top-M bound, ties going by ascending key.
"""
import math

import numpy as np
import pytest

import oracle
import workloads as wl
from tests._compare import assert_same_state, sort_terms

pytestmark = pytest.mark.gpu

itpp = pytest.importorskip("paper_2601_14400_gb300")


def _pair(H, dtau, delta, cap, policy, separate, **kw):
    g = itpp.Propagator(H.n, H.gate_x, H.gate_z, H.alpha, dtau, delta, cap, policy, **kw)
    if separate:
        g.profile_enable(True)
    return g, oracle.Oracle(H.n, H.gate_x, H.gate_z, H.alpha, dtau, delta, cap, policy)


# (without a threshold the first layer's bound lies octaves below the second's:
# the limit predicted from it may lie above the identity)
# bounds beside the smallest partition (128 strings), a pass's capacity (512
# and 1,024), what one CTA selects among (4,096) and its list in shared memory
@pytest.mark.parametrize("separate", [False, True])
@pytest.mark.parametrize("cap", [2, 127, 129, 513, 1023, 1025, 4095, 4097, 30011])
def test_bounds_beside_the_kernels_sizes(cap, separate):
    H = wl.tfim_1d(24, 1.0, 1.1, periodic=True)      # uniform: classes of equal |c|
    g, o = _pair(H, 0.05, 0.0 if cap < 1024 else 1e-9, cap, 1, separate)
    for layer in range(4):
        g.apply_trotter_layer(1)
        o.apply_layers(1)
        assert_same_state(g.terms(), o.terms(), f"cap {cap} layer {layer}")


# few sites: the windows do not fit and gates go by their pair key; with a
# large target every partition is longer than a pass.  Couplings that drop make
# gates keep fewer than the bound, which merges them again in full.
@pytest.mark.parametrize("n,target", [(6, 0), (9, 0), (9, 2048), (12, 64), (12, 2048)])
def test_dense_states_and_merges_in_full(n, target):
    H = wl.tfim_1d(n, 1.0, 0.9, periodic=True)
    kw = {"partition_target": target} if target else {}
    cap = 1500 if n == 9 else 3000
    g, o = _pair(H, 0.1, 1e-9, cap, 1, False, **kw)
    h, _ = _pair(H, 0.1, 1e-9, cap, 1, True, **kw)
    for layer in range(6):
        if layer == 3:
            for p in (g, h):
                p.set_alpha(np.asarray(H.alpha) * 0.2)
        g.apply_trotter_layer(1)
        h.apply_trotter_layer(1)
        if layer < 3:
            o.apply_layers(1)
            assert_same_state(g.terms(), o.terms(), f"n {n} layer {layer}")
        assert_same_state(g.terms(), sort_terms(*h.terms()), f"n {n} layer {layer}, both paths")
    if n > 6:
        assert h.stats()["merge_retries"] > 0


# one layer in one launch at its largest bound, against separate launches
def test_largest_bound_of_one_launch():
    H = wl.tfim_2d(9, 1.0, 3.04)                      # 81 sites: two words
    a = itpp.Propagator(H.n, H.gate_x, H.gate_z, H.alpha, 0.02, 1e-5, 1 << 20, 1)
    b = itpp.Propagator(H.n, H.gate_x, H.gate_z, H.alpha, 0.02, 1e-5, 1 << 20, 1)
    b.profile_enable(True)
    for p in (a, b):
        p.apply_trotter_layer(2)
    assert a.count() == 1 << 20
    assert_same_state(a.terms(), sort_terms(*b.terms()), "2^20 terms")


# The identity as a gate, a wide gate (its own window) and a weight cutoff.
@pytest.mark.parametrize("separate", [False, True])
@pytest.mark.parametrize("n,max_weight", [(20, 0), (20, 3), (70, 0), (70, 4)])
def test_wide_and_identity_gates_and_weights(n, max_weight, separate):
    H = wl.random_pauli_hamiltonian(n, 10, 7, max_weight=12 if n > 60 else 9)
    H.gate_x[4] = 0
    H.gate_z[4] = 0
    kw = {"max_weight": max_weight} if max_weight else {}
    g, o = _pair(H, 0.2, 1e-6, 700, 1, separate, **kw)
    if max_weight:
        o = oracle.Oracle(H.n, H.gate_x, H.gate_z, H.alpha, 0.2, 1e-6, 700, 1,
                          max_weight=max_weight)
    for layer in range(3):
        g.apply_trotter_layer(1)
        o.apply_layers(1)
        assert_same_state(g.terms(), o.terms(), f"n {n} layer {layer}")


# Equal magnitudes by the thousand: one gate whose cosh and sinh are the same
# number doubles a state of M strings, and the bound keeps M of the 2 M
# children; with one class of magnitudes all of them tie and the keys decide.
@pytest.mark.parametrize("separate", [False, True])
@pytest.mark.parametrize("classes", [1, 3])
@pytest.mark.parametrize("n,M", [(40, 100), (40, 700), (40, 2100), (40, 9000), (80, 300),
                                 (80, 2100), (80, 9000)])
def test_ties_by_key(n, M, classes, separate):
    W = (n + 63) // 64
    rng = np.random.default_rng([n, M])
    sites = n - 1                                     # the last site stays the identity
    x = np.zeros((2 * M, W), dtype=np.uint64)
    z = np.zeros((2 * M, W), dtype=np.uint64)
    for a in (x, z):
        for w in range(W):
            bits = min(64, sites - 64 * w)
            a[:, w] = rng.integers(0, 1 << 63, 2 * M, dtype=np.uint64) & np.uint64((1 << bits) - 1)
    x[0] = z[0] = 0
    keys = np.unique(np.concatenate([x, z], axis=1), axis=0)[:M]   # the identity first
    assert keys.shape[0] == M and not keys[0].any()
    x, z = keys[:, :W].copy(), keys[:, W:].copy()
    c = np.array([1.0, 0.5, 0.25])[np.arange(M) % classes]
    gx = np.zeros((1, W), dtype=np.uint64)
    gz = np.zeros((1, W), dtype=np.uint64)
    gz[0, sites // 64] = np.uint64(1 << (sites % 64))
    assert math.cosh(20.0) == math.sinh(20.0)
    p = itpp.Propagator(n, gx, gz, np.array([20.0]), 1.0, 0.0, M, 1)
    if separate:
        p.profile_enable(True)
    p.set_terms(x, z, c)
    p.apply_trotter_layer(1)
    # the children: K with c cosh, Q.K with c sinh; larger first, then by key
    kids = np.concatenate([np.concatenate([x, z], axis=1),
                           np.concatenate([x ^ gx, z ^ gz], axis=1)])
    mag = np.concatenate([c, c])
    order = np.lexsort(tuple(kids[:, j] for j in range(2 * W - 1, -1, -1)) + (-mag,))[:M]
    want = {tuple(int(v) for v in kids[i]): mag[i] for i in order}
    px, pz, pc = p.terms()
    got = {tuple(int(v) for v in np.concatenate([a, b])): abs(v) for a, b, v in zip(px, pz, pc)}
    assert got.keys() == want.keys()
    # a product with cosh and one with its reciprocal: two roundings, and one
    # of the reciprocal
    assert max(abs(got[k] - want[k]) / want[k] for k in want) <= 3 * 2.0 ** -53


# Coefficients far above the identity's, with no threshold: every child is kept.
@pytest.mark.parametrize("separate", [False, True])
@pytest.mark.parametrize("c0", [1.5, 3.0, 2.0 ** 40, 2.0 ** 300])
@pytest.mark.parametrize("delta", [0.0, 1e-300])
def test_large_coefficients_keep_their_children(delta, c0, separate):
    n, M = 20, 300
    x = np.arange(M, dtype=np.uint64)[:, None]        # X on the low sites
    z = np.zeros((M, 1), dtype=np.uint64)
    c = np.full(M, c0)
    c[0] = 1.0
    gz = np.array([[1 << 19]], dtype=np.uint64)
    p = itpp.Propagator(n, np.zeros_like(gz), gz, np.array([0.5]), 1.0, delta, 1 << 12, 0)
    if separate:
        p.profile_enable(True)
    p.set_terms(x, z, c)
    p.apply_trotter_layer(1)
    px, pz, pc = p.terms()
    got = {(int(a[0]), int(b[0])): abs(v) for a, b, v in zip(px, pz, pc)}
    t = math.sinh(0.5) / math.cosh(0.5)
    want = {(k, q): c[k] * (t if q else 1.0) for k in range(M) for q in (0, 1 << 19)}
    assert got.keys() == want.keys()
    assert max(abs(got[k] - want[k]) / want[k] for k in want) <= 6 * 2.0 ** -53


# more instances than CTAs, one instance, and a few over all of them
@pytest.mark.parametrize("B,n,cap", [(1, 24, 9000), (3, 20, 5000), (700, 7, 300)])
def test_batch_teams(B, n, cap):
    hams = [wl.tfim_1d(n, 1.0, 0.6 + 0.4 * b / B) for b in range(B)]
    bp = itpp.BatchPropagator(hams, 0.05, 1e-8, cap, 1)
    bp.apply_trotter_layer(3)
    for b in sorted({0, B // 2, B - 1}):
        H = hams[b]
        o = oracle.Oracle(H.n, H.gate_x, H.gate_z, H.alpha, 0.05, 1e-8, cap, 1)
        o.apply_layers(3)
        assert_same_state(bp.terms(b), o.terms(), f"instance {b} of {B}")


# The gradient's recompute: no select, one bin of it in one CTA's list, and a
# bin to narrow (one class of equal |c| above 4,096 needs many terms: the
# uniform chain gives hundreds).  The oracle's adjoint agrees to the order of
# its sums.
@pytest.mark.parametrize("n,cap,layers", [(8, 511, 4), (8, 513, 4), (12, 9000, 4)])
def test_gradient_recompute_at_the_bound(n, cap, layers):
    H = wl.tfim_1d(n, 1.0, 0.9, periodic=True)
    O = wl.energy_observable(H)
    g = itpp.Propagator(H.n, H.gate_x, H.gate_z, H.alpha, 0.05, 0.0, cap, 1)
    f_g, d_g = g.adjoint(layers, O, ckpt_every=2)
    o = oracle.Oracle(H.n, H.gate_x, H.gate_z, H.alpha, 0.05, 0.0, cap, 1)
    f_o, d_o = oracle.FrozenAdjoint(o, layers).grad_alpha(O, H.n_gates)
    assert abs(f_g - f_o) <= 1e-12 * max(1.0, abs(f_o))
    assert np.max(np.abs(d_g - d_o)) <= 1e-10 * np.max(np.abs(d_o))


# A warp's queue of pairs at its edges, the identity among the observable's
# strings and strings named twice.
@pytest.mark.parametrize("M", [1, 31, 33, 1000])
@pytest.mark.parametrize("m", [1, 9, 40])
def test_squared_state_pairs(M, m):
    H = wl.tfim_1d(12, 1.0, 0.9, periodic=True)
    E = wl.energy_observable(H)
    ox = np.concatenate([np.zeros_like(E.x[:1]), E.x, E.x])[:m].copy()
    oz = np.concatenate([np.zeros_like(E.z[:1]), E.z, E.z])[:m].copy()
    O = wl.Observable(H.n, ox, oz, np.linspace(-1.0, 1.5, m))
    g = itpp.Propagator(H.n, H.gate_x, H.gate_z, H.alpha, 0.1, 0.0, M, 1)
    o = oracle.Oracle(H.n, H.gate_x, H.gate_z, H.alpha, 0.1, 0.0, M, 1)
    g.apply_trotter_layer(2)
    o.apply_layers(2)
    v, num, pur = g.expect_psd(O)
    ov, onum, opur, _ = o.expect_psd(O)
    for a, b in ((v, ov), (num, onum), (pur, opur)):
        assert abs(a - b) <= 1e-10 * max(1.0, abs(b))


# The table of an observable's strings: one thread each, and several.
@pytest.mark.parametrize("m", [1, 1023, 1025, 4096])
def test_observable_table(m):
    H = wl.tfim_1d(16, 1.0, 1.2, periodic=True)
    g, o = _pair(H, 0.05, 1e-6, 1 << 14, 1, False)
    g.apply_trotter_layer(2)
    o.apply_layers(2)
    ox, oz, oc = o.terms()
    rng = np.random.default_rng(m)
    pick = rng.integers(0, ox.shape[0], m)            # many twice
    x, z = ox[pick].copy(), oz[pick].copy()
    x[1::3] ^= np.uint64(1 << 9)                      # ... and strings that may be absent
    at = {(int(a[0]), int(b[0])): c for a, b, c in zip(ox, oz, oc)}
    want = np.array([at.get((int(a[0]), int(b[0])), 0.0) for a, b in zip(x, z)])
    got = g.coeffs(x, z)
    assert (got.view(np.uint64) == want.view(np.uint64)).all()


# A layer captured on the caller's stream and replayed: one launch (0) and a
# chain of them (128 threads).
@pytest.mark.parametrize("block", [0, 128])
def test_layer_under_capture(block):
    torch = pytest.importorskip("torch")
    H = wl.tfim_1d(24, 1.0, 1.1, periodic=True)
    s = torch.cuda.Stream()
    g = itpp.Propagator(H.n, H.gate_x, H.gate_z, H.alpha, 0.05, 1e-9, 3000, 1,
                        stream=s, block_threads=block)
    g.apply_trotter_layer(2)
    g.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        g.apply_trotter_layer(1)
    with torch.cuda.stream(s):
        graph.replay()
        graph.replay()
    torch.cuda.synchronize()
    o = oracle.Oracle(H.n, H.gate_x, H.gate_z, H.alpha, 0.05, 1e-9, 3000, 1)
    o.apply_layers(4)
    assert_same_state(g.terms(), o.terms(), f"block {block}")
