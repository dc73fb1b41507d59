"""Bounds and states at the edge of what the run kernel's lists and strides hold."""
import numpy as np
import pytest

import oracle
import workloads as wl
from tests._compare import assert_same_state, sort_terms

pytestmark = pytest.mark.gpu

itpp = pytest.importorskip("paper_2601_14400_gb300")


def key_hash(x, z):
    """The partition hash of one-word keys (MurmurHash3 of their 32-bit halves)."""
    m = np.uint64(0xffffffff)

    def rotl(v, r):
        return ((v << np.uint64(r)) | (v >> np.uint64(32 - r))) & m

    h = np.full(x.shape, 0x9747b28c, dtype=np.uint64)
    for word in (x & m, x >> np.uint64(32), z & m, z >> np.uint64(32)):
        k = rotl(word * np.uint64(0xcc9e2d51) & m, 15) * np.uint64(0x1b873593) & m
        h = (rotl(h ^ k, 13) * np.uint64(5) + np.uint64(0xe6546b64)) & m
    h ^= np.uint64(16)
    h = (h ^ (h >> np.uint64(16))) * np.uint64(0x85ebca6b) & m
    h = (h ^ (h >> np.uint64(13))) * np.uint64(0xc2b2ae35) & m
    return h ^ (h >> np.uint64(16))


def piled_hamiltonian(m, n=40):
    """m wide strings whose hashes lie in the lowest sixteenth, then a wide gate
    whose pivot none of them has: at that gate the strings themselves, which the
    threshold keeps while it drops their products, all fall into the first
    partition."""
    rng = np.random.default_rng(m)
    x = rng.integers(0, 1 << (n - 1), 64 * m, dtype=np.uint64)
    z = rng.integers(0, 1 << n, 64 * m, dtype=np.uint64)
    ok = key_hash(x, z) < np.uint64(1 << 28)
    gx = np.append(x[ok][:m], np.uint64(1 << (n - 1)))[:, None]
    gz = np.append(z[ok][:m], np.uint64((1 << (n - 1)) - 1))[:, None]
    assert gx.shape[0] == m + 1
    return wl.Hamiltonian(n, gx, gz, np.full(m + 1, 1.0))


PILE_DTAU, PILE_DELTA = 0.01, 1e-3


# Few strings and one class of magnitudes: a gate doubles the state, and the
# select of a first gate lists every child there is.
@pytest.mark.parametrize("M", [114, 115, 120, 127, 128, 129])
@pytest.mark.parametrize("batch", [False, True])
def test_list_holds_every_child(M, batch):
    # seven commuting strings of angle 3: tanh(3)^7 = 0.966, half an octave holds
    # all of their products
    n = 40
    x = np.zeros((8, 1), dtype=np.uint64)
    z = (np.uint64(1) << np.arange(8, dtype=np.uint64))[:, None]
    H = wl.Hamiltonian(n, x, z, np.full(8, 3.0))
    o = oracle.Oracle(n, x, z, H.alpha, 1.0, 0.0, M, 1)
    o.apply_layers(2)
    if batch:
        p = itpp.BatchPropagator([H, H], 1.0, 0.0, M, 1, table_load_pct=50)
        p.apply_trotter_layer(2)
        got = p.terms(1)
    else:
        p = itpp.Propagator(n, x, z, H.alpha, 1.0, 0.0, M, 1)
        p.apply_trotter_layer(2)
        got = p.terms()
    assert_same_state(got, o.terms(), f"M {M}")


# Every string in one partition: the scatter by pair key finds no room at first.
@pytest.mark.parametrize("B,cap", [(1, 300), (2, 300), (3, 900)])
def test_scatter_of_a_piled_state(B, cap):
    H = piled_hamiltonian(cap - 2)
    bp = itpp.BatchPropagator([H] * B, PILE_DTAU, PILE_DELTA, cap, 1)
    bp.apply_trotter_layer(2)
    o = oracle.Oracle(H.n, H.gate_x, H.gate_z, H.alpha, PILE_DTAU, PILE_DELTA, cap, 1)
    o.apply_layers(2)
    for b in range(B):
        assert_same_state(bp.terms(b), o.terms(), f"instance {b} of {B}")


# The smallest partitions a caller can ask for: more of them than by default, so
# that the piled state finds no room where it does by default.
def test_smallest_partition_target():
    cap = 192
    H = piled_hamiltonian(cap - 4)
    scatters = []
    for target in (0, 64):
        bp = itpp.BatchPropagator([H], PILE_DTAU, PILE_DELTA, cap, 1, partition_target=target)
        bp.apply_trotter_layer(1)
        scatters.append(bp.stats(0)["repartitions"])
        o = oracle.Oracle(H.n, H.gate_x, H.gate_z, H.alpha, PILE_DTAU, PILE_DELTA, cap, 1)
        o.apply_layers(1)
        assert_same_state(bp.terms(0), o.terms(), f"target {target}")
    assert scatters[0] == H.n_gates < scatters[1]


# The autotuner tries partitions of 64 strings, which the piled state overflows
# where the default size holds it: whatever it picks runs.
def test_autotune_picks_a_shape_that_runs():
    cap = 192
    H = piled_hamiltonian(cap - 4)
    bp = itpp.BatchPropagator([H, H], PILE_DTAU, PILE_DELTA, cap, 1)
    bp.autotune(probe_layers=2)
    bp.apply_trotter_layer(2)
    counts, status = bp.counts()
    assert not status.any()
    o = oracle.Oracle(H.n, H.gate_x, H.gate_z, H.alpha, PILE_DTAU, PILE_DELTA, cap, 1)
    o.apply_layers(2)
    assert_same_state(bp.terms(1), o.terms(), "after the autotuner")


# Weights whose double is not a number of the type.
def test_squared_state_large_weights():
    n = 4
    g = itpp.Propagator(n, np.zeros((0, 1), np.uint64), np.zeros((0, 1), np.uint64),
                        np.zeros(0), 0.1, 0.0, 16, 0)
    x = np.zeros((2, 1), dtype=np.uint64)
    z = np.array([[0], [1]], dtype=np.uint64)
    g.set_terms(x, z, np.array([1.0, 0.125]))
    O = wl.Observable(n, x[1:], z[1:], np.array([1.2e308]))
    v, num, pur = g.expect_psd(O)
    assert pur == 1.0 + 0.125 ** 2
    assert num == 2.0 * (1.2e308 * 0.125)             # each member of the pair once
    assert v == num / pur


# A state that falls below its bound: the limit predicted for the select no
# longer applies, and gates are not merged twice for it.
@pytest.mark.parametrize("separate", [False, True])
def test_below_the_bound(separate):
    H = wl.tfim_1d(24, 1.0, 1.1, periodic=True)
    g = itpp.Propagator(H.n, H.gate_x, H.gate_z, H.alpha, 0.05, 1e-9, 3000, 1)
    if separate:
        g.profile_enable(True)
    g.apply_trotter_layer(3)
    assert g.count() == 3000
    c = np.abs(g.terms()[2])
    g.truncate(float(np.median(c)))
    g.set_alpha(np.zeros(H.n_gates))                  # nothing grows
    before = g.stats()["merge_retries"]
    want = sort_terms(*g.terms())
    g.apply_trotter_layer(3)
    assert_same_state(g.terms(), want, "gates of angle zero")
    assert g.stats()["merge_retries"] - before <= 1
    # and back at the bound, as a handle that starts from this state
    h = itpp.Propagator(H.n, H.gate_x, H.gate_z, H.alpha, 0.05, 1e-9, 3000, 1)
    h.set_terms(*want)
    for p in (g, h):
        p.set_alpha(H.alpha)
        p.apply_trotter_layer(2)
    assert g.count() == 3000
    assert_same_state(g.terms(), sort_terms(*h.terms()), "back at the bound")


# The identity among the gates where gates are merged in full: every string is
# its own partner.
@pytest.mark.parametrize("separate", [False, True])
@pytest.mark.parametrize("n,cap", [(1, 1), (9, 300), (40, 129), (40, 3000), (80, 300)])
def test_identity_gates_merged_in_full(n, cap, separate):
    H = wl.random_pauli_hamiltonian(n, 24, 5, max_weight=min(n, 3))
    H.gate_x[::3] = 0
    H.gate_z[::3] = 0
    g = itpp.Propagator(H.n, H.gate_x, H.gate_z, H.alpha, 0.3, 1e-9, cap, 1)
    if separate:
        g.profile_enable(True)
    o = oracle.Oracle(H.n, H.gate_x, H.gate_z, H.alpha, 0.3, 1e-9, cap, 1)
    for layer in range(4):
        g.apply_trotter_layer(1)
        o.apply_layers(1)
        assert_same_state(g.terms(), o.terms(), f"n {n} layer {layer}")


# A gate on every site, Y on most: few bits of a key lie outside it, and long
# partitions are merged in classes of strings all the same.
@pytest.mark.parametrize("separate", [False, True])
@pytest.mark.parametrize("n,layers", [(8, 6), (9, 5)])
def test_long_partitions_of_a_wide_gate(n, layers, separate):
    H = wl.tfim_1d(n, 1.0, 0.9, periodic=True)
    all_sites = np.uint64((1 << n) - 1)
    gx = np.concatenate([H.gate_x, [[all_sites]], [[all_sites >> np.uint64(1)]]])
    gz = np.concatenate([H.gate_z, [[all_sites]], [[all_sites]]])
    alpha = np.concatenate([H.alpha, [0.7, -0.4]])
    cap = 20000
    g = itpp.Propagator(n, gx, gz, alpha, 0.1, 1e-9, cap, 1, partition_target=2048)
    if separate:
        g.profile_enable(True)
    o = oracle.Oracle(n, gx, gz, alpha, 0.1, 1e-9, cap, 1)
    for layer in range(layers):
        g.apply_trotter_layer(1)
        o.apply_layers(1)
        assert_same_state(g.terms(), o.terms(), f"n {n} layer {layer}")
    assert g.count() > 4096
