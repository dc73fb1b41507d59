"""Captured gates and reads, replayed in any order with eager calls.

A replay changes the state without the host taking part, so where the state
lies (one run, or a window's partitions) is known on the device alone.
"""
import ctypes

import numpy as np
import pytest

import oracle
import workloads as wl
from tests._compare import assert_same_state, rel_close, sort_terms

pytestmark = pytest.mark.gpu

itpp = pytest.importorskip("paper_2601_14400_gb300")

N, DTAU, DELTA, CAP = 24, 0.05, 1e-9, 3000


def _handle(block, stream=None):
    H = wl.tfim_1d(N, 1.0, 1.1, periodic=True)
    return H, itpp.Propagator(H.n, H.gate_x, H.gate_z, H.alpha, DTAU, DELTA, CAP, 1,
                              stream=stream, block_threads=block)


# Whole layers in one launch (0) and a chain of launches (128 threads).
@pytest.mark.parametrize("block", [0, 128])
@pytest.mark.parametrize("read", ["terms", "expect", "coeffs"])
def test_reads_between_replays(block, read):
    torch = pytest.importorskip("torch")
    s = torch.cuda.Stream()
    H, g = _handle(block, s)
    O = wl.energy_observable(H)
    o = oracle.Oracle(H.n, H.gate_x, H.gate_z, H.alpha, DTAU, DELTA, CAP, 1)
    g.apply_trotter_layer(2)
    o.apply_layers(2)
    g.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        g.apply_trotter_layer(1)
    for replay in range(3):
        with torch.cuda.stream(s):
            graph.replay()
        o.apply_layers(1)
        if read == "terms":
            assert_same_state(g.terms(), o.terms(), f"block {block} replay {replay}")
        elif read == "expect":
            assert rel_close(g.expect(O), o.expect(O)), (block, replay)
        else:
            at = {(int(a[0]), int(b[0])): c for a, b, c in zip(*o.terms())}
            want = [at.get((int(a[0]), int(b[0])), 0.0) for a, b in zip(O.x, O.z)]
            assert list(g.coeffs(O.x, O.z)) == want, (block, replay)


# A read captured while the state was one run, replayed when it is not.
@pytest.mark.parametrize("block", [0, 128])
def test_read_captured_before_the_gates(block):
    torch = pytest.importorskip("torch")
    s = torch.cuda.Stream()
    H, g = _handle(block, s)
    O = wl.energy_observable(H)
    ox = torch.from_numpy(O.x.astype(np.int64)).cuda()
    oz = torch.from_numpy(O.z.astype(np.int64)).cuda()
    ow = torch.from_numpy(np.ascontiguousarray(O.w, dtype=np.float64)).cuda()
    m = int(ow.shape[0])
    out = torch.zeros(m + 1, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()

    def expect():
        p = [ctypes.c_void_p(t.data_ptr()) for t in (ox, oz, ow, out)]
        st = itpp.lib().itpp_expect_device(g.handle, p[0], p[1], p[2], m, p[3])
        assert st == itpp.ITPP_OK

    expect()                                          # allocates its scratch
    g.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        expect()
    o = oracle.Oracle(H.n, H.gate_x, H.gate_z, H.alpha, DTAU, DELTA, CAP, 1)
    for layer in range(2):
        g.apply_trotter_layer(1)
        o.apply_layers(1)
        with torch.cuda.stream(s):
            graph.replay()
        torch.cuda.synchronize()
        assert rel_close(float(out[m]), o.expect(O)), (block, layer)
    assert_same_state(g.terms(), o.terms(), f"block {block}")


# Gates one by one around a replayed layer: the replay leaves the partitions
# of the layer's last window behind.
@pytest.mark.parametrize("block", [0, 128])
@pytest.mark.parametrize("first", [1, 2, 3])
def test_gates_around_a_replay(block, first):
    torch = pytest.importorskip("torch")
    s = torch.cuda.Stream()
    H, g = _handle(block, s)
    _, h = _handle(0)
    g.apply_trotter_layer(2)
    h.apply_trotter_layer(2)
    g.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        g.apply_trotter_layer(1)
    for k in range(first):
        g.apply_gate(k)
        h.apply_gate(k)
    with torch.cuda.stream(s):
        graph.replay()
    h.apply_trotter_layer(1)
    for k in range(first, first + 3):
        g.apply_gate(k)
        h.apply_gate(k)
    assert_same_state(g.terms(), sort_terms(*h.terms()), f"block {block} first {first}")
