"""Schedules longer than a launch of the run kernel, and several handles at once."""
import threading

import numpy as np
import pytest

import oracle
import workloads as wl
from tests._compare import assert_same_state

pytestmark = pytest.mark.gpu

itpp = pytest.importorskip("paper_2601_14400_gb300")


# Schedules that one launch does not hold: two launches a layer.
@pytest.mark.parametrize("cap", [300, 5000])
def test_layers_of_more_than_256_gates(cap):
    H = wl.tfim_2d(11, 1.0, 3.04)
    assert H.n_gates > 256
    g = itpp.Propagator(H.n, H.gate_x, H.gate_z, H.alpha, 0.02, 1e-9, cap, 1)
    o = oracle.Oracle(H.n, H.gate_x, H.gate_z, H.alpha, 0.02, 1e-9, cap, 1)
    for layer in range(3):
        g.apply_trotter_layer(1)
        o.apply_layers(1)
        assert_same_state(g.terms(), o.terms(), f"layer {layer}")


def test_gradient_of_more_than_256_gates():
    H = wl.tfim_2d(11, 1.0, 3.04)
    O = wl.energy_observable(H)
    g = itpp.Propagator(H.n, H.gate_x, H.gate_z, H.alpha, 0.02, 1e-6, 3000, 1)
    f_g, d_g = g.adjoint(2, O, ckpt_every=1)
    o = oracle.Oracle(H.n, H.gate_x, H.gate_z, H.alpha, 0.02, 1e-6, 3000, 1)
    f_o, d_o = oracle.FrozenAdjoint(o, 2).grad_alpha(O, H.n_gates)
    assert abs(f_g - f_o) <= 1e-12 * max(1.0, abs(f_o))
    assert np.max(np.abs(d_g - d_o)) <= 1e-10 * np.max(np.abs(d_o))


# Both want the whole device: their launches follow one another.
@pytest.mark.parametrize("block", [0, 128])
def test_two_handles_in_two_threads(block):
    torch = pytest.importorskip("torch")
    H = wl.tfim_1d(24, 1.0, 1.1, periodic=True)
    caps = (3000, 5001)
    got = [None, None]
    torch.zeros(1, device="cuda")

    def work(i):
        s = torch.cuda.Stream()
        g = itpp.Propagator(H.n, H.gate_x, H.gate_z, H.alpha, 0.05, 1e-9, caps[i], 1,
                            stream=s, block_threads=block)
        for _ in range(20):
            g.reset()
            for _ in range(4):
                g.apply_trotter_layer(1)
        got[i] = g.terms()

    t = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for a in t:
        a.start()
    for a in t:
        a.join()
    for i in range(2):
        o = oracle.Oracle(H.n, H.gate_x, H.gate_z, H.alpha, 0.05, 1e-9, caps[i], 1)
        o.apply_layers(4)
        assert_same_state(got[i], o.terms(), f"handle {i}")
